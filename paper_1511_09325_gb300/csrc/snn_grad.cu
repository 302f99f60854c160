// snn_grad.cu -- a differentiable form of the network of arxiv 1511.09325,
// Sec. 2, and its reverse-mode gradient.
//
// The paper simulates the spiking network only.  This file adds the standard
// surrogate-gradient treatment of the same recursion, on the same synapse
// table (F32W records: target code, fixed-point weight):
//
//   X_E,i(t), X_I,i(t): sums of w s_j(t - d) over excitatory / inhibitory sources
//   I_i = a[E][p_i] X_E,i + a[I][p_i] X_I,i + J (lam + sqrt(lam) xi_i(t))
//   g_i = max(0, 1 - s_i(t-1) - s_i(t-2));  U_i = g (V_i + I_i) + (1 - g) V_reset
//   s_i = [U_i >= theta] (hard) or sigmoid(beta (U_i - theta)) (soft)
//   V' = U - s (U - V_reset);  c' = c + dc s
//   V(t+1) = P_VV V' + P_VC c';  c(t+1) = P_CC c',  P_VC,E = g_c kappa
//
// with xi_i(t) the normal draw of Philox stream SURR (quantile table of the
// top 16 bits), lam = nu_ext h, and the loss (r_E - r_E*)^2 + (r_I - r_I*)^2
// on the population rates.  In hard mode the backward pass uses the
// surrogate derivative ds/dU = 1 / (1 + beta |U - theta|)^2; in soft mode the
// exact one.  Parameters: a_EE, a_EI, a_IE, a_II (a_XY scales the synapses
// from X onto Y), g_c and nu_ext.
//
// Forward: grad_deliver_kernel (one warp per source row, pull by delay: the
// input of step t is every bucket d of every row weighted by s_j(t - d), summed
// as int64 fixed point in 2^-32 mV, so the sums do not depend on the order;
// a row whose last d_max spikes are all zero leaves after one load of their bit
// mask)
// and grad_update_kernel (one thread per neuron; hard mode is the spiking
// model's arithmetic, one float rounding per operation).  The state (V, c and
// the spike history of d_max + 1 steps) is checkpointed every `ckpt` steps.
// Backward: segment by segment from the end, the forward is recomputed from
// the segment's checkpoint while a tape of eight values per neuron and step is
// recorded, then the adjoint recursion runs back through the segment:
// grad_gather_kernel (one warp per source row: the adjoint of the delayed
// delivery is a gather over the row's outgoing synapses of the targets' input
// adjoints at t + d, summed in the order in which they were drawn) and
// grad_backward_kernel (one thread per neuron: the adjoint of every line above;
// parameter partials accumulate per neuron in FP64 and are summed in a
// fixed order).  Every sum has a fixed order, so a run is reproducible bit
// for bit.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <memory>
#include <new>
#include <string>
#include <vector>

#include "snn_device.cuh"
#include "snn_internal.h"

using namespace snn;

namespace {

constexpr int kThreads = 256;
constexpr int kTape = 8;  // V, I, U, g, s, c', X_E, X_I
constexpr float kTwoM32 = 2.3283064365386963e-10f;  // 2^-32
constexpr float kTwoM16 = 1.52587890625e-05f;       // 2^-16
constexpr float kTwoM24 = 5.9604644775390625e-08f;  // 2^-24

struct GradParams {
  long long N, accw;          // neurons; words of an array in acc order
  int npc, npc4, nexc, ncol, dmin, ndel, nslot, rowcap, unit, planes, hard, T;
  const uint32_t* ctile;      // geometry of the net (see snn_internal.h)
  const uint32_t* colv;
  const uint32_t* nbg;
  uint32_t* vtile;            // [ncol] first word of each virtual column's tile
  uint32_t* ord;              // the rows' draw order (see BuildParams), null: as stored
  uint8_t* ord_end;
  int ord_units;
  uint32_t seed_lo, seed_hi;
  float beta, theta, vr, dc, pvv, pcc, pvc_e, pvc_i, kappa, J, lam, sqlam;
  float a[4];  // a_EE, a_EI, a_IE, a_II
  float dlds_e, dlds_i;
  const uint2* syn;
  const uint8_t* bend;
  const float* q;
  float* V;
  float* C;
  float* shist;               // [nslot][N] s of the last nslot steps
  uint32_t* active;           // [N] bit d - 1: s(t - d) != 0 (t the step due next)
  uint32_t bucket_mask;       // ndel low bits
  unsigned long long* xe;     // [accw] input sums from E sources, 2^-32 mV, acc order
  unsigned long long* xin;    // [accw] the same from I sources
  float* tape;                // [ckpt][kTape][N]
  double* rate_part;          // [update blocks][2]
  float* vbar;
  float* cbar;
  float* ibe;                 // [nslot][accw] a[E][p_i] * adjoint of I_i(t), acc order
  float* ibi;                 // [nslot][accw] a[I][p_i] * adjoint of I_i(t)
  float* gb;                  // [3][N] -adjoint of g_i(t) where the gate is open
  float* sg;                  // [N] gathered adjoints of s_j(t), rows in table order
  double* gacc;               // [6][N] parameter partials per neuron
  double* gsum;               // [6] their sums
};

// Ring position of step s >= 0 (steps are below 2^31: 32-bit remainder).
__device__ __forceinline__ long long ring(long long s, int n) {
  return (long long)((uint32_t)s % (uint32_t)n);
}

__device__ __forceinline__ float normal_draw(const GradParams& P, long long i, long long t) {
  const uint4 x = philox4x32_10(make_uint4((uint32_t)(i >> 2), (uint32_t)t, kTagSurr, 0u),
                                P.seed_lo, P.seed_hi);
  const uint32_t w = (i & 3) == 0 ? x.x : (i & 3) == 1 ? x.y : (i & 3) == 2 ? x.z : x.w;
  return P.q[w >> 16];
}

// Initial state: V_i uniform in [0, theta) from the spiking net's INIT
// stream (word i mod 4 of Philox(i / 4, 0, INIT)), c = 0.
__global__ void __launch_bounds__(kThreads) grad_init_kernel(const GradParams P) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= P.N) return;
  const uint4 x = philox4x32_10(make_uint4((uint32_t)(i >> 2), 0u, kTagInit, 0u), P.seed_lo,
                                P.seed_hi);
  const uint32_t u = (i & 3) == 0 ? x.x : (i & 3) == 1 ? x.y : (i & 3) == 2 ? x.z : x.w;
  P.V[i] = __fmul_rn(P.theta, __fmul_rn(__uint2float_rn(u >> 8), kTwoM24));
  P.C[i] = 0.f;
  P.active[i] = 0u;
}

// Word of neuron i in arrays in acc order.
__device__ __forceinline__ long long acc_word(const GradParams& P, long long i) {
  const uint32_t c = (uint32_t)i / (uint32_t)P.npc;
  return (long long)P.colv[c] * P.npc4 + ((uint32_t)i - c * (uint32_t)P.npc);
}

// A source row: its records, and where its records' targets lie: in parts
// from word `tile` on, out parts through the row `nb` of the neighbour table.
struct GradRow {
  const uint2* rec;
  const uint8_t* ends;
  const uint32_t* nb;
  uint32_t tile;
  bool exc;
};
__device__ __forceinline__ GradRow grad_row(const GradParams& P, long long j) {
  const uint32_t c = (uint32_t)j / (uint32_t)P.npc;
  const uint32_t l = (uint32_t)j - c * (uint32_t)P.npc;
  const uint32_t v = P.colv[c];
  const size_t at = (size_t)v * P.npc + l;
  GradRow r;
  r.rec = P.syn + at * (size_t)P.rowcap;
  r.ends = P.bend + at * (size_t)(P.planes * 16);
  r.nb = P.nbg + (size_t)v * 64;
  r.tile = (v - (P.ctile[c] & 63u)) * (uint32_t)P.npc4;
  r.exc = (int)l < P.nexc;
  return r;
}
// Word of the target of a record with code `code` of an in or out part.
__device__ __forceinline__ uint32_t target_word(const GradRow& r, bool in, uint32_t code) {
  return in ? r.tile + code : __ldg(r.nb + ((code >> 11) & 63u)) + (code & 2047u);
}

// Bucket ends (slots) in lanes 0..ndel-1 of the warp; the bucket holding
// slot k is the first b with end_b > k, found by a fixed five-step search
// over the lanes (every lane takes part, whatever its k).
__device__ __forceinline__ int bucket_of(int k, int end_lane, int ndel) {
  int lo = 0, hi = ndel - 1;
#pragma unroll
  for (int step = 0; step < 5; ++step) {
    const int mid = (lo + hi) >> 1;
    const int e = __shfl_sync(0xFFFFFFFFu, end_lane, mid);
    if (e > k)
      hi = mid;
    else
      lo = min(mid + 1, hi);
  }
  return lo;
}

// Input of step t: every bucket d of every source row j, weighted by
// s_j(t - d), into the row's population accumulator.  One warp per row: P.active
// holds, per neuron, a bit d - 1 for every d with s(t - d) != 0, and the warp
// leaves after one load when no bucket has a spike; otherwise it streams the
// row four records per lane (16-byte loads; a bucket part is a whole number of
// 8-slot units, so the four records of a lane share it).
__global__ void __launch_bounds__(kThreads) grad_deliver_kernel(const GradParams P, long long t) {
  grid_wait();
  grid_go();
  const long long j = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (j >= P.N) return;
  const uint32_t act = (P.active[j] >> (P.dmin - 1)) & P.bucket_mask;
  if (act == 0u) return;
  const GradRow R = grad_row(P, j);
  float s_lane = 0.f;
  int end_lane = 0x7FFFFFFF, mid_lane = 0;
  if (lane < P.ndel) {
    const uint32_t e = *reinterpret_cast<const uint16_t*>(R.ends + desc_end(lane));
    mid_lane = (int)(e & 0xFFu) * P.unit;
    end_lane = (int)(e >> 8) * P.unit;
    if (act >> lane & 1u) s_lane = P.shist[ring(t - (P.dmin + lane), P.nslot) * P.N + j];
  }
  unsigned long long* acc = R.exc ? P.xe : P.xin;
  const int row_end = __shfl_sync(0xFFFFFFFFu, end_lane, P.ndel - 1);
  const uint2* row = R.rec;
  for (int k0 = 0; k0 < row_end; k0 += 128) {
    const int k = k0 + 4 * lane;
    const int b = bucket_of(k, end_lane, P.ndel);
    const float s = __shfl_sync(0xFFFFFFFFu, s_lane, b);
    const bool in = k < __shfl_sync(0xFFFFFFFFu, mid_lane, b);
    if (k < row_end && s != 0.f) {
      const uint4 r01 = __ldcs(reinterpret_cast<const uint4*>(row + k));
      const uint4 r23 = __ldcs(reinterpret_cast<const uint4*>(row + k + 2));
      const uint32_t tg[4] = {r01.x, r01.z, r23.x, r23.z};
      const uint32_t wf[4] = {r01.y, r01.w, r23.y, r23.w};
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if (tg[q] & kPad) continue;
        const int32_t wfx = (int32_t)wf[q];
        const long long v = P.hard ? (long long)wfx * 65536ll
                                   : __float2ll_rn(__fmul_rn(__fmul_rn(s, (float)wfx), 65536.f));
        atomicAdd(acc + target_word(R, in, tg[q]), (unsigned long long)v);
      }
    }
  }
}

// Bits of P.active at step t from the spike history (after a checkpoint).
__global__ void __launch_bounds__(kThreads) grad_active_kernel(const GradParams P, long long t) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= P.N) return;
  uint32_t act = 0u;
  for (int d = 1; d < P.nslot && d <= t; ++d)
    act |= P.shist[ring(t - d, P.nslot) * P.N + i] != 0.f ? 1u << (d - 1) : 0u;
  P.active[i] = act;
}

// Neuron update of step t; records the tape at slot `slot` (>= 0) and adds
// the spikes of each population to this block's rate partial sums when
// `rates` is set.
__global__ void __launch_bounds__(kThreads) grad_update_kernel(const GradParams P, long long t,
                                                              int slot, int rates) {
  grid_wait();
  grid_go();
  __shared__ float s_sum[kThreads / 32][2];
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  float s = 0.f;
  bool exc = false;
  if (i < P.N) {
    const long long iw = acc_word(P, i);
    const float XE = __fmul_rn(__ll2float_rn((long long)P.xe[iw]), kTwoM32);
    const float XI = __fmul_rn(__ll2float_rn((long long)P.xin[iw]), kTwoM32);
    P.xe[iw] = 0ull;
    P.xin[iw] = 0ull;
    exc = (int)((uint32_t)i % (uint32_t)P.npc) < P.nexc;
    const float xi = normal_draw(P, i, t);
    const float e = __fmul_rn(P.J, __fadd_rn(P.lam, __fmul_rn(P.sqlam, xi)));
    const float aE = exc ? P.a[0] : P.a[1];
    const float aI = exc ? P.a[2] : P.a[3];
    const float I = __fadd_rn(__fadd_rn(__fmul_rn(aE, XE), __fmul_rn(aI, XI)), e);
    const float s1 = t >= 1 ? P.shist[ring(t - 1, P.nslot) * P.N + i] : 0.f;
    const float s2 = t >= 2 ? P.shist[ring(t - 2, P.nslot) * P.N + i] : 0.f;
    const float V = P.V[i], c = P.C[i];
    float g, U, Vp, cp;
    if (P.hard) {
      g = (s1 == 0.f && s2 == 0.f) ? 1.f : 0.f;
      U = g != 0.f ? __fadd_rn(V, I) : P.vr;
      s = U >= P.theta ? 1.f : 0.f;
      Vp = s != 0.f ? P.vr : U;
      cp = s != 0.f ? __fadd_rn(c, P.dc) : c;
    } else {
      g = fmaxf(__fsub_rn(__fsub_rn(1.f, s1), s2), 0.f);
      U = __fadd_rn(__fmul_rn(g, __fadd_rn(V, I)), __fmul_rn(__fsub_rn(1.f, g), P.vr));
      const float z = __fmul_rn(P.beta, __fsub_rn(U, P.theta));
      const float ez = expf(-fabsf(z));
      s = z >= 0.f ? 1.f / (1.f + ez) : ez / (1.f + ez);
      Vp = __fsub_rn(U, __fmul_rn(s, __fsub_rn(U, P.vr)));
      cp = __fadd_rn(c, __fmul_rn(P.dc, s));
    }
    const float pvc = exc ? P.pvc_e : P.pvc_i;
    P.V[i] = __fmaf_rn(cp, pvc, __fmul_rn(Vp, P.pvv));
    P.C[i] = __fmul_rn(cp, P.pcc);
    P.shist[ring(t, P.nslot) * P.N + i] = s;
    P.active[i] = P.active[i] << 1 | (s != 0.f ? 1u : 0u);
    if (slot >= 0) {
      float* tp = P.tape + (long long)slot * kTape * P.N + i;
      const float vals[kTape] = {V, I, U, g, s, cp, XE, XI};
#pragma unroll
      for (int k = 0; k < kTape; ++k) tp[(long long)k * P.N] = vals[k];
    }
  }
  if (!rates) return;
  // this block's spikes per population, in a fixed order
  float se = exc ? s : 0.f, si = (i < P.N && !exc) ? s : 0.f;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    se += __shfl_xor_sync(0xFFFFFFFFu, se, o);
    si += __shfl_xor_sync(0xFFFFFFFFu, si, o);
  }
  if ((threadIdx.x & 31) == 0) {
    s_sum[threadIdx.x >> 5][0] = se;
    s_sum[threadIdx.x >> 5][1] = si;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double te = 0.0, ti = 0.0;
    for (int w = 0; w < kThreads / 32; ++w) {
      te += (double)s_sum[w][0];
      ti += (double)s_sum[w][1];
    }
    P.rate_part[2 * blockIdx.x] += te;
    P.rate_part[2 * blockIdx.x + 1] += ti;
  }
}

// Adjoint of s_j(tau) through its outgoing synapses: the sum over the buckets d
// with tau + d < T of w * (a[p_j][p_i] * adjoint of I_i(tau + d)).
// The order of the FP32 sum is part of the result: the row's synapses, bucket by
// bucket, in the order in which they were drawn, each bucket padded to 8 places;
// lane e of the row's warp adds places 4 e .. 4 e + 3 of every run of 128, and the
// lanes' sums are added as a tree.  Where no synapse leaves its tile (a net of one
// tile, units of 8 slots) the table itself lies in that order; else P.ord gives
// the slots of each unit of 8 places (see write_order in snn_build.cu).

// One warp per row, the targets' adjoints read from L2 (MAP: the rows' order is
// P.ord's, its words loaded a run ahead).  Each record needs one scattered 4-byte
// read of an adjoint, a 32-byte sector of the L2, which bounds it.  MAP on 12x12
// columns, 60 steps forward and backward: 54.5 ms with five blocks per SM, 56.1 with
// six, 56.5 with eight.
template <bool MAP>
__global__ void __launch_bounds__(kThreads, MAP ? 5 : 1)
    grad_gather_kernel(const GradParams P, long long tau) {
  const long long at = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;  // row of the table
  const int lane = threadIdx.x & 31;
  if (at >= P.N) return;
  const uint32_t v = (uint32_t)at / (uint32_t)P.npc;
  const bool exc = (int)((uint32_t)at - v * (uint32_t)P.npc) < P.nexc;
  const float* ib = exc ? P.ibe : P.ibi;
  const uint32_t* nb = P.nbg + (size_t)v * 64;
  const uint32_t tile = P.vtile[v];
  long long off_lane = -1;    // ring offset of bucket `lane`'s step, -1 beyond T
  int end_lane = 0x7FFFFFFF;  // end of bucket `lane` in places
  int slot_lane = 0;          // its end in slots (MAP)
  if (lane < P.ndel) {
    const long long dst = tau + P.dmin + lane;
    off_lane = dst < P.T ? ring(dst, P.nslot) * P.accw : -1;
    slot_lane = (int)P.bend[at * (P.planes * 16) + desc_end(lane) + 1] * P.unit;
    end_lane = MAP ? (int)P.ord_end[at * P.ndel + lane] * 8 : slot_lane;
  }
  const int row_end = __shfl_sync(0xFFFFFFFFu, end_lane, P.ndel - 1);
  const uint2* row = P.syn + at * (long long)P.rowcap;
  const uint32_t* ord = MAP ? P.ord + at * (long long)P.ord_units : nullptr;
  float acc = 0.f;
  uint32_t u_next = MAP && 4 * lane < row_end ? __ldg(ord + (lane >> 1)) : 0u;  // a run ahead
#pragma unroll (MAP ? 1 : 2)
  for (int k0 = 0; k0 < row_end; k0 += 128) {
    const int k = k0 + 4 * lane;
    const int b = bucket_of(k, end_lane, P.ndel);
    const long long off = __shfl_sync(0xFFFFFFFFu, off_lane, b);
    const int slot_end = MAP ? __shfl_sync(0xFFFFFFFFu, slot_lane, b) : 0;
    const uint32_t u = u_next;
    if (MAP && k + 128 < row_end) u_next = __ldg(ord + ((k + 128) >> 3));
    if (k < row_end && off >= 0) {
      const float* ibs = ib + off;
      uint32_t code[4], w[4] = {0u, 0u, 0u, 0u};
      uint32_t in = 0xFu;  // bit q: record q is an in record
      if (MAP) {
        const uint32_t h = (uint32_t)k & 4u;
        in = u >> h & 0xFu;
        const uint32_t before = __popc(u & ((1u << h) - 1u));  // in records of the unit's first half
        uint32_t ip = (u >> 8 & 0xFFFu) + before, op = (u >> 20) + h - before;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          // places beyond the bucket's synapses: pads, or beyond its slots
          const int s = (int)(in >> q & 1u ? ip++ : op++);
          const uint2 x = __ldg(row + min(s, slot_end - 1));
          code[q] = s < slot_end ? x.x : kPad;
          w[q] = x.y;
        }
      } else {
        const uint4 x = __ldcs(reinterpret_cast<const uint4*>(row + k));
        const uint4 y = __ldcs(reinterpret_cast<const uint4*>(row + k + 2));
        code[0] = x.x; code[1] = x.z; code[2] = y.x; code[3] = y.z;
        w[0] = x.y; w[1] = x.w; w[2] = y.y; w[3] = y.w;
      }
      if (MAP) {  // (no load under a branch, where it would be waited for)
        float v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const uint32_t out = __ldg(nb + (code[q] >> 11 & 63u)) + (code[q] & 2047u);
          v[q] = __ldg(ibs + (code[q] & kPad ? 0u : in >> q & 1u ? tile + code[q] : out));
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (!(code[q] & kPad)) acc = __fmaf_rn((float)(int32_t)w[q], v[q], acc);
      } else {
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (!(code[q] & kPad)) acc = __fmaf_rn((float)(int32_t)w[q], ibs[tile + code[q]], acc);
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xFFFFFFFFu, acc, o);
  if (lane == 0) P.sg[at] = __fmul_rn(acc, kTwoM16);
}

// The same for a net of one tile whose adjoints of a step fit shared memory twice:
// a block takes a run of rows of one population, up to kGatherRows per warp, and
// goes through the buckets; the adjoints at tau + d are copied to shared memory
// while the bucket before is summed, and each row's records of a bucket are
// loaded while the bucket before is summed.  The lanes' sums of all rows stay in
// registers.
// The adjoints come from shared memory instead of L2; what is left is the table
// (4x4: 197 MB, 31 us of DRAM time) and a barrier per bucket, with 17 of 32 lanes
// at work on a bucket of 62 synapses.  4x4, 500 steps forward and backward: 44.6
// ms, by the warps of grad_gather_kernel 57.9 ms; 4x3 (200 steps) 16.9 and 19.9 ms;
// 3x3 13.9 and 15.1 ms.  2x2 and smaller nets have too few rows to hide the
// barriers (300 steps of 2x2: 15.3 and 14.1 ms).
constexpr int kGatherThreads = 512;  // one block per SM
constexpr int kGatherWarps = kGatherThreads / 32;
constexpr int kGatherRows = 9;       // rows per warp, at most
constexpr int kGatherBufs = 4;       // windows in shared memory, at most

template <int ROWS>
__global__ void __launch_bounds__(kGatherThreads, 1)
    grad_gather_tile_kernel(const GradParams P, long long tau, int nb, int bufs, int per_block, int blocks_e) {
  extern __shared__ __align__(16) float s_ib[];  // [bufs][accw]
  const bool exc = (int)blockIdx.x < blocks_e;
  const uint32_t npop = (uint32_t)(exc ? P.nexc : P.npc - P.nexc);  // rows of a column
  const uint32_t r0 = (uint32_t)(exc ? blockIdx.x : blockIdx.x - blocks_e) * (uint32_t)per_block;
  const uint32_t rows = npop * (uint32_t)P.ncol;
  const uint32_t r1 = min(rows, r0 + (uint32_t)per_block);
  const float* ib = exc ? P.ibe : P.ibi;
  const int lane = threadIdx.x & 31;
  const uint32_t words = (uint32_t)P.accw;
  auto window = [&](int b, int buf) {  // bucket b's adjoints on their way to buffer `buf`
    if (b < nb) {
      const float* src = ib + ring(tau + P.dmin + b, P.nslot) * P.accw;
      const uint32_t dst = (uint32_t)__cvta_generic_to_shared(s_ib + buf * words);
      for (uint32_t i = threadIdx.x * 4u; i < words; i += kGatherThreads * 4u)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + i * 4u), "l"(src + i) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  for (int b = 0; b + 1 < bufs; ++b) window(b, b);
  float acc[ROWS];
  int end_lane[ROWS];  // lane b: end of bucket b of each row, in slots
  uint32_t row[ROWS];  // rows of the table
  uint4 x[ROWS], y[ROWS];
  const uint32_t rw = r0 + (threadIdx.x >> 5);
#pragma unroll
  for (int i = 0; i < ROWS; ++i) {
    const uint32_t r = min(rw + (uint32_t)(i * kGatherWarps), rows - 1u);
    const uint32_t c = r / npop;
    row[i] = c * (uint32_t)P.npc + (exc ? 0u : (uint32_t)P.nexc) + (r - c * npop);
    end_lane[i] = 0;
    if (rw + (uint32_t)(i * kGatherWarps) < r1 && lane < P.ndel)
      end_lane[i] = (int)P.bend[(size_t)row[i] * (uint32_t)(P.planes * 16) + desc_end(lane) + 1] * kSlotUnit;
    acc[i] = 0.f;
  }
  // the lane's place in the bucket of slots beg .. end - 1 (beyond it if k >= end)
  auto place = [&](int beg) { return beg + 4 * ((lane - (beg >> 2)) & 31); };
  auto load = [&](int i, int beg, int end) {  // lanes beyond the bucket repeat its last group
    const int k = max(0, min(place(beg), end - 4));
    const uint4* p = reinterpret_cast<const uint4*>(P.syn + (size_t)row[i] * (uint32_t)P.rowcap + k);
    x[i] = __ldcs(p);
    y[i] = __ldcs(p + 1);
  };
#pragma unroll
  for (int i = 0; i < ROWS; ++i) load(i, 0, __shfl_sync(0xFFFFFFFFu, end_lane[i], 0));
  int buf = 0;  // bucket b's buffer
  for (int b = 0; b < nb; ++b) {
    // all but the last bufs - 2 windows have arrived
    if (bufs == 2)
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    else if (bufs == 3)
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    else
      asm volatile("cp.async.wait_group 2;" ::: "memory");
    __syncthreads();
    window(b + bufs - 1, buf ? buf - 1 : bufs - 1);
    const float* win = s_ib + buf * words;
    buf = buf + 1 < bufs ? buf + 1 : 0;
    auto add = [&](float a, const uint4& p, const uint4& q, bool on) {
      const uint32_t code[4] = {p.x, p.z, q.x, q.z}, w[4] = {p.y, p.w, q.y, q.w};
      float v[4];
#pragma unroll
      for (int m = 0; m < 4; ++m) v[m] = on && !(code[m] & kPad) ? win[code[m]] : 0.f;
#pragma unroll
      for (int m = 0; m < 4; ++m)
        if (on && !(code[m] & kPad)) a = __fmaf_rn((float)(int32_t)w[m], v[m], a);
      return a;
    };
#pragma unroll
    for (int i = 0; i < ROWS; ++i) {
      const int beg = b ? __shfl_sync(0xFFFFFFFFu, end_lane[i], b - 1) : 0;
      const int end = __shfl_sync(0xFFFFFFFFu, end_lane[i], b);
      const int nxt = b + 1 < nb ? __shfl_sync(0xFFFFFFFFu, end_lane[i], b + 1) : end;
      acc[i] = add(acc[i], x[i], y[i], place(beg) < end);
      load(i, end, nxt);
      for (int k = place(beg) + 128; k < end; k += 128) {
        const uint4* p = reinterpret_cast<const uint4*>(P.syn + (size_t)row[i] * (uint32_t)P.rowcap + k);
        acc[i] = add(acc[i], __ldcs(p), __ldcs(p + 1), true);
      }
    }
  }
#pragma unroll
  for (int i = 0; i < ROWS; ++i) {
    float a = acc[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xFFFFFFFFu, a, o);
    if (lane == 0 && rw + (uint32_t)(i * kGatherWarps) < r1) P.sg[row[i]] = __fmul_rn(a, kTwoM16);
  }
}

// One step of the adjoint recursion for step tau (tape slot `slot`): takes the
// adjoints of V(tau+1), c(tau+1) and leaves those of V(tau), c(tau).
__global__ void __launch_bounds__(kThreads) grad_backward_kernel(const GradParams P, long long tau,
                                                                int slot) {
  grid_wait();
  grid_go();
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= P.N) return;
  const bool exc = (int)((uint32_t)i % (uint32_t)P.npc) < P.nexc;
  const float* tp = P.tape + (long long)slot * kTape * P.N + i;
  const float V = tp[0], I = tp[P.N], U = tp[2 * P.N], g = tp[3 * P.N], s = tp[4 * P.N];
  const float cp = tp[5 * P.N], XE = tp[6 * P.N], XI = tp[7 * P.N];
  const uint32_t c = (uint32_t)i / (uint32_t)P.npc, l = (uint32_t)i - c * (uint32_t)P.npc;
  const uint32_t v = P.colv[c];
  // the adjoint of s(tau) through the synapses (none that ends before T: 0)
  const float sg = tau + P.dmin < P.T ? P.sg[(size_t)v * P.npc + l] : 0.f;
  float sbar = (exc ? P.dlds_e : P.dlds_i) + sg + P.gb[ring(tau + 1, 3) * P.N + i] +
               P.gb[ring(tau + 2, 3) * P.N + i];
  const float vb1 = P.vbar[i], cb1 = P.cbar[i];
  const float pvc = exc ? P.pvc_e : P.pvc_i;
  // V(tau+1) = P_VV V' + P_VC c',  c(tau+1) = P_CC c'
  const float vpbar = P.pvv * vb1;
  const float cpbar = P.pcc * cb1 + pvc * vb1;
  double* ga = P.gacc + i;
  if (exc) ga[4 * P.N] += (double)vb1 * (double)cp * (double)P.kappa;
  // V' = U - s (U - V_reset),  c' = c + dc s
  float ubar = vpbar * (1.f - s);
  sbar += -vpbar * (U - P.vr) + cpbar * P.dc;
  // the spike nonlinearity: surrogate (hard) or exact (soft) derivative
  float dsdu;
  if (P.hard) {
    const float den = 1.f + P.beta * fabsf(U - P.theta);
    dsdu = 1.f / (den * den);
  } else {
    dsdu = P.beta * s * (1.f - s);
  }
  ubar += sbar * dsdu;
  // U = g (V + I) + (1 - g) V_reset
  const float ib = ubar * g;
  P.vbar[i] = ib;
  P.cbar[i] = cpbar;
  P.gb[ring(tau, 3) * P.N + i] = g > 0.f ? -ubar * (V + I - P.vr) : 0.f;
  const float aE = exc ? P.a[0] : P.a[1];
  const float aI = exc ? P.a[2] : P.a[3];
  const long long iw = ring(tau, P.nslot) * P.accw + (long long)v * P.npc4 + l;
  P.ibe[iw] = aE * ib;
  P.ibi[iw] = aI * ib;
  // I = a[E][p] X_E + a[I][p] X_I + J (lam + sqrt(lam) xi),  h = 1 ms
  ga[(exc ? 0 : 1) * P.N] += (double)ib * (double)XE;
  ga[(exc ? 2 : 3) * P.N] += (double)ib * (double)XI;
  const float xi = normal_draw(P, i, tau);
  ga[5 * P.N] += (double)ib * (double)P.J * (1.0 + (double)xi / (2.0 * (double)P.sqlam));
}

// First word of the tile of every virtual column, one block per tile.
__global__ void __launch_bounds__(kThreads) grad_tile_words_kernel(const GradParams P, const uint2* tinfo) {
  const uint2 ti = tinfo[blockIdx.x];
  for (uint32_t k = threadIdx.x; k < ti.y; k += blockDim.x) P.vtile[ti.x + k] = ti.x * (uint32_t)P.npc4;
}

// Sums of the six parameters' partials over the neurons, one block per
// parameter, in a fixed order.
constexpr int kSumThreads = 1024;
__global__ void __launch_bounds__(kSumThreads) grad_sum_kernel(const GradParams P) {
  __shared__ double s_sum[kSumThreads];
  const double* p = P.gacc + (size_t)blockIdx.x * P.N;
  double sum = 0.0;
#pragma unroll 4
  for (long long i = threadIdx.x; i < P.N; i += kSumThreads) sum += p[i];
  s_sum[threadIdx.x] = sum;
  for (int o = kSumThreads / 2; o > 0; o >>= 1) {
    __syncthreads();
    if ((int)threadIdx.x < o) s_sum[threadIdx.x] += s_sum[threadIdx.x + o];
  }
  if (threadIdx.x == 0) P.gsum[blockIdx.x] = s_sum[0];
}

}  // namespace

struct snn_grad {
  NetView v{};
  long long T = 0;
  int ckpt = 0, nseg = 0, hard = 1, nslot = 0, ublocks = 0, wblocks = 0;
  float beta = 5.f;
  double targets[2] = {3.0, 8.0};
  double kappa = 0.0, pvv = 0.0, pcc = 0.0;
  GradParams P{};
  float* q = nullptr;
  float* ck = nullptr;  // [nseg][(2 + nslot) N]: V, c, s history at each segment start
  std::vector<void*> bufs;
  std::string err;
};

namespace {

int gfail(snn_grad* g, int code, const std::string& msg) {
  if (g) g->err = msg;
  return code == SNN_OK ? code : fail_global(code, msg);
}

#define SNN_GCUDA(g, call)                                                              \
  do {                                                                                  \
    cudaError_t e_ = (call);                                                            \
    if (e_ != cudaSuccess)                                                              \
      return gfail((g), e_ == cudaErrorMemoryAllocation ? SNN_ENOMEM : SNN_ECUDA,       \
                   std::string(#call ": ") + cudaGetErrorString(e_));                   \
  } while (0)

template <class T>
int galloc(snn_grad* g, T** p, size_t count) {
  void* d = nullptr;
  const size_t bytes = count * sizeof(T) > 0 ? count * sizeof(T) : 256;
  cudaError_t e = cudaMalloc(&d, bytes);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return gfail(g, e == cudaErrorMemoryAllocation ? SNN_ENOMEM : SNN_ECUDA,
                 "cudaMalloc of " + std::to_string(bytes) + " bytes: " + cudaGetErrorString(e));
  }
  g->bufs.push_back(d);
  *p = static_cast<T*>(d);
  return SNN_OK;
}

void grad_release(snn_grad* g) {
  for (void* p : g->bufs) cudaFree(p);
  g->bufs.clear();
}

// The tile kernel for `per` rows per block.
const void* gather_tile_fn(long long per) {
  return per <= 5 * kGatherWarps   ? reinterpret_cast<const void*>(grad_gather_tile_kernel<5>)
         : per <= 7 * kGatherWarps ? reinterpret_cast<const void*>(grad_gather_tile_kernel<7>)
                                   : reinterpret_cast<const void*>(grad_gather_tile_kernel<kGatherRows>);
}

// Gather of step tau, by the tile kernel where the rows lie in draw order, two
// steps' adjoints fit a block's shared memory and there are more than three rows
// per warp of a full wave.  Its blocks: one wave, as few rows per block as that
// allows.  A plain launch: launched while the backward kernel
// still holds registers, its blocks would not fit in one wave.
cudaError_t launch_gather(snn_grad* g, long long tau) {
  const NetView& v = g->v;
  int nb = (int)std::min<long long>(v.ndel, g->T - tau - v.dmin);
  if (nb <= 0) return cudaSuccess;
  const size_t win = (size_t)v.acc_words * 4;
  if (g->P.ord || 2 * win > kSmemBudget || v.N <= 3 * kGatherWarps * v.num_sms) {
    void* args[] = {&g->P, &tau};
    return launch_overlapped(g->P.ord ? reinterpret_cast<const void*>(grad_gather_kernel<true>)
                                      : reinterpret_cast<const void*>(grad_gather_kernel<false>),
                             dim3((unsigned)g->wblocks), kThreads, 0, args, false, v.stream);
  }
  const long long ncol = v.N / v.npc;
  const long long re = ncol * v.nexc, ri = v.N - re;
  const long long most = kGatherWarps * kGatherRows;
  long long per = std::min(most, (v.N + v.num_sms - 1) / v.num_sms);
  while (per < most && (re + per - 1) / per + (ri + per - 1) / per > v.num_sms) ++per;
  int per_block = (int)per, blocks_e = (int)((re + per - 1) / per);
  const int blocks = blocks_e + (int)((ri + per - 1) / per);
  int bufs = (int)std::min<size_t>(kGatherBufs, kSmemBudget / win);
  void* args[] = {&g->P, &tau, &nb, &bufs, &per_block, &blocks_e};
  return launch_overlapped(gather_tile_fn(per), dim3((unsigned)blocks), kGatherThreads, bufs * win, args, false,
                           v.stream);
}

cudaError_t launch_forward_step(snn_grad* g, long long t, int slot, int rates) {
  const GradParams& P = g->P;
  cudaStream_t st = g->v.stream;
  void* dargs[] = {const_cast<GradParams*>(&P), &t};
  void* uargs[] = {const_cast<GradParams*>(&P), &t, &slot, &rates};
  const cudaError_t e = launch_overlapped(reinterpret_cast<const void*>(grad_deliver_kernel),
                                          dim3((unsigned)g->wblocks), kThreads, 0, dargs, true, st);
  if (e != cudaSuccess) return e;
  return launch_overlapped(reinterpret_cast<const void*>(grad_update_kernel), dim3((unsigned)g->ublocks),
                           kThreads, 0, uargs, true, st);
}

}  // namespace

extern "C" {

int snn_grad_build(snn_net* net, int64_t n_steps, int32_t checkpoint_every, int32_t hard,
                   float beta, const double* target_rates, snn_grad** out) try {
  if (!out) return fail_global(SNN_EINVAL, "out is NULL");
  *out = nullptr;
  NetView v{};
  if (!net || net_view(net, &v) != SNN_OK)
    return fail_global(SNN_EINVAL, "net is NULL or a shard");
  if (v.precision != SNN_EXACT_F32W)
    return fail_global(SNN_EINVAL, "the differentiable form needs an SNN_EXACT_F32W net");
  if (n_steps < 1 || n_steps > (1LL << 31)) return fail_global(SNN_EINVAL, "n_steps must be >= 1");
  if (checkpoint_every < 1) return fail_global(SNN_EINVAL, "checkpoint_every must be >= 1");
  if (!(beta > 0.f) || !std::isfinite(beta)) return fail_global(SNN_EINVAL, "beta must be > 0");
  if (v.neuron.tau_c == v.neuron.tau_m)
    return fail_global(SNN_EINVAL, "tau_c must differ from tau_m");
  struct Release {
    void operator()(snn_grad* g) const {
      grad_release(g);
      delete g;
    }
  };
  std::unique_ptr<snn_grad, Release> own(new (std::nothrow) snn_grad());
  snn_grad* const g = own.get();
  if (!g) return fail_global(SNN_ENOMEM, "host allocation failed");
  g->bufs.reserve(32);
  g->v = v;
  g->T = n_steps;
  g->ckpt = (int)std::min<long long>(checkpoint_every, n_steps);
  g->nseg = (int)((n_steps + g->ckpt - 1) / g->ckpt);
  g->hard = hard ? 1 : 0;
  g->beta = beta;
  if (target_rates) {
    g->targets[0] = target_rates[0];
    g->targets[1] = target_rates[1];
  }
  g->nslot = v.dmin + v.ndel;  // d_max + 1
  const long long N = v.N;
  g->ublocks = (int)((N + kThreads - 1) / kThreads);
  g->wblocks = (int)((N * 32 + kThreads - 1) / kThreads);
  for (int rows : {5, 7, kGatherRows})
    if (cudaFuncSetAttribute(gather_tile_fn(rows * kGatherWarps), cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kSmemBudget) != cudaSuccess)
      return fail_global(SNN_ECUDA, "the gather kernel does not fit on the device");
  // propagators in FP64 as the spiking tables compute them (h = 1 ms)
  const double tm = v.neuron.tau_m, tc = v.neuron.tau_c;
  g->pvv = std::exp(-1.0 / tm);
  g->pcc = std::exp(-1.0 / tc);
  g->kappa = -tm * tc / (tc - tm) * (g->pcc - g->pvv);

  GradParams& P = g->P;
  P.N = N;
  P.accw = v.acc_words;
  P.npc = v.npc;
  P.npc4 = v.npc4;
  P.ncol = (int)(N / v.npc);
  P.unit = v.unit;
  P.planes = v.planes;
  P.ctile = v.ctile;
  P.colv = v.colv;
  P.nbg = v.nbg;
  P.nexc = v.nexc;
  P.dmin = v.dmin;
  P.ndel = v.ndel;
  P.bucket_mask = v.ndel == 32 ? 0xFFFFFFFFu : (1u << v.ndel) - 1u;
  P.nslot = g->nslot;
  P.rowcap = v.rowcap;
  P.hard = g->hard;
  P.T = (int)n_steps;
  P.seed_lo = (uint32_t)(v.seed & 0xFFFFFFFFu);
  P.seed_hi = (uint32_t)(v.seed >> 32);
  P.beta = beta;
  P.theta = v.neuron.theta;
  P.vr = v.neuron.v_reset;
  P.dc = v.neuron.dc;
  P.pvv = (float)g->pvv;
  P.pcc = (float)g->pcc;
  P.kappa = (float)g->kappa;
  P.J = v.neuron.j_ext_mV;
  P.syn = static_cast<const uint2*>(v.syn);
  P.bend = v.bend;

  int rc = SNN_OK;
  const size_t n = (size_t)N, accw = (size_t)v.acc_words;
  if (!rc) rc = galloc(g, &g->q, 65536);
  if (!rc) rc = galloc(g, &P.V, n);
  if (!rc) rc = galloc(g, &P.C, n);
  if (!rc) rc = galloc(g, &P.shist, n * g->nslot);
  if (!rc) rc = galloc(g, &P.active, n);
  if (!rc) rc = galloc(g, &P.gsum, 6);
  if (!rc) rc = galloc(g, &P.xe, accw);
  if (!rc) rc = galloc(g, &P.xin, accw);
  if (!rc) rc = galloc(g, &P.tape, n * kTape * g->ckpt);
  if (!rc) rc = galloc(g, &P.rate_part, (size_t)g->ublocks * 2);
  if (!rc) rc = galloc(g, &P.vbar, n);
  if (!rc) rc = galloc(g, &P.cbar, n);
  if (!rc) rc = galloc(g, &P.ibe, accw * g->nslot);
  if (!rc) rc = galloc(g, &P.ibi, accw * g->nslot);
  if (!rc) rc = galloc(g, &P.gb, n * 3);
  if (!rc) rc = galloc(g, &P.sg, n);
  if (!rc) rc = galloc(g, &P.gacc, n * 6);
  if (!rc) rc = galloc(g, &g->ck, n * (2 + g->nslot) * g->nseg);
  if (!rc) rc = galloc(g, &P.vtile, (size_t)(N / v.npc));
  // rows whose synapses lie in another order than they were drawn in
  const bool map = v.ntile > 1 || v.unit != kSlotUnit;
  P.ord_units = v.ord_units;
  if (!rc && map) rc = galloc(g, &P.ord, n * v.ord_units);
  if (!rc && map) rc = galloc(g, &P.ord_end, n * v.ndel);
  if (rc) return fail_global(rc, g->err);
  P.q = g->q;
  const std::vector<double>& qd = quantile_table();
  std::vector<float> qf(qd.size());
  for (size_t k = 0; k < qd.size(); ++k) qf[k] = (float)qd[k];
  cudaError_t e = cudaMemcpyAsync(g->q, qf.data(), qf.size() * 4, cudaMemcpyHostToDevice, v.stream);
  if (e == cudaSuccess) {
    grad_tile_words_kernel<<<(unsigned)v.ntile, kThreads, 0, v.stream>>>(P, v.tinfo);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess && map) {
    BuildParams bp = v.build;
    bp.ord = P.ord;
    bp.ord_end = P.ord_end;
    bp.ord_units = P.ord_units;
    e = launch_draw_order(bp, v.paper, v.num_sms, v.stream);
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(v.stream);
  if (e != cudaSuccess)
    return fail_global(SNN_ECUDA, std::string("gradient tables: ") + cudaGetErrorString(e));
  *out = own.release();
  return SNN_OK;
}
SNN_CATCH(fail_global(SNN_ENOMEM, kNoHostMemory))

int snn_grad_run(snn_grad* g, const double* theta, double* loss, double* rates, double* grad) try {
  if (!g || !theta || !loss) return gfail(g, SNN_EINVAL, "null argument");
  for (int k = 0; k < 6; ++k)
    if (!std::isfinite(theta[k])) return gfail(g, SNN_EINVAL, "parameters must be finite");
  if (!(theta[5] > 0.0)) return gfail(g, SNN_EINVAL, "nu_ext must be positive");
  GradParams& P = g->P;
  for (int k = 0; k < 4; ++k) P.a[k] = (float)theta[k];
  P.pvc_e = (float)(theta[4] * g->kappa);
  P.pvc_i = (float)((double)g->v.neuron.gc_inh * g->kappa);
  const double lam = theta[5] * 1.0;  // nu_ext (kHz) * h (1 ms)
  P.lam = (float)lam;
  P.sqlam = (float)std::sqrt(lam);
  cudaStream_t st = g->v.stream;
  const long long N = g->v.N;
  const size_t n = (size_t)N, accw = (size_t)g->v.acc_words;
  const size_t ckw = n * (2 + g->nslot);  // floats per checkpoint

  // forward, saving a checkpoint at the start of every segment
  grad_init_kernel<<<g->ublocks, kThreads, 0, st>>>(P);
  SNN_GCUDA(g, cudaGetLastError());
  SNN_GCUDA(g, cudaMemsetAsync(P.shist, 0, n * g->nslot * 4, st));
  SNN_GCUDA(g, cudaMemsetAsync(P.xe, 0, accw * 8, st));
  SNN_GCUDA(g, cudaMemsetAsync(P.xin, 0, accw * 8, st));
  SNN_GCUDA(g, cudaMemsetAsync(P.rate_part, 0, (size_t)g->ublocks * 16, st));
  for (long long t = 0; t < g->T; ++t) {
    if (t % g->ckpt == 0) {
      float* ck = g->ck + (size_t)(t / g->ckpt) * ckw;
      SNN_GCUDA(g, cudaMemcpyAsync(ck, P.V, n * 4, cudaMemcpyDeviceToDevice, st));
      SNN_GCUDA(g, cudaMemcpyAsync(ck + n, P.C, n * 4, cudaMemcpyDeviceToDevice, st));
      SNN_GCUDA(g, cudaMemcpyAsync(ck + 2 * n, P.shist, n * g->nslot * 4,
                                   cudaMemcpyDeviceToDevice, st));
    }
    SNN_GCUDA(g, launch_forward_step(g, t, -1, 1));
  }
  std::vector<double> part((size_t)g->ublocks * 2);
  SNN_GCUDA(g, cudaMemcpyAsync(part.data(), P.rate_part, part.size() * 8, cudaMemcpyDeviceToHost, st));
  SNN_GCUDA(g, cudaStreamSynchronize(st));
  double se = 0.0, si = 0.0;
  for (int b = 0; b < g->ublocks; ++b) {
    se += part[2 * b];
    si += part[2 * b + 1];
  }
  const long long ncol = N / g->v.npc;
  const double NE = (double)ncol * g->v.nexc, NI = (double)N - NE;
  const double rE = NE > 0 ? 1000.0 * se / ((double)g->T * NE) : 0.0;
  const double rI = NI > 0 ? 1000.0 * si / ((double)g->T * NI) : 0.0;
  *loss = (rE - g->targets[0]) * (rE - g->targets[0]) + (rI - g->targets[1]) * (rI - g->targets[1]);
  if (rates) {
    rates[0] = rE;
    rates[1] = rI;
  }
  if (!grad) return SNN_OK;

  // backward: recompute each segment from its checkpoint, then run back
  P.dlds_e = NE > 0 ? (float)(2.0 * (rE - g->targets[0]) * 1000.0 / ((double)g->T * NE)) : 0.f;
  P.dlds_i = NI > 0 ? (float)(2.0 * (rI - g->targets[1]) * 1000.0 / ((double)g->T * NI)) : 0.f;
  SNN_GCUDA(g, cudaMemsetAsync(P.vbar, 0, n * 4, st));
  SNN_GCUDA(g, cudaMemsetAsync(P.cbar, 0, n * 4, st));
  SNN_GCUDA(g, cudaMemsetAsync(P.ibe, 0, accw * g->nslot * 4, st));
  SNN_GCUDA(g, cudaMemsetAsync(P.ibi, 0, accw * g->nslot * 4, st));
  SNN_GCUDA(g, cudaMemsetAsync(P.gb, 0, n * 3 * 4, st));
  SNN_GCUDA(g, cudaMemsetAsync(P.gacc, 0, n * 6 * 8, st));
  for (int seg = g->nseg - 1; seg >= 0; --seg) {
    const long long t0 = (long long)seg * g->ckpt;
    const long long t1 = std::min<long long>(g->T, t0 + g->ckpt);
    const float* ck = g->ck + (size_t)seg * ckw;
    SNN_GCUDA(g, cudaMemcpyAsync(P.V, ck, n * 4, cudaMemcpyDeviceToDevice, st));
    SNN_GCUDA(g, cudaMemcpyAsync(P.C, ck + n, n * 4, cudaMemcpyDeviceToDevice, st));
    SNN_GCUDA(g, cudaMemcpyAsync(P.shist, ck + 2 * n, n * g->nslot * 4, cudaMemcpyDeviceToDevice,
                                 st));
    grad_active_kernel<<<g->ublocks, kThreads, 0, st>>>(P, t0);
    for (long long t = t0; t < t1; ++t) SNN_GCUDA(g, launch_forward_step(g, t, (int)(t - t0), 0));
    for (long long tau = t1 - 1; tau >= t0; --tau) {
      SNN_GCUDA(g, launch_gather(g, tau));
      int slot = (int)(tau - t0);
      void* args[] = {&P, &tau, &slot};
      SNN_GCUDA(g, launch_overlapped(reinterpret_cast<const void*>(grad_backward_kernel),
                                     dim3((unsigned)g->ublocks), kThreads, 0, args, true, st));
    }
    SNN_GCUDA(g, cudaGetLastError());
  }
  grad_sum_kernel<<<6, kSumThreads, 0, st>>>(P);
  SNN_GCUDA(g, cudaGetLastError());
  SNN_GCUDA(g, cudaMemcpyAsync(grad, P.gsum, 6 * sizeof(double), cudaMemcpyDeviceToHost, st));
  SNN_GCUDA(g, cudaStreamSynchronize(st));
  return SNN_OK;
}
SNN_CATCH(gfail(g, SNN_ENOMEM, kNoHostMemory))

const char* snn_grad_last_error(const snn_grad* g) { return g ? g->err.c_str() : ""; }

void snn_grad_destroy(snn_grad* g) {
  if (!g) return;
  cudaStreamSynchronize(g->v.stream);
  grad_release(g);
  delete g;
}

}  // extern "C"
