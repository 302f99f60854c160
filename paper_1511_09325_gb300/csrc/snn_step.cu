// snn_step.cu -- the two kernels of one 1 ms step.
//
// update_kernel (neuron update, arxiv 1511.09325 Sec. 2 LIF + SFA):
//   grid-stride over chunks of 128 neurons, one warp each; one lane owns 4
//   consecutive neurons and one Philox4x32-10 block (counter (i/4, t, EXT, 0))
//   whose 4 words give their external Poisson counts.  It reads and clears
//   their recurrent input, applies refractoriness, threshold, reset and the
//   exact propagator with explicitly rounded FP32 operations.  A chunk's
//   spikes go to their delivery tile's list of the step (one atomic per tile and
//   chunk) as descriptors -- the spiker's row and its bucket ends, copied from
//   the build's table -- and to the block's record region.  The item counts of
//   the next delivery (isum, gsum) are kept up to date here; spike and
//   external-event totals go to per-block partial sums.  Warps work without
//   each other, so no barrier waits for the chunk with the most spikes.  Bound
//   by instruction issue (59 % of slots at 96x96; 406 instructions per chunk
//   without spikes, most of them Philox) and by the state's 26 bytes per
//   neuron.  Measured at 96x96, 11.4 M neurons, Down / mean / Up state: 64 / 74 /
//   87 us a step; with tiles of 1024 neurons per block, counted and placed
//   between barriers, 89 / 99 / 111 us.
//
// deliver_kernel (event-driven delivery, Sec. 1), "pull by delay": the input
//   of step t+1 is the sum over delays d of bucket d of every neuron that
//   spiked at step t+1-d, so only one accumulator (resident in L2) receives
//   additions, not a d_max-slot ring.  The (delay bucket, spiker) items of the
//   last d_max steps, ordered by (tile, bucket, spiker), form one virtual list
//   split by cost over a persistent grid of one block per SM.  A part of a
//   tile with enough items keeps a shared-memory window over the tile's
//   columns, where about four fifths of the tile's synapses land (the local
//   half and most of the near stencil; a bucket's "in" part, whose records
//   name the window's word directly); those are summed there with
//   shared-memory reductions and the window is added once to the accumulator
//   by bulk asynchronous reductions.  The "out" parts go to L2 as
//   fire-and-forget int32 reductions through the tile's neighbour table.  A
//   warp resolves 32 items at a time (one per lane: list entry, bucket ends)
//   and deals their 32-byte sectors to its lanes through a list in shared
//   memory, in parts and then out parts, so that a round of 32 sectors runs
//   one code path; the next batch's entries and ends are loaded meanwhile.
//   Integer addition makes the result independent of the order.
//   Bound in dense states by the L2: an FP16 item is about 300 bytes of DRAM
//   reads (47 ps of the chip's time) and 12 scattered L2 reductions (61 ps at
//   the measured 204 G/s), and takes 100 ps; own-tile synapses (50 reductions
//   in shared memory, 21 ps) hide behind both.  Measured, us a step (before:
//   rows without parts, one table lookup per record): 2x2 FP32 10.6 (26.2),
//   24x24 FP32 44 (66), 48x48 FP32 128 (162), 96x96 FP16 358 (376; Down state
//   89 (116), Up state 747 (760)).
#include <algorithm>

#include "snn_device.cuh"
#include "snn_internal.h"

namespace snn {
namespace {

constexpr int kUpdateThreads = 256;
constexpr int kDeliverThreads = 768;   // one delivery block per SM (24 warps, 2 rounds in flight)
constexpr int kBatchThreads = 512;     // batch kernel: 2 update sub-blocks or one delivery block
constexpr int kUpdateSubs = kBatchThreads / kUpdateThreads;
// Precision of a kernel: SNN_EXACT_F32W, SNN_EXACT_F16W, or F16W with a weight of
// 64 mV or more (see half_fx).
constexpr int kF16Wide = 2;
template <int PREC>
__device__ constexpr bool f16() {
  return PREC != SNN_EXACT_F32W;
}
constexpr int kDepth = 2;        // rounds of 32-byte sectors in flight per lane
constexpr int kUpdateWarps = kUpdateThreads / 32;
constexpr int kChunk = 128;      // neurons of a warp's chunk (four per lane)
// Sector list of a warp: kListCap entries (a multiple of 32) at places p +
// p / 32, so that lanes that write runs of about 8 entries meet few bank
// conflicts.  A batch of 32 items of the default networks has about 290
// entries; a longer one is streamed in pieces.
constexpr int kListCap = 320;
constexpr int kListWords = kListCap + kListCap / 32 + 2;

struct NeuronOut {
  float v, c;
  uint32_t r;
  bool spike;
};

// One neuron, one step; every float operation rounded as written.  Selects, no
// branches: a refractory neuron (r > 0) discards its input and is clamped to
// V_reset.
__device__ __forceinline__ NeuronOut neuron_step(float v, float c, uint32_t r,
                                                 int32_t I, float pvc,
                                                 const StepParams& P) {
  NeuronOut o;
  const float u = __fadd_rn(v, __fmul_rn(__int2float_rn(I), 1.52587890625e-05f));
  const bool active = r == 0u;
  o.spike = active && u >= P.theta;
  const float w = active && !o.spike ? u : P.vr;
  const float ca = o.spike ? __fadd_rn(c, P.dc) : c;
  o.r = active ? (o.spike ? (uint32_t)P.nref : 0u) : r - 1u;
  o.v = __fmaf_rn(ca, pvc, __fmul_rn(w, P.pvv));
  o.c = __fmul_rn(ca, P.pcc);
  return o;
}

// Fire-and-forget int32 reductions into the accumulator and into shared
// memory.  No compiler memory barrier: nothing the streaming
// loops read aliases the window or the accumulator.
__device__ __forceinline__ void red_add_nz(const int32_t* p, int32_t v) {  // nothing for v = 0
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.s32 p, %1, 0;\n\t"
      "@p red.global.add.s32 [%0], %1;\n\t}" ::"l"(p), "r"(v));
}
__device__ __forceinline__ void red_shared(uint32_t a, int32_t v) {
  asm volatile("red.shared.add.s32 [%0], %1;" ::"r"(a), "r"(v));
}

// Loads of the neuron state, read once per step: no L1 allocation, so that
// L1 capacity does not bound the loads a block keeps in flight.
__device__ __forceinline__ float4 ld_stream(const float4* p) {
  float4 v;
  asm volatile("ld.global.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "l"(p));
  return v;
}
__device__ __forceinline__ int4 ld_stream(const int4* p) {
  int4 v;
  asm volatile("ld.global.L1::no_allocate.v4.s32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p));
  return v;
}
__device__ __forceinline__ uint32_t ld_stream(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.global.L1::no_allocate.u32 %0, [%1];" : "=r"(v) : "l"(p));
  return v;
}

// Poisson count of word x by inversion.  Entry b of the table (one per top
// byte of x) holds bits 0-6: the thresholds <= b << 24; bits 8-31: the low 24
// bits of the one threshold inside the bin, less one (2^24 - 1: none inside);
// bit 7: more than one inside, scan from the count.  So x << 8 > entry exactly
// when x has reached the bin's threshold.
__device__ __forceinline__ uint32_t poisson_entry(const StepParams& P, int b) {
  const int k = P.pois_guide[b];
  const uint32_t lo = (uint32_t)b << 24;
  const bool in1 = k < P.n_pois_thr && (P.pois_thr[k] - lo) >> 24 == 0u;
  const bool in2 = k + 1 < P.n_pois_thr && (P.pois_thr[k + 1] - lo) >> 24 == 0u;
  return (in1 ? (P.pois_thr[k] - lo - 1u) << 8 : 0xFFFFFF00u) | (in2 ? 128u : 0u) | (uint32_t)k;
}

// Barrier of an update body: the whole block (bar 0) or one 256-thread
// sub-block of the batch kernel (named barrier `bar`).
__device__ __forceinline__ void body_sync(int bar) {
  if (bar == 0)
    __syncthreads();
  else
    asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(kUpdateThreads) : "memory");
}

// Slot of step s >= 0 (a 64-bit remainder is about 100 instructions).
__device__ __forceinline__ int slot_of(const StepParams& P, long long s) {
  return (s >> 32) == 0 ? (int)((uint32_t)s % (uint32_t)P.nslot) : (int)(s % P.nslot);
}

// Records the first inconsistency a kernel finds; the host turns it into
// SNN_ESTATE.
__device__ __forceinline__ void set_status(const StepParams& P, unsigned code) {
  atomicOr(&P.ctl->status, code);
  if (P.hstatus != nullptr) *reinterpret_cast<volatile unsigned*>(P.hstatus) = code;
}

// Quotient of x by d from m = min(floor(2^32 / d), 2^32 - 1): the estimate
// is at most one below the quotient, so one correction step finishes it.
__device__ __forceinline__ uint32_t div_by(uint32_t x, uint32_t d, uint32_t m) {
  uint32_t q = __umulhi(x, m);
  if (x - q * d >= d) ++q;
  return q;
}

// The next place at *count for each lane of `live`, all of which make this call:
// one atomic for the lanes of the same `key` (mostly one; the lanes of a key have
// the same counter).
__device__ __forceinline__ unsigned next_place(unsigned live, unsigned* count, uint32_t key) {
  const unsigned lane = threadIdx.x & 31u;
  const unsigned peers = __match_any_sync(live, key);
  const int lead = __ffs(peers) - 1;
  unsigned pos = 0u;
  if ((int)lane == lead) pos = atomicAdd(count, (unsigned)__popc(peers));
  return __shfl_sync(peers, pos, lead) + (unsigned)__popc(peers & ((1u << lane) - 1u));
}

// Shared memory of one update body.
struct UpdateSmem {
  uint32_t pois[256];
  unsigned rc;                   // records written in this step
  unsigned items;                // change of gsum
  uint32_t id[kUpdateWarps][kChunk];  // the spikes of a warp's chunk
  unsigned long long syn[kUpdateWarps];  // synaptic events per warp
  unsigned ksum[kUpdateWarps];
};

// Update body vb of vgrid for step t, run by kUpdateThreads threads (thread
// index tid, barrier `bar`): every warp takes chunks of kChunk neurons, lane e
// of a chunk the quad of neurons 4 e .. 4 e + 3, and works without the other
// warps.  A chunk's spikes are then dealt to the lanes, one each: a lane finds
// its spike's column and takes the next place of the column's tile's list; the
// chunk takes its places in the body's record region by one atomic.  Body vb
// owns ext_part[vb], spk_part[vb], syn_part[vb] and record region vb of the
// net, so the grid size must be the same every step.  Each spike goes to its
// tile's list of the step (or to one compact list of ids, without ccnt) and to
// the body's record region as (step << 32 | id).  A shard (SHARD, P.sg.on)
// updates its own columns only, draws the external input with global neuron
// indices and records global indices; the halo's columns take part in the
// count bookkeeping.  The step is t_of(), called when the state may be read.
template <bool SHARD, class F>
__device__ __forceinline__ void update_body(const StepParams& P, F&& t_of, int vb, int vgrid,
                                            UpdateSmem& S, int tid, int bar) {
  const int lane = tid & 31, warp = tid >> 5;
  const uint32_t npc = (uint32_t)P.npc;
  const uint32_t quads = (uint32_t)((P.N + 3) / 4);  // below 2^29
  const uint32_t stride = (uint32_t)vgrid * (uint32_t)(kUpdateWarps * 32);  // quads
  // A quad's input: one 16-byte access where columns are whole quads (or acc
  // is indexed by the neuron); else word by word, in its first neuron's column
  // and the next one (columns of 2 or 3 neurons: see below).
  const bool whole = (npc & 3u) == 0u;
  const bool direct = P.colv == nullptr || whole;
  const bool split = !direct && npc >= 4u;

  // The state of the warp's next chunk is requested before the current chunk
  // is processed, and the virtual index of the column(s) of the one after it
  // (which its input's address needs), so their latency overlaps the work.
  // l: place of the quad's first neuron in its column; a: quad of its input, or
  // word of the first neuron's input with a2 the word that neuron would have
  // in front of the next column.
  float4 pv = make_float4(0.f, 0.f, 0.f, 0.f), pc = pv;
  uint32_t pr = 0u;
  int4 pa = make_int4(0, 0, 0, 0);
  auto place = [&](uint32_t q, uint32_t* l, uint32_t* v, uint32_t* v2) {
    const uint32_t c = div_by(4u * q, npc, P.npc_m);
    *l = 4u * q - c * npc;
    *v = P.colv != nullptr && q < quads ? __ldg(P.colv + c) : 0u;
    *v2 = split && q < quads && c + 1u < (uint32_t)P.ncol ? __ldg(P.colv + c + 1u) : 0u;
  };
  auto input = [&](uint32_t q, uint32_t l, uint32_t v, uint32_t v2, uint32_t* a, uint32_t* a2) {
    const unsigned long long w = (unsigned long long)v * (uint32_t)P.npc4 + l;
    *a = P.colv == nullptr ? q : whole ? (uint32_t)(w >> 2) : (uint32_t)w;
    *a2 = v2 * (uint32_t)P.npc4 + l - npc;
  };
  // word of neuron 4 q + e's input (split)
  auto word = [&](uint32_t l, uint32_t a, uint32_t a2, uint32_t e) -> int32_t* {
    return P.acc + (size_t)(uint32_t)((l + e < npc ? a : a2) + e);
  };
  auto load = [&](uint32_t q, uint32_t l, uint32_t a, uint32_t a2) {
    if (q < quads) {
      pv = ld_stream(reinterpret_cast<const float4*>(P.V) + q);
      pc = ld_stream(reinterpret_cast<const float4*>(P.C) + q);
      pr = ld_stream(reinterpret_cast<const uint32_t*>(P.R) + q);
      if (direct) {
        pa = ld_stream(reinterpret_cast<const int4*>(P.acc) + a);
      } else if (split) {
        const uint32_t n = (uint32_t)min(4ll, P.N - 4ll * q);
        pa.x = *word(l, a, a2, 0u);
        pa.y = n > 1u ? *word(l, a, a2, 1u) : 0;
        pa.z = n > 2u ? *word(l, a, a2, 2u) : 0;
        pa.w = n > 3u ? *word(l, a, a2, 3u) : 0;
      }
    }
  };
  uint32_t q = (uint32_t)vb * (uint32_t)(kUpdateWarps * 32) + (uint32_t)tid;
  uint32_t l, l_nxt, v, v2, v_nxt, v2_nxt, a, a2;
  place(q, &l, &v, &v2);
  place(q + stride, &l_nxt, &v_nxt, &v2_nxt);
  input(q, l, v, v2, &a, &a2);
  body_sync(bar);  // the shared memory may still be read by a previous body
  S.pois[tid] = poisson_entry(P, tid);
  const long long t = t_of();
  load(q, l, a, a2);
  const int slot = slot_of(P, t);
  if (tid == 0) {
    S.rc = 0u;
    S.items = 0u;
    if (vb == 0) P.ctl->td = t;  // the step's delivery
  }
  const unsigned long long rc0 = P.rcnt[vb];
  unsigned ksum = 0u;
  unsigned long long syn = 0ull;  // out-degrees of this thread's spikes (with deg)
  body_sync(bar);

  // Each tile's item count (isum, their sum gsum) moves on by one step: it
  // covers the steps t - d_max + 1 .. t - d_min + 1 that this step's delivery
  // reads, less step t itself (d_min = 1), whose spikes the delivery adds.
  // Step t - d_max, whose slot is (t + 1) mod (d_max + 1), goes out.
  if (P.ccnt != nullptr) {
    const long long s_in = P.dmin == 1 ? t - 1 : t + 1 - P.dmin;
    const unsigned* cin_ = s_in >= 0 ? P.ccnt + (size_t)slot_of(P, s_in) * P.ntile * kCntStride : nullptr;
    const unsigned* cout_ = P.ccnt + (size_t)slot_of(P, t + 1) * P.ntile * kCntStride;
    for (long long m = (long long)vb * kUpdateThreads + tid; m < P.ntile;
         m += (long long)vgrid * kUpdateThreads) {
      const unsigned d = (cin_ ? cin_[m * kCntStride] : 0u) - cout_[m * kCntStride];
      if (d) {
        atomicAdd(P.isum + m * kCntStride, d);
        atomicAdd(&S.items, d);
      }
    }
  }
  if (SHARD)  // halo spikes per column that the step's ingest will count
    for (long long c = (long long)vb * kUpdateThreads + tid; c < P.ncol;
         c += (long long)vgrid * kUpdateThreads)
      P.icnt[c] = 0u;

  for (; q - (uint32_t)lane < quads; q += stride) {
    const float4 v4 = pv, c4 = pc;
    const uint32_t r4 = pr;
    int4 a4 = pa;
    const uint32_t a_own = a, a2_own = a2, l_own = l;
    l = l_nxt;
    input(q + stride, l, v_nxt, v2_nxt, &a, &a2);
    load(q + stride, l, a, a2);
    place(q + 2u * stride, &l_nxt, &v_nxt, &v2_nxt);

    uint32_t gq = q;  // global quad of the four neurons
    bool own = q < quads;
    if (SHARD && own) {
      const int col = (int)((4u * q - l_own) / npc);
      const int cy = col / P.W, cx = col - cy * P.W;
      own = cx >= P.sg.tx0 && cx < P.sg.tx0 + P.sg.tw && cy >= P.sg.ty0 && cy < P.sg.ty0 + P.sg.th;
      int gx, gy;
      shard_global_col(P.sg, cx, cy, &gx, &gy);
      gq = (((uint32_t)gy * (uint32_t)P.sg.GW + (uint32_t)gx) * npc + l_own) >> 2;
    }
    unsigned spk = 0u;  // bit e: neuron 4 q + e fired
    if (own) {
      const uint4 x = philox4x32_10(make_uint4(gq, (uint32_t)t, kTagExt, 0u), P.key);
      if (direct) {
        reinterpret_cast<int4*>(P.acc)[a_own] = make_int4(0, 0, 0, 0);
      } else if (split) {
#pragma unroll
        for (uint32_t e = 0; e < 4u; ++e)
          if (4ll * q + e < P.N) *word(l_own, a_own, a2_own, e) = 0;
      } else {
        int32_t in[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const long long i = 4ll * q + e;
          in[e] = 0;
          if (i < P.N) {
            const uint32_t c = div_by((uint32_t)i, npc, P.npc_m);
            int32_t* w = P.acc + (size_t)P.colv[c] * P.npc4 + ((uint32_t)i - c * npc);
            in[e] = *w;
            *w = 0;
          }
        }
        a4 = make_int4(in[0], in[1], in[2], in[3]);
      }
      const float vin[4] = {v4.x, v4.y, v4.z, v4.w};
      const float cin[4] = {c4.x, c4.y, c4.z, c4.w};
      const int32_t ain[4] = {a4.x, a4.y, a4.z, a4.w};
      const uint32_t xin[4] = {x.x, x.y, x.z, x.w};
      int kp[4];
      uint32_t ent[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) ent[e] = S.pois[xin[e] >> 24];
#pragma unroll
      for (int e = 0; e < 4; ++e) kp[e] = (int)(ent[e] & 127u) + ((xin[e] << 8) > ent[e] ? 1 : 0);
      if ((ent[0] | ent[1] | ent[2] | ent[3]) & 128u) {
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (ent[e] & 128u) {
            int k = (int)(ent[e] & 127u);
            while (k < P.n_pois_thr && xin[e] >= P.pois_thr[k]) ++k;
            kp[e] = k;
          }
      }
      float vout[4], cout[4];
      uint32_t rout = 0u;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        uint32_t le = l_own + (uint32_t)e;
        if (!whole) {  // n_per_col may be 2
          le -= le >= npc ? npc : 0u;
          le -= le >= npc ? npc : 0u;
        }
        const int32_t I = ain[e] + kp[e] * P.jx;
        const uint32_t r = r4 >> (8 * e) & 0xFFu;
        const NeuronOut o = neuron_step(vin[e], cin[e], r, I, le < (uint32_t)P.nexc ? P.pvc_e : P.pvc_i, P);
        vout[e] = o.v;
        cout[e] = o.c;
        rout |= o.r << (8 * e);
        spk |= o.spike ? 1u << e : 0u;
      }
      if (q == quads - 1u && (P.N & 3)) {  // the last quad ends early
        const int live = (int)(P.N & 3);
        spk &= (1u << live) - 1u;
#pragma unroll
        for (int e = 1; e < 4; ++e)
          if (e >= live) kp[e] = 0;
      }
      ksum += (unsigned)(kp[0] + kp[1] + kp[2] + kp[3]);
      reinterpret_cast<float4*>(P.V)[q] = make_float4(vout[0], vout[1], vout[2], vout[3]);
      reinterpret_cast<float4*>(P.C)[q] = make_float4(cout[0], cout[1], cout[2], cout[3]);
      reinterpret_cast<uint32_t*>(P.R)[q] = rout;
    }
    if (__ballot_sync(0xFFFFFFFFu, spk != 0u) == 0u) continue;

    // the chunk's spikes in a row, and their places in the record region
    unsigned n = 0u;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const unsigned b = __ballot_sync(0xFFFFFFFFu, spk >> e & 1u);
      if (spk >> e & 1u) S.id[warp][n + __popc(b & ((1u << lane) - 1u))] = 4u * q + (uint32_t)e;
      n += (unsigned)__popc(b);
    }
    unsigned rec = 0u;
    if (lane == 0) rec = atomicAdd(&S.rc, n);
    rec = __shfl_sync(0xFFFFFFFFu, rec, 0);
    __syncwarp();
    for (unsigned k0 = 0u; k0 < n; k0 += 32u) {
      const unsigned k = k0 + (unsigned)lane;
      uint32_t row = 0u;             // the spike's row in bend
      unsigned long long at = 0ull;  // its place in the lists
      const unsigned live = n - k0 < 32u ? (1u << (n - k0)) - 1u : 0xFFFFFFFFu;  // lanes with k < n
      if (k < n) {
        const uint32_t id = S.id[warp][k];
        const uint32_t c = div_by(id, npc, P.npc_m), il = id - c * npc;
        if (P.ccnt != nullptr) {
          const uint32_t ct = __ldg(P.ctile + c);
          row = __ldg(P.colv + c) * npc + il;
          const size_t ts = (size_t)slot * P.ntile + (ct >> 6);
          const unsigned place = next_place(live, P.ccnt + ts * kCntStride, ct >> 6);
          at = ((unsigned long long)slot * P.planes * P.ntile + (ct >> 6)) * P.tcap + place;
          if (P.rlist != nullptr) P.rlist[ts * P.tcap + place] = (uint16_t)((ct & 63u) * npc + il);
        } else {
          P.ids[next_place(live, P.cnt + slot, 0u)] = id;
        }
        atomicAdd(&P.colcnt[2ull * c + (il < (uint32_t)P.nexc ? 0u : 1u)], 1ull);
        if (P.deg != nullptr) syn += P.deg[id];
        uint32_t gid = id;
        if (SHARD) {
          const int cy = (int)c / P.W, cx = (int)c - cy * P.W;
          int gx, gy;
          shard_global_col(P.sg, cx, cy, &gx, &gy);
          gid = ((uint32_t)gy * (uint32_t)P.sg.GW + (uint32_t)gx) * npc + il;
        }
        const unsigned long long ri = rc0 + rec + k;
        if ((long long)ri < P.rec_region)
          P.rec[(long long)vb * P.rec_region + (long long)ri] = ((unsigned long long)(unsigned)t << 32) | gid;
      }
      // descriptors: four lanes copy one spike's planes into its list
      if (P.list != nullptr) {
        const size_t plane = (size_t)P.ntile * P.tcap;
        for (unsigned s0 = 0u; s0 < min(n - k0, 32u); s0 += 8u) {
          const int src = (int)(s0 + ((unsigned)lane >> 2));
          const uint32_t rs = __shfl_sync(0xFFFFFFFFu, row, src);
          const unsigned long long as = __shfl_sync(0xFFFFFFFFu, at, src);
          if (k0 + (unsigned)src < n)
            for (int p = lane & 3; p < P.planes; p += 4)
              P.list[as + p * plane] = P.bend[(size_t)rs * P.planes + p];
        }
      }
    }
    __syncwarp();
  }

  // external and synaptic events: per-body partial sums
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    ksum += __shfl_xor_sync(0xFFFFFFFFu, ksum, o);
    syn += __shfl_xor_sync(0xFFFFFFFFu, syn, o);
  }
  if (lane == 0) {
    S.ksum[warp] = ksum;
    S.syn[warp] = syn;
  }
  body_sync(bar);
  if (tid == 0) {
    unsigned long long tot = 0ull, tsyn = 0ull;
    for (int w = 0; w < kUpdateWarps; ++w) {
      tot += S.ksum[w];
      tsyn += S.syn[w];
    }
    if (S.items) atomicAdd(P.gsum, S.items);
    // (reductions: nothing waits for the old values)
    atomicAdd(P.ext_part + vb, tot);
    atomicAdd(P.spk_part + vb, (unsigned long long)S.rc);
    if (P.syn_part != nullptr)
      atomicAdd(P.syn_part + vb, P.deg != nullptr ? tsyn : (unsigned long long)S.rc * (unsigned)P.K);
    if ((long long)(rc0 + S.rc) > P.rec_region) P.ctl->rec_overflow = 1u;
    P.rcnt[vb] = rc0 + S.rc;
  }
}

template <bool SHARD>
__global__ void __launch_bounds__(kUpdateThreads, 4) update_kernel(const StepParams P) {
  __shared__ UpdateSmem S;
  update_body<SHARD>(
      P,
      [&]() -> long long {
        grid_wait();
        grid_go();
        return P.ctl->t;
      },
      (int)blockIdx.x, (int)gridDim.x, S, (int)threadIdx.x, 0);
}

// ---------------------------------------------------------------------------
// Delivery.
// ---------------------------------------------------------------------------

struct DeliverSmem {
  unsigned long long wsum[3][32]; // per-warp sums of the range scan
  int rt[2];                      // tiles holding the ends of the block's range
  unsigned ri[2];                 // item places of the ends inside them
};

// Sums, over the block's threads, of three 64-bit values, and the exclusive
// prefix of the first.  Contains one barrier.
__device__ __forceinline__ void block_scan3(unsigned long long a, unsigned long long b,
                                            unsigned long long c, DeliverSmem& S,
                                            unsigned long long* a_excl, unsigned long long* a_total,
                                            unsigned long long* b_total, unsigned long long* c_total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nwarps = (int)(blockDim.x >> 5);
  unsigned long long incl = a;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long u = __shfl_up_sync(0xFFFFFFFFu, incl, o);
    b += __shfl_xor_sync(0xFFFFFFFFu, b, o);
    c += __shfl_xor_sync(0xFFFFFFFFu, c, o);
    if (lane >= o) incl += u;
  }
  if (lane == 31) {
    S.wsum[0][warp] = incl;
    S.wsum[1][warp] = b;
    S.wsum[2][warp] = c;
  }
  __syncthreads();
  unsigned long long w = lane < nwarps ? S.wsum[0][lane] : 0ull;
  unsigned long long before = lane < warp ? w : 0ull;
  b = lane < nwarps ? S.wsum[1][lane] : 0ull;
  c = lane < nwarps ? S.wsum[2][lane] : 0ull;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    w += __shfl_xor_sync(0xFFFFFFFFu, w, o);
    before += __shfl_xor_sync(0xFFFFFFFFu, before, o);
    b += __shfl_xor_sync(0xFFFFFFFFu, b, o);
    c += __shfl_xor_sync(0xFFFFFFFFu, c, o);
  }
  *a_excl = before + incl - a;
  *a_total = w;
  *b_total = b;
  *c_total = c;
}

// What a warp needs of the part it streams: items a .. b - 1 of a tile.
struct Part {
  const unsigned char* syn;  // the tile's first row
  const uint4* lst;          // lane b: bucket b's descriptors (lists of rows: its
                             // u16 rows), less its first item's place
  const uint4* bend;         // lists of rows: the tile's first descriptor, else null
  int planes;
  unsigned pfx;              // lane b: items of the tile before bucket b
  unsigned a, b;
};

// Item `item` of the part: its descriptor's plane and its bucket.  The
// buckets' prefixes lie in the lanes; a five-step search over them finds the
// last bucket that starts at or before the item.  Beyond the part: bucket -1.
// ROWS: the net may keep lists of rows.
template <bool ROWS>
__device__ __forceinline__ int load_item(const Part& T, unsigned item, uint4* d) {
  int lo = 0;
#pragma unroll
  for (int step = 16; step > 0; step >>= 1) {
    const unsigned v = __shfl_sync(0xFFFFFFFFu, T.pfx, lo + step);
    if (v <= item) lo += step;
  }
  const unsigned long long l = __shfl_sync(0xFFFFFFFFu, (unsigned long long)T.lst, lo);
  if (item >= T.b) return -1;
  if (ROWS && T.bend != nullptr) {
    const uint32_t row = __ldcs(reinterpret_cast<const uint16_t*>(l) + item);
    *d = __ldg(T.bend + (size_t)row * T.planes + lo / kPlaneBuckets);
  } else {
    *d = __ldcs(reinterpret_cast<const uint4*>(l) + item);
  }
  return lo;
}

// Row (bits 0 .. 15) and bucket ends (units): bytes beg, mid, end of an item.
__device__ __forceinline__ uint2 item_bounds(const uint4& d, int bucket) {
  if (bucket < 0) return make_uint2(0u, 0u);
  const int i = bucket % kPlaneBuckets;  // its ends: the i-th halfword of words 1 .. 3
  const uint32_t w = i < 2 ? d.y : i < 4 ? d.z : d.w;
  const uint32_t me = i & 1 ? w >> 16 : w & 0xFFFFu;
  const uint32_t before = i & 1 ? w >> 8 : i == 0 ? d.x >> 16 : i == 2 ? d.y >> 24 : d.z >> 24;
  return make_uint2(d.x & 0xFFFFu, (before & 0xFFu) | me << 8);
}

// Sector-list entries.  F16W: sector (25 bits) | k << 25 | sign of the source
// << 31; F32W: sector (26 bits) | k << 26.  A sector is counted from the
// tile's first row: a tile has at most 50 176 rows of at most 255 units of 2
// (F16W) or 4 (F32W) sectors.
template <int PREC>
__device__ constexpr uint32_t sector_bits() {
  return f16<PREC>() ? 25u : 26u;
}

// One 32-byte sector of the table, read once.  The L2 fetches 64 bytes around
// it, not the default 128: a bucket (about 270 bytes at a random place) then
// takes about 300 bytes of DRAM traffic instead of 360 (96x96 FP16 Up state:
// 745 us a step, 850 us with the default).  The load is predicated, not
// branched around: a load under a branch is waited for at the branch's end,
// which leaves one round in flight whatever the depth.
struct Sector {
  uint32_t w[8];
};
__device__ __forceinline__ void ld_sector(Sector& s, const unsigned char* p, bool on) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.u32 p, %9, 0;\n\t"
      "@p ld.global.L1::no_allocate.L2::evict_first.L2::64B.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n\t}"
      : "+r"(s.w[0]), "+r"(s.w[1]), "+r"(s.w[2]), "+r"(s.w[3]), "+r"(s.w[4]), "+r"(s.w[5]),
        "+r"(s.w[6]), "+r"(s.w[7])
      : "l"(p), "r"((uint32_t)on));
}

// Weight of an F16W record, rint(half * 2^16) with the scale's sign.  One rounded
// multiply-add: x * (+-2^16) + 1.5 * 2^23 lands in [2^23, 2^24), where the float
// grid is the integers, so the low mantissa bits hold the rounded product.  That
// holds for weights below 64 mV; nets with larger ones (kF16Wide) convert.
template <int PREC>
__device__ __forceinline__ int32_t half_fx(uint32_t half_bits, float scale) {
  const float h = __half2float(__ushort_as_half((unsigned short)half_bits));
  if (PREC == kF16Wide) return __float2int_rn(__fmul_rn(h, scale));
  return __float_as_int(__fmaf_rn(h, scale, 12582912.0f)) - 0x4B400000;
}

// Delivers the records of one in sector: into the window at win_s (WIN), else
// into the accumulator words of the tile at `acc`.
template <int PREC, bool WIN>
__device__ __forceinline__ void deliver_in(const Sector& s, uint32_t win_s, const int32_t* acc) {
  if (f16<PREC>()) {
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int32_t wfx = half_fx<PREC>(s.w[q] >> 16, 65536.0f);
      if (WIN)
        red_shared(win_s + 4u * (s.w[q] & 0xFFFFu), wfx);
      else
        red_add_nz(acc + (s.w[q] & 0xFFFFu), wfx);
    }
  } else {
#pragma unroll
    for (int q = 0; q < 8; q += 2) {
      const int32_t wfx = (int32_t)s.w[q + 1];
      if (WIN)
        red_shared(win_s + 4u * s.w[q], wfx);  // a pad's bit 31 leaves the address
      else if (wfx != 0)  // a pad's code has bit 31 set
        red_add_nz(acc + s.w[q], wfx);
    }
  }
}

// Delivers the records of one out sector through the neighbour-table row of
// the source's column (in shared memory for WIN, else in global memory).
template <int PREC, bool WIN>
__device__ __forceinline__ void deliver_out(const Sector& s, float scale, uint32_t nb_s,
                                            const uint32_t* nb_g, const int32_t* acc) {
  constexpr int kN = f16<PREC>() ? 8 : 4, kW = 8 / kN;
  uint32_t base[kN];
#pragma unroll
  for (int q = 0; q < kN; ++q) {
    const uint32_t code = s.w[kW * q];
    if (WIN)
      asm volatile("ld.shared.u32 %0, [%1];" : "=r"(base[q]) : "r"(nb_s + ((code >> 9) & 0xFCu)));
    else
      base[q] = __ldg(nb_g + ((code >> 11) & 63u));
  }
#pragma unroll
  for (int q = 0; q < kN; ++q) {
    const uint32_t code = s.w[kW * q];
    const int32_t wfx = f16<PREC>() ? half_fx<PREC>(code >> 17, scale) : (int32_t)s.w[kW * q + kW - 1];
    red_add_nz(acc + (base[q] + (code & 2047u)), wfx);
  }
}

// One warp streams its share of a part: batches of bs items, batch q by warp
// q mod the block's warps (counted from warp `w0`).  WIN: the part's window
// and neighbour table are in shared memory.
template <int PREC, int DEPTH, bool ROWS, bool WIN>
__device__ __forceinline__ void stream_part(const StepParams& P, const Part& T, const int32_t* acc_t,
                                            const uint32_t* nb_g, unsigned bs, int w0, uint32_t win_s,
                                            uint32_t nb_s, uint32_t* list) {
  const int lane = threadIdx.x & 31;
  const unsigned nw = blockDim.x >> 5;
  const unsigned warp = ((threadIdx.x >> 5) + nw - (unsigned)w0) % nw;
  constexpr uint32_t kSecMask = (1u << sector_bits<PREC>()) - 1u;
  static_assert(kListCap % (32 * DEPTH) == 0, "a piece of a batch is whole groups of rounds");
  const unsigned step = bs * nw;
  unsigned it0 = T.a + warp * bs;
  if (it0 >= T.b) return;
  // this lane's item of the batch at i: none beyond the batch or the part
  auto item_at = [&](unsigned i, uint4* d) -> int {
    return load_item<ROWS>(T, (unsigned)lane < bs && i < T.b ? i + lane : 0xFFFFFFFFu, d);
  };
  uint4 raw = make_uint4(0u, 0u, 0u, 0u);
  int nb = item_at(it0, &raw);
  uint2 cur = item_bounds(raw, nb);
  for (;;) {
    // the next batch's descriptors are loaded while this one is streamed
    nb = item_at(it0 + step, &raw);
    // sectors of the current batch: the in parts' at 0 .. n_in - 1, the out
    // parts' from the next multiple of 32
    const int beg = (int)(cur.y & 0xFFu), mid = (int)(cur.y >> 8 & 0xFFu), end = (int)(cur.y >> 16);
    const int u_in = (mid - beg) * P.unit_sec, u_out = (end - mid) * P.unit_sec;
    uint32_t incl = (uint32_t)u_in | (uint32_t)u_out << 16;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if (lane >= o) incl += v;
    }
    const uint32_t tot = __shfl_sync(0xFFFFFFFFu, incl, 31);
    const int n_in = (int)(tot & 0xFFFFu), n_out = (int)(tot >> 16);
    const int r_in = (n_in + 31) >> 5, rounds = r_in + ((n_out + 31) >> 5);
    const int lim_out = r_in * 32 + n_out;
    for (int c0 = 0; c0 < rounds * 32; c0 += kListCap) {
      __syncwarp();
      {
        // this lane's entries inside [c0, c0 + kListCap)
        const uint32_t k = div_by(cur.x, (uint32_t)P.npc, P.npc_m), l = cur.x - k * (uint32_t)P.npc;
        uint32_t tag = cur.x * (uint32_t)P.row_sec + (uint32_t)(beg * P.unit_sec);
        tag |= k << sector_bits<PREC>();
        if (f16<PREC>() && (int)l >= P.nexc) tag |= 0x80000000u;
        const int p_in = (int)(incl & 0xFFFFu) - u_in - c0;
        const int p_out = r_in * 32 + (int)(incl >> 16) - u_out - c0;
        for (int p = max(p_in, 0); p < min(p_in + u_in, kListCap); ++p)
          list[p + (p >> 5)] = tag + (uint32_t)(p - p_in);
        for (int p = max(p_out, 0); p < min(p_out + u_out, kListCap); ++p)
          list[p + (p >> 5)] = tag + (uint32_t)(u_in + p - p_out);
      }
      __syncwarp();
      const int r0 = c0 >> 5, r1 = min(rounds, r0 + (kListCap >> 5));
      Sector sec[DEPTH] = {};
      uint32_t en[DEPTH];
      auto fetch = [&](int r, Sector& x, uint32_t& e) {
        const int p = r * 32 + lane;
        const bool on = r < r1 && p < (r < r_in ? n_in : lim_out);
        e = on ? list[(r - r0) * 33 + lane] : 0u;
        ld_sector(x, T.syn + (size_t)(e & kSecMask) * 32u, on);
      };
#pragma unroll
      for (int d = 0; d < DEPTH; ++d) fetch(r0 + d, sec[d], en[d]);
      for (int r = r0; r < r1; r += DEPTH) {
#pragma unroll
        for (int d = 0; d < DEPTH; ++d) {
          const int rr = r + d;
          if (rr < r_in) {
            if (rr * 32 + lane < n_in) deliver_in<PREC, WIN>(sec[d], win_s, acc_t);
          } else if (rr < r1 && rr * 32 + lane < lim_out) {
            const uint32_t kk = f16<PREC>() ? (en[d] >> 25) & 63u : en[d] >> 26;
            deliver_out<PREC, WIN>(sec[d], __uint_as_float(0x47800000u | (en[d] & 0x80000000u)),
                                   nb_s + kk * 256u, nb_g + kk * 64u, P.acc);
          }
          fetch(rr + DEPTH, sec[d], en[d]);
        }
      }
    }
    it0 += step;
    if (it0 >= T.b || it0 < step) break;
    cur = item_bounds(raw, nb);
  }
}

// What the range split knows of a tile.
struct TileLoad {
  unsigned items;                // (bucket, spiker) items that this step delivers
  unsigned old;                  // those of the steps before (isum)
  unsigned win_items, cost_win;  // see StepParams
};
// A tile costs its items plus a fixed part: cost_win when its items reach the
// window threshold -- the set-up and flush of the window -- else kCostPart
// when it has items.
__device__ __forceinline__ unsigned tile_cost(const TileLoad& l) {
  return l.items + (l.items >= l.win_items ? l.cost_win : (l.items ? kCostPart : 0u));
}
// Item of a tile on which cost point x (< its cost) falls: the fixed part is
// laid out before the items.
__device__ __forceinline__ unsigned item_at_cost(const TileLoad& l, unsigned x) {
  const unsigned fixed = tile_cost(l) - l.items;
  return x > fixed ? x - fixed : 0u;
}

// The tiles of one net, for deliver_blocks.
struct NetTiles {
  const StepParams& P;
  const unsigned* now;  // counts of step t per tile (d_min = 1)
  long long t;
  __device__ __forceinline__ NetTiles(const StepParams& p) : P(p), now(nullptr), t(0) {}
  __device__ __forceinline__ void start(long long step) {
    t = step;
    if (P.dmin == 1) now = P.ccnt + (size_t)slot_of(P, t) * P.ntile * kCntStride;
  }
  __device__ __forceinline__ int count() const { return P.ntile; }
  __device__ __forceinline__ unsigned min_items() const { return P.min_items; }
  __device__ __forceinline__ TileLoad load(int g) const {
    TileLoad l;
    l.old = P.isum[(size_t)g * kCntStride];
    l.items = l.old + (now ? now[(size_t)g * kCntStride] : 0u);
    l.win_items = P.win_items;
    l.cost_win = P.cost_win;
    return l;
  }
  // clears the counts that the next update fills (step t - d_max, whose slot
  // it is, is no longer read)
  __device__ __forceinline__ void clear(int g) const {
    P.ccnt[((size_t)slot_of(P, t + 1) * P.ntile + g) * kCntStride] = 0u;
  }
  // block-uniform: parameters and own index of tile g
  __device__ __forceinline__ const StepParams& net(int g, int* tile) const {
    *tile = g;
    return P;
  }
  __device__ __forceinline__ void check(int vb, unsigned long long old_total) const {
    if (vb == 0 && threadIdx.x == 0 && (unsigned)old_total != *P.gsum) set_status(P, kStatusCounts);
  }
};

// Delivery block vb of vgrid (NT threads) for one step.  The step's items,
// ordered by (tile, delay bucket, spiker), are split into at most vgrid
// contiguous ranges of equal cost and at least min_items items each; a cost
// point maps to the item it falls on, so consecutive blocks' ranges tile the
// items.  Block vb locates the tiles and items its range spans from the tiles'
// counts and walks the tiles that have items.  A tile's part with at least
// win_items items is delivered through the shared-memory window, a smaller one
// without any block-wide set-up.  Counts that disagree with the spike lists
// set the status word; items beyond the lists are not delivered.  `dyn` is the
// block's dynamic shared memory: window, neighbour table, sector lists (for
// windows of at most win_words words and max_cols columns).  The step is
// t_of(), called when the lists may be read.
template <int PREC, int DEPTH, int NT, bool ROWS, class Tiles, class F>
__device__ __forceinline__ void deliver_blocks(Tiles& tiles, F&& t_of, int vb, int vgrid, int win_words,
                                               int max_cols, DeliverSmem& S, unsigned char* dyn) {
  const int tid = threadIdx.x;
  const int lane = tid & 31;
  constexpr int kWarps = NT / 32;
  int32_t* const win = reinterpret_cast<int32_t*>(dyn);
  uint32_t* const nbs = reinterpret_cast<uint32_t*>(win + win_words);
  uint32_t* const list = nbs + max_cols * 64 + (tid >> 5) * kListWords;
  // the window is cleared first
  for (int i = tid; i < win_words >> 2; i += NT) reinterpret_cast<int4*>(win)[i] = make_int4(0, 0, 0, 0);
  const long long t = t_of();
  tiles.start(t);
  const int ntile = tiles.count();

  // the block's range: items i0 of tile t0 to i1 (exclusive) of tile t1
  int t0, t1;
  unsigned i0, i1;
  TileLoad mine = {0u, 0u, 0u, 0u};  // up to 32 tiles: lane's tile, in every warp
  if (ntile <= 32) {
    if (lane < ntile) mine = tiles.load(lane);
    const unsigned cost = tile_cost(mine);
    unsigned long long incl = cost;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long u = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if (lane >= o) incl += u;
    }
    // a tile has at most 50 176 rows and 32 buckets: the sums fit 32 bits
    const unsigned total = __reduce_add_sync(0xFFFFFFFFu, mine.items);
    const unsigned old = __reduce_add_sync(0xFFFFFFFFu, mine.old);
    const unsigned long long ctotal = __shfl_sync(0xFFFFFFFFu, incl, 31);
    tiles.check(vb, old);
    if (vb == 0 && tid < ntile) tiles.clear(tid);
    const unsigned want = (total + tiles.min_items() - 1u) / tiles.min_items();
    const unsigned nact = min(want, (unsigned)vgrid);
    if ((unsigned)vb >= nact) return;
    auto find = [&](unsigned i, int* tile, unsigned* item) {
      const unsigned long long x = ctotal * i / nact;
      const unsigned after = __ballot_sync(0xFFFFFFFFu, incl > x);  // tiles that end beyond x
      const int m = after ? __ffs(after) - 1 : 0;
      const unsigned it = __shfl_sync(0xFFFFFFFFu, item_at_cost(mine, (unsigned)(x - (incl - cost))), m);
      *tile = after ? m : ntile;
      *item = after ? it : 0u;
    };
    find((unsigned)vb, &t0, &i0);
    find((unsigned)vb + 1u, &t1, &i1);
  } else {
    const int per = (ntile + NT - 1) / NT;
    const int g0 = tid * per;
    unsigned long long items = 0ull, cost = 0ull, old = 0ull;
    for (int g = g0; g < g0 + per && g < ntile; ++g) {
      const TileLoad l = tiles.load(g);
      items += l.items;
      old += l.old;
      cost += tile_cost(l);
    }
    for (long long g = (long long)vb * NT + tid; g < ntile; g += (long long)vgrid * NT) tiles.clear((int)g);
    unsigned long long cexcl = 0ull, ctotal = 0ull, total = 0ull, old_total = 0ull;
    block_scan3(cost, items, old, S, &cexcl, &ctotal, &total, &old_total);
    tiles.check(vb, old_total);
    const unsigned long long want = (total + tiles.min_items() - 1) / tiles.min_items();
    const int nact = (int)(want < (unsigned long long)vgrid ? want : (unsigned long long)vgrid);
    if (vb >= nact) return;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const unsigned long long x = ctotal * (unsigned long long)(vb + i) / (unsigned long long)nact;
      if (x >= ctotal) {
        if (tid == 0) {
          S.rt[i] = ntile;
          S.ri[i] = 0u;
        }
      } else if (x >= cexcl && x < cexcl + cost) {
        unsigned long long rc = cexcl;
        for (int g = g0; g < g0 + per && g < ntile; ++g) {
          const TileLoad l = tiles.load(g);
          const unsigned c = tile_cost(l);
          if (x < rc + c) {
            S.rt[i] = g;
            S.ri[i] = item_at_cost(l, (unsigned)(x - rc));
            break;
          }
          rc += c;
        }
      }
    }
    __syncthreads();
    t0 = S.rt[0];
    t1 = S.rt[1];
    i0 = S.ri[0];
    i1 = S.ri[1];
  }

  const uint32_t win_s = (uint32_t)__cvta_generic_to_shared(win);
  const uint32_t nb_s = (uint32_t)__cvta_generic_to_shared(nbs);
  bool clean = true;      // the window is clear and no flush reads it
  int rot = 0;            // first warp of the next part without window
  for (int c0 = ntile <= 32 ? 0 : t0; c0 <= t1 && c0 < ntile; c0 += 32) {
    const unsigned xs = ntile <= 32 ? mine.items : c0 + lane < ntile ? tiles.load(c0 + lane).items : 0u;
    unsigned have = __ballot_sync(0xFFFFFFFFu, xs != 0u && c0 + lane >= t0 && c0 + lane <= t1);
    while (have) {
      const int m = __ffs(have) - 1;
      have &= have - 1u;
      const int g = c0 + m;
      const unsigned x = __shfl_sync(0xFFFFFFFFu, xs, m);
      const unsigned a = g == t0 ? i0 : 0u;
      const unsigned b = g == t1 ? min(i1, x) : x;
      if (a >= b) continue;
      int tile;
      const StepParams& P = tiles.net(g, &tile);
      // lane b: the slot of bucket b's step (-1: before step 0) and the tile's
      // count; a list holds at most tcap spikes
      const long long s = t + 1 - (P.dmin + lane);
      const int slot_l = lane < P.ndel && s >= 0 ? slot_of(P, s) : -1;
      const long long ts = (long long)slot_l * P.ntile + tile;
      const unsigned n = slot_l >= 0 ? min(P.ccnt[ts * kCntStride], (unsigned)P.tcap) : 0u;
      const uint2 ti = P.tinfo[tile];
      unsigned incl = n;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned u = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += u;
      }
      const unsigned found = __shfl_sync(0xFFFFFFFFu, incl, 31);
      if (found != x && tid == 0) set_status(P, kStatusCounts);
      Part T;
      T.syn = static_cast<const unsigned char*>(P.syn) + (size_t)ti.x * P.npc * P.row_sec * 32u;
      T.pfx = lane < P.ndel ? incl - n : 0xFFFFFFFFu;
      T.lst = P.list + ((((long long)slot_l * P.planes + lane / kPlaneBuckets) * P.ntile + tile) * P.tcap -
                        (long long)T.pfx);
      T.bend = nullptr;
      T.planes = 0;
      if (ROWS && P.rlist != nullptr) {
        T.lst = reinterpret_cast<const uint4*>(P.rlist + (ts * P.tcap - (long long)T.pfx));
        T.bend = P.bend + (size_t)ti.x * P.npc * P.planes;
        T.planes = P.planes;
      }
      int32_t* const acc_t = P.acc + (size_t)ti.x * P.npc4;
      const uint32_t* nb_g = P.nbg + (size_t)ti.x * 64;
      const int cols = (int)ti.y;
      T.a = a;
      T.b = min(b, found);
      if (b - a >= P.win_items) {
        if (!clean) {
          // the issuing threads' bulk reductions have read the window
          if (tid < kMaxTileCols) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
          __syncthreads();
          for (int i = tid; i < (cols * P.npc4) >> 2; i += NT)
            reinterpret_cast<int4*>(win)[i] = make_int4(0, 0, 0, 0);
        }
        for (int i = tid; i < cols * 16; i += NT)
          reinterpret_cast<uint4*>(nbs)[i] = __ldg(reinterpret_cast<const uint4*>(nb_g) + i);
        __syncthreads();
        // the same number of batches for every warp, as few as can be (delivery
        // of 24x24 FP32, mean state: 47.7 us with batches of a quarter of a
        // warp's items rounded down, 45.2 rounded up, 43.8 so)
        const unsigned per_warp = (b - a + 32u * kWarps - 1u) / (32u * kWarps);
        const unsigned bs = max(2u, (b - a + per_warp * kWarps - 1u) / (per_warp * kWarps));
        stream_part<PREC, DEPTH, ROWS, true>(P, T, acc_t, nb_g, bs, 0, win_s, nb_s, list);
        // add the window to the accumulator: one asynchronous bulk reduction
        // (element-wise atomic in L2) per column, issued once every warp's
        // reductions are visible to the async proxy
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
        if (tid < cols) {
          const uint32_t bytes = (uint32_t)P.npc4 * 4u;
          asm volatile(
              "cp.reduce.async.bulk.global.shared::cta.bulk_group.add.s32 [%0], [%1], %2;\n\t"
              "cp.async.bulk.commit_group;" ::"l"(acc_t + (size_t)tid * P.npc4),
              "r"(win_s + (uint32_t)tid * bytes), "r"(bytes)
              : "memory");
        }
        clean = false;
      } else {
        // few items: every warp takes batches of its own, as many as fill the block
        const unsigned nit = T.b > T.a ? T.b - T.a : 0u;
        unsigned bs = (nit + kWarps - 1) / kWarps;
        bs = bs < 2u ? 2u : (bs > 32u ? 32u : bs);
        stream_part<PREC, DEPTH, ROWS, false>(P, T, acc_t, nb_g, bs, rot, win_s, nb_s, list);
        rot = (int)((rot + (nit + bs - 1) / bs) % kWarps);
      }
    }
  }
  // the bulk reductions must have been performed (not only have read the
  // window) before the block goes on: the batch kernel's next phase reads the
  // accumulator after a grid barrier
  if (tid < kMaxTileCols) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

// ROWS: for nets with lists of rows.  Those take 42 bytes per neuron instead of
// 1344 (20 delays), but an item's descriptor is then 16 bytes at a random place
// instead of the next 16 bytes of a list, which is slower (96x96 FP16, an early
// form of this kernel: 1077 against 892 us a step in an Up state, 132 against
// 118 in a Down state), so they are kept only where the others do not fit.
template <int PREC, bool ROWS>
__global__ void __launch_bounds__(kDeliverThreads, 1) deliver_kernel(const StepParams P) {
  extern __shared__ __align__(16) unsigned char s_dyn[];
  __shared__ DeliverSmem S;
  NetTiles tiles(P);
  deliver_blocks<PREC, kDepth, kDeliverThreads, ROWS>(
      tiles,
      [&]() -> long long {
        grid_wait();
        grid_go();
        const long long t = P.ctl->td;
        if (blockIdx.x == 0 && threadIdx.x == 0) P.ctl->t = t + 1;  // the next update's step
        return t;
      },
      (int)blockIdx.x, (int)gridDim.x, P.tcols * P.npc4, P.tcols, S, s_dyn);
}

// ---------------------------------------------------------------------------
// Batched form: many independent nets advanced by one persistent launch.
// Every step runs the update bodies of all nets (two 256-thread sub-blocks
// per block, each with its own named barrier), a grid barrier, the delivery
// of all nets, and a second barrier.  Virtual update body g belongs to net k
// with first[k] <= g < first[k + 1] and is the standalone kernel's block body.
// The delivery treats the tiles of all nets as one sequence, which the blocks
// split by cost as the standalone kernel's blocks split one net's tiles, so
// every net computes exactly what its own kernels compute.  (A virtual
// delivery block per net and column before: 1356 for the 64-net sweep, each
// with its own search for its range: 225 us a step; now 133 us.)
// ---------------------------------------------------------------------------

// The tiles of all nets of a batch, for deliver_blocks.
struct BatchTiles {
  const BatchParams& B;
  StepParams& cur;  // shared memory: the parameters of net `k`
  int k;
  long long t;
  __device__ __forceinline__ BatchTiles(const BatchParams& b, StepParams& p) : B(b), cur(p), k(-1), t(0) {}
  __device__ __forceinline__ void start(long long step) { t = step; }
  __device__ __forceinline__ int count() const { return B.n_tiles; }
  __device__ __forceinline__ unsigned min_items() const { return B.min_items; }
  __device__ __forceinline__ TileLoad load(int g) const {
    const BatchTile& b = B.tiles[g];
    TileLoad l;
    l.old = *b.isum;
    l.items = l.old;
    if (b.dmin == 1) l.items += b.ccnt[(size_t)((uint32_t)(t % b.nslot)) * b.stride];
    l.win_items = b.win_items;
    l.cost_win = b.cost_win;
    return l;
  }
  __device__ __forceinline__ void clear(int g) const {
    const BatchTile& b = B.tiles[g];
    b.ccnt[(size_t)((uint32_t)((t + 1) % b.nslot)) * b.stride] = 0u;
  }
  __device__ __forceinline__ const StepParams& net(int g, int* tile) {
    const BatchTile& b = B.tiles[g];
    *tile = b.tile;
    if (b.net != k) {
      k = b.net;
      __syncthreads();  // every warp is done with the net before
      for (int w = threadIdx.x; w < (int)(sizeof(StepParams) / 4); w += kBatchThreads)
        reinterpret_cast<uint32_t*>(&cur)[w] = reinterpret_cast<const uint32_t*>(B.nets + k)[w];
      __syncthreads();
    }
    return cur;
  }
  __device__ __forceinline__ void check(int, unsigned long long) const {}
};

// Bounded grid barrier (all blocks are co-resident: cooperative launch).  A
// block that polls spin_limit times without the generation moving sets *err
// and gives up; every later barrier then returns false at once.
__device__ __forceinline__ bool grid_barrier(const BatchParams& B, unsigned* s_ok) {
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned ok = 1u;
    volatile unsigned* gen = B.bar + 1;
    volatile unsigned* err = B.bar + 2;
    if (*err) {
      ok = 0u;
    } else {
      const unsigned g = *gen;
      __threadfence();
      const unsigned expected = gridDim.x + B.extra_arrivals;
      if (atomicAdd(B.bar, 1u) == expected - 1u) {
        B.bar[0] = 0u;
        __threadfence();
        atomicAdd(B.bar + 1, 1u);
      } else {
        long long polls = 0;
        while (*gen == g) {
          if (*err) {
            ok = 0u;
            break;
          }
          if (++polls > B.spin_limit) {
            atomicExch(B.bar + 2, 1u);
            ok = 0u;
            break;
          }
          __nanosleep(64);
        }
      }
      __threadfence();
    }
    *s_ok = ok;
  }
  __syncthreads();
  return *s_ok != 0u;
}

// Net of virtual body g: the last k with first[k] <= g.
__device__ __forceinline__ int net_of(const int* first, int n, int g) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (first[mid] <= g)
      lo = mid;
    else
      hi = mid - 1;
  }
  return lo;
}

template <int PREC, int INFL, bool ROWS>
__global__ void __launch_bounds__(kBatchThreads, 2) batch_kernel(const BatchParams B) {
  extern __shared__ __align__(16) unsigned char s_dyn[];
  __shared__ StepParams s_p[kUpdateSubs];  // the nets of the current virtual bodies
  __shared__ DeliverSmem SD;
  __shared__ int s_uf[kMaxBatch + 1];
  __shared__ unsigned s_ok;
  UpdateSmem* SU = reinterpret_cast<UpdateSmem*>(s_dyn);  // one per sub-block
  const int sub = threadIdx.x / kUpdateThreads;
  const int stid = threadIdx.x - sub * kUpdateThreads;
  const int n = B.n_nets;
  for (int k = threadIdx.x; k <= n; k += blockDim.x) s_uf[k] = B.u_first[k];
  __syncthreads();
  const int total_u = s_uf[n];
  constexpr int kParamWords = (int)(sizeof(StepParams) / 4);
  for (long long step = 0; step < B.n_steps; ++step) {
    const long long t = B.t0 + step;
    for (int g = blockIdx.x * kUpdateSubs + sub; g < total_u; g += gridDim.x * kUpdateSubs) {
      const int k = net_of(s_uf, n, g);
      body_sync(1 + sub);
      for (int w = stid; w < kParamWords; w += kUpdateThreads)
        reinterpret_cast<uint32_t*>(&s_p[sub])[w] = reinterpret_cast<const uint32_t*>(B.nets + k)[w];
      body_sync(1 + sub);
      update_body<false>(s_p[sub], [&]() -> long long { return t; }, g - s_uf[k], s_uf[k + 1] - s_uf[k],
                         SU[sub], stid, 1 + sub);
    }
    if (!grid_barrier(B, &s_ok)) return;
    BatchTiles tiles(B, s_p[0]);
    deliver_blocks<PREC, INFL, kBatchThreads, ROWS>(tiles, [&]() -> long long { return t; }, (int)blockIdx.x,
                                                    (int)gridDim.x, B.win_words, B.max_cols, SD, s_dyn);
    // each net's tiles must sum to its own total
    for (int k = (int)blockIdx.x * (kBatchThreads / 32) + (int)(threadIdx.x >> 5); k < n;
         k += (int)gridDim.x * (kBatchThreads / 32)) {
      unsigned old = 0u;
      for (int g = B.t_first[k] + (int)(threadIdx.x & 31); g < B.t_first[k + 1]; g += 32) old += *B.tiles[g].isum;
      old = __reduce_add_sync(0xFFFFFFFFu, old);
      if ((threadIdx.x & 31) == 0 && old != *B.nets[k].gsum) set_status(B.nets[k], kStatusCounts);
    }
    if (!grid_barrier(B, &s_ok)) return;
  }
  if (blockIdx.x == 0)
    for (int k = threadIdx.x; k < n; k += blockDim.x) B.nets[k].ctl->t = B.t0 + B.n_steps;
}

// Spike-record drain, one kernel.  Block b copies the records kept in region
// b (rcnt[b], at most `region`; records are step << 32 | id) as separate id
// and step arrays, starting at the number of records kept in the regions
// before b, to the mapped host buffers when all kept records fit them
// (map_cap) and to the device stage otherwise.  Block 0 writes the header
// {records kept, 1 if any were dropped, first step, last step} to mapped host
// memory (each region is in step order, so its first and last
// records bound its steps).  The last block to finish resets the region
// counters and the overflow flag.
__global__ void __launch_bounds__(256) drain_records_kernel(
    unsigned long long* rcnt, int nreg, long long region, const unsigned long long* rec,
    Ctl* ctl, unsigned long long* map_hdr, uint32_t* stage_ids,
    uint32_t* stage_steps, uint32_t* map_ids, uint32_t* map_steps, long long map_cap) {
  __shared__ unsigned long long s_pre[8], s_tot[8];
  __shared__ unsigned s_tmin[8], s_tmax[8], s_lost[8];
  __shared__ bool s_last;
  const int b = blockIdx.x;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  unsigned long long pre = 0ull, tot = 0ull;
  unsigned tmin = 0xFFFFFFFFu, tmax = 0u, lost = 0u;
  for (int r = threadIdx.x; r < nreg; r += blockDim.x) {
    const unsigned long long v = rcnt[r];
    const unsigned long long kept = (long long)v < region ? v : (unsigned long long)region;
    lost |= (long long)v > region ? 1u : 0u;
    tot += kept;
    if (r < b) pre += kept;
    if (b == 0 && kept > 0ull) {
      const unsigned first = (unsigned)(rec[(long long)r * region] >> 32);
      const unsigned lastt = (unsigned)(rec[(long long)r * region + (long long)kept - 1] >> 32);
      tmin = min(tmin, first);
      tmax = max(tmax, lastt);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    pre += __shfl_xor_sync(0xFFFFFFFFu, pre, o);
    tot += __shfl_xor_sync(0xFFFFFFFFu, tot, o);
    tmin = min(tmin, __shfl_xor_sync(0xFFFFFFFFu, tmin, o));
    tmax = max(tmax, __shfl_xor_sync(0xFFFFFFFFu, tmax, o));
    lost |= __shfl_xor_sync(0xFFFFFFFFu, lost, o);
  }
  if (lane == 0) {
    s_pre[w] = pre;
    s_tot[w] = tot;
    s_tmin[w] = tmin;
    s_tmax[w] = tmax;
    s_lost[w] = lost;
  }
  __syncthreads();
  pre = 0ull;
  tot = 0ull;
  tmin = 0xFFFFFFFFu;
  tmax = 0u;
  lost = 0u;
  for (int k = 0; k < (int)(blockDim.x >> 5); ++k) {
    pre += s_pre[k];
    tot += s_tot[k];
    tmin = min(tmin, s_tmin[k]);
    tmax = max(tmax, s_tmax[k]);
    lost |= s_lost[k];
  }
  if (b == 0 && threadIdx.x == 0) {
    const unsigned long long h[4] = {tot, (lost || ctl->rec_overflow) ? 1ull : 0ull,
                                     (unsigned long long)tmin, (unsigned long long)tmax};
    for (int k = 0; k < 4; ++k) map_hdr[k] = h[k];
  }
  const bool to_map = (long long)tot <= map_cap;
  uint32_t* ids = (to_map ? map_ids : stage_ids) + pre;
  uint32_t* steps = (to_map ? map_steps : stage_steps) + pre;
  const unsigned long long v = rcnt[b];
  const long long kept = (long long)v < region ? (long long)v : region;
  const unsigned long long* src = rec + (long long)b * region;
  for (long long k = threadIdx.x; k < kept; k += blockDim.x) {
    const unsigned long long r = src[k];
    ids[k] = (uint32_t)r;
    steps[k] = (uint32_t)(r >> 32);
  }
  // the counters are read by every block: the last one to finish resets them
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    s_last = atomicAdd(&ctl->drained, 1u) == (unsigned)nreg - 1u;
  }
  __syncthreads();
  if (s_last) {
    __threadfence();
    for (int r = threadIdx.x; r < nreg; r += blockDim.x) rcnt[r] = 0ull;
    if (threadIdx.x == 0) {
      ctl->rec_overflow = 0u;
      ctl->drained = 0u;
    }
  }
}

// Lists neuron l of column c at place r of its tile's list of the step: its row,
// or its descriptor (plane 0; the other planes follow at the stride of all
// tiles' lists).
__device__ __forceinline__ void list_spike(const StepParams& P, long long slot, uint32_t ct, unsigned r,
                                           uint32_t c, uint32_t l) {
  if (P.rlist != nullptr) {
    P.rlist[(slot * P.ntile + (ct >> 6)) * P.tcap + r] = (uint16_t)((ct & 63u) * (uint32_t)P.npc + l);
    return;
  }
  const long long at = (slot * P.planes * P.ntile + (ct >> 6)) * P.tcap + r;
  const uint4* d = P.bend + ((size_t)P.colv[c] * P.npc + l) * P.planes;
  const long long stride = (long long)P.ntile * P.tcap;
  for (int p = 0; p < P.planes; ++p) P.list[at + p * stride] = d[p];
}

// Counts the records a drain would return: header {records kept, 1 if any were
// dropped} to mapped host memory (one block).
__global__ void __launch_bounds__(1024) count_records_kernel(const unsigned long long* rcnt, int nreg,
                                                             long long region, const Ctl* ctl,
                                                             unsigned long long* map_hdr) {
  __shared__ unsigned long long s_kept[32];
  unsigned long long kept = 0ull;
  unsigned lost = ctl->rec_overflow;
  for (int r = threadIdx.x; r < nreg; r += blockDim.x) {
    const unsigned long long v = rcnt[r];
    kept += (long long)v < region ? v : (unsigned long long)region;
    lost |= (long long)v > region ? 1u : 0u;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) kept += __shfl_xor_sync(0xFFFFFFFFu, kept, o);
  if ((threadIdx.x & 31) == 0) s_kept[threadIdx.x >> 5] = kept;
  const int any = __syncthreads_or((int)lost);
  if (threadIdx.x == 0) {
    kept = 0ull;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) kept += s_kept[w];
    map_hdr[0] = kept;
    map_hdr[1] = any ? 1ull : 0ull;
  }
}

// Shard: the received spikes of step t (global indices ids[0 .. n)) that
// belong to halo columns join the step's lists as the update kernel's own
// spikes do, at the next place of the tile's list.  Indices of the shard's
// own columns and of columns outside its local grid are skipped.  An index
// beyond the global network, or more than n_per_col spikes for one column
// (a duplicated index), is skipped and sets the status word.
__global__ void __launch_bounds__(256) ingest_kernel(const StepParams P, const uint32_t* ids,
                                                     long long n) {
  const long long t = P.ctl->t;
  const long long slot = t % P.nslot;
  const unsigned long long ng = (unsigned long long)P.sg.GW * (unsigned long long)P.sg.GH *
                                (unsigned long long)P.npc;
  const int lane = threadIdx.x & 31;
  // (whole warps: the lanes that list a spike take their places together)
  for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k - lane < n;
       k += (long long)gridDim.x * blockDim.x) {
    uint32_t c = 0u, l = 0u;  // local column and place in it
    bool halo = false;
    if (k < n) {
      const uint32_t g = ids[k];
      if ((unsigned long long)g >= ng) {
        set_status(P, kStatusIngest);
      } else {
        const uint32_t gc = g / (uint32_t)P.npc;
        l = g - gc * (uint32_t)P.npc;
        const int gy = (int)(gc / (uint32_t)P.sg.GW), gx = (int)gc - gy * P.sg.GW;
        const int lx = wrap(gx - P.sg.ex0, P.sg.GW), ly = wrap(gy - P.sg.ey0, P.sg.GH);
        const bool own = lx >= P.sg.tx0 && lx < P.sg.tx0 + P.sg.tw && ly >= P.sg.ty0 &&
                         ly < P.sg.ty0 + P.sg.th;  // listed by the update kernel
        halo = lx < P.W && ly < P.H && !own;
        c = (uint32_t)(ly * P.W + lx);
        if (halo && atomicAdd(P.icnt + c, 1u) >= (unsigned)P.npc) {
          set_status(P, kStatusIngest);
          halo = false;
        }
      }
    }
    const unsigned live = __ballot_sync(0xFFFFFFFFu, halo);
    if (halo) {
      // at most n_per_col spikes of each of its columns: the list has room
      const uint32_t ct = P.ctile[c];
      const long long tile_slot = slot * P.ntile + (ct >> 6);
      const unsigned r = next_place(live, P.ccnt + tile_slot * kCntStride, ct >> 6);
      list_spike(P, slot, ct, r, c, l);
    }
  }
}

// Sum of the per-block spike counts (measurement helper).
__global__ void sum_parts_kernel(const unsigned long long* part, int n, unsigned long long* out) {
  unsigned long long s = 0ull;
  for (int i = threadIdx.x; i < n; i += 32) s += part[i];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
  if (threadIdx.x == 0) *out = s;
}

}  // namespace

int update_grid(long long N, int num_sms) {
  int per_sm = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, update_kernel<false>, kUpdateThreads, 0);
  if (per_sm < 1) per_sm = 1;
  const long long tiles = ((N + 3) / 4 + kUpdateThreads - 1) / kUpdateThreads;
  const long long g = (long long)per_sm * num_sms;
  return (int)(tiles < g ? tiles : g);
}

namespace {
template <int PREC>
const void* deliver_fn(bool rows) {
  return rows ? reinterpret_cast<const void*>(deliver_kernel<PREC, true>)
              : reinterpret_cast<const void*>(deliver_kernel<PREC, false>);
}
const void* deliver_fn(const StepParams& p, int precision) {
  const bool rows = p.rlist != nullptr;
  if (p.wide) return deliver_fn<kF16Wide>(rows);
  return precision == SNN_EXACT_F16W ? deliver_fn<SNN_EXACT_F16W>(rows) : deliver_fn<SNN_EXACT_F32W>(rows);
}
}  // namespace

cudaError_t launch_update(const StepParams& p, int grid, bool overlap, cudaStream_t st) {
  const void* fn = p.sg.on ? reinterpret_cast<const void*>(update_kernel<true>)
                           : reinterpret_cast<const void*>(update_kernel<false>);
  void* args[] = {const_cast<StepParams*>(&p)};
  return launch_overlapped(fn, dim3((unsigned)grid), kUpdateThreads, 0, args, overlap, st);
}

cudaError_t launch_ingest(const StepParams& p, const uint32_t* ids, long long n, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  const long long blocks = (n + 255) / 256;
  ingest_kernel<<<(unsigned)(blocks < 1024 ? blocks : 1024), 256, 0, st>>>(p, ids, n);
  return cudaGetLastError();
}

size_t deliver_smem(int cols, int npc4, bool batch) {
  const int warps = (batch ? kBatchThreads : kDeliverThreads) / 32;
  return ((size_t)cols * npc4 + (size_t)cols * 64 + (size_t)warps * kListWords) * 4;
}

// Delivery grid: one block per SM (a persistent grid).
int deliver_grid(const StepParams& p, int precision, int num_sms) {
  const size_t smem = deliver_smem(p.tcols, p.npc4, false);
  const void* fn = deliver_fn(p, precision);
  int per_sm = 0;
  // the attribute belongs to the kernel, not to the net: always the budget
  if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)std::max(smem, kSmemBudget)) != cudaSuccess)
    return 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kDeliverThreads, smem);
  return per_sm > 0 ? num_sms : 0;
}

cudaError_t launch_deliver(const StepParams& p, int precision, int grid, bool overlap, cudaStream_t st) {
  void* args[] = {const_cast<StepParams*>(&p)};
  return launch_overlapped(deliver_fn(p, precision), dim3((unsigned)grid), kDeliverThreads,
                           deliver_smem(p.tcols, p.npc4, false), args, overlap, st);
}

cudaError_t launch_drain_records(const StepParams& p, int nreg, uint32_t* stage_ids,
                                 uint32_t* stage_steps, unsigned long long* map_hdr, uint32_t* map_ids,
                                 uint32_t* map_steps, long long map_cap, cudaStream_t st) {
  drain_records_kernel<<<nreg, 256, 0, st>>>(p.rcnt, nreg, p.rec_region, p.rec, p.ctl,
                                             map_hdr, stage_ids, stage_steps, map_ids, map_steps,
                                             map_cap);
  return cudaGetLastError();
}

cudaError_t launch_count_records(const StepParams& p, int nreg, unsigned long long* map_hdr,
                                 cudaStream_t st) {
  count_records_kernel<<<1, 1024, 0, st>>>(p.rcnt, nreg, p.rec_region, p.ctl, map_hdr);
  return cudaGetLastError();
}

namespace {
template <int PREC, int INFL, bool ROWS>
void* batch_fn() {
  return reinterpret_cast<void*>(batch_kernel<PREC, INFL, ROWS>);
}
// The batch tuner's schedule `infl` (2 or 4) selects 1 or 2 rounds of
// sectors in flight per lane (always 1 for lists of rows and wide weights).
void* batch_kernel_ptr(int precision, int infl, bool rows, bool wide) {
  if (wide) return batch_fn<kF16Wide, 1, true>();
  if (rows) return precision == SNN_EXACT_F16W ? batch_fn<1, 1, true>() : batch_fn<0, 1, true>();
  if (precision == SNN_EXACT_F16W) return infl == 2 ? batch_fn<1, 1, false>() : batch_fn<1, 2, false>();
  return infl == 2 ? batch_fn<0, 1, false>() : batch_fn<0, 2, false>();
}
}  // namespace

static_assert(2 * (kBatchSmemBudget + kUpdateSubs * sizeof(StepParams) + sizeof(DeliverSmem) +
                   (kMaxBatch + 1) * sizeof(int) + 64 + 1024) <= 228 * 1024,
              "two blocks of the batch kernel fit an SM");

size_t batch_smem(int win_words, int max_cols) {
  return std::max(kUpdateSubs * sizeof(UpdateSmem),
                  ((size_t)win_words + (size_t)max_cols * 64 + (size_t)(kBatchThreads / 32) * kListWords) * 4);
}

int batch_grid(int precision, int infl, bool rows, bool wide, int num_sms, size_t smem) {
  void* fn = batch_kernel_ptr(precision, infl, rows, wide);
  if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)std::max(smem, kBatchSmemBudget)) != cudaSuccess)
    return 0;
  int per_sm = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kBatchThreads, smem);
  return per_sm * num_sms;
}

cudaError_t launch_batch(const BatchParams& b, int precision, int infl, bool rows, bool wide, int grid,
                         size_t smem, cudaStream_t st) {
  void* args[] = {const_cast<BatchParams*>(&b)};
  return cudaLaunchCooperativeKernel(batch_kernel_ptr(precision, infl, rows, wide), dim3(grid),
                                     dim3(kBatchThreads), args, smem, st);
}

cudaError_t launch_sum_parts(const unsigned long long* part, int n, unsigned long long* out,
                             cudaStream_t st) {
  sum_parts_kernel<<<1, 32, 0, st>>>(part, n, out);
  return cudaGetLastError();
}

}  // namespace snn
