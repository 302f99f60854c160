// snn_build.cu -- on-device construction of the delay-bucketed synapse table.
//
// Connectivity of arxiv 1511.09325, Sec. 2, as read by this library: synapse
// k of neuron j (column (x, y), index l_j in it) draws one Philox4x32-10 block
// (counter (j, k, CONN, 0)) = (x0, x1, x2, x3):
//   k <  k_local : target in the own column, l = u_{n-1}(x0), skipping l_j;
//   k >= k_local : stencil offset = first m with x1 < thr[m] (P ~ exp(-r/lambda)),
//                  target l = u_n(x0) in column ((x+dx) mod W, (y+dy) mod H);
//   delay d = d_min + u_ndel(x2);  weight = table[population][x3 >> 16].
// A delay bucket has two parts (see snn_internal.h): the synapses that end in
// the source's own delivery tile, stored as words of the tile's window, and
// the others, stored as a stencil offset and an index.
// One warp owns one row: a first pass counts the synapses of every bucket part, a
// second pass regenerates them and stores each into its part in k order (warp
// match + popc rank), then the parts' tails are padded.  Both run in one kernel,
// where the counting hides behind the stores (96x96: 126 ms, 178 ms as two
// kernels), with the rows' stride estimated; a row that is longer is reported and
// left out, and the build counts all rows first then, as it does where memory is
// short.  Rows are stored, and walked, in virtual column order.  The same walk reads rows back in the order in which they
// were drawn, and checks that the stored ends, records and padding are where the
// draws say.
// A shard (see ShardGeo) draws every synapse with the neuron's global index
// and keeps only those whose target column is one of its own (local and
// global stencil arithmetic agree for such targets: the halo is as wide as
// the stencil, or the local grid spans the whole global side).
#include <cuda_fp16.h>

#include "snn_device.cuh"
#include "snn_internal.h"

namespace snn {
namespace {

constexpr int kBuildWarps = 8;
constexpr int kDropped = 0xFE;  // offset class: not kept by the shard
constexpr int kOut = 0xFF;      // offset class: another tile
constexpr int kModeCount = 0, kModeFill = 1, kModeRead = 2, kModeOrder = 3;

// Shared tables of a block and its warps' rows.
struct RowSmem {
  unsigned cnt[kBuildWarps][64];       // synapses per bucket part (2 b, 2 b + 1)
  unsigned cur[kBuildWarps][64];       // next slot of each part
  unsigned rd[kBuildWarps][32];        // readback: next entry of each delay; draw
                                       // order: next place of each bucket
  uint32_t mask[kBuildWarps][64];      // draw order: bit p: place p is an in record
  uint8_t cls[kBuildWarps][kMaxOff + 1];  // target's place in the tile per offset
  uint32_t thr[kMaxOff];
  uint8_t guide[256];                  // offsets whose threshold is <= (b << 24)
  int8_t dx[kMaxOff + 1], dy[kMaxOff + 1];  // the last entry is (0, 0)
};

// The row a warp works on.
struct Row {
  long long j;        // its neuron (real, local index)
  uint32_t jj;        // the index its draws are keyed on
  int lj, cx, cy;
  int x0, y0, tw;     // first column and width of its tile
  size_t at;          // its place in syn and bend
};

template <bool PAPER>
__device__ __forceinline__ void load_offsets(const BuildParams& P, RowSmem& S) {
  const int n = PAPER ? P.n_poff : P.n_off;
  for (int m = threadIdx.x; m <= kMaxOff; m += blockDim.x) {
    S.dx[m] = m < n ? (PAPER ? P.poff_dx[m] : P.off_dx[m]) : (int8_t)0;
    S.dy[m] = m < n ? (PAPER ? P.poff_dy[m] : P.off_dy[m]) : (int8_t)0;
    if (m < kMaxOff) S.thr[m] = P.stencil_thr[m];
  }
  __syncthreads();
  for (int b = threadIdx.x; b < 256; b += blockDim.x) {
    int g = 0;
    while (g + 1 < P.n_off && S.thr[g] <= (uint32_t)b << 24) ++g;
    S.guide[b] = (uint8_t)g;
  }
  __syncthreads();
}

// Row of neuron l of column c, and the class of every stencil offset of it:
// the target column's place in the tile, kOut, or kDropped.
template <bool PAPER>
__device__ __forceinline__ Row open_row(const BuildParams& P, RowSmem& S, int c, int l) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  Row r;
  r.j = (long long)c * P.npc + l;
  r.lj = l;
  r.cy = c / P.W;
  r.cx = c - r.cy * P.W;
  int gx, gy;
  shard_global_col(P.sg, r.cx, r.cy, &gx, &gy);
  r.jj = P.sg.on ? ((uint32_t)gy * (uint32_t)P.sg.GW + (uint32_t)gx) * (uint32_t)P.npc + (uint32_t)l
                 : (uint32_t)r.j;
  r.x0 = r.cx / P.tw * P.tw;
  r.y0 = r.cy / P.th * P.th;
  r.tw = min(P.tw, P.W - r.x0);
  const int th = min(P.th, P.H - r.y0);
  r.at = (size_t)P.colv[c] * P.npc + l;
  const int n = PAPER ? P.n_poff : P.n_off;
  __syncwarp();
  for (int m = lane; m <= kMaxOff; m += 32) {
    const int dx = S.dx[m], dy = S.dy[m];
    const int ox = wrap(r.cx + dx, P.W) - r.x0, oy = wrap(r.cy + dy, P.H) - r.y0;
    int v = (unsigned)ox < (unsigned)r.tw && (unsigned)oy < (unsigned)th ? oy * r.tw + ox : kOut;
    if (P.sg.on && (m < n || m == kMaxOff) &&
        !shard_owns_global(P.sg, P.W, P.H, wrap(gx + dx, P.sg.GW), wrap(gy + dy, P.sg.GH)))
      v = kDropped;
    S.cls[w][m] = (uint8_t)v;
  }
  __syncwarp();
  return r;
}

// Stencil offset of word x: the first m with x < thr[m] (the last catches all).
__device__ __forceinline__ int offset_of(const BuildParams& P, const RowSmem& S, uint32_t x) {
  int m = S.guide[x >> 24];
  while (m + 1 < P.n_off && x >= S.thr[m]) ++m;
  return m;
}

// A bucket in draw order: its synapses, of both parts, from place 8 * first on,
// in 8-place units first .. end - 1 (the calling lane's bucket).
struct DrawBucket {
  unsigned first, end;
};
__device__ __forceinline__ DrawBucket draw_bucket(const BuildParams& P, unsigned ci, unsigned co) {
  const unsigned lane = threadIdx.x & 31u;
  const unsigned u = (ci + co + 7u) / 8u;
  unsigned incl = u;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned v = __shfl_up_sync(0xFFFFFFFFu, incl, o);
    if (lane >= (unsigned)o) incl += v;
  }
  return DrawBucket{incl - u, incl};
}

// Parts' sizes (S.cnt) to bucket ends and first slots; lane b holds bucket b.
// Returns the row's units.
template <int MODE>
__device__ __forceinline__ unsigned open_parts(const BuildParams& P, RowSmem& S, const Row& r) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned unit = (unsigned)P.unit;
  const unsigned ci = lane < P.ndel ? S.cnt[w][2 * lane] : 0u;
  const unsigned co = lane < P.ndel ? S.cnt[w][2 * lane + 1] : 0u;
  const unsigned ui = (ci + unit - 1u) / unit, uo = (co + unit - 1u) / unit;
  unsigned incl = ui + uo, icnt = ci + co;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned v = __shfl_up_sync(0xFFFFFFFFu, incl, o);
    const unsigned c = __shfl_up_sync(0xFFFFFFFFu, icnt, o);
    if (lane >= o) {
      incl += v;
      icnt += c;
    }
  }
  const unsigned excl = incl - ui - uo;
  S.cur[w][2 * lane] = excl * unit;
  S.cur[w][2 * lane + 1] = (excl + ui) * unit;
  const uint32_t row = (uint32_t)((r.cy - r.y0) * r.tw + (r.cx - r.x0)) * (uint32_t)P.npc + (uint32_t)r.lj;
  if (MODE == kModeRead) {
    S.rd[w][lane] = icnt - ci - co;
    // the stored descriptor says the same
    const uint8_t* d = P.bend + r.at * P.planes * 16;
    bool bad = lane < P.ndel && *reinterpret_cast<const uint16_t*>(d + desc_end(lane)) != (excl + ui | incl << 8);
    if (lane < P.ndel && lane % kPlaneBuckets == 0)
      bad = bad || *reinterpret_cast<const uint32_t*>(d + desc_start(lane) - 2) != (row | excl << 16);
    if (bad) atomicOr(P.rd_bad, 1u);
  } else if (MODE == kModeOrder) {
    const DrawBucket d = draw_bucket(P, ci, co);
    S.rd[w][lane] = 8u * d.first;
    S.mask[w][lane] = 0u;
    S.mask[w][lane + 32] = 0u;
    if (lane < P.ndel) P.ord_end[r.at * P.ndel + lane] = (uint8_t)d.end;
  } else {
    uint8_t* d = P.bend + r.at * P.planes * 16;
    if (lane < P.planes * kPlaneBuckets)
      *reinterpret_cast<uint16_t*>(d + desc_end(lane)) =
          (uint16_t)(min(excl + ui, 255u) | min(incl, 255u) << 8);
    if (lane < P.planes * kPlaneBuckets && lane % kPlaneBuckets == 0)
      *reinterpret_cast<uint32_t*>(d + desc_start(lane) - 2) = row | min(excl, 255u) << 16;
  }
  __syncwarp();
  return __shfl_sync(0xFFFFFFFFu, incl, 31);
}

// First slots of the parts from the stored bucket ends (S.cur; lane b: bucket b).
__device__ __forceinline__ void stored_parts(const BuildParams& P, RowSmem& S, const Row& r) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane < P.ndel) {
    const uint8_t* d = P.bend + r.at * P.planes * 16;
    const int at = lane % kPlaneBuckets ? desc_end(lane) - 1 : desc_start(lane);
    S.cur[w][2 * lane] = (unsigned)d[at] * (unsigned)P.unit;
    S.cur[w][2 * lane + 1] = (unsigned)d[desc_end(lane)] * (unsigned)P.unit;
  }
  __syncwarp();
}

// Whether a stored record is padding.
template <int PREC>
__device__ __forceinline__ bool is_pad(const BuildParams& P, size_t s, bool out) {
  if (PREC != SNN_EXACT_F16W) return static_cast<const uint2*>(P.syn)[s].x & kPad;
  const uint32_t rec = static_cast<const uint32_t*>(P.syn)[s];
  return out ? (rec & 0x3800u) == kPadF16 : (rec >> 16 & 0x7FFFu) == kPadHalf;
}

// Readback: the slots behind a part's last synapse must be padding.
template <int PREC>
__device__ __forceinline__ void check_pads(const BuildParams& P, RowSmem& S, const Row& r) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned unit = (unsigned)P.unit;
  bool bad = false;
  for (int part = 0; lane < P.ndel && part < 2; ++part) {
    const unsigned at = S.cur[w][2 * lane + part];
    const unsigned end = (at + unit - 1u) / unit * unit;
    for (unsigned s = at; s < end; ++s) bad = bad || !is_pad<PREC>(P, r.at * (size_t)P.rowcap + s, part == 1);
  }
  if (bad) atomicOr(P.rd_bad, 1u);
  __syncwarp();
}

// Places (or reads back) one synapse per lane: part bb = 2 bucket + (0 in,
// 1 out) or 64 for none.
template <int PREC, int MODE>
__device__ __forceinline__ void place(const BuildParams& P, RowSmem& S, const Row& r, int bb, int m,
                                      uint32_t l, uint32_t wbits, long long out0) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  const bool valid = bb < 64;
  const unsigned peers = __match_any_sync(0xFFFFFFFFu, bb);
  const unsigned rank = __popc(peers & lt);
  const unsigned pos = S.cur[w][bb & 63] + rank;
  unsigned dpeers = 0u, dpos = 0u;
  if (MODE == kModeRead || MODE == kModeOrder) {
    dpeers = __match_any_sync(0xFFFFFFFFu, bb >> 1);
    dpos = S.rd[w][(bb >> 1) & 31] + __popc(dpeers & lt);
  }
  __syncwarp();
  if (valid) {
    const size_t s = r.at * (size_t)P.rowcap + pos;
    const bool out = bb & 1;
    if (MODE == kModeFill) {
      const uint32_t code = out ? (uint32_t)((S.dy[m] + 3) << 3 | (S.dx[m] + 3)) << 11 | l
                                : (uint32_t)S.cls[w][m] * (uint32_t)P.npc4 + l;
      if (PREC == SNN_EXACT_F16W) {
        const uint32_t mag = wbits & 0x7FFFu;
        const uint32_t half = (mag == kPadHalf ? 0u : mag) | (r.lj < P.nexc ? 0u : 0x8000u);
        static_cast<uint32_t*>(P.syn)[s] = out ? mag << 17 | code : half << 16 | code;
      } else {
        // the FP32 weight, delivered as round(w * 2^16) in the input's units
        const int32_t wfx = __float2int_rn(__fmul_rn(__uint_as_float(wbits), 65536.0f));
        static_cast<uint2*>(P.syn)[s] = make_uint2(code, (uint32_t)wfx);
      }
    } else if (MODE == kModeOrder) {
      if (!out) atomicOr(&S.mask[w][dpos >> 5 & 63u], 1u << (dpos & 31u));
    } else {
      uint32_t code;
      int32_t wfx;
      if (is_pad<PREC>(P, s, out)) atomicOr(P.rd_bad, 1u);
      if (PREC == SNN_EXACT_F16W) {
        const uint32_t rec = static_cast<const uint32_t*>(P.syn)[s];
        code = out ? rec & 0x1FFFFu : rec & 0xFFFFu;
        const uint32_t mag = out ? rec >> 17 : rec >> 16 & 0x7FFFu;
        const float f = __half2float(__ushort_as_half((unsigned short)mag));
        wfx = __float2int_rn(__fmul_rn(r.lj < P.nexc ? f : -f, 65536.0f));
      } else {
        const uint2 rec = static_cast<const uint2*>(P.syn)[s];
        code = rec.x;
        wfx = (int32_t)rec.y;
      }
      int tx, ty;
      uint32_t tl;
      if (out) {
        tx = wrap(r.cx + (int)(code >> 11 & 7u) - 3, P.W);
        ty = wrap(r.cy + (int)(code >> 14 & 7u) - 3, P.H);
        tl = code & 2047u;
      } else {
        const int k = (int)(code / (uint32_t)P.npc4);
        ty = r.y0 + k / r.tw;
        tx = r.x0 + k % r.tw;
        tl = code - (uint32_t)k * (uint32_t)P.npc4;
      }
      const long long o = out0 + dpos;
      P.rd_target[o] = ((long long)ty * P.W + tx) * P.npc + tl;
      P.rd_delay[o] = P.dmin + (bb >> 1);
      P.rd_wfx[o] = wfx;
    }
    if (rank == 0) S.cur[w][bb] += __popc(peers);
    if ((MODE == kModeRead || MODE == kModeOrder) && (dpeers & lt) == 0u)
      S.rd[w][bb >> 1] += __popc(dpeers);
  }
  __syncwarp();
}

// Pads every part of the row up to its end (lane b: bucket b).  An in pad
// names the source's own word, so that pads of different rows fall on
// different words.
template <int PREC>
__device__ __forceinline__ void pad_parts(const BuildParams& P, RowSmem& S, const Row& r) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t own = (uint32_t)((r.cy - r.y0) * r.tw + (r.cx - r.x0)) * (uint32_t)P.npc4 + (uint32_t)r.lj;
  if (lane < P.ndel) {
    const unsigned unit = (unsigned)P.unit;
    for (int part = 0; part < 2; ++part) {
      const unsigned at = S.cur[w][2 * lane + part];
      const unsigned end = (at + unit - 1u) / unit * unit;
      for (unsigned s = at; s < end; ++s) {
        const size_t o = r.at * (size_t)P.rowcap + s;
        if (PREC == SNN_EXACT_F16W)
          static_cast<uint32_t*>(P.syn)[o] = part ? kPadF16 : kPadHalf << 16 | own;
        else
          static_cast<uint2*>(P.syn)[o] = make_uint2(part ? kPad : kPad | own, 0u);
      }
    }
  }
  __syncwarp();
}

// Writes the row's draw order: a word per unit of 8 places in draw order, bits
// 0-7: which places hold in records, bits 8-19 and 20-31: the slots of the
// first in and out records at or after the unit's start.
__device__ __forceinline__ void write_order(const BuildParams& P, RowSmem& S, const Row& r) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned unit = (unsigned)P.unit;
  const unsigned ci = lane < P.ndel ? S.cnt[w][2 * lane] : 0u;
  const unsigned co = lane < P.ndel ? S.cnt[w][2 * lane + 1] : 0u;
  const DrawBucket d = draw_bucket(P, ci, co);
  // lane b: bucket b's in records before it in the row, and its parts' first units
  const unsigned ui = (ci + unit - 1u) / unit, uo = (co + unit - 1u) / unit;
  unsigned uincl = ui + uo, cincl = ci;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned u = __shfl_up_sync(0xFFFFFFFFu, uincl, o);
    const unsigned c = __shfl_up_sync(0xFFFFFFFFu, cincl, o);
    if (lane >= o) {
      uincl += u;
      cincl += c;
    }
  }
  const unsigned in0 = (uincl - ui - uo) * unit, out0 = (uincl - uo) * unit;
  const unsigned units = __shfl_sync(0xFFFFFFFFu, d.end, 31);
  unsigned before = 0u;  // in records of the units before
  for (unsigned u0 = 0u; u0 < units; u0 += 32u) {
    const unsigned u = u0 + (unsigned)lane;
    const uint32_t m = u < units ? S.mask[w][u >> 2 & 63u] >> (8u * (u & 3u)) & 0xFFu : 0u;
    unsigned incl = (unsigned)__popc(m);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned v = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if (lane >= o) incl += v;
    }
    // the unit's bucket: the first with end > u
    int b = 0;
#pragma unroll
    for (int step = 16; step > 0; step >>= 1) {
      const unsigned e = __shfl_sync(0xFFFFFFFFu, d.end, b + step - 1);
      if (e <= u) b += step;
    }
    b = min(b, 31);
    const unsigned n_in = before + incl - (unsigned)__popc(m) -
                          __shfl_sync(0xFFFFFFFFu, cincl - ci, b);  // of the bucket, before u
    const unsigned f = __shfl_sync(0xFFFFFFFFu, d.first, b);
    const unsigned i0 = __shfl_sync(0xFFFFFFFFu, in0, b), o0 = __shfl_sync(0xFFFFFFFFu, out0, b);
    if (u < units && u < (unsigned)P.ord_units)
      P.ord[r.at * (size_t)P.ord_units + u] = m | (i0 + n_in) << 8 | (o0 + 8u * (u - f) - n_in) << 20;
    before += __shfl_sync(0xFFFFFFFFu, incl, 31);
  }
  __syncwarp();
}

// Rows of the fixed law, one warp per row; MODE fill builds them (max_units[0]: the
// longest row beyond the stride, else untouched), read writes rows j0 .. j0 +
// n_rows - 1 to the rd_* arrays, count finds the longest, order writes the rows'
// draw order.
template <int PREC, int MODE>
__global__ void __launch_bounds__(kBuildWarps * 32) build_rows_kernel(const BuildParams P) {
  __shared__ RowSmem S;
  load_offsets<false>(P, S);
  const int w = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const long long nwarps = (long long)gridDim.x * kBuildWarps;
  const uint32_t ndel = (uint32_t)P.ndel;
  const long long rows = MODE == kModeRead ? P.n_rows : P.N;

  for (long long i = (long long)blockIdx.x * kBuildWarps + w; i < rows; i += nwarps) {
    const uint32_t j = (uint32_t)(MODE == kModeRead ? P.j0 + i : i);
    const int c = (int)(j / (uint32_t)P.npc);
    const Row r = open_row<false>(P, S, c, (int)(j - (uint32_t)c * (uint32_t)P.npc));
    S.cnt[w][lane] = 0u;
    S.cnt[w][lane + 32] = 0u;
    __syncwarp();
    // pass 1: synapses per bucket part
    unsigned nkept = 0u;
    for (int k = lane; k < P.K; k += 32) {
      const uint4 x = philox4x32_10(make_uint4(r.jj, (uint32_t)k, kTagConn, 0u), P.seed_lo, P.seed_hi);
      const int cl = S.cls[w][k < P.k_local ? kMaxOff : offset_of(P, S, x.y)];
      if (cl != kDropped) {
        atomicAdd(&S.cnt[w][2 * below(x.z, ndel) + (cl == kOut ? 1 : 0)], 1u);
        ++nkept;
      }
    }
    if (MODE == kModeFill && P.deg != nullptr) {
      nkept = __reduce_add_sync(0xFFFFFFFFu, nkept);
      if (lane == 0) P.deg[j] = nkept;
    }
    __syncwarp();
    const unsigned units = open_parts<MODE>(P, S, r);
    if (MODE == kModeCount || (MODE == kModeFill && (int)units * P.unit > P.rowcap)) {
      if (lane == 0) atomicMax(P.max_units, units);
      continue;
    }

    const uint32_t* wt = P.wtab + (r.lj < P.nexc ? 0 : 65536);
    const long long out0 = MODE == kModeRead ? P.rd_off[i] : 0;
    // pass 2: regenerate and place every synapse
    for (int k0 = 0; k0 < P.K; k0 += 32) {
      const int k = k0 + lane;
      const uint4 x = philox4x32_10(make_uint4(r.jj, (uint32_t)k, kTagConn, 0u), P.seed_lo, P.seed_hi);
      int m = kMaxOff;
      uint32_t l;
      if (k < P.k_local) {
        l = below(x.x, (uint32_t)(P.npc - 1));
        l += (l >= (uint32_t)r.lj) ? 1u : 0u;
      } else {
        m = offset_of(P, S, x.y);
        l = below(x.x, (uint32_t)P.npc);
      }
      const int cl = S.cls[w][m];
      const int bb = k < P.K && cl != kDropped ? 2 * (int)below(x.z, ndel) + (cl == kOut ? 1 : 0) : 64;
      place<PREC, MODE>(P, S, r, bb, m, l, MODE == kModeFill ? wt[x.w >> 16] : 0u, out0);
    }
    if (MODE == kModeFill) pad_parts<PREC>(P, S, r);
    if (MODE == kModeRead) check_pads<PREC>(P, S, r);
    if (MODE == kModeOrder) write_order(P, S, r);
  }
}

// Initial state: V_i uniform in [0, theta) at 24-bit resolution from word
// i mod 4 of Philox(i / 4, 0, INIT); calcium and refractoriness zero.
// A shard draws with the global index i (n_per_col is a multiple of 4 there,
// so a quad of local neurons is a quad of global ones).
__global__ void __launch_bounds__(256) init_state_kernel(const StepParams P) {
  const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long i0 = q * 4;
  if (i0 >= P.N) return;
  uint32_t gq = (uint32_t)q;
  if (P.sg.on) {
    const int col = (int)((uint32_t)i0 / (uint32_t)P.npc);
    const int l = (int)((uint32_t)i0 - (uint32_t)col * (uint32_t)P.npc);
    const int cy = col / P.W;
    int gx, gy;
    shard_global_col(P.sg, col - cy * P.W, cy, &gx, &gy);
    gq = (((uint32_t)gy * (uint32_t)P.sg.GW + (uint32_t)gx) * (uint32_t)P.npc + (uint32_t)l) >> 2;
  }
  const uint4 u = philox4x32_10(make_uint4(gq, 0u, kTagInit, 0u), P.seed_lo, P.seed_hi);
  const float s = 5.9604644775390625e-08f;  // 2^-24
  float4 v;
  v.x = __fmul_rn(P.theta, __fmul_rn(__uint2float_rn(u.x >> 8), s));
  v.y = __fmul_rn(P.theta, __fmul_rn(__uint2float_rn(u.y >> 8), s));
  v.z = __fmul_rn(P.theta, __fmul_rn(__uint2float_rn(u.z >> 8), s));
  v.w = __fmul_rn(P.theta, __fmul_rn(__uint2float_rn(u.w >> 8), s));
  reinterpret_cast<float4*>(P.V)[q] = v;
  reinterpret_cast<float4*>(P.C)[q] = make_float4(0.f, 0.f, 0.f, 0.f);
  reinterpret_cast<uchar4*>(P.R)[q] = make_uchar4(0, 0, 0, 0);
}

// Paper connectivity law (Sec. 2): candidate c of neuron j -- the column's
// other neurons in ascending order, then the n_per_col neurons of each kept
// remote offset -- is kept iff word c mod 4 of Philox(j, c / 4, PCONN) is
// below its threshold.  The k-th kept candidate is synapse k, whose delay and
// weight come from Philox(j, k, CONN) as under the fixed law.  One warp per
// row; in pass it, lane e takes candidates 128 it + 4 e .. + 3, so a warp
// scan of the lanes' kept counts ranks them.  The count pass writes the
// bucket ends, the out-degree and the largest row; the fill pass makes the
// same draws and places every synapse, then pads the parts; the read pass
// counts and then reads back, and the order pass likewise.
template <int PREC, int MODE>
__global__ void __launch_bounds__(kBuildWarps * 32) paper_rows_kernel(const BuildParams P) {
  __shared__ RowSmem S;
  __shared__ unsigned long long s_pthr[kMaxOff];
  for (int m = threadIdx.x; m < kMaxOff; m += blockDim.x) s_pthr[m] = m < P.n_poff ? P.poff_thr[m] : 0ull;
  load_offsets<true>(P, S);
  const int w = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const long long nwarps = (long long)gridDim.x * kBuildWarps;
  const uint32_t ndel = (uint32_t)P.ndel;
  const long long rows = MODE == kModeRead ? P.n_rows : P.N;

  for (long long i = (long long)blockIdx.x * kBuildWarps + w; i < rows; i += nwarps) {
    const uint32_t j = (uint32_t)(MODE == kModeRead ? P.j0 + i : i);
    const int col = (int)(j / (uint32_t)P.npc);
    const Row r = open_row<true>(P, S, col, (int)(j - (uint32_t)col * (uint32_t)P.npc));
    const uint32_t* wt = P.wtab + (r.lj < P.nexc ? 0 : 65536);
    const long long out0 = MODE == kModeRead ? P.rd_off[i] : 0;
    S.cnt[w][lane] = 0u;
    S.cnt[w][lane + 32] = 0u;
    if (MODE == kModeFill) stored_parts(P, S, r);
    __syncwarp();
    // one walk over the candidates; `placing`: place them, else count them
    auto walk = [&](bool placing) -> unsigned {
      unsigned k_run = 0u;
      for (long long c0 = 0; c0 < P.n_cand; c0 += 128) {
        const long long cb = c0 + 4 * lane;
        const uint4 x = philox4x32_10(make_uint4(r.jj, (uint32_t)(cb >> 2), kTagPConn, 0u), P.seed_lo,
                                      P.seed_hi);
        const uint32_t words[4] = {x.x, x.y, x.z, x.w};
        unsigned bits = 0u;
        int lq[4], mq[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const long long c = cb + q;
          lq[q] = 0;
          mq[q] = kMaxOff;
          if (c >= P.n_cand) continue;
          unsigned long long thr;
          if (c < P.npc - 1) {
            thr = P.plocal_thr;
            lq[q] = (int)c + ((int)c >= r.lj ? 1 : 0);
          } else {
            const long long rr = c - (P.npc - 1);
            const int m = (int)((uint32_t)rr / (uint32_t)P.npc);
            thr = s_pthr[m];
            mq[q] = m;
            lq[q] = (int)(rr - (long long)m * P.npc);
          }
          if ((unsigned long long)words[q] < thr) bits |= 1u << q;
        }
        const unsigned nb = (unsigned)__popc(bits);
        unsigned incl = nb;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const unsigned v = __shfl_up_sync(0xFFFFFFFFu, incl, o);
          if (lane >= o) incl += v;
        }
        const unsigned kb = k_run + incl - nb;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          int bb = 64;
          uint32_t wbits = 0u;
          if ((bits >> q) & 1u) {
            const unsigned k = kb + (unsigned)__popc(bits & ((1u << q) - 1u));
            const uint4 y = philox4x32_10(make_uint4(r.jj, k, kTagConn, 0u), P.seed_lo, P.seed_hi);
            bb = 2 * (int)below(y.z, ndel) + (S.cls[w][mq[q]] == kOut ? 1 : 0);
            if (MODE == kModeFill) wbits = wt[y.w >> 16];
          }
          if (!placing) {
            if (bb < 64) atomicAdd(&S.cnt[w][bb], 1u);
          } else {
            place<PREC, MODE>(P, S, r, bb, mq[q], (uint32_t)lq[q], wbits, out0);
          }
        }
        k_run += __shfl_sync(0xFFFFFFFFu, incl, 31);
      }
      __syncwarp();
      return k_run;
    };
    if (MODE != kModeFill) {
      const unsigned deg = walk(false);
      const unsigned units = open_parts<MODE>(P, S, r);
      if (MODE == kModeCount) {
        unsigned u8 = lane < P.ndel ? (S.cnt[w][2 * lane] + S.cnt[w][2 * lane + 1] + 7u) / 8u : 0u;
        u8 = __reduce_add_sync(0xFFFFFFFFu, u8);
        if (lane == 0) {
          atomicMax(P.max_units, units);
          atomicMax(P.max_units + 1, u8);
          P.deg[j] = deg;
        }
      }
    }
    if (MODE != kModeCount) walk(true);
    if (MODE == kModeFill) pad_parts<PREC>(P, S, r);
    if (MODE == kModeRead) check_pads<PREC>(P, S, r);
    if (MODE == kModeOrder) write_order(P, S, r);
  }
}

// Geometry tables, one thread per column and stencil offset (offset fields of 7
// name no column).
__global__ void __launch_bounds__(256) geometry_kernel(int W, int H, int tw, int th, int npc4, uint32_t* ctile,
                                                       uint32_t* colv, uint2* tinfo, uint32_t* nbg) {
  const long long n = (long long)W * H * 64;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(i >> 6), off = (int)(i & 63);
    const int y = c / W, x = c - y * W;
    const TilePlace p = tile_place(W, H, tw, th, x, y);
    const int dx = (off & 7) - 3, dy = (off >> 3) - 3;
    nbg[(size_t)p.v * 64 + off] =
        dx > 3 || dy > 3 ? 0u
                         : tile_place(W, H, tw, th, wrap(x + dx, W), wrap(y + dy, H)).v * (uint32_t)npc4;
    if (off) continue;
    ctile[c] = p.tile << 6 | p.k;
    colv[c] = p.v;
    if (p.k == 0u) tinfo[p.tile] = make_uint2(p.v, (unsigned)(p.w * p.h));
  }
}

}  // namespace

cudaError_t launch_geometry(int W, int H, int tw, int th, int npc4, uint32_t* ctile, uint32_t* colv,
                            uint2* tinfo, uint32_t* nbg, cudaStream_t st) {
  const long long blocks = ((long long)W * H * 64 + 255) / 256;
  geometry_kernel<<<(unsigned)(blocks < 65536 ? blocks : 65536), 256, 0, st>>>(W, H, tw, th, npc4, ctile, colv,
                                                                               tinfo, nbg);
  return cudaGetLastError();
}

cudaError_t launch_build_count(const BuildParams& bp, int num_sms, cudaStream_t st) {
  build_rows_kernel<SNN_EXACT_F32W, kModeCount><<<num_sms * 8, kBuildWarps * 32, 0, st>>>(bp);
  return cudaGetLastError();
}

cudaError_t launch_paper_count(const BuildParams& bp, int num_sms, cudaStream_t st) {
  paper_rows_kernel<SNN_EXACT_F32W, kModeCount><<<num_sms * 8, kBuildWarps * 32, 0, st>>>(bp);
  return cudaGetLastError();
}

cudaError_t launch_paper_fill(const BuildParams& bp, int precision, int num_sms,
                              cudaStream_t st) {
  if (precision == SNN_EXACT_F16W)
    paper_rows_kernel<SNN_EXACT_F16W, kModeFill><<<num_sms * 8, kBuildWarps * 32, 0, st>>>(bp);
  else
    paper_rows_kernel<SNN_EXACT_F32W, kModeFill><<<num_sms * 8, kBuildWarps * 32, 0, st>>>(bp);
  return cudaGetLastError();
}

cudaError_t launch_build(const BuildParams& bp, int precision, int num_sms,
                         cudaStream_t st) {
  const int grid = num_sms * 8;
  if (precision == SNN_EXACT_F16W)
    build_rows_kernel<SNN_EXACT_F16W, kModeFill><<<grid, kBuildWarps * 32, 0, st>>>(bp);
  else
    build_rows_kernel<SNN_EXACT_F32W, kModeFill><<<grid, kBuildWarps * 32, 0, st>>>(bp);
  return cudaGetLastError();
}

cudaError_t launch_read_rows(const BuildParams& bp, int precision, bool paper, cudaStream_t st) {
  const unsigned grid = (unsigned)((bp.n_rows + kBuildWarps - 1) / kBuildWarps);
  const bool f16 = precision == SNN_EXACT_F16W;
  if (paper && f16)
    paper_rows_kernel<SNN_EXACT_F16W, kModeRead><<<grid, kBuildWarps * 32, 0, st>>>(bp);
  else if (paper)
    paper_rows_kernel<SNN_EXACT_F32W, kModeRead><<<grid, kBuildWarps * 32, 0, st>>>(bp);
  else if (f16)
    build_rows_kernel<SNN_EXACT_F16W, kModeRead><<<grid, kBuildWarps * 32, 0, st>>>(bp);
  else
    build_rows_kernel<SNN_EXACT_F32W, kModeRead><<<grid, kBuildWarps * 32, 0, st>>>(bp);
  return cudaGetLastError();
}

cudaError_t launch_draw_order(const BuildParams& bp, bool paper, int num_sms, cudaStream_t st) {
  if (paper)
    paper_rows_kernel<SNN_EXACT_F32W, kModeOrder><<<num_sms * 8, kBuildWarps * 32, 0, st>>>(bp);
  else
    build_rows_kernel<SNN_EXACT_F32W, kModeOrder><<<num_sms * 8, kBuildWarps * 32, 0, st>>>(bp);
  return cudaGetLastError();
}

cudaError_t launch_init_state(const StepParams& p, cudaStream_t st) {
  const long long quads = (p.N + 3) / 4;
  const unsigned grid = (unsigned)((quads + 255) / 256);
  init_state_kernel<<<grid, 256, 0, st>>>(p);
  return cudaGetLastError();
}

}  // namespace snn
