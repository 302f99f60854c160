// snn_internal.h -- types shared by the translation units of the library.
//
// Device data layout of one net (all arrays are library-owned, 256 B aligned).
// The grid is covered by delivery tiles of tw x th columns; a column's
// virtual index v counts the columns tile by tile (tiles in row-major order,
// row-major inside a tile), so the columns of a tile are consecutive and the
// k-th column of a tile is v = first + k.
//   syn    outgoing-synapse table.  Row of neuron l of virtual column v at
//          (v * npc + l) * rowcap slots.  A row holds the neuron's synapses
//          grouped by delay bucket b = d - d_min; a bucket holds the synapses
//          that end in the source's own tile ("in"), then the others ("out"),
//          each part padded to whole units of 8 slots (16 where a row would
//          exceed 255 units of 8).
//            in, F16W:  u32 = half(16, signed) << 16 | code(16)
//            in, F32W:  { code, int32 round(w * 2^16) }
//              code = k * npc4 + l: word of the target in its tile's window
//              (k the target column's place in the tile)
//            out, F16W: u32 = half_magnitude(15) << 17 | off(6) << 11 | l(11)
//            out, F32W: { off << 11 | l, int32 round(w * 2^16) }
//              off = (dy + 3) << 3 | (dx + 3): stencil offset of the target
//              column; F16W: the sign is the source population's (Dale)
//          padding records deliver 0 (kPadHalf / kPadF16 / kPad).
//   bend   [ncol * npc][planes] of 16 bytes, rows in the order of syn: a
//          spiker's descriptor.  Plane p covers buckets 6p .. 6p + 5: bytes 0-1
//          the neuron's row in its tile (k * npc + l), byte 2 the start of
//          bucket 6p, bytes 4 + 2i and 5 + 2i the ends of the in and out parts
//          of bucket 6p + i, in units.
//   V, C   float[Npad] membrane potential (mV) and calcium.
//   R      u8[Npad] remaining refractory steps.
//   acc    int32[ncol * npc4] recurrent input of the next step, 2^-16 mV
//          units; neuron l of virtual column v at v * npc4 + l (npc4 = npc
//          rounded up to 4), so a tile's input is one run of words.
//   list   [d_max + 1][planes][ntile][tcap] of 16 bytes: descriptors of the
//          spikes of the last d_max + 1 steps (slot t % (d_max + 1)) per tile,
//          in no fixed order; ccnt[slot][tile] of them (one counter per 32
//          bytes).  The items of a bucket read one plane of one list in order.
//   rlist  u16[d_max + 1][ntile][tcap]: the spikers' rows in their tiles, in
//          place of `list` where the device has no room for it.
//   isum   u32[ntile] (bucket, spiker) items of each tile over the steps that
//          the delivery of step t reads, less step t itself (one counter per 32
//          bytes); gsum: their sum.
//   ctile  u32[ncol] tile << 6 | k of each real column; colv: its virtual index.
//   tinfo  {first virtual column, columns} of each tile.
//   nbg    u32[ncol][64] first word in acc of the column at each stencil offset
//          of each virtual column.
//   cnt    u32 spikes of the step (compact-list form only).
//   ctl    control block (step counters, overflow flag, status).
//   rec    u64 spike records (step << 32 | id), one region per update block,
//          rcnt[b] records in region b since the last drain.
//   colcnt u64[ncol][2] spike counts per column and population.
//   ext_part, spk_part  u64[update grid] external events and spikes counted
//          by each update block.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "snn.h"

namespace snn {

constexpr uint32_t kTagConn = 1u;  // Philox counter word 2 of each stream
constexpr uint32_t kTagExt = 2u;
constexpr uint32_t kTagInit = 3u;
constexpr uint32_t kTagSurr = 4u;  // normal draws of the differentiable form
constexpr uint32_t kTagPConn = 5u; // candidate draws of the paper connectivity law
constexpr int kMaxDelays = 32;   // d_max <= 32
constexpr int kPlaneBuckets = 6; // buckets that a 16-byte plane of a descriptor covers
constexpr int kSlotUnit = 8;     // bucket parts are padded to 8 (or 16) synapse slots
constexpr int kMaxPoisThr = 127; // Poisson thresholds below 2^32
constexpr int kMaxOff = 48;      // remote stencil offsets (radius <= 3)
// Padding records.  F32W: bit 31 of the code set, weight 0.  F16W: an in
// record of the half 2^-24, which rounds to 0 input units (a synapse of that
// weight is stored as the half 0 instead), or an out record of weight 0 and
// stencil field dx + 3 = 7, which no synapse uses (|dx| <= 3).
constexpr uint32_t kPad = 0x80000000u;
constexpr uint32_t kPadHalf = 1u;
constexpr uint32_t kPadF16 = 7u << 11;
constexpr int kMaxGridSide = 16383;     // columns per grid side (14-bit coordinates)
constexpr int kMaxTile = 8;             // delivery tile side, columns
constexpr int kMaxTileCols = kMaxTile * kMaxTile;
constexpr int kCntStride = 8;           // words from one tile counter to the next
// Dynamic shared memory of a delivery block: of a net of its own (one block per
// SM) and of the batch kernel (two per SM, with their static part and the 1 KB
// that the system keeps of each block in the SM's 228 KB: with 110 KB, tiles of
// more than 111 376 bytes left one block per SM); the window alone takes at most
// kWindowBudget.
constexpr size_t kSmemBudget = 224 * 1024;
constexpr size_t kBatchSmemBudget = 108 * 1024;
constexpr size_t kWindowBudget = 196 * 1024;
// Words of a tile's window per item of the fewest that make a part use the
// window, and per item of its fixed cost in the range split (set-up and
// flush); the fixed cost, in items, of a tile with fewer but some items.
// Without a window each of an item's ~62 synapses is an L2 reduction (about
// 1.3 per ns and SM), with one the window's words are cleared and added once
// (about 7.5 words per ns and SM).  Measured (us per delivery over 1000 steps from
// step 600 on: 8x8 FP16, 24x24 FP16, 24x24 FP32, 96x96 FP16): a window from 1 item
// per 87 words on 15.9, 37.5, 42.4, 417; 175: 15.4, 33.9, 39.8, 416; 250: 15.2,
// 33.6, 39.5, 417; 350: 15.1, 33.6, 39.5, 417.  A cost of 1 item per 30 words 15.5,
// 34.4, 40.5, 422; 44: 15.3, 33.8, 39.9, 417; 60: 15.2, 33.6, 39.5, 417; 88: 15.0,
// 33.5, 39.2, 417.
constexpr int kWinWordsPerItem = 250;
constexpr int kCostWordsPerItem = 60;
constexpr unsigned kCostPart = 32;

// Tables computed on the host in FP64 and rounded once.
struct HostTables {
  int n_off = 0;
  int8_t off_dx[kMaxOff] = {}, off_dy[kMaxOff] = {};
  uint32_t stencil_thr[kMaxOff] = {};  // first n_off - 1 used; last is 2^32
  int n_pois_thr = 0;                  // thresholds below 2^32
  uint32_t pois_thr[kMaxPoisThr + 1] = {};
  uint8_t pois_guide[256] = {};        // #thresholds <= (b << 24)
  std::vector<uint32_t> wtab;          // [2][65536] stored weight bits
  float pvv = 0, pcc = 0, pvc[2] = {0, 0};
  int32_t jx = 0;
  int nref = 0;
  int k_local = 0;
  // paper connectivity law (SNN_CONN_PAPER)
  int n_poff = 0;
  int8_t poff_dx[kMaxOff] = {}, poff_dy[kMaxOff] = {};
  unsigned long long poff_thr[kMaxOff] = {};  // candidate kept iff word < thr
  unsigned long long plocal_thr = 0;
  long long n_cand = 0;                        // candidates per neuron
};

int make_host_tables(const snn_neuron_params& np, const snn_synapse_params& sp,
                     int precision, HostTables* out, std::string* err);
// The neuron-update part only: Poisson table, propagators, J_ext, refractory.
int make_neuron_tables(const snn_neuron_params& np, HostTables* out, std::string* err);
// Standard-normal quantiles at (m + 0.5) / 65536, m < 65536 (computed once).
const std::vector<double>& quantile_table();

// Device control block.
struct Ctl {
  long long t;                  // step index of the next update (set by the delivery)
  long long td;                 // step index of the next delivery (set by the update)
  unsigned int drained;         // blocks done with the current record drain
  unsigned int rec_overflow;    // set when a record did not fit its region
  unsigned int status;          // nonzero: a delivery found inconsistent counts
};

// Status codes a kernel leaves in Ctl::status (and the mapped host word).
constexpr unsigned kStatusCounts = 1u;  // item counts disagree with the spike lists
constexpr unsigned kStatusIngest = 2u;  // a shard received an index it cannot list

// A shard: a net over a local grid E of W x H columns (its own columns and a
// halo of stencil_radius columns around them, clipped to the global grid)
// whose local column (lx, ly) is global column ((ex0 + lx) mod GW,
// (ey0 + ly) mod GH).  Only the columns of T = [tx0, tx0 + tw) x [ty0, ty0 +
// th) (local coordinates) are its own: it updates their neurons and keeps the
// synapses that end in them; the halo's spikes arrive from other shards.
// Random draws and spike records use global neuron indices.  A whole network
// is the shard with on = 0 (E = T = the grid).
struct ShardGeo {
  int on;
  int GW, GH;
  int ex0, ey0;
  int tx0, ty0, tw, th;
};

// Global column of local column (lx, ly).
__host__ __device__ inline void shard_global_col(const ShardGeo& g, int lx, int ly, int* gx,
                                                 int* gy) {
  if (!g.on) {
    *gx = lx;
    *gy = ly;
    return;
  }
  *gx = (g.ex0 + lx) % g.GW;
  *gy = (g.ey0 + ly) % g.GH;
}

// Whether global column (gx, gy) is one of the shard's own columns.
__host__ __device__ inline bool shard_owns_global(const ShardGeo& g, int W, int H, int gx, int gy) {
  if (!g.on) return true;
  const int lx = ((gx - g.ex0) % g.GW + g.GW) % g.GW;
  const int ly = ((gy - g.ey0) % g.GH + g.GH) % g.GH;
  return lx < W && ly < H && lx >= g.tx0 && lx < g.tx0 + g.tw && ly >= g.ty0 && ly < g.ty0 + g.th;
}

// The delivery tile of column (x, y) of a W x H grid, its place in the tile and
// its virtual index: tiles of tw x th columns (narrower at the right and lower
// edges), row by row.
struct TilePlace {
  uint32_t tile, k, v;
  int w, h;  // the tile's size
};
__host__ __device__ inline TilePlace tile_place(int W, int H, int tw, int th, int x, int y) {
  const int tx = x / tw, ty = y / th, x0 = tx * tw, y0 = ty * th;
  TilePlace p;
  p.w = W - x0 < tw ? W - x0 : tw;
  p.h = H - y0 < th ? H - y0 : th;
  p.tile = (uint32_t)ty * (uint32_t)((W + tw - 1) / tw) + (uint32_t)tx;
  p.k = (uint32_t)((y - y0) * p.w + x - x0);
  p.v = (uint32_t)y0 * (uint32_t)W + (uint32_t)(x0 * p.h) + p.k;
  return p;
}

// Everything a step kernel needs, passed by value (constant bank).
struct StepParams {
  long long N;
  int npc, npc4, nexc, W, H, K, dmin, ndel, nslot;
  int ncol, ntile;
  int tcap;                // list entries per slot and tile
  int tcols;               // columns of the largest tile
  int planes;              // 16-byte planes of a spike descriptor
  int row_sec, unit_sec;   // 32-byte sectors of a row and of a bucket unit
  int wide;                // F16W: some weight is 64 mV or more
  unsigned min_items;      // fewest items a delivery block takes (fewer blocks run)
  unsigned win_items;      // fewest items of a part that uses the window (2^32 - 1: none does)
  unsigned cost_win;       // fixed cost (in items) of a tile with a window
  uint32_t npc_m;          // floor(2^32 / n_per_col) (capped)
  uint32_t seed_lo, seed_hi;
  uint32_t key[20];        // the seed's Philox keys of the ten rounds
  float theta, vr, dc, pvv, pcc, pvc_e, pvc_i;
  int32_t jx;
  int nref;
  int n_pois_thr;
  uint32_t pois_thr[kMaxPoisThr + 1];
  uint8_t pois_guide[256];
  float* V;
  float* C;
  uint8_t* R;
  int32_t* acc;
  uint32_t* ids;   // compact spike-id list (noalloc form only)
  uint4* list;     // spike lists per slot, plane and tile (with ccnt)
  uint16_t* rlist; // lists of rows instead (list is null then)
  const uint32_t* ctile;
  const uint32_t* colv;   // null: acc is indexed by the real neuron index
  const uint2* tinfo;
  const uint32_t* nbg;
  unsigned* hstatus;  // mapped host copy of Ctl::status (may be null)
  unsigned* cnt;
  unsigned* ccnt;  // list lengths per slot and tile; null: one compact list
  unsigned* isum;  // items per tile of the delivery window (with ccnt)
  unsigned* gsum;  // their sum
  unsigned* icnt;  // shard: halo spikes of each column listed this step
  const uint4* bend;
  const void* syn;
  Ctl* ctl;
  unsigned long long* rec;
  long long rec_region;          // records per update block
  unsigned long long* rcnt;      // records written per region since the last drain
  unsigned long long* colcnt;
  unsigned long long* ext_part;  // external-event partial sums, one per update block
  unsigned long long* spk_part;  // spike partial sums, one per update block
  const uint32_t* deg;           // out-degree per neuron (paper law), else null
  unsigned long long* syn_part;  // synaptic events of the spikes, one per update block
  ShardGeo sg;                   // shard geometry (sg.on = 0: a whole network)
};

// A batch of nets advanced by one persistent launch (snn_batch_*).
constexpr int kMaxBatch = 256;
struct BatchTile {          // a tile of a member
  const unsigned* isum;
  unsigned* ccnt;           // its counter in slot 0
  uint32_t stride;          // words from one slot's counters to the next
  int nslot, dmin, net, tile;
  unsigned win_items, cost_win;
};
struct BatchParams {
  StepParams* nets;         // [n_nets], device
  const int* u_first;       // [n_nets + 1] first update virtual block of each net
  const int* t_first;       // [n_nets + 1] first tile of each net
  const BatchTile* tiles;   // [n_tiles], device
  int n_nets, n_tiles;
  int win_words, max_cols;  // largest window and tile of the members
  unsigned min_items;       // fewest items a delivery block takes
  long long t0, n_steps;
  unsigned* bar;            // grid barrier: arrivals, generation, error flag
  long long spin_limit;     // polls before a barrier wait gives up
  unsigned extra_arrivals;  // arrivals expected beyond the grid (0; tests only)
};

struct BuildParams {
  long long N;
  int npc, npc4, nexc, W, H, K, k_local, dmin, ndel, rowcap, n_off;
  int tw, th;             // delivery tile, columns
  int unit;               // slots per bucket unit (8 or 16)
  int planes;
  uint32_t seed_lo, seed_hi;
  uint32_t stencil_thr[kMaxOff];
  int8_t off_dx[kMaxOff], off_dy[kMaxOff];
  const uint32_t* wtab;
  const uint32_t* colv;
  void* syn;
  uint8_t* bend;
  // paper connectivity law
  int n_poff;
  long long n_cand;
  unsigned long long poff_thr[kMaxOff];
  unsigned long long plocal_thr;
  int8_t poff_dx[kMaxOff], poff_dy[kMaxOff];
  uint32_t* deg;          // [N] out-degree of each neuron
  // [0] the largest row, in units; [1] the largest row in units of 8 slots
  // with one part per bucket (the size limit of the paper law)
  unsigned* max_units;
  ShardGeo sg;            // shard geometry (sg.on = 0: a whole network)
  // readback: rows j0 .. j0 + n_rows - 1, row r's synapses from entry rd_off[r]
  long long j0, n_rows;
  const long long* rd_off;
  long long* rd_target;
  int32_t* rd_delay;
  int32_t* rd_wfx;
  unsigned* rd_bad;       // set if a row does not hold what its draws say
  // draw order of the rows (the differentiable form's sums; see snn_grad.cu):
  // a word per 8 places of a row, and the ends of its buckets in such units
  uint32_t* ord;          // [ncol * npc][ord_units], rows in the order of syn
  uint8_t* ord_end;       // [ncol * npc][ndel]
  int ord_units;
};

// Byte of a descriptor that holds the end of the in part of bucket b (the end
// of its out part follows), and of the start of its plane's first bucket.
__host__ __device__ constexpr int desc_end(int b) {
  return b / kPlaneBuckets * 16 + 4 + 2 * (b % kPlaneBuckets);
}
__host__ __device__ constexpr int desc_start(int b) { return b / kPlaneBuckets * 16 + 2; }

// What the differentiable form reads of a net (snn_api.cu fills it).
struct NetView {
  const void* syn;
  const uint8_t* bend;
  long long N, acc_words;
  int npc, npc4, nexc, dmin, ndel, rowcap, unit, planes, precision, num_sms;
  const uint32_t* ctile;
  const uint32_t* colv;
  const uint32_t* nbg;
  const uint2* tinfo;
  int ntile, tcols;
  int ord_units;       // units of the longest row in draw order
  BuildParams build;   // the construction's draws
  bool paper;
  uint64_t seed;
  snn_neuron_params neuron;
  cudaStream_t stream;
};
int net_view(snn_net* net, NetView* v);

// min(floor(2^32 / d), 2^32 - 1): the multiplier of the kernels' divisions.
inline uint32_t recip32(uint32_t d) {
  const unsigned long long m = (1ull << 32) / (unsigned long long)d;
  return m > 0xFFFFFFFFull ? 0xFFFFFFFFu : (uint32_t)m;
}

// The seed's Philox round keys (Weyl sequences of the two key words).
inline void philox_keys(StepParams* p) {
  for (uint32_t r = 0; r < 10; ++r) {
    p->key[2 * r] = p->seed_lo + r * 0x9E3779B9u;
    p->key[2 * r + 1] = p->seed_hi + r * 0xBB67AE85u;
  }
}

// Shared host helpers (snn_api.cu).
int fail_global(int code, const std::string& msg);
// End of the function-try block of a C entry: what a host allocation throws
// becomes SNN_ENOMEM.  (The message fits a string without an allocation.)
#define SNN_CATCH(fail_call) \
  catch (...) {              \
    return fail_call;        \
  }
constexpr const char* kNoHostMemory = "no host memory";
int validate_neuron_params(const snn_neuron_params* n, std::string* why);

// Kernel launchers (snn_build.cu / snn_step.cu).
// Geometry tables (see above): the tile, place and virtual index of every column,
// every tile's first virtual column and columns, and the first word in acc of the
// column at each stencil offset of each virtual column.
cudaError_t launch_geometry(int W, int H, int tw, int th, int npc4, uint32_t* ctile, uint32_t* colv,
                            uint2* tinfo, uint32_t* nbg, cudaStream_t st);
// Fixed law: the fill pass writes bend, deg (shards), the rows of at most rowcap
// slots, and the longest of the others to max_units[0]; the count pass writes the
// longest row.
cudaError_t launch_build_count(const BuildParams& bp, int num_sms, cudaStream_t st);
cudaError_t launch_build(const BuildParams& bp, int precision, int num_sms,
                         cudaStream_t st);
// Paper connectivity law: the count pass writes bend, deg and max_units; the
// fill pass (same draws) writes the rows.
cudaError_t launch_paper_count(const BuildParams& bp, int num_sms, cudaStream_t st);
cudaError_t launch_paper_fill(const BuildParams& bp, int precision, int num_sms,
                              cudaStream_t st);
// Readback of rows in the order they were drawn, within a row by delay.
cudaError_t launch_read_rows(const BuildParams& bp, int precision, bool paper, cudaStream_t st);
// The rows' draw order (bp.ord, bp.ord_end), drawn again.
cudaError_t launch_draw_order(const BuildParams& bp, bool paper, int num_sms, cudaStream_t st);
cudaError_t launch_init_state(const StepParams& p, cudaStream_t st);
// `overlap`: programmatic dependent launch (step graphs, where update and
// delivery alternate); else a plain launch.
cudaError_t launch_update(const StepParams& p, int grid, bool overlap, cudaStream_t st);
int update_grid(long long N, int num_sms);
// Delivery: dynamic shared memory of one block of a net's own kernel or of
// the batch kernel (window, neighbour table, the warps' sector lists) for
// tiles of `cols` columns of npc4 words, and the persistent grid (0 if it
// does not fit).
size_t deliver_smem(int cols, int npc4, bool batch);
int deliver_grid(const StepParams& p, int precision, int num_sms);
cudaError_t launch_deliver(const StepParams& p, int precision, int grid, bool overlap, cudaStream_t st);
// Compact the per-block record regions into id and step arrays and reset
// them; header = {records kept, 1 if records were dropped, first step, last
// step}, written to the mapped host header map_hdr.  The arrays go to the mapped
// host buffers when they hold at most map_cap records, else to the device stage.
constexpr long long kMappedRecords = 1LL << 18;  // mapped host records per net
cudaError_t launch_drain_records(const StepParams& p, int nreg, uint32_t* stage_ids,
                                 uint32_t* stage_steps, unsigned long long* map_hdr, uint32_t* map_ids,
                                 uint32_t* map_steps, long long map_cap, cudaStream_t st);
// Counts the records a drain would return: {kept, 1 if records were dropped}
// to the mapped host header.
cudaError_t launch_count_records(const StepParams& p, int nreg, unsigned long long* map_hdr,
                                 cudaStream_t st);
// Batch kernel: dynamic shared memory for members whose largest window has
// win_words words and whose largest tile has max_cols columns, its grid (0 if it does not fit), its launch.
size_t batch_smem(int win_words, int max_cols);
// `rows`: some member keeps lists of rows; `wide`: some member has wide weights.
int batch_grid(int precision, int infl, bool rows, bool wide, int num_sms, size_t smem);
cudaError_t launch_batch(const BatchParams& b, int precision, int infl, bool rows, bool wide, int grid,
                         size_t smem, cudaStream_t st);
// Shard: list the received spikes (global indices ids[0 .. n)) of the halo
// columns in the step's lists, as the update kernel lists its own.
cudaError_t launch_ingest(const StepParams& p, const uint32_t* ids, long long n, cudaStream_t st);
cudaError_t launch_sum_parts(const unsigned long long* part, int n, unsigned long long* out,
                             cudaStream_t st);

}  // namespace snn
