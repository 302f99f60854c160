// snn_api.cu -- the C ABI: net lifetime, graph-captured step loop, readback.
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstring>
#include <memory>
#include <new>
#include <string>
#include <vector>

#include "snn_internal.h"

using namespace snn;

struct snn_net {
  // configuration
  int W = 0, H = 0, npc = 0, nexc = 0, K = 0, dmin = 0, ndel = 0, nslot = 0;
  int precision = 0, rowcap = 0, rec_size = 0, num_sms = 0, update_grid = 0;
  bool wide = false;  // F16W with a weight of 64 mV or more
  bool agg = true;
  int deliver_grid = 0;
  int npc4 = 0, unit = kSlotUnit;     // words of a column in acc; slots of a bucket unit
  int planes = 1;                     // planes of a spike descriptor
  int ord_units = 0;                  // 8-slot units of the longest row, one part per bucket
  int tw = 1, th = 1, ntile = 1;      // delivery tiles
  bool batch_member = false;          // windows sized for the batch kernel's blocks
  unsigned min_items = 256;  // fewest items a delivery block takes
  unsigned win_items = 0;  // fewest items of a windowed tile part
  unsigned cost_win = 0;     // range split's fixed cost of a tile with a window
  long long N = 0, Npad = 0, ncol = 0;
  uint64_t seed = 0;
  snn_neuron_params neuron{};
  HostTables tables;
  StepParams sp{};
  // device memory
  void* syn = nullptr;
  uint8_t* bend = nullptr;
  float* V = nullptr;
  float* C = nullptr;
  uint8_t* R = nullptr;
  int32_t* acc = nullptr;
  uint4* list = nullptr;                  // spike lists
  uint16_t* rlist = nullptr;              // or lists of rows
  bool lean = false;                      // lists of rows
  uint32_t* ctile = nullptr;              // geometry tables (see snn_internal.h)
  uint32_t* colv = nullptr;
  uint2* tinfo = nullptr;
  uint32_t* nbg = nullptr;
  unsigned* icnt = nullptr;
  BuildParams bp{};                       // the construction's draws, for readback
  unsigned* hstatus = nullptr;            // status word (pinned, mapped)
  unsigned* hstatus_dev = nullptr;
  unsigned* ccnt = nullptr;
  uint32_t* deg = nullptr;                 // out-degree per neuron (paper law)
  unsigned long long* syn_part = nullptr;  // synaptic events per update block
  long long total_syn = 0;                 // synapses of the whole net
  int connectivity = SNN_CONN_FIXED;
  unsigned* isum = nullptr;
  unsigned* gsum = nullptr;
  unsigned* max_units = nullptr;           // the construction's longest row
  Ctl* ctl = nullptr;
  unsigned long long* rec = nullptr;
  long long rec_cap = 0;     // requested total record capacity
  long long rec_region = 0;  // records per update block
  unsigned long long* rcnt = nullptr;
  unsigned long long* stage = nullptr;   // large drains on the device: ids then steps (u32)
  unsigned long long* hhdr = nullptr;    // drain header (pinned, mapped)
  unsigned long long* hhdr_dev = nullptr;
  uint32_t* hmap = nullptr;              // small drains: ids then steps (pinned, mapped)
  uint32_t* hmap_dev = nullptr;
  long long hmap_cap = 0;                // records
  uint32_t* hstage = nullptr;            // large drains: ids then steps (pinned host)
  long long hstage_cap = 0;              // records
  unsigned long long* colcnt = nullptr;
  unsigned long long* ext_part = nullptr;
  unsigned long long* spk_part = nullptr;
  size_t device_bytes = 0;
  // execution
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  cudaGraphExec_t graph_one = nullptr;
  cudaGraphExec_t graph_many = nullptr;
  int graph_many_steps = 64;
  long long rate_window_start = 0;
  bool in_batch = false;  // stepped only through its snn_batch
  // shard (snn_build_shard): geometry, the half step due next (0 update,
  // 1 delivery), and the received spike indices (pinned host stage, device
  // copy, and an event recorded once the ingest kernel has read them)
  ShardGeo sg{};
  int shard_phase = 0;
  uint32_t* ingest = nullptr;
  uint32_t* hingest = nullptr;
  long long ingest_cap = 0;
  cudaEvent_t ingest_ev = nullptr;
  cudaEvent_t copy_ev[2] = {nullptr, nullptr};  // halves of the pinned copies out
  std::string err;
};

namespace {

thread_local std::string g_err;

int fail(snn_net* net, int code, const std::string& msg) {
  if (net)
    net->err = msg;
  else
    g_err = msg;
  return code;
}

}  // namespace

namespace snn {

int fail_global(int code, const std::string& msg) { return fail(nullptr, code, msg); }

int validate_neuron_params(const snn_neuron_params* n, std::string* why) {
  auto bad = [&](const char* m) {
    *why = m;
    return SNN_EINVAL;
  };
  if (!n) return bad("null parameter struct");
  if (n->n_per_col < 2 || n->n_per_col > 2048) return bad("n_per_col must be in 2..2048");
  if (n->n_exc < 0 || n->n_exc > n->n_per_col) return bad("n_exc must be in 0..n_per_col");
  if (!(n->tau_m > 0.f) || !(n->tau_c > 0.f)) return bad("time constants must be positive");
  if (!(n->t_ref >= 0.f) || n->t_ref > 200.f) return bad("t_ref must be in 0..200 ms");
  if (!(n->nu_ext_kHz >= 0.f) || n->nu_ext_kHz > 40.f) return bad("nu_ext_kHz must be in 0..40");
  if (!std::isfinite(n->theta) || !std::isfinite(n->v_reset) || !std::isfinite(n->dc) ||
      !std::isfinite(n->gc_exc) || !std::isfinite(n->gc_inh) || !std::isfinite(n->j_ext_mV))
    return bad("non-finite neuron parameter");
  return SNN_OK;
}

}  // namespace snn

namespace {

int cuda_fail(snn_net* net, cudaError_t e, const char* what) {
  return fail(net, e == cudaErrorMemoryAllocation ? SNN_ENOMEM : SNN_ECUDA,
              std::string(what) + ": " + cudaGetErrorString(e));
}

#define SNN_CUDA(net, call)                                   \
  do {                                                        \
    cudaError_t e_ = (call);                                  \
    if (e_ != cudaSuccess) return cuda_fail((net), e_, #call); \
  } while (0)

template <class T>
int dalloc(snn_net* net, T** p, size_t bytes) {
  void* v = nullptr;
  cudaError_t e = cudaMalloc(&v, bytes ? bytes : 256);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return fail(net, e == cudaErrorMemoryAllocation ? SNN_ENOMEM : SNN_ECUDA,
                "cudaMalloc of " + std::to_string(bytes) + " bytes: " + cudaGetErrorString(e));
  }
  *p = static_cast<T*>(v);
  net->device_bytes += bytes;
  return SNN_OK;
}

void free_graphs(snn_net* net) {
  if (net->graph_one) cudaGraphExecDestroy(net->graph_one);
  if (net->graph_many) cudaGraphExecDestroy(net->graph_many);
  net->graph_one = net->graph_many = nullptr;
}

void release(snn_net* net) {
  free_graphs(net);
  if (net->hhdr) cudaFreeHost(net->hhdr);
  if (net->hmap) cudaFreeHost(net->hmap);
  if (net->hstage) cudaFreeHost(net->hstage);
  if (net->hstatus) cudaFreeHost(net->hstatus);
  if (net->ingest) cudaFree(net->ingest);
  if (net->hingest) cudaFreeHost(net->hingest);
  if (net->ingest_ev) cudaEventDestroy(net->ingest_ev);
  for (cudaEvent_t ev : net->copy_ev)
    if (ev) cudaEventDestroy(ev);
  void* ptrs[] = {net->syn, net->bend, net->V, net->C, net->R, net->acc, net->list, net->rlist, net->ctile,
                  net->colv, net->tinfo, net->nbg, net->icnt, net->ccnt, net->deg, net->syn_part,
                  net->isum, net->gsum, net->max_units, net->ctl, net->rec, net->rcnt, net->stage,
                  net->colcnt, net->ext_part, net->spk_part};
  for (void* p : ptrs)
    if (p) cudaFree(p);
  if (net->own_stream && net->stream) cudaStreamDestroy(net->stream);
}

int validate(int gw, int gh, const snn_neuron_params* n, const snn_synapse_params* s,
             int precision, std::string* why) {
  auto bad = [&](const char* m) {
    *why = m;
    return SNN_EINVAL;
  };
  if (!n || !s) return bad("null parameter struct");
  if (gw < 1 || gh < 1) return bad("grid must be at least 1x1");
  if (gw > kMaxGridSide || gh > kMaxGridSide) return bad("grid_w and grid_h must be at most 16383");
  const int nrc = snn::validate_neuron_params(n, why);
  if (nrc != SNN_OK) return nrc;
  if (s->k_out < 1) return bad("k_out must be positive");
  if (!(s->frac_local >= 0.f && s->frac_local <= 1.f)) return bad("frac_local must be in [0, 1]");
  if (!(s->lambda_cols > 0.f)) return bad("lambda_cols must be positive");
  if (s->stencil_radius < 1 || s->stencil_radius > 3) return bad("stencil_radius must be 1..3");
  if (s->d_min < 1 || s->d_max < s->d_min || s->d_max > kMaxDelays)
    return bad("delays must satisfy 1 <= d_min <= d_max <= 32");
  if (s->periodic != 1) return bad("only periodic grids are supported");
  if (!std::isfinite(s->w_exc_mV) || !std::isfinite(s->w_inh_mV) || !std::isfinite(s->w_cv))
    return bad("non-finite weight parameter");
  if (precision != SNN_EXACT_F32W && precision != SNN_EXACT_F16W) return bad("unknown precision");
  const int ndel = s->d_max - s->d_min + 1;
  if (s->connectivity != SNN_CONN_FIXED && s->connectivity != SNN_CONN_PAPER)
    return bad("connectivity must be SNN_CONN_FIXED or SNN_CONN_PAPER");
  if (s->connectivity == SNN_CONN_FIXED &&
      (s->k_out + (kSlotUnit - 1) * ndel + kSlotUnit - 1) / kSlotUnit > 255)
    return bad("k_out too large for 8-bit bucket ends");
  if (s->connectivity == SNN_CONN_PAPER &&
      (!(s->p_local >= 0.f && s->p_local <= 1.f) || !(s->remote_a >= 0.f && s->remote_a <= 1.f) ||
       !(s->remote_sigma > 0.f) || !std::isfinite(s->remote_sigma) || !(s->remote_cutoff > 0.f)))
    return bad("paper law: p_local and remote_a in [0, 1], remote_sigma and remote_cutoff > 0");
  if (s->connectivity == SNN_CONN_PAPER &&
      (double)s->remote_a * std::exp(-16.0 / (2.0 * (double)s->remote_sigma * s->remote_sigma)) >=
          (double)s->remote_cutoff)
    return bad("the paper law keeps offsets beyond the 7x7 stencil");
  const long long N = (long long)gw * gh * n->n_per_col;
  if (N >= (1LL << 31) - 4) return bad("too many neurons");
  return SNN_OK;
}

// Fewest items a delivery block takes (fewer blocks run when a step has few
// items).  Measured (us per delivery, mean state) with 128, 64, 32 and 16: 2x2
// FP32 12.1, 11.2, 10.8, 10.6; 8x8 FP16 18.4, 16.8, 15.2, 15.1.
constexpr unsigned kMinItems = 16;
constexpr unsigned kBatchMinItems = 256;

// Delivery tiles: the largest square tile (side <= kMaxTile) whose window,
// neighbour table and the warps' sector lists fit the shared memory of a
// delivery block -- one block per SM for a net of its own, two per SM in the
// batch kernel -- then evened out over the grid's sides (24 columns make four
// tiles of 6, 8 make two of 4).  The largest tile keeps most synapses in the
// window (6x6: 80 %).  Measured at 96x96 (FP16, us per delivery in Down and Up
// states): 6x6 tiles 101 and 746; 5x5 187 and 792; 4x4 with a window of the 20
// most-hit columns around each 168 and 701.
void choose_tiles(snn_net* net) {
  net->npc4 = (net->npc + 3) / 4 * 4;
  const size_t budget = net->batch_member ? kBatchSmemBudget : kSmemBudget;
  int t = std::min(kMaxTile, std::max(net->W, net->H));
  for (; t > 1; --t) {
    const int cols = std::min(t, net->W) * std::min(t, net->H);
    if (deliver_smem(cols, net->npc4, net->batch_member) <= budget &&
        (size_t)cols * net->npc4 * 4 <= kWindowBudget)
      break;
  }
  auto even = [](int side, int t) {
    const int n = (side + t - 1) / t;
    return (side + n - 1) / n;
  };
  net->tw = even(net->W, std::min(t, net->W));
  net->th = even(net->H, std::min(t, net->H));
  const int words = net->tw * net->th * net->npc4;
  net->win_items = (unsigned)std::max(32, words / kWinWordsPerItem);
  net->cost_win = (unsigned)std::max(32, words / kCostWordsPerItem);
  net->ntile = ((net->W + net->tw - 1) / net->tw) * ((net->H + net->th - 1) / net->th);
}

// Slots of a bucket unit and of a row for rows of at most K synapses: units of 8
// slots, or of 16 where a row could exceed the 255 units that its bucket ends
// count; a row's slots as estimated for the longest row of the fixed law -- a part's
// padding is 0 .. unit - 1 slots, about equally often, so the sum over the parts
// stays within six standard deviations of its mean in nets of any size that fits
// (1240 synapses in 40 parts: 1472; the longest of 96x96 columns has 1448) unless
// the parts are short; then the longest row is counted.
void choose_unit(snn_net* net, int K) {
  const int n = std::min(K, 2 * net->ndel);  // parts that hold a synapse
  int most = 0;                              // slots of the longest row possible
  for (net->unit = kSlotUnit;; net->unit *= 2) {
    most = (K + (net->unit - 1) * n + net->unit - 1) / net->unit * net->unit;
    if (most / net->unit <= 255 || net->unit == 2 * kSlotUnit) break;
  }
  const double u = net->unit;
  const double slots = K + n * (u - 1.0) / 2.0 + 6.0 * std::sqrt(n * (u * u - 1.0) / 12.0);
  net->rowcap = std::min(most, ((int)slots / net->unit + 1) * net->unit);
}

// A kernel found inconsistent counts: the net's stepping is no longer exact.
int check_status(snn_net* net) {
  const unsigned st = net->hstatus ? *reinterpret_cast<volatile unsigned*>(net->hstatus) : 0u;
  if (st & kStatusIngest)
    return fail(net, SNN_ESTATE,
                "a shard received a spike index beyond the network or more spikes of one column "
                "than it has neurons; the net's state is no longer exact");
  if (st != 0u)
    return fail(net, SNN_ESTATE,
                "a delivery found item counts that disagree with the spike lists; the net's "
                "state is no longer exact");
  return SNN_OK;
}

int capture(snn_net* net, int steps, cudaGraphExec_t* out) {
  cudaGraph_t g = nullptr;
  SNN_CUDA(net, cudaStreamBeginCapture(net->stream, cudaStreamCaptureModeThreadLocal));
  cudaError_t le = cudaSuccess;
  for (int s = 0; s < steps && le == cudaSuccess; ++s) {
    // the graph's first kernel follows whatever the stream holds: a plain launch
    le = launch_update(net->sp, net->update_grid, s > 0, net->stream);
    if (le == cudaSuccess)
      le = launch_deliver(net->sp, net->precision, net->deliver_grid, true, net->stream);
  }
  cudaError_t ee = cudaStreamEndCapture(net->stream, &g);
  if (le != cudaSuccess) {
    if (g) cudaGraphDestroy(g);
    return cuda_fail(net, le, "kernel launch during capture");
  }
  if (ee != cudaSuccess) return cuda_fail(net, ee, "cudaStreamEndCapture");
  cudaError_t ie = cudaGraphInstantiate(out, g, 0);
  cudaGraphDestroy(g);
  if (ie != cudaSuccess) return cuda_fail(net, ie, "cudaGraphInstantiate");
  return SNN_OK;
}

void fill_step_params(snn_net* net) {
  StepParams& p = net->sp;
  const HostTables& t = net->tables;
  p.N = net->N;
  p.npc = net->npc;
  p.nexc = net->nexc;
  p.W = net->W;
  p.H = net->H;
  p.K = net->K;
  p.dmin = net->dmin;
  p.ndel = net->ndel;
  p.nslot = net->nslot;
  p.row_sec = net->rowcap * net->rec_size / 32;
  p.unit_sec = net->unit * net->rec_size / 32;
  p.ncol = (int)net->ncol;
  p.wide = net->wide ? 1 : 0;
  p.npc4 = net->npc4;
  p.ntile = net->ntile;
  p.tcols = net->tw * net->th;
  p.tcap = p.tcols * net->npc;
  p.min_items = net->min_items;
  p.win_items = net->agg ? net->win_items : 0xFFFFFFFFu;  // no windows: none is paid for either
  p.cost_win = net->cost_win;
  p.npc_m = recip32((uint32_t)net->npc);
  p.seed_lo = (uint32_t)(net->seed & 0xFFFFFFFFu);
  p.seed_hi = (uint32_t)(net->seed >> 32);
  philox_keys(&p);
  p.pvv = t.pvv;
  p.pcc = t.pcc;
  p.pvc_e = t.pvc[0];
  p.pvc_i = t.pvc[1];
  p.jx = t.jx;
  p.nref = t.nref;
  p.n_pois_thr = t.n_pois_thr;
  std::memcpy(p.pois_thr, t.pois_thr, sizeof(p.pois_thr));
  std::memcpy(p.pois_guide, t.pois_guide, sizeof(p.pois_guide));
  p.V = net->V;
  p.C = net->C;
  p.R = net->R;
  p.acc = net->acc;
  p.ids = nullptr;
  p.list = net->list;
  p.rlist = net->rlist;
  p.planes = net->planes;
  p.ctile = net->ctile;
  p.colv = net->colv;
  p.tinfo = net->tinfo;
  p.nbg = net->nbg;
  p.icnt = net->icnt;
  p.hstatus = net->hstatus_dev;
  p.cnt = nullptr;
  p.ccnt = net->ccnt;
  // a shard keeps the out-degree of its rows (synapses into its own columns)
  // for snn_row_lengths; its spikes count the full k_out synaptic events
  p.deg = net->sg.on ? nullptr : net->deg;
  p.syn_part = net->syn_part;
  p.sg = net->sg;
  p.isum = net->isum;
  p.gsum = net->gsum;
  p.bend = reinterpret_cast<const uint4*>(net->bend);
  p.syn = net->syn;
  p.ctl = net->ctl;
  p.rec = net->rec;
  p.rec_region = net->rec_region;
  p.rcnt = net->rcnt;
  p.colcnt = net->colcnt;
  p.ext_part = net->ext_part;
  p.spk_part = net->spk_part;
}

// Whether a net whose arrays still to be allocated take `small` bytes with lists
// of rows and `large` with lists of descriptors (`had`: allocated already), on a
// device with `free` bytes, takes the descriptors: only where they leave room for a
// second net of this size if there is room for two without them, and half as much
// in any case (for a differentiable view, or the caller's own arrays).
// Descriptors are about 1300 of an FP16 net's 7300 or an FP32 net's 13 200 bytes
// per neuron; lists of rows cost time: 1000 steps of 96x96 FP16 451 instead of 408
// ms, of 48x48 FP32 149 instead of 140 ms.
bool roomy_lists(size_t free, size_t had, size_t small, size_t large) {
  constexpr size_t kSlack = 48u << 20;  // rounding of two dozen allocations
  const size_t other = had + small;     // the second net, without descriptors
  if (large + kSlack + other / 2 > free) return false;
  return large + kSlack + other <= free || small + kSlack + other > free;
}

int build_impl(snn_net* net, int gw, int gh, const snn_neuron_params* np,
               const snn_synapse_params* sp, uint64_t seed, int precision) {
  std::string why;
  int rc = validate(gw, gh, np, sp, precision, &why);
  if (rc != SNN_OK) return fail(net, rc, why);
  net->W = gw;
  net->H = gh;
  net->npc = np->n_per_col;
  net->nexc = np->n_exc;
  net->K = sp->k_out;
  net->dmin = sp->d_min;
  net->ndel = sp->d_max - sp->d_min + 1;
  net->nslot = sp->d_max + 1;
  net->precision = precision;
  net->seed = seed;
  net->neuron = *np;
  net->ncol = (long long)gw * gh;
  net->N = net->ncol * np->n_per_col;
  net->Npad = (net->N + 3) / 4 * 4;
  net->rec_size = precision == SNN_EXACT_F16W ? 4 : 8;
  net->planes = (net->ndel + kPlaneBuckets - 1) / kPlaneBuckets;
  choose_unit(net, sp->k_out);
  net->ord_units = (sp->k_out + (kSlotUnit - 1) * std::min(sp->k_out, net->ndel) + kSlotUnit - 1) / kSlotUnit;
  net->rec_cap = 1LL << 24;
  rc = make_host_tables(*np, *sp, precision, &net->tables, &why);
  if (rc != SNN_OK) return fail(net, rc, why);
  constexpr uint32_t kHalf64 = 0x5400u;  // 64 as a half
  if (precision == SNN_EXACT_F16W)
    for (uint32_t w : net->tables.wtab) net->wide = net->wide || w >= kHalf64;
  net->sp.theta = np->theta;
  net->sp.vr = np->v_reset;
  net->sp.dc = np->dc;

  int dev = 0;
  SNN_CUDA(net, cudaGetDevice(&dev));
  SNN_CUDA(net, cudaDeviceGetAttribute(&net->num_sms, cudaDevAttrMultiProcessorCount, dev));
  net->update_grid = update_grid(net->N, net->num_sms);
  choose_tiles(net);
  fill_step_params(net);
  net->deliver_grid = deliver_grid(net->sp, precision, net->num_sms);
  if (net->deliver_grid < 1) return fail(net, SNN_ECUDA, "delivery kernel does not fit on the device");
  net->rec_region = (net->rec_cap + net->update_grid - 1) / net->update_grid;

  net->connectivity = sp->connectivity;
  BuildParams& bp = net->bp;
  bp.N = net->N;
  bp.npc = net->npc;
  bp.nexc = net->nexc;
  bp.W = net->W;
  bp.H = net->H;
  bp.K = net->K;
  bp.k_local = net->tables.k_local;
  bp.dmin = net->dmin;
  bp.ndel = net->ndel;
  bp.n_off = net->tables.n_off;
  bp.seed_lo = (uint32_t)(seed & 0xFFFFFFFFu);
  bp.seed_hi = (uint32_t)(seed >> 32);
  std::memcpy(bp.stencil_thr, net->tables.stencil_thr, sizeof(bp.stencil_thr));
  std::memcpy(bp.off_dx, net->tables.off_dx, sizeof(bp.off_dx));
  std::memcpy(bp.off_dy, net->tables.off_dy, sizeof(bp.off_dy));
  bp.n_poff = net->tables.n_poff;
  bp.n_cand = net->tables.n_cand;
  std::memcpy(bp.poff_thr, net->tables.poff_thr, sizeof(bp.poff_thr));
  bp.plocal_thr = net->tables.plocal_thr;
  std::memcpy(bp.poff_dx, net->tables.poff_dx, sizeof(bp.poff_dx));
  std::memcpy(bp.poff_dy, net->tables.poff_dy, sizeof(bp.poff_dy));
  bp.sg = net->sg;
  bp.npc4 = net->npc4;
  bp.tw = net->tw;
  bp.th = net->th;
  bp.unit = net->unit;
  bp.planes = net->planes;
  if ((rc = dalloc(net, &net->ctile, (size_t)net->ncol * 4))) return rc;
  if ((rc = dalloc(net, &net->colv, (size_t)net->ncol * 4))) return rc;
  if ((rc = dalloc(net, &net->tinfo, (size_t)net->ntile * sizeof(uint2)))) return rc;
  if ((rc = dalloc(net, &net->nbg, (size_t)net->ncol * 64 * 4))) return rc;
  SNN_CUDA(net, launch_geometry(gw, gh, net->tw, net->th, net->npc4, net->ctile, net->colv, net->tinfo, net->nbg,
                                net->stream));
  bp.colv = net->colv;
  if ((rc = dalloc(net, &net->bend, (size_t)net->N * net->planes * 16))) return rc;
  net->total_syn = net->N * (long long)net->K;
  if (net->sg.on && (rc = dalloc(net, &net->deg, (size_t)net->N * 4))) return rc;
  const bool paper = net->connectivity == SNN_CONN_PAPER;
  if (paper && (rc = dalloc(net, &net->deg, (size_t)net->N * 4))) return rc;
  unsigned max_units[2] = {0u, 0u};
  if ((rc = dalloc(net, &net->max_units, 8))) return rc;
  bp.max_units = net->max_units;
  bp.bend = net->bend;
  bp.deg = net->deg;
  // runs a pass over the rows and reads max_units back
  auto pass = [&](auto&& launch) -> cudaError_t {
    cudaError_t ce = cudaMemsetAsync(bp.max_units, 0, 8, net->stream);
    if (ce == cudaSuccess) ce = launch();
    if (ce == cudaSuccess)
      ce = cudaMemcpyAsync(max_units, bp.max_units, 8, cudaMemcpyDeviceToHost, net->stream);
    return ce == cudaSuccess ? cudaStreamSynchronize(net->stream) : ce;
  };
  // the longest row sets the row stride of the table
  auto count_rows = [&]() -> int {
    const cudaError_t ce = pass([&] {
      return paper ? launch_paper_count(bp, net->num_sms, net->stream)
                   : launch_build_count(bp, net->num_sms, net->stream);
    });
    if (ce != cudaSuccess) return cuda_fail(net, ce, "connectivity count pass");
    net->rowcap = (int)std::max(1u, max_units[0]) * net->unit;
    return SNN_OK;
  };
  if (paper) {
    // bucket ends, out-degrees and the longest row; 16 slots only where a row needs them
    for (net->unit = kSlotUnit;; net->unit *= 2) {
      bp.unit = net->unit;
      if ((rc = count_rows())) return rc;
      if (max_units[0] <= 255u || net->unit == 2 * kSlotUnit) break;
    }
    if (max_units[1] > 255u || max_units[0] > 255u)
      return fail(net, SNN_EINVAL, "a row of the paper law needs more than 2040 slots");
    net->ord_units = (int)std::max(1u, max_units[1]);
  }
  // Spike lists: of descriptors (planes x 16 bytes per neuron and step) or, where
  // the device has little room, of rows (2 bytes).
  const size_t tcap = (size_t)net->tw * net->th * net->npc;
  const size_t list_len = (size_t)net->nslot * net->ntile * tcap;
  size_t syn_bytes = (size_t)net->N * net->rowcap * net->rec_size;
  const size_t acc_bytes = (size_t)net->ncol * net->npc4 * 4;
  const size_t ccnt_bytes = (size_t)net->nslot * net->ntile * kCntStride * 4;
  const size_t isum_bytes = (size_t)net->ntile * kCntStride * 4;
  const size_t icnt_bytes = net->sg.on ? (size_t)net->ncol * 4 : 0;
  const size_t rec_bytes = (size_t)net->rec_region * net->update_grid * 8;
  const size_t col_bytes = (size_t)net->ncol * 2 * 8;
  const size_t wtab_bytes = net->tables.wtab.size() * 4;
  const size_t rest = (size_t)net->Npad * 9 + acc_bytes + ccnt_bytes + isum_bytes + icnt_bytes +
                      2 * rec_bytes + col_bytes + wtab_bytes;
  size_t free_bytes = 0, all_bytes = 0;
  SNN_CUDA(net, cudaMemGetInfo(&free_bytes, &all_bytes));
  if (!roomy_lists(free_bytes, net->device_bytes, syn_bytes + rest + list_len * 2,
                   syn_bytes + rest + list_len * net->planes * 16))
    net->lean = true;
  const bool rows = net->lean;
  if (rows && !paper && (rc = count_rows())) return rc;
  auto alloc_table = [&]() -> int {
    bp.rowcap = net->rowcap;
    syn_bytes = (size_t)net->N * net->rowcap * net->rec_size;
    const int arc = dalloc(net, &net->syn, syn_bytes);
    bp.syn = net->syn;
    return arc;
  };
  if ((rc = alloc_table())) return rc;
  if ((rc = dalloc(net, &net->V, (size_t)net->Npad * 4))) return rc;
  if ((rc = dalloc(net, &net->C, (size_t)net->Npad * 4))) return rc;
  if ((rc = dalloc(net, &net->R, (size_t)net->Npad))) return rc;
  if ((rc = dalloc(net, &net->acc, acc_bytes))) return rc;
  if (rows) {
    if ((rc = dalloc(net, &net->rlist, list_len * 2))) return rc;
  } else if ((rc = dalloc(net, &net->list, list_len * net->planes * 16))) {
    return rc;
  }
  if ((rc = dalloc(net, &net->ccnt, ccnt_bytes))) return rc;
  if ((rc = dalloc(net, &net->isum, isum_bytes))) return rc;
  if ((rc = dalloc(net, &net->gsum, 4))) return rc;
  if (icnt_bytes && (rc = dalloc(net, &net->icnt, icnt_bytes))) return rc;
  if ((rc = dalloc(net, &net->ctl, sizeof(Ctl)))) return rc;
  if ((rc = dalloc(net, &net->rec, rec_bytes))) return rc;
  if ((rc = dalloc(net, &net->rcnt, (size_t)net->update_grid * 8))) return rc;
  if ((rc = dalloc(net, &net->stage, rec_bytes))) return rc;
  SNN_CUDA(net, cudaHostAlloc(&net->hstatus, 16, cudaHostAllocMapped));
  SNN_CUDA(net, cudaHostGetDevicePointer(&net->hstatus_dev, net->hstatus, 0));
  *net->hstatus = 0u;
  SNN_CUDA(net, cudaHostAlloc(&net->hhdr, 32, cudaHostAllocMapped));
  SNN_CUDA(net, cudaHostGetDevicePointer(&net->hhdr_dev, net->hhdr, 0));
  net->hmap_cap = std::min<long long>(net->rec_region * net->update_grid, kMappedRecords);
  SNN_CUDA(net, cudaHostAlloc(&net->hmap, (size_t)net->hmap_cap * 8, cudaHostAllocMapped));
  SNN_CUDA(net, cudaHostGetDevicePointer(&net->hmap_dev, net->hmap, 0));
  if ((rc = dalloc(net, &net->colcnt, col_bytes))) return rc;
  if ((rc = dalloc(net, &net->ext_part, (size_t)net->update_grid * 8))) return rc;
  if ((rc = dalloc(net, &net->spk_part, (size_t)net->update_grid * 8))) return rc;
  if ((rc = dalloc(net, &net->syn_part, (size_t)net->update_grid * 8))) return rc;
  uint32_t* wtab = nullptr;
  if ((rc = dalloc(net, &wtab, wtab_bytes))) return rc;
  net->device_bytes -= wtab_bytes;

  cudaError_t e = cudaMemcpyAsync(wtab, net->tables.wtab.data(), wtab_bytes, cudaMemcpyHostToDevice,
                                  net->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(net->ctl, 0, sizeof(Ctl), net->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(net->acc, 0, acc_bytes, net->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(net->ccnt, 0, ccnt_bytes, net->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(net->isum, 0, isum_bytes, net->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(net->gsum, 0, 4, net->stream);
  if (e == cudaSuccess && net->icnt)
    e = cudaMemsetAsync(net->icnt, 0, (size_t)net->ncol * 4, net->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(net->colcnt, 0, (size_t)net->ncol * 16, net->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(net->ext_part, 0, (size_t)net->update_grid * 8, net->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(net->spk_part, 0, (size_t)net->update_grid * 8, net->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(net->syn_part, 0, (size_t)net->update_grid * 8, net->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(net->rcnt, 0, (size_t)net->update_grid * 8, net->stream);
  bp.wtab = wtab;
  auto fill = [&] {
    return paper ? launch_paper_fill(bp, precision, net->num_sms, net->stream)
                 : launch_build(bp, precision, net->num_sms, net->stream);
  };
  if (e == cudaSuccess) e = pass(fill);
  if (e == cudaSuccess && !paper && max_units[0] > 0u) {
    // a row is longer than estimated: the table again, by the rows' count
    cudaFree(net->syn);
    net->syn = nullptr;
    net->device_bytes -= syn_bytes;
    rc = count_rows();
    if (!rc) rc = alloc_table();
    if (!rc) e = pass(fill);
  }
  cudaFree(wtab);
  if (rc) return rc;
  fill_step_params(net);
  if (rows && deliver_grid(net->sp, precision, net->num_sms) < 1)
    return fail(net, SNN_ECUDA, "delivery kernel does not fit on the device");
  if (e == cudaSuccess) e = launch_init_state(net->sp, net->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(net->stream);
  if (e != cudaSuccess) return cuda_fail(net, e, "network construction");
  if (net->deg) {
    // paper law: the rows' out-degrees; shard: the synapses into its own columns
    std::vector<uint32_t> deg((size_t)net->N);
    SNN_CUDA(net, cudaMemcpyAsync(deg.data(), net->deg, deg.size() * 4, cudaMemcpyDeviceToHost,
                                  net->stream));
    SNN_CUDA(net, cudaStreamSynchronize(net->stream));
    net->total_syn = 0;
    for (uint32_t d : deg) net->total_syn += d;
  }
  return SNN_OK;
}

int sync(snn_net* net) {
  SNN_CUDA(net, cudaStreamSynchronize(net->stream));
  return SNN_OK;
}

// Copies `bytes` of device memory to pageable host memory `dst`.  A larger
// copy goes through the two halves of the pinned record buffer (which no call
// leaves in use), one half filled by the GPU while the other is copied out:
// a pageable copy into fresh heap memory ran at 1.4 GB/s (state of 48x48
// columns, 25.8 MB: 18 ms; staged: 2.6 ms).  Arrays of 32 MB and more, which the
// allocator maps by large pages, are faster copied directly (96x96, 103 MB: 6.4
// ms direct, 9.8 ms staged).
int copy_out(snn_net* net, void* dst, const void* src, size_t bytes) {
  const size_t half = (size_t)net->hmap_cap * 4 / 4096 * 4096;
  if (bytes <= 65536 || bytes >= (32u << 20) || half == 0) {
    SNN_CUDA(net, cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDeviceToHost, net->stream));
    return SNN_OK;
  }
  for (cudaEvent_t& ev : net->copy_ev)
    if (!ev) SNN_CUDA(net, cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
  char* const buf = reinterpret_cast<char*>(net->hmap);
  const size_t parts = (bytes + half - 1) / half;
  for (size_t k = 0; k <= parts; ++k) {
    if (k < parts) {
      SNN_CUDA(net, cudaMemcpyAsync(buf + (k & 1) * half, static_cast<const char*>(src) + k * half,
                                    std::min(half, bytes - k * half), cudaMemcpyDeviceToHost, net->stream));
      SNN_CUDA(net, cudaEventRecord(net->copy_ev[k & 1], net->stream));
    }
    if (k > 0) {
      SNN_CUDA(net, cudaEventSynchronize(net->copy_ev[(k - 1) & 1]));
      std::memcpy(static_cast<char*>(dst) + (k - 1) * half, buf + ((k - 1) & 1) * half,
                  std::min(half, bytes - (k - 1) * half));
    }
  }
  return SNN_OK;
}

Ctl read_ctl(snn_net* net, cudaError_t* e) {
  Ctl c{};
  *e = cudaMemcpyAsync(&c, net->ctl, sizeof(Ctl), cudaMemcpyDeviceToHost, net->stream);
  if (*e == cudaSuccess) *e = cudaStreamSynchronize(net->stream);
  return c;
}

}  // namespace

namespace snn {

int net_view(snn_net* net, NetView* v) {
  if (!net) return SNN_EINVAL;
  if (net->sg.on) return SNN_ESTATE;
  v->syn = net->syn;
  v->bend = net->bend;
  v->N = net->N;
  v->acc_words = net->ncol * (long long)net->npc4;
  v->npc = net->npc;
  v->npc4 = net->npc4;
  v->unit = net->unit;
  v->planes = net->planes;
  v->ctile = net->ctile;
  v->colv = net->colv;
  v->nbg = net->nbg;
  v->tinfo = net->tinfo;
  v->ntile = net->ntile;
  v->tcols = net->tw * net->th;
  v->ord_units = net->ord_units;
  v->build = net->bp;
  v->build.unit = net->unit;
  v->build.rowcap = net->rowcap;
  v->paper = net->connectivity == SNN_CONN_PAPER;
  v->nexc = net->nexc;
  v->dmin = net->dmin;
  v->ndel = net->ndel;
  v->rowcap = net->rowcap;
  v->precision = net->precision;
  v->num_sms = net->num_sms;
  v->seed = net->seed;
  v->neuron = net->neuron;
  v->stream = net->stream;
  return SNN_OK;
}

}  // namespace snn

namespace {

int build_net(int grid_w, int grid_h, const snn_neuron_params* neuron,
              const snn_synapse_params* synapse, uint64_t seed, int precision,
              void* cuda_stream, bool batch_member, snn_net** out,
              const ShardGeo* shard = nullptr, bool lean = false) {
  if (!out) return fail(nullptr, SNN_EINVAL, "out is NULL");
  *out = nullptr;
  std::string why;
  const int vrc = validate(grid_w, grid_h, neuron, synapse, precision, &why);
  if (vrc != SNN_OK) return fail(nullptr, vrc, why);
  snn_net* net = new (std::nothrow) snn_net();
  if (!net) return fail(nullptr, SNN_ENOMEM, "host allocation failed");
  net->batch_member = batch_member;
  net->lean = lean;
  net->min_items = batch_member ? kBatchMinItems : kMinItems;
  if (shard) net->sg = *shard;
  if (cuda_stream) {
    net->stream = static_cast<cudaStream_t>(cuda_stream);
  } else {
    cudaError_t e = cudaStreamCreateWithFlags(&net->stream, cudaStreamNonBlocking);
    if (e != cudaSuccess) {
      delete net;
      return fail(nullptr, SNN_ECUDA, std::string("cudaStreamCreate: ") + cudaGetErrorString(e));
    }
    net->own_stream = true;
  }
  int rc = SNN_OK;
  try {
    rc = build_impl(net, grid_w, grid_h, neuron, synapse, seed, precision);
  } catch (...) {
    rc = fail(net, SNN_ENOMEM, kNoHostMemory);
  }
  if (rc != SNN_OK) {
    const bool smaller = rc == SNN_ENOMEM && !net->lean;
    g_err = net->err;
    release(net);
    delete net;
    // the room went to others meanwhile: once more with the smaller lists
    if (smaller)
      return build_net(grid_w, grid_h, neuron, synapse, seed, precision, cuda_stream, batch_member, out, shard,
                       true);
    return rc;
  }
  *out = net;
  return SNN_OK;
}

}  // namespace

extern "C" {

int snn_build(int grid_w, int grid_h, const snn_neuron_params* neuron,
              const snn_synapse_params* synapse, uint64_t seed, int precision,
              void* cuda_stream, snn_net** out) {
  return build_net(grid_w, grid_h, neuron, synapse, seed, precision, cuda_stream, false, out);
}

}  // extern "C"

namespace {

// Local grid of the shard of tile (x0, y0, w, h): the tile and a halo of R
// columns on each side, or the whole grid side where the two would meet.
// *ew, *eh receive the local grid's size.
int shard_geometry(int grid_w, int grid_h, int x0, int y0, int w, int h, int R, ShardGeo* g, int* ew,
                   int* eh) {
  if (grid_w < 1 || grid_h < 1 || grid_w > kMaxGridSide || grid_h > kMaxGridSide)
    return fail(nullptr, SNN_EINVAL, "grid_w and grid_h must be in 1..16383");
  if (x0 < 0 || y0 < 0 || w < 1 || h < 1 || x0 > grid_w - w || y0 > grid_h - h)
    return fail(nullptr, SNN_EINVAL, "the shard's tile must lie inside the grid");
  if (R < 1 || R > 3) return fail(nullptr, SNN_EINVAL, "stencil_radius must be 1..3");
  *g = ShardGeo{};
  g->on = 1;
  g->GW = grid_w;
  g->GH = grid_h;
  g->tw = w;
  g->th = h;
  *ew = grid_w;
  *eh = grid_h;
  if (w + 2 * R < grid_w) {
    *ew = w + 2 * R;
    g->ex0 = (x0 - R + grid_w) % grid_w;
    g->tx0 = R;
  } else {
    g->ex0 = 0;
    g->tx0 = x0;
  }
  if (h + 2 * R < grid_h) {
    *eh = h + 2 * R;
    g->ey0 = (y0 - R + grid_h) % grid_h;
    g->ty0 = R;
  } else {
    g->ey0 = 0;
    g->ty0 = y0;
  }
  return SNN_OK;
}

void geometry_words(const ShardGeo& g, int ew, int eh, int32_t* geo, int n) {
  const int32_t v[10] = {g.GW, g.GH, ew, eh, g.ex0, g.ey0, g.tx0, g.ty0, g.tw, g.th};
  for (int i = 0; i < n && i < 10; ++i) geo[i] = v[i];
}

}  // namespace

extern "C" {

int snn_shard_geometry(int grid_w, int grid_h, int x0, int y0, int w, int h, int stencil_radius,
                       int32_t* geo, int n) {
  if (!geo) return fail(nullptr, SNN_EINVAL, "geo is NULL");
  ShardGeo g{};
  int ew = 0, eh = 0;
  const int rc = shard_geometry(grid_w, grid_h, x0, y0, w, h, stencil_radius, &g, &ew, &eh);
  if (rc != SNN_OK) return rc;
  geometry_words(g, ew, eh, geo, n);
  return SNN_OK;
}

int snn_build_shard(int grid_w, int grid_h, int x0, int y0, int w, int h,
                    const snn_neuron_params* neuron, const snn_synapse_params* synapse,
                    uint64_t seed, int precision, void* cuda_stream, snn_net** out) {
  if (!out) return fail(nullptr, SNN_EINVAL, "out is NULL");
  *out = nullptr;
  std::string why;
  const int vrc = validate(grid_w, grid_h, neuron, synapse, precision, &why);
  if (vrc != SNN_OK) return fail(nullptr, vrc, why);
  if (synapse->connectivity != SNN_CONN_FIXED)
    return fail(nullptr, SNN_EINVAL, "shards support SNN_CONN_FIXED only");
  if (neuron->n_per_col % 4 != 0)
    return fail(nullptr, SNN_EINVAL, "shards need n_per_col to be a multiple of 4");
  ShardGeo g{};
  int ew = 0, eh = 0;
  const int grc = shard_geometry(grid_w, grid_h, x0, y0, w, h, synapse->stencil_radius, &g, &ew, &eh);
  if (grc != SNN_OK) return grc;
  return build_net(ew, eh, neuron, synapse, seed, precision, cuda_stream, false, out, &g);
}

int snn_shard_update(snn_net* net) {
  if (!net) return fail(nullptr, SNN_EINVAL, "net is NULL");
  if (!net->sg.on) return fail(net, SNN_ESTATE, "not a shard: use snn_step");
  if (net->shard_phase != 0) return fail(net, SNN_ESTATE, "snn_shard_deliver is due first");
  int rc = check_status(net);
  if (rc) return rc;
  SNN_CUDA(net, launch_update(net->sp, net->update_grid, false, net->stream));
  net->shard_phase = 1;
  return SNN_OK;
}

int snn_shard_deliver(snn_net* net, const int32_t* ids, int64_t n, int32_t ids_on_device) {
  if (!net) return fail(nullptr, SNN_EINVAL, "net is NULL");
  if (!net->sg.on) return fail(net, SNN_ESTATE, "not a shard: use snn_step");
  if (n < 0 || (n > 0 && !ids)) return fail(net, SNN_EINVAL, "bad spike index array");
  if (net->shard_phase != 1) return fail(net, SNN_ESTATE, "snn_shard_update is due first");
  const uint32_t* src = reinterpret_cast<const uint32_t*>(ids);
  const bool staged = n > 0 && !ids_on_device;
  if (staged) {
    // the previous staged indices must have been read before the stage is reused
    if (net->ingest_ev) SNN_CUDA(net, cudaEventSynchronize(net->ingest_ev));
    else SNN_CUDA(net, cudaEventCreateWithFlags(&net->ingest_ev, cudaEventDisableTiming));
    if (n > net->ingest_cap) {
      const long long want = std::max<long long>(n, 1 << 16);
      if (net->ingest) cudaFree(net->ingest);
      if (net->hingest) cudaFreeHost(net->hingest);
      net->device_bytes -= (size_t)net->ingest_cap * 4;
      net->ingest = nullptr;
      net->hingest = nullptr;
      net->ingest_cap = 0;
      if (int rc = dalloc(net, &net->ingest, (size_t)want * 4)) return rc;
      SNN_CUDA(net, cudaMallocHost(&net->hingest, (size_t)want * 4));
      net->ingest_cap = want;
    }
    std::memcpy(net->hingest, ids, (size_t)n * 4);
    SNN_CUDA(net, cudaMemcpyAsync(net->ingest, net->hingest, (size_t)n * 4, cudaMemcpyHostToDevice,
                                  net->stream));
    src = net->ingest;
  }
  SNN_CUDA(net, launch_ingest(net->sp, src, n, net->stream));
  if (staged) SNN_CUDA(net, cudaEventRecord(net->ingest_ev, net->stream));
  SNN_CUDA(net, launch_deliver(net->sp, net->precision, net->deliver_grid, false, net->stream));
  net->shard_phase = 0;
  return SNN_OK;
}

int snn_shard_info(snn_net* net, int32_t* geo, int n) {
  if (!net || !geo) return fail(net, SNN_EINVAL, "null argument");
  if (!net->sg.on) return fail(net, SNN_ESTATE, "not a shard");
  geometry_words(net->sg, net->W, net->H, geo, n);
  return SNN_OK;
}

int snn_step(snn_net* net, int64_t n_steps) {
  if (!net) return fail(nullptr, SNN_EINVAL, "net is NULL");
  if (net->in_batch) return fail(net, SNN_ESTATE, "net belongs to a batch: use snn_batch_step");
  if (net->sg.on)
    return fail(net, SNN_ESTATE, "a shard steps by snn_shard_update and snn_shard_deliver");
  if (n_steps < 0) return fail(net, SNN_EINVAL, "n_steps must be >= 0");
  int rc = check_status(net);
  if (rc) return rc;
  if (n_steps == 0) return SNN_OK;
  if (n_steps >= net->graph_many_steps && !net->graph_many)
    if ((rc = capture(net, net->graph_many_steps, &net->graph_many))) return rc;
  if (!net->graph_one)
    if ((rc = capture(net, 1, &net->graph_one))) return rc;
  int64_t left = n_steps;
  while (left >= net->graph_many_steps) {
    SNN_CUDA(net, cudaGraphLaunch(net->graph_many, net->stream));
    left -= net->graph_many_steps;
  }
  while (left-- > 0) SNN_CUDA(net, cudaGraphLaunch(net->graph_one, net->stream));
  return SNN_OK;
}

int snn_step_profiled(snn_net* net, int64_t n_steps, double* ms, double* bytes) try {
  if (!net) return fail(nullptr, SNN_EINVAL, "net is NULL");
  if (net->in_batch) return fail(net, SNN_ESTATE, "net belongs to a batch: use snn_batch_step");
  if (net->sg.on)
    return fail(net, SNN_ESTATE, "a shard steps by snn_shard_update and snn_shard_deliver");
  if (n_steps < 0) return fail(net, SNN_EINVAL, "n_steps must be >= 0");
  if (n_steps >= 1LL << 40) return fail(net, SNN_ENOMEM, kNoHostMemory);  // three events a step
  std::vector<cudaEvent_t> ev((size_t)n_steps * 3 + 1);
  std::vector<unsigned long long> hspk((size_t)n_steps + 1, 0ull);
  unsigned long long* dspk = nullptr;  // spikes so far, after each step
  int rc = dalloc(net, &dspk, ((size_t)n_steps + 1) * 8);
  if (rc) return rc;
  net->device_bytes -= ((size_t)n_steps + 1) * 8;
  size_t made = 0;
  cudaError_t e = cudaSuccess;
  for (; made < ev.size() && e == cudaSuccess; ++made) e = cudaEventCreate(&ev[made]);
  if (e != cudaSuccess) --made;
  if (e == cudaSuccess) e = launch_sum_parts(net->spk_part, net->update_grid, dspk, net->stream);
  for (int64_t s = 0; s < n_steps && e == cudaSuccess; ++s) {
    e = cudaEventRecord(ev[3 * s], net->stream);
    if (e == cudaSuccess) e = launch_update(net->sp, net->update_grid, false, net->stream);
    if (e == cudaSuccess) e = cudaEventRecord(ev[3 * s + 1], net->stream);
    if (e == cudaSuccess)
      e = launch_deliver(net->sp, net->precision, net->deliver_grid, false, net->stream);
    if (e == cudaSuccess) e = cudaEventRecord(ev[3 * s + 2], net->stream);
    if (e == cudaSuccess)
      e = launch_sum_parts(net->spk_part, net->update_grid, dspk + s + 1, net->stream);
  }
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(hspk.data(), dspk, hspk.size() * 8, cudaMemcpyDeviceToHost, net->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(net->stream);
  double t_up = 0.0, t_dl = 0.0, b_up = 0.0, b_dl = 0.0;
  const double neuron_bytes = 26.0 * (double)net->N;
  for (int64_t s = 0; s < n_steps && e == cudaSuccess; ++s) {
    float a = 0.f, b = 0.f;
    e = cudaEventElapsedTime(&a, ev[3 * s], ev[3 * s + 1]);
    if (e == cudaSuccess) e = cudaEventElapsedTime(&b, ev[3 * s + 1], ev[3 * s + 2]);
    t_up += a;
    t_dl += b;
    const double S = (double)(hspk[s + 1] - hspk[s]);
    b_up += neuron_bytes + 12.0 * S;
    b_dl += S * ((double)net->total_syn / (double)net->N * net->rec_size + 6.0 * net->ndel);
  }
  if (e != cudaSuccess) rc = cuda_fail(net, e, "profiled step");
  for (size_t i = 0; i < made; ++i) cudaEventDestroy(ev[i]);
  cudaFree(dspk);
  if (rc == SNN_OK) {
    if (ms) {
      ms[0] = t_up;
      ms[1] = t_dl;
    }
    if (bytes) {
      bytes[0] = b_up;
      bytes[1] = b_dl;
    }
  }
  return rc;
}
SNN_CATCH(fail(net, SNN_ENOMEM, kNoHostMemory))

namespace {

int reset_records(snn_net* net) {
  const unsigned zero32 = 0u;
  SNN_CUDA(net, cudaMemsetAsync(net->rcnt, 0, (size_t)net->update_grid * 8, net->stream));
  SNN_CUDA(net, cudaMemcpyAsync((char*)net->ctl + offsetof(Ctl, rec_overflow), &zero32, 4,
                                cudaMemcpyHostToDevice, net->stream));
  SNN_CUDA(net, cudaStreamSynchronize(net->stream));
  return SNN_OK;
}

}  // namespace

int snn_pending_spikes(snn_net* net, int64_t* n_out) {
  if (!net || !n_out) return fail(net, SNN_EINVAL, "null argument");
  SNN_CUDA(net, launch_count_records(net->sp, net->update_grid, net->hhdr_dev, net->stream));
  SNN_CUDA(net, cudaStreamSynchronize(net->stream));
  *n_out = (int64_t)net->hhdr[0];
  return SNN_OK;
}

int snn_read_spikes(snn_net* net, int32_t* steps, int32_t* ids, int64_t cap, int64_t* n_out) try {
  if (!net || !n_out || cap < 0 || (cap > 0 && (!steps || !ids)))
    return fail(net, SNN_EINVAL, "bad argument");
  *n_out = 0;
  // compact the regions on the device into id and step arrays and reset
  // them; a drain of at most hmap_cap records lands in mapped host memory
  // directly, a larger one is copied from the device stage afterwards
  const long long stage_cap = net->rec_region * net->update_grid;
  uint32_t* stage_ids = reinterpret_cast<uint32_t*>(net->stage);
  SNN_CUDA(net, launch_drain_records(net->sp, net->update_grid, stage_ids, stage_ids + stage_cap,
                                     net->hhdr_dev, net->hmap_dev,
                                     net->hmap_dev + net->hmap_cap, net->hmap_cap, net->stream));
  SNN_CUDA(net, cudaStreamSynchronize(net->stream));
  if (int src = check_status(net)) return src;
  const long long kept = (long long)net->hhdr[0];
  bool lost = net->hhdr[1] != 0ull || kept > cap;
  const uint32_t tmin = (uint32_t)net->hhdr[2], tmax = (uint32_t)net->hhdr[3];
  const long long n = kept < cap ? kept : cap;
  const uint32_t* hid = net->hmap;
  const uint32_t* hst = net->hmap + net->hmap_cap;
  if (n > 0 && kept > net->hmap_cap) {
    if (n > net->hstage_cap) {
      if (net->hstage) cudaFreeHost(net->hstage);
      net->hstage = nullptr;
      net->hstage_cap = 0;
      const long long want = std::max<long long>(n, 1 << 16);
      SNN_CUDA(net, cudaMallocHost(&net->hstage, (size_t)want * 8));
      net->hstage_cap = want;
    }
    SNN_CUDA(net, cudaMemcpyAsync(net->hstage, stage_ids, (size_t)n * 4, cudaMemcpyDeviceToHost,
                                  net->stream));
    SNN_CUDA(net, cudaMemcpyAsync(net->hstage + net->hstage_cap, stage_ids + stage_cap,
                                  (size_t)n * 4, cudaMemcpyDeviceToHost, net->stream));
    SNN_CUDA(net, cudaStreamSynchronize(net->stream));
    hid = net->hstage;
    hst = net->hstage + net->hstage_cap;
  }
  if (n > 0) {
    if (tmin == tmax) {
      // one step (the usual read after every step): the ids as they are
      std::memcpy(ids, hid, (size_t)n * 4);
      std::fill(steps, steps + n, (int32_t)tmin);
    } else {
      // each region is in step order: a counting sort by step puts the
      // window in step order (within a step the order stays unspecified)
      std::vector<long long> pos((size_t)(tmax - tmin) + 2, 0);
      for (long long k = 0; k < n; ++k) ++pos[(size_t)(hst[k] - tmin) + 1];
      for (size_t i = 1; i < pos.size(); ++i) pos[i] += pos[i - 1];
      for (long long k = 0; k < n; ++k) {
        const long long o = pos[hst[k] - tmin]++;
        steps[o] = (int32_t)hst[k];
        ids[o] = (int32_t)hid[k];
      }
    }
    *n_out = n;
  }
  if (lost) return fail(net, SNN_EOVERFLOW, "spike records dropped (buffer or cap too small)");
  return SNN_OK;
}
SNN_CATCH(fail(net, SNN_ENOMEM, kNoHostMemory))

int snn_set_record_capacity(snn_net* net, int64_t capacity) {
  if (!net || capacity < 1) return fail(net, SNN_EINVAL, "bad argument");
  int rc = sync(net);
  if (rc) return rc;
  const long long region = (capacity + net->update_grid - 1) / net->update_grid;
  unsigned long long* nr = nullptr;
  cudaError_t e = cudaMalloc(&nr, (size_t)region * net->update_grid * 8);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return cuda_fail(net, e, "cudaMalloc record buffer");
  }
  unsigned long long* ns = nullptr;
  e = cudaMalloc(&ns, (size_t)region * net->update_grid * 8);
  if (e != cudaSuccess) {
    cudaGetLastError();
    cudaFree(nr);
    return cuda_fail(net, e, "cudaMalloc record staging buffer");
  }
  cudaFree(net->rec);
  cudaFree(net->stage);
  net->device_bytes -= 2 * (size_t)net->rec_region * net->update_grid * 8;
  net->device_bytes += 2 * (size_t)region * net->update_grid * 8;
  net->rec = nr;
  net->stage = ns;
  net->rec_cap = capacity;
  net->rec_region = region;
  fill_step_params(net);
  free_graphs(net);
  return reset_records(net);
}

int snn_read_rates(snn_net* net, float* hz, int64_t n, float* pop_hz) try {
  if (!net) return fail(nullptr, SNN_EINVAL, "net is NULL");
  if (hz && n < 2 * net->ncol) return fail(net, SNN_EINVAL, "hz array too small");
  cudaError_t e;
  Ctl c = read_ctl(net, &e);
  if (e != cudaSuccess) return cuda_fail(net, e, "read control block");
  if (int src = check_status(net)) return src;
  std::vector<unsigned long long> cnt((size_t)net->ncol * 2);
  SNN_CUDA(net, cudaMemcpyAsync(cnt.data(), net->colcnt, cnt.size() * 8, cudaMemcpyDeviceToHost,
                                net->stream));
  SNN_CUDA(net, cudaMemsetAsync(net->colcnt, 0, cnt.size() * 8, net->stream));
  SNN_CUDA(net, cudaStreamSynchronize(net->stream));
  const long long window = c.t - net->rate_window_start;
  net->rate_window_start = c.t;
  const double secs = (double)window * 1e-3;
  const double nE = (double)net->nexc, nI = (double)(net->npc - net->nexc);
  // a shard's own columns (the halo's spikes are counted by their owners)
  const double own_cols = net->sg.on ? (double)net->sg.tw * net->sg.th : (double)net->ncol;
  double totE = 0.0, totI = 0.0;
  for (long long k = 0; k < net->ncol; ++k) {
    totE += (double)cnt[2 * k];
    totI += (double)cnt[2 * k + 1];
    if (hz) {
      hz[2 * k] = (secs > 0 && nE > 0) ? (float)((double)cnt[2 * k] / (nE * secs)) : 0.f;
      hz[2 * k + 1] = (secs > 0 && nI > 0) ? (float)((double)cnt[2 * k + 1] / (nI * secs)) : 0.f;
    }
  }
  if (pop_hz) {
    pop_hz[0] = (secs > 0 && nE > 0) ? (float)(totE / (nE * own_cols * secs)) : 0.f;
    pop_hz[1] = (secs > 0 && nI > 0) ? (float)(totI / (nI * own_cols * secs)) : 0.f;
  }
  return SNN_OK;
}
SNN_CATCH(fail(net, SNN_ENOMEM, kNoHostMemory))

int snn_stats(snn_net* net, double* recurrent_events, double* external_events, int64_t* steps) try {
  if (!net) return fail(nullptr, SNN_EINVAL, "net is NULL");
  cudaError_t e;
  Ctl c = read_ctl(net, &e);
  if (e != cudaSuccess) return cuda_fail(net, e, "read control block");
  std::vector<unsigned long long> ext((size_t)net->update_grid), syn((size_t)net->update_grid);
  SNN_CUDA(net, cudaMemcpyAsync(ext.data(), net->ext_part, ext.size() * 8, cudaMemcpyDeviceToHost,
                                net->stream));
  SNN_CUDA(net, cudaMemcpyAsync(syn.data(), net->syn_part, syn.size() * 8, cudaMemcpyDeviceToHost,
                                net->stream));
  SNN_CUDA(net, cudaStreamSynchronize(net->stream));
  if (int src = check_status(net)) return src;
  unsigned long long se = 0ull, sy = 0ull;
  for (size_t b = 0; b < ext.size(); ++b) {
    se += ext[b];
    sy += syn[b];
  }
  // every spike counts its neuron's out-degree (k_out under the fixed law)
  if (recurrent_events) *recurrent_events = (double)sy;
  if (external_events) *external_events = (double)se;
  if (steps) *steps = (int64_t)c.t;
  return SNN_OK;
}
SNN_CATCH(fail(net, SNN_ENOMEM, kNoHostMemory))

int snn_get_state(snn_net* net, float* v, float* c, uint8_t* refractory) {
  if (!net) return fail(nullptr, SNN_EINVAL, "net is NULL");
  const size_t N = (size_t)net->N;
  int rc = SNN_OK;
  if (v) rc = copy_out(net, v, net->V, N * 4);
  if (c && !rc) rc = copy_out(net, c, net->C, N * 4);
  if (refractory && !rc) rc = copy_out(net, refractory, net->R, N);
  return rc ? rc : sync(net);
}

int snn_read_synapses(snn_net* net, int64_t j0, int64_t n, int64_t* target, int32_t* delay,
                      int32_t* wfx) try {
  if (!net || j0 < 0 || n < 0 || j0 + n > net->N || (n > 0 && (!target || !delay || !wfx)))
    return fail(net, SNN_EINVAL, "bad argument");
  if (n == 0) return SNN_OK;
  std::vector<int32_t> len((size_t)n);
  int rc = snn_row_lengths(net, j0, n, len.data());
  if (rc) return rc;
  // the device walks each row's draws again and decodes the records in that
  // order, a bounded number of rows at a time: in the drain's stage, which is
  // idle between reads, or where that is too small in a buffer of its own
  constexpr int64_t kRows = 4096, kFewRows = 32;
  int32_t longest = 0;
  for (int32_t l : len) longest = std::max(longest, l);
  const int64_t in_stage = (net->rec_region * net->update_grid - 1) / (1 + 2 * (int64_t)longest);
  const bool staged = in_stage >= std::min(n, kFewRows);
  const int64_t m = std::min(n, staged ? std::min(in_stage, kRows) : kRows);
  size_t most = 0;
  std::vector<long long> off;
  off.reserve((size_t)m);
  for (int64_t r0 = 0; r0 < n; r0 += m) {
    size_t k = 0;
    for (int64_t r = r0; r < std::min(n, r0 + m); ++r) k += (size_t)len[r];
    most = std::max(most, k);
  }
  // error word, offsets, targets, delays, weights
  unsigned char* buf = reinterpret_cast<unsigned char*>(net->stage);
  const size_t off_bytes = 8 + (size_t)m * 8, b8 = most * 8, b4 = most * 4;
  if (!staged) {
    rc = dalloc(net, &buf, off_bytes + b8 + 2 * b4);
    if (rc) return rc;
    net->device_bytes -= off_bytes + b8 + 2 * b4;
  }
  BuildParams bp = net->bp;
  bp.syn = net->syn;
  bp.bend = net->bend;
  bp.unit = net->unit;
  bp.rowcap = net->rowcap;
  bp.rd_bad = reinterpret_cast<unsigned*>(buf);
  bp.rd_off = reinterpret_cast<long long*>(buf + 8);
  bp.rd_target = reinterpret_cast<long long*>(buf + off_bytes);
  bp.rd_delay = reinterpret_cast<int32_t*>(buf + off_bytes + b8);
  bp.rd_wfx = reinterpret_cast<int32_t*>(buf + off_bytes + b8 + b4);
  unsigned bad = 0u;
  cudaError_t e = cudaMemsetAsync(bp.rd_bad, 0, 4, net->stream);
  size_t at = 0;
  for (int64_t r0 = 0; r0 < n && e == cudaSuccess; r0 += m) {
    bp.j0 = j0 + r0;
    bp.n_rows = std::min(n - r0, m);
    off.assign((size_t)bp.n_rows, 0);
    size_t k = 0;
    for (int64_t r = 0; r < bp.n_rows; ++r) {
      off[(size_t)r] = (long long)k;
      k += (size_t)len[r0 + r];
    }
    e = cudaMemcpyAsync(buf + 8, off.data(), off.size() * 8, cudaMemcpyHostToDevice, net->stream);
    if (e == cudaSuccess)
      e = launch_read_rows(bp, net->precision, net->connectivity == SNN_CONN_PAPER, net->stream);
    if (e == cudaSuccess && k > 0) {
      e = cudaMemcpyAsync(target + at, bp.rd_target, k * 8, cudaMemcpyDeviceToHost, net->stream);
      if (e == cudaSuccess)
        e = cudaMemcpyAsync(delay + at, bp.rd_delay, k * 4, cudaMemcpyDeviceToHost, net->stream);
      if (e == cudaSuccess)
        e = cudaMemcpyAsync(wfx + at, bp.rd_wfx, k * 4, cudaMemcpyDeviceToHost, net->stream);
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(net->stream);
    at += k;
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(&bad, bp.rd_bad, 4, cudaMemcpyDeviceToHost, net->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(net->stream);
  if (!staged) cudaFree(buf);
  if (e != cudaSuccess) return cuda_fail(net, e, "synapse readback");
  if (bad) return fail(net, SNN_ESTATE, "a row of the table does not hold the synapses drawn for it");
  return SNN_OK;
}
SNN_CATCH(fail(net, SNN_ENOMEM, kNoHostMemory))

int snn_row_lengths(snn_net* net, int64_t j0, int64_t n, int32_t* counts) {
  if (!net || j0 < 0 || n < 0 || j0 + n > net->N || (n > 0 && !counts))
    return fail(net, SNN_EINVAL, "bad argument");
  if (n == 0) return SNN_OK;
  if (!net->deg) {
    for (int64_t r = 0; r < n; ++r) counts[r] = net->K;
    return SNN_OK;
  }
  SNN_CUDA(net, cudaMemcpyAsync(counts, net->deg + j0, (size_t)n * 4, cudaMemcpyDeviceToHost,
                                net->stream));
  return sync(net);
}

int snn_info(snn_net* net, int64_t* info, int n) {
  if (!net || !info) return fail(net, SNN_EINVAL, "null argument");
  const int64_t v[9] = {net->N, (int64_t)net->total_syn, (int64_t)net->device_bytes,
                        net->N * (int64_t)net->rowcap * net->rec_size, net->rowcap,
                        net->precision, net->tw, net->deliver_grid, net->update_grid};
  for (int i = 0; i < n && i < 9; ++i) info[i] = v[i];
  return SNN_OK;
}

const char* snn_last_error(const snn_net* net) {
  return net ? net->err.c_str() : g_err.c_str();
}

static TilePlace place_of(const snn_net* net, int64_t column) {
  return tile_place(net->W, net->H, net->tw, net->th, (int)(column % net->W), (int)(column / net->W));
}

int snn_debug_offset_count(snn_net* net, int64_t column, int32_t delta, int32_t group_only) {
  if (!net) return fail(nullptr, SNN_EINVAL, "net is NULL");
  if (column < 0 || column >= net->ncol) return fail(net, SNN_EINVAL, "column out of range");
  int rc = sync(net);
  if (rc) return rc;
  unsigned* const tile = net->isum + (size_t)place_of(net, column).tile * kCntStride;
  unsigned word = 0u;
  if (!group_only) {
    SNN_CUDA(net, cudaMemcpy(&word, tile, 4, cudaMemcpyDeviceToHost));
    word += (unsigned)delta;
    SNN_CUDA(net, cudaMemcpy(tile, &word, 4, cudaMemcpyHostToDevice));
  }
  SNN_CUDA(net, cudaMemcpy(&word, net->gsum, 4, cudaMemcpyDeviceToHost));
  word += (unsigned)delta;
  SNN_CUDA(net, cudaMemcpy(net->gsum, &word, 4, cudaMemcpyHostToDevice));
  return SNN_OK;
}

int snn_debug_flip_byte(snn_net* net, int64_t neuron, int64_t byte, int32_t mask, int32_t in_table) {
  if (!net) return fail(nullptr, SNN_EINVAL, "net is NULL");
  const int64_t row_bytes = in_table ? (int64_t)net->rowcap * net->rec_size : (int64_t)net->planes * 16;
  if (neuron < 0 || neuron >= net->N || byte < 0 || byte >= row_bytes)
    return fail(net, SNN_EINVAL, "neuron or byte out of range");
  int rc = sync(net);
  if (rc) return rc;
  const int64_t row = (int64_t)place_of(net, neuron / net->npc).v * net->npc + neuron % net->npc;
  uint8_t* const at = (in_table ? static_cast<uint8_t*>(net->syn) : net->bend) + row * row_bytes + byte;
  uint8_t v = 0;
  SNN_CUDA(net, cudaMemcpy(&v, at, 1, cudaMemcpyDeviceToHost));
  v = (uint8_t)(v ^ (uint8_t)mask);
  SNN_CUDA(net, cudaMemcpy(at, &v, 1, cudaMemcpyHostToDevice));
  return SNN_OK;
}

void snn_destroy(snn_net* net) {
  if (!net) return;
  if (net->stream) cudaStreamSynchronize(net->stream);
  release(net);
  delete net;
}

}  // extern "C"

// ---------------------------------------------------------------------------
// Batched form: independent nets advanced together by one persistent launch.
// ---------------------------------------------------------------------------
struct snn_batch {
  std::vector<snn_net*> nets;
  int precision = 0, num_sms = 0;
  int infl = 4;            // 16-byte chunks in flight in the delivery loop
  int agg = 1;             // block windows for the local half of the synapses
  unsigned min_items = kBatchMinItems;  // fewest items a delivery block takes
  int choice = -1;         // autotuner's pick (-1: not tuned)
  std::vector<int> first;  // [2][n + 1]: first update virtual blocks, first tiles
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  StepParams* d_nets = nullptr;
  int* d_first = nullptr;  // first, on the device
  BatchTile* d_tiles = nullptr;
  unsigned* d_bar = nullptr;
  long long t = 0;
  long long spin_limit = 1LL << 25;
  unsigned extra_arrivals = 0u;
  std::string err;
};

namespace {

int bfail(snn_batch* b, int code, const std::string& msg) {
  if (b)
    b->err = msg;
  else
    g_err = msg;
  return code;
}

#define SNN_BCUDA(b, call)                                                            \
  do {                                                                                \
    cudaError_t e_ = (call);                                                          \
    if (e_ != cudaSuccess) return bfail((b), SNN_ECUDA, std::string(#call ": ") +     \
                                                           cudaGetErrorString(e_));   \
  } while (0)

void batch_release(snn_batch* b) {
  for (snn_net* n : b->nets) snn_destroy(n);
  b->nets.clear();
  if (b->d_nets) cudaFree(b->d_nets);
  if (b->d_first) cudaFree(b->d_first);
  if (b->d_tiles) cudaFree(b->d_tiles);
  if (b->d_bar) cudaFree(b->d_bar);
  if (b->own_stream && b->stream) cudaStreamDestroy(b->stream);
}

// Upload the members' step parameters with the batch's window setting.
int batch_upload(snn_batch* b) {
  std::vector<StepParams> ps(b->nets.size());
  std::vector<BatchTile> tiles;
  for (size_t k = 0; k < b->nets.size(); ++k) {
    b->nets[k]->agg = b->agg != 0;
    fill_step_params(b->nets[k]);
    ps[k] = b->nets[k]->sp;
    const StepParams& p = ps[k];
    for (int m = 0; m < p.ntile; ++m) {
      BatchTile bt{};
      bt.isum = p.isum + (size_t)m * kCntStride;
      bt.ccnt = p.ccnt + (size_t)m * kCntStride;
      bt.stride = (uint32_t)(p.ntile * kCntStride);
      bt.nslot = p.nslot;
      bt.dmin = p.dmin;
      bt.net = (int)k;
      bt.tile = m;
      bt.win_items = p.win_items;
      bt.cost_win = p.cost_win;
      tiles.push_back(bt);
    }
  }
  SNN_BCUDA(b, cudaMemcpyAsync(b->d_tiles, tiles.data(), tiles.size() * sizeof(BatchTile),
                               cudaMemcpyHostToDevice, b->stream));
  SNN_BCUDA(b, cudaMemcpyAsync(b->d_nets, ps.data(), ps.size() * sizeof(StepParams),
                               cudaMemcpyHostToDevice, b->stream));
  SNN_BCUDA(b, cudaStreamSynchronize(b->stream));
  return SNN_OK;
}

int batch_run(snn_batch* b, long long n_steps) {
  if (n_steps == 0) return SNN_OK;
  // members' buffers may have been reallocated (record capacity): refresh
  const int urc = batch_upload(b);
  if (urc != SNN_OK) return urc;
  const int n = (int)b->nets.size();
  BatchParams bp{};
  bp.nets = b->d_nets;
  bp.u_first = b->d_first;
  bp.t_first = b->d_first + (n + 1);
  bp.tiles = b->d_tiles;
  bp.n_nets = n;
  bp.n_tiles = b->first.back();
  bp.min_items = b->min_items;
  bp.t0 = b->t;
  bp.n_steps = n_steps;
  bp.bar = b->d_bar;
  bp.spin_limit = b->spin_limit;
  bp.extra_arrivals = b->extra_arrivals;
  for (const snn_net* net : b->nets) {
    bp.win_words = std::max(bp.win_words, net->sp.tcols * net->sp.npc4);
    bp.max_cols = std::max(bp.max_cols, net->sp.tcols);
  }
  const size_t smem = batch_smem(bp.win_words, bp.max_cols);
  bool rows = false, wide = false;
  for (const snn_net* net : b->nets) {
    rows = rows || net->rlist != nullptr;
    wide = wide || net->wide;
  }
  const int grid = batch_grid(b->precision, b->infl, rows, wide, b->num_sms, smem);
  if (grid < 1) return bfail(b, SNN_ECUDA, "batch kernel does not fit on the device");
  SNN_BCUDA(b, cudaMemsetAsync(b->d_bar, 0, 3 * sizeof(unsigned), b->stream));
  SNN_BCUDA(b, launch_batch(bp, b->precision, b->infl, rows, wide, grid, smem, b->stream));
  unsigned flags[3] = {0u, 0u, 0u};
  SNN_BCUDA(b, cudaMemcpyAsync(flags, b->d_bar, sizeof(flags), cudaMemcpyDeviceToHost, b->stream));
  SNN_BCUDA(b, cudaStreamSynchronize(b->stream));
  if (flags[2]) return bfail(b, SNN_ETIMEOUT, "a grid barrier wait gave up");
  b->t += n_steps;
  return SNN_OK;
}

}  // namespace

extern "C" {

int snn_batch_build(int n_nets, const int32_t* grid_w, const int32_t* grid_h,
                    const snn_neuron_params* neuron, const snn_synapse_params* synapse,
                    const uint64_t* seeds, int precision, void* cuda_stream, snn_batch** out) try {
  if (!out) return bfail(nullptr, SNN_EINVAL, "out is NULL");
  *out = nullptr;
  if (n_nets < 1 || n_nets > kMaxBatch) return bfail(nullptr, SNN_EINVAL, "n_nets must be in 1..256");
  if (!grid_w || !grid_h || !neuron || !synapse || !seeds)
    return bfail(nullptr, SNN_EINVAL, "null argument");
  for (int k = 0; k < n_nets; ++k) {
    std::string why;
    const int rc = validate(grid_w[k], grid_h[k], neuron + k, synapse + k, precision, &why);
    if (rc != SNN_OK) return bfail(nullptr, rc, "net " + std::to_string(k) + ": " + why);
  }
  struct Release {
    void operator()(snn_batch* b) const {
      batch_release(b);
      delete b;
    }
  };
  std::unique_ptr<snn_batch, Release> b(new (std::nothrow) snn_batch());
  if (!b) return bfail(nullptr, SNN_ENOMEM, "host allocation failed");
  b->precision = precision;
  if (cuda_stream) {
    b->stream = static_cast<cudaStream_t>(cuda_stream);
  } else {
    cudaError_t e = cudaStreamCreateWithFlags(&b->stream, cudaStreamNonBlocking);
    if (e != cudaSuccess)
      return bfail(nullptr, SNN_ECUDA, std::string("cudaStreamCreate: ") + cudaGetErrorString(e));
    b->own_stream = true;
  }
  int rc = SNN_OK;
  b->first.assign(2 * (size_t)(n_nets + 1), 0);
  b->nets.reserve((size_t)n_nets);
  bool lean = false;
  for (int k = 0; k < n_nets && rc == SNN_OK; ++k) {
    snn_net* net = nullptr;
    rc = build_net(grid_w[k], grid_h[k], neuron + k, synapse + k, seeds[k], precision, b->stream,
                   true, &net, nullptr, lean);
    if (rc == SNN_ENOMEM && !lean) {
      // the members before took more memory than they need: once more, all lean
      for (snn_net* n : b->nets) snn_destroy(n);
      b->nets.clear();
      lean = true;
      rc = SNN_OK;
      k = -1;
      continue;
    }
    if (rc != SNN_OK) break;
    net->in_batch = true;
    b->nets.push_back(net);
    b->num_sms = net->num_sms;
    // update: the net's own grid (its partial sums and record regions)
    b->first[k + 1] = b->first[k] + net->update_grid;
    b->first[(n_nets + 1) + k + 1] = b->first[(n_nets + 1) + k] + net->ntile;
  }
  if (rc != SNN_OK) return rc;  // with the member's message
  cudaError_t e = cudaMalloc(&b->d_nets, sizeof(StepParams) * (size_t)n_nets);
  if (e == cudaSuccess) e = cudaMalloc(&b->d_first, b->first.size() * sizeof(int));
  if (e == cudaSuccess) e = cudaMalloc(&b->d_tiles, (size_t)b->first.back() * sizeof(BatchTile));
  if (e == cudaSuccess) e = cudaMalloc(&b->d_bar, 4 * sizeof(unsigned));
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(b->d_first, b->first.data(), b->first.size() * sizeof(int),
                        cudaMemcpyHostToDevice, b->stream);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return bfail(nullptr, e == cudaErrorMemoryAllocation ? SNN_ENOMEM : SNN_ECUDA,
                 std::string("batch buffers: ") + cudaGetErrorString(e));
  }
  rc = batch_upload(b.get());
  if (rc != SNN_OK) return bfail(nullptr, rc, b->err);
  *out = b.release();
  return SNN_OK;
}
SNN_CATCH(bfail(nullptr, SNN_ENOMEM, kNoHostMemory))

int snn_batch_step(snn_batch* b, int64_t n_steps) try {
  if (!b) return bfail(nullptr, SNN_EINVAL, "batch is NULL");
  if (n_steps < 0) return bfail(b, SNN_EINVAL, "n_steps must be >= 0");
  return batch_run(b, n_steps);
}
SNN_CATCH(bfail(b, SNN_ENOMEM, kNoHostMemory))

snn_net* snn_batch_net(snn_batch* b, int k) {
  if (!b || k < 0 || k >= (int)b->nets.size()) return nullptr;
  return b->nets[k];
}

int snn_batch_tune(snn_batch* b, int64_t steps_per_trial, int32_t* choice) try {
  if (!b || steps_per_trial < 1) return bfail(b, SNN_EINVAL, "bad argument");
  // every variant computes the same sums, so the trials simply advance the
  // simulation; two interleaved rounds even out changes in activity.  Stage
  // 0 times the four delivery schedules, stage 1 the delivery densities (the
  // fewest items a block takes) with the schedule that won.
  const int infl[4] = {4, 4, 2, 2}, agg[4] = {1, 0, 1, 0};
  const unsigned min_items[4] = {64, 128, 256, 512};
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  cudaError_t ce = cudaEventCreate(&e0);
  if (ce == cudaSuccess) ce = cudaEventCreate(&e1);
  if (ce != cudaSuccess) {
    if (e0) cudaEventDestroy(e0);
    return bfail(b, SNN_ECUDA, std::string("tuner events: ") + cudaGetErrorString(ce));
  }
  int rc = SNN_OK;
  int pick[2] = {0, 0};
  for (int stage = 0; stage < 2 && rc == SNN_OK; ++stage) {
    double ms[4] = {0, 0, 0, 0};
    for (int round = 0; round < 2 && rc == SNN_OK; ++round) {
      for (int v = 0; v < 4 && rc == SNN_OK; ++v) {
        if (stage == 0) {
          b->infl = infl[v];
          b->agg = agg[v];
          rc = batch_upload(b);
        } else {
          b->min_items = min_items[v];
        }
        if (rc) break;
        cudaError_t e = cudaEventRecord(e0, b->stream);
        if (e == cudaSuccess) {
          rc = batch_run(b, steps_per_trial);
          if (rc) break;
          e = cudaEventRecord(e1, b->stream);
        }
        if (e == cudaSuccess) e = cudaEventSynchronize(e1);
        float x = 0.f;
        if (e == cudaSuccess) e = cudaEventElapsedTime(&x, e0, e1);
        if (e != cudaSuccess) {
          rc = bfail(b, SNN_ECUDA, std::string("tuner timing: ") + cudaGetErrorString(e));
          break;
        }
        ms[v] += x;
      }
    }
    for (int v = 1; v < 4; ++v)
      if (ms[v] < ms[pick[stage]]) pick[stage] = v;
    if (rc == SNN_OK && stage == 0) {
      b->infl = infl[pick[0]];
      b->agg = agg[pick[0]];
      rc = batch_upload(b);
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (rc != SNN_OK) return rc;
  b->min_items = min_items[pick[1]];
  b->choice = pick[0] + 4 * pick[1];
  if (choice) *choice = b->choice;
  return SNN_OK;
}
SNN_CATCH(bfail(b, SNN_ENOMEM, kNoHostMemory))

int snn_batch_set_wait(snn_batch* b, int64_t spin_limit, int32_t extra_arrivals) {
  if (!b || spin_limit < 1 || extra_arrivals < 0) return bfail(b, SNN_EINVAL, "bad argument");
  b->spin_limit = spin_limit;
  b->extra_arrivals = (unsigned)extra_arrivals;
  return SNN_OK;
}

const char* snn_batch_last_error(const snn_batch* b) { return b ? b->err.c_str() : g_err.c_str(); }

void snn_batch_destroy(snn_batch* b) {
  if (!b) return;
  if (b->stream) cudaStreamSynchronize(b->stream);
  batch_release(b);
  delete b;
}


}  // extern "C"
