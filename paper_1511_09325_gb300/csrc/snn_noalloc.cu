// snn_noalloc.cu -- one neuron-update step on caller-owned buffers, with no
// allocation of any kind.
//
// Some callers cannot let a library call cudaMalloc: a process whose device
// memory is already reserved by another framework's caching allocator or a
// fixed arena, or a real-time loop that cannot afford the implicit
// synchronisation of an allocation.  For them the
// neuron-update kernel of snn_step.cu runs here on their own state arrays; its
// scratch (step counter, spike-list cursor, per-block partial sums and the
// per-column spike counters) lives in one file-scope device array below, of a
// fixed size, which every GPU that loads the library holds until exit.
//
// The call is bound by its launches and one synchronisation: clear, update,
// results (each started while the one before runs) and one 16-byte copy; 24x24
// columns 36 us, with eight separate operations 58 us.
#include <algorithm>
#include <cstddef>
#include <mutex>
#include <string>

#include "snn_device.cuh"
#include "snn_internal.h"

using namespace snn;

namespace {

constexpr int kNoAllocMaxCols = 16384;   // columns per call
constexpr int kNoAllocMaxBlocks = 2048;  // update blocks per call
constexpr int kMaxDevices = 64;

// Byte offsets inside the scratch array.
constexpr size_t kOffCtl = 0;                                       // Ctl
constexpr size_t kOffCnt = 256;                                     // u32 spike count
constexpr size_t kOffOut = 264;                                     // u64 spikes, sum of ext_part
constexpr size_t kOffExt = 512;                                     // u64[blocks]
constexpr size_t kOffSpk = kOffExt + 8 * (size_t)kNoAllocMaxBlocks;  // u64[blocks]
constexpr size_t kOffRc = kOffSpk + 8 * (size_t)kNoAllocMaxBlocks;   // u64[blocks]
constexpr size_t kOffCol = kOffRc + 8 * (size_t)kNoAllocMaxBlocks;   // u64[2 * columns]
constexpr size_t kScratchBytes = kOffCol + 16 * (size_t)kNoAllocMaxCols;  // 311 808 B

static_assert(sizeof(Ctl) <= kOffCnt, "control block overlaps the counters");

__device__ __align__(256) unsigned char g_update_scratch[kScratchBytes];

// Clears the first `words` 8-byte words of the scratch, with the step index in
// the control block.
constexpr int kThreads = 1024;
__global__ void __launch_bounds__(kThreads) begin_kernel(unsigned long long* scratch, int words,
                                                         long long t) {
  grid_go();
  for (int i = blockIdx.x * kThreads + threadIdx.x; i < words; i += gridDim.x * kThreads)
    scratch[i] = i == (int)(offsetof(Ctl, t) / 8) ? (unsigned long long)t : 0ull;
}

// Results after the update: the spike count and the external events, side by
// side, and a copy of the column counts when wanted.
__global__ void __launch_bounds__(kThreads) end_kernel(const unsigned* cnt, const unsigned long long* ext_part,
                                                       int nparts, unsigned long long* out,
                                                       const unsigned long long* colcnt,
                                                       unsigned long long* col_counts, int ncounts) {
  grid_wait();
  for (int i = blockIdx.x * kThreads + threadIdx.x; i < ncounts; i += gridDim.x * kThreads)
    col_counts[i] = colcnt[i];
  if (blockIdx.x != 0 || threadIdx.x >= 32) return;
  unsigned long long s = 0ull;
  for (int i = threadIdx.x; i < nparts; i += 32) s += ext_part[i];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
  if (threadIdx.x == 0) {
    out[0] = *cnt;
    out[1] = s;
  }
}

std::mutex g_mu;
void* g_scratch_addr[kMaxDevices] = {};

// Device address of the scratch array on `dev` (which must be current).  The
// first call on a device looks it up; later calls reuse it, which assumes the
// device is not reset (cudaDeviceReset reloads the module) in between.
int scratch_address(int dev, unsigned char** out) {
  std::lock_guard<std::mutex> lock(g_mu);
  if (dev < 0 || dev >= kMaxDevices) return fail_global(SNN_EINVAL, "device ordinal out of range");
  if (!g_scratch_addr[dev]) {
    void* p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_update_scratch);
    if (e != cudaSuccess)
      return fail_global(SNN_ECUDA, std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e));
    g_scratch_addr[dev] = p;
  }
  *out = static_cast<unsigned char*>(g_scratch_addr[dev]);
  return SNN_OK;
}

bool aligned(const void* p, size_t a) { return ((uintptr_t)p % a) == 0; }

}  // namespace

extern "C" int snn_update_noalloc(int grid_w, int grid_h, const snn_neuron_params* neuron,
                                  uint64_t seed, int64_t step, float* v, float* c,
                                  uint8_t* refractory, int32_t* input, uint32_t* spikes,
                                  int64_t* n_spikes, int64_t* ext_events,
                                  unsigned long long* col_counts, void* cuda_stream) {
  std::string why;
  const int vrc = validate_neuron_params(neuron, &why);
  if (vrc != SNN_OK) return fail_global(vrc, why);
  if (grid_w < 1 || grid_h < 1) return fail_global(SNN_EINVAL, "grid must be at least 1x1");
  const long long ncol = (long long)grid_w * grid_h;
  if (ncol > kNoAllocMaxCols)
    return fail_global(SNN_EINVAL, "snn_update_noalloc handles at most 16384 columns");
  if (step < 0 || step > 0xFFFFFFFFLL) return fail_global(SNN_EINVAL, "step must be in 0..2^32-1");
  if (!v || !c || !refractory || !input || !spikes || !n_spikes)
    return fail_global(SNN_EINVAL, "null buffer");
  if (!aligned(v, 16) || !aligned(c, 16) || !aligned(input, 16) || !aligned(refractory, 4) ||
      !aligned(spikes, 4) || !aligned(col_counts, 8))
    return fail_global(SNN_EINVAL,
                       "v, c, input must be 16-byte, refractory and spikes 4-byte, col_counts "
                       "8-byte aligned");

  HostTables tb;
  int rc = make_neuron_tables(*neuron, &tb, &why);
  if (rc != SNN_OK) return fail_global(rc, why);
  int dev = 0, num_sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&num_sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return fail_global(SNN_ECUDA, std::string("device query: ") + cudaGetErrorString(e));
  unsigned char* base = nullptr;
  rc = scratch_address(dev, &base);
  if (rc != SNN_OK) return rc;

  const long long N = ncol * neuron->n_per_col;
  int grid = update_grid(N, num_sms);
  if (grid > kNoAllocMaxBlocks) grid = kNoAllocMaxBlocks;

  StepParams p{};
  p.N = N;
  p.npc = neuron->n_per_col;
  p.nexc = neuron->n_exc;
  p.W = grid_w;
  p.H = grid_h;
  p.nslot = 1;
  p.npc_m = recip32((uint32_t)neuron->n_per_col);
  p.ncol = (int)ncol;
  p.seed_lo = (uint32_t)(seed & 0xFFFFFFFFu);
  p.seed_hi = (uint32_t)(seed >> 32);
  philox_keys(&p);
  p.theta = neuron->theta;
  p.vr = neuron->v_reset;
  p.dc = neuron->dc;
  p.pvv = tb.pvv;
  p.pcc = tb.pcc;
  p.pvc_e = tb.pvc[0];
  p.pvc_i = tb.pvc[1];
  p.jx = tb.jx;
  p.nref = tb.nref;
  p.n_pois_thr = tb.n_pois_thr;
  for (int k = 0; k <= kMaxPoisThr; ++k) p.pois_thr[k] = tb.pois_thr[k];
  for (int k = 0; k < 256; ++k) p.pois_guide[k] = tb.pois_guide[k];
  p.V = v;
  p.C = c;
  p.R = refractory;
  p.acc = input;
  p.ids = spikes;
  p.ctl = reinterpret_cast<Ctl*>(base + kOffCtl);
  p.cnt = reinterpret_cast<unsigned*>(base + kOffCnt);
  p.ext_part = reinterpret_cast<unsigned long long*>(base + kOffExt);
  p.spk_part = reinterpret_cast<unsigned long long*>(base + kOffSpk);
  p.rcnt = reinterpret_cast<unsigned long long*>(base + kOffRc);
  p.colcnt = reinterpret_cast<unsigned long long*>(base + kOffCol);
  p.rec = nullptr;  // no spike records: the spike list is the output
  p.rec_region = 0;

  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  // Three kernels and one copy back: everything the update accumulates into
  // starts at zero, and the step index goes into the control block; then the
  // results.  (A memset, a copy in, the update, a sum and three copies before:
  // each of the copies to or from pageable memory waited for the stream.)
  const int words = (int)((kOffCol + 16 * (size_t)ncol) / 8), ncounts = col_counts ? 2 * (int)ncol : 0;
  begin_kernel<<<std::min(num_sms, (words + kThreads - 1) / kThreads), kThreads, 0, st>>>(
      reinterpret_cast<unsigned long long*>(base), words, step);
  e = cudaGetLastError();
  if (e == cudaSuccess) e = launch_update(p, grid, true, st);
  unsigned long long* d_out = reinterpret_cast<unsigned long long*>(base + kOffOut);
  unsigned long long out[2] = {0ull, 0ull};
  if (e == cudaSuccess) {
    const unsigned* cnt = p.cnt;
    const unsigned long long* ext = p.ext_part;
    const unsigned long long* col = p.colcnt;
    int nparts = grid, nc = ncounts;
    void* args[] = {&cnt, &ext, &nparts, &d_out, &col, &col_counts, &nc};
    e = launch_overlapped(reinterpret_cast<const void*>(end_kernel),
                          dim3((unsigned)std::max(1, std::min(num_sms, (ncounts + kThreads - 1) / kThreads))),
                          kThreads, 0, args, true, st);
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(out, d_out, sizeof(out), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess)
    return fail_global(SNN_ECUDA, std::string("snn_update_noalloc: ") + cudaGetErrorString(e));
  *n_spikes = (int64_t)out[0];
  if (ext_events) *ext_events = (int64_t)out[1];
  return SNN_OK;
}
