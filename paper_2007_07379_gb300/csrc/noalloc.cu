// A plain Gibbs run that allocates no memory: its scratch (run header,
// tables, chain state, counters) lives in one file-scope device array.
//
// This serves callers that cannot allocate device memory at the point of the
// call: for example a plug-in whose host application owns every device
// allocation, or code running while a memory budget is frozen.  Such a
// caller passes only its inputs (a compiled model, a run configuration) and
// its outputs (device buffers for the counts); nothing is allocated here.
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>

#include "pb_internal.h"
#include "sweep_common.cuh"

namespace pb {
cudaError_t launch_sweeps_plain(const RunModelDev* d_rm, int n_models, uint32_t total_groups,
                                uint32_t n_sweeps, int cons, int prod, int units, int max_col, int nc,
                                bool wgt, size_t smem_bytes, WsHeader* hdr, cudaStream_t st);
cudaError_t sweep_plain_prepare();
}  // namespace pb

using namespace pb;

namespace {

// The scratch array: 16 MiB, held by every GPU that loads the library.
constexpr size_t kScratchBytes = 16u << 20;
static __device__ __align__(256) unsigned char g_pb_scratch[kScratchBytes];

// Per device, set up once with that device current: the device address of
// g_pb_scratch (the name itself is only a host-side stand-in) and the sweep
// kernels' shared-memory opt-in.  The cache assumes the device's context is
// not reset while the library is loaded (cudaDeviceReset would invalidate
// both; a process that resets a device must not call this entry point
// afterwards).
constexpr int kMaxDevices = 64;
void* g_scratch_addr[kMaxDevices];
std::mutex g_scratch_mutex;

int scratch_address(void** out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return PB_ECUDA;
  if (dev < 0 || dev >= kMaxDevices) return PB_ERANGE;
  std::lock_guard<std::mutex> lock(g_scratch_mutex);
  if (!g_scratch_addr[dev]) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_pb_scratch) != cudaSuccess || p == nullptr) return PB_ECUDA;
    if (sweep_plain_prepare() != cudaSuccess) return PB_ECUDA;
    g_scratch_addr[dev] = p;
  }
  *out = g_scratch_addr[dev];
  return PB_OK;
}

inline size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

// The start of a call: a cleared header (sweep index 0, status 0), the run
// entry, cleared counters and the initial chains (a CTA per chain group, more
// where there are many counters).  The entry comes as a kernel parameter, which
// a launch copies: nothing that outlives the call points at its stack.
struct NoallocRun {
  RunModelDev rm;
  ModelDev md;
  const uint32_t* init;
  WsHeader* d_hdr;
  RunModelDev* d_rm;
  ModelDev* d_md;
};
__device__ void put_words(void* dst, const void* src, size_t bytes) {
  for (uint32_t i = threadIdx.x; i < bytes / 4; i += blockDim.x)
    static_cast<uint32_t*>(dst)[i] = src ? static_cast<const uint32_t*>(src)[i] : 0u;
}
__global__ void __launch_bounds__(256) noalloc_begin_kernel(const __grid_constant__ NoallocRun run) {
  extern __shared__ __align__(16) uint32_t smem[];
  const uint32_t n_counts = run.rm.bins * 8u;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n_counts; i += gridDim.x * blockDim.x)
    run.rm.hist[i] = 0ull;
  if (blockIdx.x == 0) {
    if (threadIdx.x == 0) *run.rm.valid = *run.rm.samples = 0ull;
    put_words(run.d_hdr, nullptr, sizeof(WsHeader));
    put_words(run.d_rm, &run.rm, sizeof(RunModelDev));
    put_words(run.d_md, &run.md, sizeof(ModelDev));
  }
  // (no header for the status of a bad table: it is being cleared, and the
  // sweeps check the tables again)
  if (blockIdx.x < run.rm.groups) init_group(run.rm, run.md, blockIdx.x, run.init, smem, nullptr);
}
static_assert(sizeof(WsHeader) % 4 == 0 && sizeof(RunModelDev) % 4 == 0 && sizeof(ModelDev) % 4 == 0,
              "copied by words");

}  // namespace

extern "C" PB_API int pb_gibbs_run_noalloc(const pb_model* m, const pb_run_cfg* cfg,
                                           uint32_t n_sweeps, unsigned long long* d_counts,
                                           unsigned long long* d_totals, uintptr_t stream) {
  if (!m || !cfg || !d_counts || !d_totals) return PB_EINVAL;
  if (cfg->sampler != PB_GIBBS || cfg->alphas != nullptr || cfg->n_alphas != 0) return PB_EINVAL;
  if (cfg->chains == 0 || cfg->record_every == 0) return PB_EINVAL;
  if (m->wgt) return PB_EINVAL;  // general one-qubit gates: use pb_run_create
  if (m->n > 16) return PB_ERANGE;
  if (n_sweeps > (1u << 26)) return PB_ERANGE;
  if ((uint64_t)cfg->group0 + (cfg->chains + 31) / 32 > 0xFFFFFFFFull) return PB_ERANGE;
  // The call copies its tables from host memory: it cannot be recorded into
  // a CUDA graph (a replay would read the model's tables, which may be gone).
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(reinterpret_cast<cudaStream_t>(stream), &cap) != cudaSuccess)
    return PB_ECUDA;
  if (cap != cudaStreamCaptureStatusNone) return PB_ESTATE;

  const int n = m->n, d = m->d;
  const size_t npb = (size_t)n * d;
  const uint32_t groups = (cfg->chains + 31) / 32;
  const uint32_t bins = 1u << n;

  // Layout of the scratch (one model, one batch).
  size_t off = 0;
  const size_t o_hdr = off; off = align256(off + sizeof(WsHeader));
  const size_t o_rm = off; off = align256(off + sizeof(RunModelDev));
  const size_t o_md = off; off = align256(off + sizeof(ModelDev));
  const TableOffsets tab = table_offsets(npb);
  const size_t o_tab = off; off = align256(off + tab.bytes);
  const size_t o_state = off; off = align256(off + (size_t)groups * npb * 4);
  // counters: the run keeps them in the caller's buffers; the scratch has
  // room for them where those are not aligned for 64-bit atomics
  const size_t o_hist = off; off = align256(off + (size_t)bins * 8 * 8);
  const size_t o_cnt = off; off = align256(off + 2 * 8);
  if (off > kScratchBytes) return PB_ERANGE;

  void* base_v = nullptr;
  int rc = scratch_address(&base_v);
  if (rc != PB_OK) return rc;
  char* base = static_cast<char*>(base_v);
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);

  // Shape as for a single-model run.
  int maxcol = 1, nc = 2;  // largest class; colour steps per sweep
  for (int c = 0; c < 4; ++c) {
    maxcol = std::max(maxcol, m->col_off[c + 1] - m->col_off[c]);
    if (m->col_off[c + 1] > m->col_off[c]) nc = std::max(nc, c + 1);
  }
  // histogram placement: the rule of a single-model run (shared memory for
  // up to 4096 bins when the CTA still fits)
  auto hist_fits = [&](int units) {
    return bins <= 4096u && plain_smem_bytes(n, d, bins, units) <= kSweepSmemMax;
  };
  auto smem_for = [&](int units) {
    return plain_smem_bytes(n, d, hist_fits(units) ? bins : 0, units);
  };
  int dev = 0, sms = 1;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return PB_ECUDA;
  const PlainDefault ps = plain_shape(n * d, maxcol, groups, sms, smem_for);
  const bool hist_smem = hist_fits(ps.units);
  const int units = plain_launch_units(n * d, ps.units, n_sweeps);
  const size_t smem = plain_smem_bytes(n, d, hist_smem ? bins : 0, units);
  if (smem > kSweepSmemMax) return PB_ERANGE;

  NoallocRun run{};
  ModelDev& md = run.md;
  md.n = n;
  md.d = d;
  md.nw = n_words(n, d);
  md.h = m->h;
  md.beta = m->beta;
  for (int k = 0; k < 4; ++k) md.thr[k] = m->thr[k];
  for (int k = 0; k < 5; ++k) md.col_off[k] = m->col_off[k];
  md.max_col = maxcol;
  for (int k = 0; k < 4; ++k) md.n_rec[k] = m->n_rec[k];

  RunModelDev& r = run.rm;
  r.model = reinterpret_cast<const ModelDev*>(base + o_md);
  r.md = md;
  r.desc = reinterpret_cast<const Desc*>(base + o_tab + tab.desc);
  r.rec = reinterpret_cast<const Rec*>(base + o_tab + tab.rec);
  r.state = reinterpret_cast<uint32_t*>(base + o_state);
  const bool direct = (((uintptr_t)d_counts | (uintptr_t)d_totals) & 7u) == 0;
  unsigned long long* counts = direct ? d_counts : reinterpret_cast<unsigned long long*>(base + o_hist);
  unsigned long long* totals = direct ? d_totals : reinterpret_cast<unsigned long long*>(base + o_cnt);
  r.hist = counts;
  r.valid = totals;
  r.samples = totals + 1;
  r.alpha_sorted = nullptr;
  r.alpha_slot = nullptr;
  r.amp = nullptr;
  r.n_alphas = 0;
  r.bins = bins;
  r.chains = cfg->chains;
  r.groups = groups;
  r.n_batches = 1;
  r.burn_in = cfg->burn_in;
  r.record_every = cfg->record_every;
  r.seed_lo = (uint32_t)cfg->seed;
  r.seed_hi = (uint32_t)(cfg->seed >> 32);
  r.group_base = 0;
  r.group0 = cfg->group0;
  r.hist_smem = hist_smem ? 1u : 0u;
  run.init = reinterpret_cast<const uint32_t*>(base + o_tab + tab.init);
  run.d_hdr = reinterpret_cast<WsHeader*>(base + o_hdr);
  run.d_rm = reinterpret_cast<RunModelDev*>(base + o_rm);
  run.d_md = reinterpret_cast<ModelDev*>(base + o_md);

  // The tables go up as one block that the model keeps, one kernel does the
  // rest of a call's start, and the kernels count in the caller's buffers:
  // one copy and two launches (6 qubits, 256 chains, 32 sweeps: 26.7 us a
  // call; 30.6 with the whole block built on the stack, two clears and two
  // launches; 83.6 with a copy for every table).
  if (cudaMemcpyAsync(base + o_tab, m->tables.data(), tab.bytes, cudaMemcpyHostToDevice, st) != cudaSuccess)
    return PB_ECUDA;
  const uint32_t blocks = std::max(groups, std::min(bins * 8u / 256u, 4u * (uint32_t)sms));
  noalloc_begin_kernel<<<blocks, 256, (size_t)n_words(n, d) * 4, st>>>(run);
  if (cudaGetLastError() != cudaSuccess) return PB_ECUDA;
  const RunModelDev* d_rm = run.d_rm;
  WsHeader* hdr = run.d_hdr;
  const int prod = std::min(ps.prod, plain_launch_producers(n * d, 0, hist_smem ? bins : 0, groups > (uint32_t)sms,
                                                            ps.cons, ps.units, n_sweeps));
  if (n_sweeps > 0 && launch_sweeps_plain(d_rm, 1, groups, n_sweeps, ps.cons, prod, units, maxcol, nc,
                                          false, smem, hdr, st) != cudaSuccess)
    return PB_ECUDA;
  if (!direct && (cudaMemcpyAsync(d_counts, counts, (size_t)bins * 8 * 8, cudaMemcpyDeviceToDevice, st) !=
                      cudaSuccess ||
                  cudaMemcpyAsync(d_totals, totals, 2 * 8, cudaMemcpyDeviceToDevice, st) != cudaSuccess))
    return PB_ECUDA;
  return PB_OK;
}
