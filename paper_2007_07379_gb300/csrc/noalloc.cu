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
#include <cstring>
#include <mutex>

#include "pb_internal.h"

namespace pb {
cudaError_t launch_init(const RunModelDev* d_rm, int n_models, uint32_t total_groups,
                        const uint32_t* const* d_init_tabs, size_t smem_bytes, WsHeader* hdr,
                        cudaStream_t st);
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
  // a CUDA graph (the copies would point at this call's host buffers).
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
  const size_t o_iptr = off; off = align256(off + sizeof(uint32_t*));
  const size_t o_md = off; off = align256(off + sizeof(ModelDev));
  const size_t o_desc = off; off = align256(off + npb * sizeof(Desc));
  const size_t o_rec = off; off = align256(off + npb * sizeof(Rec));
  const size_t o_init = off; off = align256(off + npb * 4);
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
  const size_t smem = smem_for(ps.units);
  if (smem > kSweepSmemMax) return PB_ERANGE;

  ModelDev md{};
  md.n = n;
  md.d = d;
  md.nw = n_words(n, d);
  md.h = m->h;
  md.beta = m->beta;
  for (int k = 0; k < 4; ++k) md.thr[k] = m->thr[k];
  for (int k = 0; k < 5; ++k) md.col_off[k] = m->col_off[k];
  md.max_col = maxcol;
  for (int k = 0; k < 4; ++k) md.n_rec[k] = m->n_rec[k];

  RunModelDev r{};
  r.model = reinterpret_cast<const ModelDev*>(base + o_md);
  r.md = md;
  r.desc = reinterpret_cast<const Desc*>(base + o_desc);
  r.rec = reinterpret_cast<const Rec*>(base + o_rec);
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
  const uint32_t* init_tab = reinterpret_cast<const uint32_t*>(base + o_init);

  // Everything below the chain words -- a cleared header (sweep index 0,
  // status 0), the run entry and the tables -- goes up as one block from the
  // stack, and the kernels count in the caller's buffers: two clears, one
  // copy and two kernels (eleven operations, each a few microseconds of a
  // short call, when every table had its own copy and the counters theirs).
  constexpr size_t kUpMax = 40 * 1024;  // n <= 16, d <= 64: at most 1024 p-bits
  alignas(16) char up[kUpMax];
  if (o_state > kUpMax) return PB_ERANGE;
  std::memset(up, 0, o_state);
  std::memcpy(up + o_md, &md, sizeof md);
  std::memcpy(up + o_rm, &r, sizeof r);
  std::memcpy(up + o_iptr, &init_tab, sizeof init_tab);
  std::memcpy(up + o_desc, m->desc.data(), npb * sizeof(Desc));
  std::memcpy(up + o_rec, m->rec.data(), npb * sizeof(Rec));
  std::memcpy(up + o_init, m->init.data(), npb * 4);
  if (cudaMemcpyAsync(base, up, o_init + npb * 4, cudaMemcpyHostToDevice, st) != cudaSuccess ||
      cudaMemsetAsync(counts, 0, (size_t)bins * 8 * 8, st) != cudaSuccess ||
      cudaMemsetAsync(totals, 0, 2 * 8, st) != cudaSuccess)
    return PB_ECUDA;
  const RunModelDev* d_rm = reinterpret_cast<const RunModelDev*>(base + o_rm);
  WsHeader* hdr = reinterpret_cast<WsHeader*>(base + o_hdr);
  if (launch_init(d_rm, 1, groups, reinterpret_cast<const uint32_t* const*>(base + o_iptr),
                  (size_t)n_words(n, d) * 4, hdr, st) != cudaSuccess)
    return PB_ECUDA;
  if (n_sweeps > 0 && launch_sweeps_plain(d_rm, 1, groups, n_sweeps, ps.cons, ps.prod, ps.units, maxcol,
                                          nc, false, smem, hdr, st) != cudaSuccess)
    return PB_ECUDA;
  if (!direct && (cudaMemcpyAsync(d_counts, counts, (size_t)bins * 8 * 8, cudaMemcpyDeviceToDevice, st) !=
                      cudaSuccess ||
                  cudaMemcpyAsync(d_totals, totals, 2 * 8, cudaMemcpyDeviceToDevice, st) != cudaSuccess))
    return PB_ECUDA;
  return PB_OK;
}
