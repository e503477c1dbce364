// Internal layout shared by the host compiler, the runtime and the kernels.
#pragma once
#include <cstddef>
#include <algorithm>
#include <cstdint>
#include <vector>

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "pbits.h"

namespace pb {

// Word indices in a chain group's shared-memory image: layer k word q sits
// at k*n + q (k = 0 is the clamped input), followed by a zero word and an
// all-ones word.
__host__ __device__ inline int zero_idx(int n, int d) { return (d + 1) * n; }
__host__ __device__ inline int ones_idx(int n, int d) { return (d + 1) * n + 1; }
__host__ __device__ inline int n_words(int n, int d) { return (d + 1) * n + 2; }

// One p-bit update (16 bytes).  Link i (i < m) demands the value
// r_i = W[a[i]] ^ W[b[i]]; the p-bit's violation count changes by
// v = sum_i (1 - 2 r_i) when it goes 0 -> 1.
struct Desc {
  uint16_t dst;   // word index of the p-bit (k*n + q)
  uint8_t mflag;  // bits 0-1: m (links), bit 2: link 0 is the p-bit's own link,
                  // bit 3: coupled (Metropolis acceptance, see Cpl),
                  // bit 4: general links (a Toffoli's, see GLink),
                  // bit 5: table acceptance (two-qubit tables, see TAcc)
  uint8_t pair;   // threshold pair: 0 (t0,t0) 1 (t1,t1) 2 (t2,t0) 3 (t3,t1)
  uint16_t a[3];
  uint16_t b[3];
};
static_assert(sizeof(Desc) == 16, "Desc must be 16 bytes");

// Record term of one p-bit (16 bytes): violation word W[vd]^W[va]^W[vb]
// (all ZERO when the p-bit has no own link; general-gate runs read
// W[vd]^W[va]^(W[vb]&W[vc]), vc = ONES except on a Toffoli target) and phase
// term w * (W[pa] & W[pb]) with w (bits 0-2) in {0, 1, 2, 4} units of pi/4.
// Plain runs keep the terms in lists: `slot` is the index among the
// violation terms (0xFFFF: none), bits 3-15 of w the index among the phase
// terms of that weight.
struct Rec {
  uint16_t vd, va, vb;
  uint16_t pa, pb;
  uint16_t w;
  uint16_t vc, slot;
};
static_assert(sizeof(Rec) == 16, "Rec must be 16 bytes");

// Coupling of one p-bit to the neighbours of its coupled general gates
// (32 bytes, by p; models with PB_U gates only).  Category c = e_in + 2 e_out
// with e_in = x ^ W[win], e_out = x ^ W[wout] (win / wout = the p-bit's own
// word where it has no such neighbour): a proposed flip is accepted always
// (amask bit c) or when the tag-6 uniform is below A[c].  B: the exact
// sampler's threshold of a coupled output.  flags bit 0: the p-bit has a
// coupling; bit 1: it is the output of a coupled gate; bits 8-31: its index
// among the coupled p-bits.
struct Cpl {
  uint16_t win, wout;
  uint32_t amask;
  uint32_t A[4];
  uint32_t B;
  uint32_t flags;
};
static_assert(sizeof(Cpl) == 32, "Cpl must be 32 bytes");

// General links of a p-bit next to a Toffoli gate (32 bytes, by p): link i
// demands r_i = W[a] ^ (W[b] & W[c]) and counts where W[e] is set (e = ZERO:
// no link; a plain link has c = e = ONES; a control's link through the
// target is active where the other control is 1).  Link 0 is the own link
// when the p-bit has one (its value for the initial path and the exact
// sampler).
struct GLink {
  uint16_t a[3], b[3], c[3], e[3];
  uint32_t pad[2];
};
static_assert(sizeof(GLink) == 32, "GLink must be 32 bytes");

// Metropolis acceptance of a p-bit next to two-qubit table gates (Eq. ET2),
// 544 bytes by p: a proposed flip of a chain is kept when bit idx of amask is
// set or the chain's tag-7 uniform is below thr[idx], idx = the bits of
// W[w[0..5]] at the chain (the in-table's other output and inputs, the
// out-table's other input and outputs; ZERO where absent) | old value << 6.
struct TAcc {
  uint16_t w[6];
  uint16_t pad[2];
  uint32_t amask[4];
  uint32_t thr[128];
};
static_assert(sizeof(TAcc) == 544, "TAcc must be 544 bytes");

// Record entry of a two-qubit table gate (80 bytes): inputs W[wx0], W[wx1],
// outputs W[wy0], W[wy1]; entry idx = x0 + 2 x1 + 4 (y0 + 2 y1): phase
// ph[idx] (2^-32 turn), zero entry (an invalid path) when bit idx of zmask.
struct TRec {
  uint16_t wx0, wx1, wy0, wy1;
  uint32_t zmask;
  uint32_t ph[16];
  uint32_t pad;
};
static_assert(sizeof(TRec) == 80, "TRec must be 80 bytes");

// Phase of one general gate (32 bytes): ph[2 y + x] = arg U_yx in units of
// 2^-32 turn, y = bit W[wout], x = bit W[win] of the chain.
struct UPh {
  uint32_t ph[4];
  uint16_t wout, win;
  uint32_t pad[3];
};
static_assert(sizeof(UPh) == 32, "UPh must be 32 bytes");

// Per-model device header (in the workspace).
struct ModelDev {
  int32_t n, d, nw;        // qubits, layers, words per group image
  int32_t h;
  uint32_t beta;
  uint32_t thr[4];
  int32_t col_off[5];      // descriptor ranges per colour class
  int32_t max_col;         // largest colour class
  int32_t wgt;             // 1: PB_U gates (complex phase sums, couplings)
  int32_t n_ug;            // PB_U gates (UPh entries)
  int32_t n_tr;            // two-qubit table gates (TRec entries)
  double log2z;            // log2 of the estimator scale
  int32_t n_rec[4];        // record terms: own links, phases of weight 1, 2, 4
  int32_t n_cp;            // coupled p-bits (Cpl::flags bit 0)
};

// Per-model run entry (device), one per model of a run.
struct RunModelDev {
  const ModelDev* model;
  const Desc* desc;        // n*d, ordered by colour class
  const Rec* rec;          // n*d
  uint32_t* state;         // groups * d * n words
  unsigned long long* hist;     // n_batches * bins * 8
  unsigned long long* valid;    // n_batches
  unsigned long long* samples;  // n_batches
  const uint32_t* alpha_sorted; // n_alphas (sorted)
  const int32_t* alpha_slot;    // original position of each sorted alpha
  double* amp;             // bins * 3 (re, im, se) output of the amplitude kernel
  int32_t n_alphas;        // 0 = full histogram
  uint32_t bins;
  uint32_t chains, groups, n_batches;
  uint32_t burn_in, record_every;
  uint32_t seed_lo, seed_hi;
  uint32_t group_base;     // first flat group index of this model in a launch
  uint32_t group0;         // global index of group 0 (Philox counter word 0)
  uint32_t hist_smem;      // 1: a CTA counts into shared memory and adds its
                           //    counts to `hist` once at the end of a launch
  int32_t amp_shift;       // amplitude scale 2^{h/2 + amp_shift} (-rank when clamped)
  // output-clamped exact sampler (PB_ELIM_CLAMP; else clamp_tab = nullptr):
  // per p-bit (1 + clamp_mw) words -- an H output's constant bit and its
  // mask over the clamp_nfree free draws
  const uint32_t* clamp_tab;
  int32_t clamp_mw, clamp_nfree, clamp_ok;  // clamp_ok = 0: alpha unreachable
  int32_t pad2;
  // models with PB_U gates (else nullptr): couplings by p, gate phases.
  // Their histogram slots per (batch, bin) are {re (double), im (double),
  // count (u64), compensation of re (double), compensation of im (double),
  // unused...} instead of 8 phase-class counters: the phase sums are
  // compensated (the sum is re + its compensation).
  const Cpl* cpl;
  const UPh* uph;
  const GLink* glk;        // models with Toffoli gates, else nullptr
  const TAcc* tacc;        // models with two-qubit table gates, else nullptr
  const TRec* trec;
  ModelDev md;             // copy of *model
};

// Workspace header at offset 0.
struct WsHeader {
  uint32_t status;         // 0 = ok, else a pb_status code set by a kernel
  uint32_t work_next;      // persistent scheduler counter
  uint32_t sweep0;         // absolute index of the next sweep
  uint32_t periods_left;   // learned runs: move periods still to run in a launch
  uint32_t ctas_done;      // CTAs of the current plain launch counted so far
  uint32_t pad[59];
};

// Dynamic shared memory the sweep and exact-sampler kernels may use per CTA
// (227 KB per block on sm_103a, less their static shared memory).
constexpr size_t kSweepSmemMax = 226 * 1024;
// Threads per sweep CTA in a run with general one-qubit gates (the general
// instantiation is compiled for at most this many).
constexpr int kSweepThreadsWgt = 512;
// Launch bound of the plain sweep kernels: the largest that leaves a thread 88
// registers (65,536 / 736), so that two CTAs of 352 threads share an SM.
// Launches have 608 threads at most (224 consumers, 352 producers and one more
// warp).
constexpr int kSweepThreadsPlain = 736;

// Plain runs work in periods of plain_period sweeps: about `units` p-bit
// updates (1 sweep at least, 16 at most, an even number above 1 because
// sweeps are recorded in pairs).
constexpr __host__ __device__ int plain_period(int npb, int units) {
  const int ps = units / npb;
  return ps < 2 ? 1 : (ps > 16 ? 16 : ps & ~1);
}
// The period of a launch: shorter where n_sweeps are few, a quarter of them so
// that the stages overlap, but no less than (up to eight sweeps of) what 16
// warps start in one task each.
constexpr __host__ __device__ int plain_launch_period(int npb, int units, uint32_t n_sweeps) {
  const int ps = plain_period(npb, units);
  if (ps < 2 || n_sweeps >= 4u * (uint32_t)ps) return ps;
  if (n_sweeps < 2u) return 1;
  const int n = (int)n_sweeps, share = ((n + 3) >> 2) & ~1, all = (n + 1) & ~1;
  int least = (1024 / npb) & ~1;
  least = least > 8 ? 8 : (least < 2 ? 2 : least);
  const int want = share > least ? share : (least < all ? least : all);
  return want < ps ? want : ps;
}
// Shared memory of a CTA: the group image, the snapshots of two periods,
// consumer entries, three periods of comparison words, record lists, the
// period's units, Philox and threshold words, undecided masks, an optional
// histogram.
inline size_t plain_smem_bytes(int n, int d, uint32_t hist_bins, int period_units) {
  const size_t npb = (size_t)n * d, ps = (size_t)plain_period((int)npb, period_units), psp = (ps + 1) & ~(size_t)1;
  const size_t units = (ps * npb + 63) & ~(size_t)63, npad = (npb + 31) & ~(size_t)31;
  const size_t iw = ((size_t)n_words(n, d) + 1 + 3) & ~(size_t)3;
  return (1 + 2 * psp) * iw * 4 + npb * 32 + (3 * units + npad) * 8 +
         (npad + 96 + units) * 4 + (28 + 144 + 4) * 4 + 2 * (units >> 5) * 4 + (size_t)hist_bins * 32;
}

// The same for a model of a general-gate run: 40 bytes a bin where it has
// general gates, and the coupled p-bits' thresholds and entries, the gate
// phases and two periods of acceptance words.
inline size_t general_smem_bytes(int n, int d, bool wgt, int n_cp, int n_ug, uint32_t hist_bins,
                                 int period_units) {
  const size_t npb = (size_t)n * d, ps = (size_t)plain_period((int)npb, period_units);
  const size_t words = wgt ? ((size_t)hist_bins * 10 + 3) & ~(size_t)3 : (size_t)hist_bins * 8;
  return plain_smem_bytes(n, d, 0, period_units) + words * 4 + (size_t)n_cp * 16 +
         (((size_t)n_cp + 1) & ~(size_t)1) * 8 + npb * 16 + (size_t)n_ug * 16 +
         (((size_t)n_ug + 3) & ~(size_t)3) * 4 + 2 * ps * ((size_t)n_cp + 1) * 16;
}

constexpr uint32_t kTagSweep = 0;
constexpr uint32_t kTagInit = 1;
constexpr uint32_t kTagMH = 2;
constexpr uint32_t kTagElim = 4;  // exact sampler's H outputs (tag 3: training rows)
constexpr uint32_t kTagClamp = 5;  // free draws of the output-clamped exact sampler
constexpr uint32_t kTagCouple = 6;  // Metropolis acceptance of coupled p-bits
constexpr uint32_t kTagTable = 7;   // acceptance next to two-qubit tables (per-chain words)

}  // namespace pb

// Compiled model (host side of pb_model).
struct pb_model {
  int n = 0, d = 0;
  uint32_t beta = 0;
  double J = 0.0;
  uint32_t thr[4] = {0, 0, 0, 0};
  int h = 0, M = 0, rank = 0;
  int col_off[5] = {0, 0, 0, 0, 0};
  std::vector<int32_t> colour;        // [d][n]
  std::vector<pb::Desc> desc;         // colour-ordered
  std::vector<pb::Rec> rec;           // by p = (k-1) n + q
  int32_t n_rec[4] = {0, 0, 0, 0};    // lengths of the record lists (ModelDev::n_rec)
  std::vector<uint32_t> init;         // by p: 0xFFFFFFFF = free output, else a | b << 16
  std::vector<pb_gate> gates;
  // general one-qubit gates
  bool wgt = false;                   // any PB_U gate
  int n_u = 0, n_coupled = 0;
  double log2z = 0.0;
  std::vector<pb::Cpl> cpl;           // by p (wgt only)
  int n_cp = 0;                       // coupled p-bits
  std::vector<pb::UPh> uph;           // one per PB_U gate
  int n_ccx = 0;                      // Toffoli gates
  std::vector<pb::GLink> glk;         // by p (Toffoli models only)
  int n_tab = 0;                      // two-qubit table gates
  std::vector<pb::TAcc> tacc;         // by p (table models only)
  std::vector<pb::TRec> trec;         // one per table gate
  std::vector<char> tables;           // models of the no-allocation run: desc, rec and init in one
                                      // block (table_offsets), which a call uploads from here
};

namespace pb {
// Models that the no-allocation run takes, and their tables' places in one
// block.
inline bool noalloc_model(const pb_model& m) { return !m.wgt && m.n <= 16; }
struct TableOffsets {
  size_t desc, rec, init, bytes;
};
inline TableOffsets table_offsets(size_t npb) {
  auto up = [](size_t x) { return (x + 255) & ~(size_t)255; };
  TableOffsets t;
  t.desc = 0;
  t.rec = up(npb * sizeof(Desc));
  t.init = up(t.rec + npb * sizeof(Rec));
  t.bytes = t.init + npb * 4;
  return t;
}

// Philox calls the producers of a general-gate launch make in one colour
// step: 3 per p-bit of the next class (12 planes ahead, two buffers).
inline int sweep_producers_wanted(const pb_model& m) {
  int maxcol = 1;
  for (int c = 0; c < 4; ++c) maxcol = std::max(maxcol, m.col_off[c + 1] - m.col_off[c]);
  return 3 * maxcol;
}
constexpr int kProducersMax = 352;
// Plain runs: default CTA shape and period for `groups` chain groups of
// models of up to npb p-bits (largest colour class maxcol) on a GPU of `sms`
// SMs; smem(units): shared memory of a CTA with that period.
// Two CTAs an SM where there are groups for them and they fit beside the
// histogram that smem counts: the roles of one hide the other's latencies
// (large workload, ms per 1e3 sweeps: 64 consumers + 256 producers, two CTAs,
// 17.2; 64 + 352, one CTA, 21.8, both before the last 0.8 came off the shape
// that was kept).  A histogram of 1024 to 4096 bins takes that room (a CTA with
// one would be alone), so full histograms of 10 to 12 qubits run one CTA an SM
// although two fit with their counts in global memory (20 layers, 65,536
// chains, ms per 1e3 sweeps, one CTA / two CTAs with global counts: 10 qubits
// 6.65 / 5.94, 11 qubits 6.41 / 5.65, 12 qubits, whose counts are in global
// memory either way, 6.72 / 5.96).
// Otherwise one CTA an SM with a consumer per p-bit of the largest class, as
// many producers as a period has tasks for and a longer period, whose tasks
// spread more evenly over the warps (mid, ms per 1e4 sweeps: 4096 units
// 4.73, 2048 4.89; learned 7.00, now 6.85, and 7.90).
struct PlainDefault {
  int cons, prod, units;
};
constexpr int kPlainUnitsOne = 4096, kPlainUnitsTwo = 2048;
template <class Smem>
inline PlainDefault plain_shape(int npb, int maxcol, uint32_t groups, int sms, Smem smem) {
  auto up32 = [](int x) { return ((x + 31) / 32) * 32; };
  PlainDefault s;
  const bool two = groups > (uint32_t)sms && 2 * smem(kPlainUnitsTwo) <= kSweepSmemMax;
  s.units = two || smem(kPlainUnitsOne) > kSweepSmemMax ? kPlainUnitsTwo : kPlainUnitsOne;
  s.cons = std::max(32, std::min(two ? 64 : 224, up32(maxcol)));
  const int ps = plain_period(npb, s.units);
  const int tasks = (ps * npb + 63) / 64 + (ps * npb + 255) / 256 + (ps + 1) / 2;
  s.prod = std::max(32, std::min(two ? 256 : 352, 32 * ((tasks + 1) / 2)));
  return s;
}
// A launch of few sweeps needs less than the run's shape: the units of its
// period, and a producer warp for two tasks of an iteration: the start of a
// period's words, their finish (ncp: coupled p-bits, whose acceptance words
// are tasks too) and its records, which with one period are iterations of
// their own, and which more CTAs an SM overlap where the groups fill the GPU
// (full; with coupled p-bits, whose records take as long as the rest, up to
// three periods).  At least a thread for every p-bit of the tables and for eight bins
// of a histogram in shared memory.
inline int plain_launch_units(int npb, int units, uint32_t n_sweeps) {
  return plain_launch_period(npb, units, n_sweeps) * npb;
}
inline int plain_launch_producers(int npb, int ncp, uint32_t hist_bins, bool full, int cons, int units,
                                  uint32_t n_sweeps) {
  if (n_sweeps >= 4u * (uint32_t)plain_period(npb, units)) return kProducersMax;
  const int ps = std::min<uint32_t>(plain_launch_period(npb, units, n_sweeps), n_sweeps);
  const int start = (ps * npb + 63) / 64, record = (ps + 1) / 2;
  const int finish = (ps * npb + 255) / 256 + (ps * ncp + 31) / 32;
  const bool apart = n_sweeps == (uint32_t)ps || (full && (ncp == 0 || n_sweeps <= 3u * (uint32_t)ps));
  const int tasks = apart ? std::max(std::max(start, finish), record) : start + finish + record;
  const int threads = std::max(npb, (int)hist_bins / 8);
  // (one more warp than producers, which counts where the groups fill the GPU)
  const int warps = full ? (tasks - 1) / 2 : (tasks + 1) / 2;
  return std::max(full ? 0 : 32, std::max(32 * warps, (threads + 31) / 32 * 32 - cons - 32));
}
}  // namespace pb

namespace pb {
// Exact sampler of plain models: a launch counts in shared memory where it adds
// two counts to every counter on average.  Below that, clearing and flushing
// the histogram cost more than counting in global memory (12 qubits, 16,384
// chains, one sample: 58.8 us against 17.6; 2000 samples of 4096 chains: equal).
constexpr __host__ __device__ bool elim_hist_pays(uint32_t bins, uint32_t n_sweeps, uint32_t record_every) {
  return 2ull * (n_sweeps / record_every) >= bins;
}
}  // namespace pb

// Proposal network (host side of pb_mlp): fp32 master weights, Adam state,
// bf16 copies for the tensor cores and the batch buffers of one call.
struct pb_mlp {
  int n = 0, d = 0, H = 0, kin = 0, npad = 0, batch = 0;
  cudaStream_t st = nullptr;
  char* ws = nullptr;
  size_t ws_bytes = 0;
  size_t off_W1 = 0, off_b1 = 0, off_W2 = 0, off_b2 = 0, off_W3 = 0, off_b3 = 0, n_params = 0;
  float *w = nullptr, *m = nullptr, *v = nullptr, *g = nullptr;
  __nv_bfloat16 *W1 = nullptr, *W2 = nullptr, *W3 = nullptr, *W2t = nullptr, *W3t = nullptr;
  // W1, W2 (in K-chunks of 64) and W3 in the tensor cores' canonical K-major
  // shared-memory layout, loaded by the fused kernel with one bulk copy each
  __nv_bfloat16 *W1p = nullptr, *W2p = nullptr, *W3p = nullptr;
  __nv_bfloat16 *X = nullptr, *Xt = nullptr, *H1 = nullptr, *H1t = nullptr, *H2 = nullptr,
                *H2t = nullptr, *dY = nullptr, *dYt = nullptr, *dZ2 = nullptr, *dZ2t = nullptr,
                *dZ1t = nullptr;
  float *logits = nullptr, *target = nullptr, *terms = nullptr, *loss = nullptr;
  // PB_ETIMEOUT once a bounded wait in one of this network's kernels expired
  // (a word of the workspace, zeroed at creation)
  uint32_t* status = nullptr;
  int step = 0;
};

namespace pb {
// Forward of `rows` rows already staged in mlp->X: logits in mlp->logits
// [rows x npad].  Gradients (forward and backward) of the rows staged in
// mlp->X, mlp->Xt (their transpose, [kin x rows]) and mlp->target: mlp->g and
// mlp->loss.
cudaError_t mlp_forward_rows(pb_mlp* p, int rows);
cudaError_t mlp_gradient_rows(pb_mlp* p, int rows);
cudaError_t mlp_adam_step(pb_mlp* p, float lr);
cudaError_t mlp_prepare();
cudaError_t mlp_forward_fused(pb_mlp* p, int rows);
cudaError_t mlp_fused_logq(pb_mlp* p, const uint32_t* P, uint32_t beta, int chains, int k, float* lq,
                           cudaStream_t st);
cudaError_t mlp_fused_sample(pb_mlp* p, const uint32_t* P, uint32_t* Pn, uint32_t beta, int chains,
                             int k, int j, int jlast, float* lqf, uint32_t k0, uint32_t k1,
                             const uint32_t* move_dev, uint32_t group0, cudaStream_t st);
cudaError_t mlp_fused_logq_dev(pb_mlp* p, const uint32_t* P, uint32_t beta, int chains,
                               const int* k_dev, float* lq, cudaStream_t st);
cudaError_t mlp_fused_sample_dev(pb_mlp* p, const uint32_t* P, uint32_t* Pn, uint32_t beta,
                                 int chains, const int* k_dev, float* lqf, uint32_t k0, uint32_t k1,
                                 const uint32_t* move_dev, uint32_t group0, cudaStream_t st);

// Learned-proposal moves on one model (learned.cu): the run's chain words,
// the network and a device region of mh_region_bytes(d, groups) bytes
// (256-byte aligned) holding the per-chain words, log q terms, the move
// counters and the layer table.
struct MhCtx {
  const pb_model* model = nullptr;
  pb_mlp* mlp = nullptr;
  uint32_t* state = nullptr;  // [group][k-1][q] chain words of the model
  uint32_t chains = 0, groups = 0, group0 = 0;
  uint64_t seed = 0;
  char* ws = nullptr;
  // a second stream and two events: the log q of the current suffix runs
  // beside the proposal draw (mh_ctx_open / mh_ctx_close)
  cudaStream_t side = nullptr;
  cudaEvent_t fork = nullptr, join = nullptr;
};
// Counters at the start of a move region: proposals accepted, moves done.
struct MhCounters {
  unsigned long long accepted;
  uint32_t moves;
  int32_t k;  // suffix start of the current move
};
size_t mh_region_bytes(int d, uint32_t groups);
cudaError_t mh_ctx_open(MhCtx& c);
void mh_ctx_close(MhCtx& c);
// True when the network takes the fused inference kernel (k_in <= 96,
// n <= 32): then a move draws its suffix start on the device.
bool mh_fused(const pb_mlp* mlp);
// Zeroes the region and uploads the layer table (synchronous on st).
cudaError_t mh_region_init(const MhCtx& c, cudaStream_t st);
// Enqueues one move with its suffix start drawn on the device from the seed
// and the move counter (fused networks; capturable, no host synchronisation).
// hdr != nullptr: the move also counts down a period of the graph loop `loop`.
cudaError_t mh_enqueue_move_dev(const MhCtx& c, cudaStream_t st, WsHeader* hdr = nullptr,
                                cudaGraphConditionalHandle loop = 0);

// What the learned-proposal code needs to know about one model of a run.
struct RunView {
  cudaStream_t st;
  uint32_t* state;  // [group][k-1][q] chain words
  const pb_model* model;
  uint32_t chains, groups, group0;
  uint64_t seed;
};
int run_view(const pb_run* r, int model, RunView* out);
}  // namespace pb
