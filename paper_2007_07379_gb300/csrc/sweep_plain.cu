// Gibbs sweeps of plain (Clifford+T and X) models (sm_103a).
//
// The heat-bath draw of p-bit p at sweep t replaces its 32 chains' word by
//   neg ^ (sel ? A : B),   A = [u < tA],  B = [u < tB],
// with tA, tB the two thresholds the p-bit's link count m allows (m = 0:
// t0, t0; 1: t1, t1; 2: t2, t0; 3: t3, t1), sel the lanes whose links agree
// and neg the majority of the demanded values.  A and B depend on the random
// numbers only, not on the chains, so they are made ahead of the sweeps that
// use them; what is left on the chains' critical path is six link loads,
// eight logic operations and a store per colour class.
//
// Work of one CTA (one group of 32 chains at a time), in periods of `ps`
// sweeps separated by one CTA barrier.  In period t
//   consumers  redraw the sweeps of period t, class by class (a barrier of
//              the consumer warps alone between classes),
//   workers    take tasks from a list: finish the words of period t + 1 whose
//              lanes planes 0..7 left undecided, record the sweeps of period
//              t - 1 (two a task) from the snapshots the consumers wrote,
//              and make the words of period t + 2 from planes 0..7.
// A word is undecided after 8 planes with probability about 1 - (1 - 2^-8)^32
// = 12 %; those units are gathered from the tasks' masks and finished densely,
// 32 to a warp, so a p-bit costs 2.2 Philox calls on average instead of the 4
// that a fixed number of planes needs to be nearly always enough.
//
// What bounds it: issue slots, and where one CTA has an SM to itself the
// consumers' chain beside them.  A word update (32 chains) costs about 8 warp
// instructions' lanes, two Philox calls being 40 % of them (a call's multiplies
// alone take 17 cycles a warp and SM), and 53-59 % of the issue slots are used:
// an SM's ~16 warps do not hide every latency.  On mid a colour step is about
// 323 cycles; on tiny (one warp of consumers) the chain of loads, logic and
// barrier is 155 cycles a step and nothing else counts.  Measured
// against the kernel this replaced (16 planes for every p-bit, the comparison
// on the consumers' path, one recorder warp, a CTA barrier per class; ms):
// mid (12 qubits, 20 layers, 4096 chains, 1e4 sweeps) 13.0 -> 4.7, large (24
// qubits, 32 layers, 65,536 chains, 1e3 sweeps) 41.9 -> 16.4, tiny (1e4
// sweeps) 9.0 -> 1.6, 256 batched circuits (300 sweeps) 15.2 -> 4.35; with
// general one-qubit gates, whose acceptance words are made ahead as well,
// general_mid (35 coupled gates, 4096 chains, 2e3 sweeps) 6.63 -> 3.1: there
// 35 % of the slots are used, the other warps waiting at a period's end for
// the last phase records (sincospif and FP64 shared atomics).
#include <cuda_runtime.h>

#include <type_traits>

#include "pb_internal.h"
#include "philox.cuh"
#include "sweep_common.cuh"

namespace pb {
namespace {

struct PlainShape {
  int cons, work, units;  // consumer threads, worker warps, units of a period (plain_period)
};

// Four planes (Philox output grp) of [u < t], most significant first.
__device__ __forceinline__ void compare_planes(uint32_t& lt, uint32_t& eq, uint32_t t, uint4 r,
                                               uint32_t grp) {
  const uint32_t R[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
  for (uint32_t w = 0; w < 4u; ++w) {
    const uint32_t T = (uint32_t)((int32_t)(t << (grp * 4u + w)) >> 31);
    lt |= eq & ~R[w] & T;
    eq &= ~(R[w] ^ T);
  }
}
// Eight planes against the threshold's bits as masks T: lt the lanes below,
// eq the lanes equal.  Least significant plane first, a plane's effect on lt
// is one three-input majority.
__device__ __forceinline__ void compare8(uint32_t& lt, uint32_t& eq, const uint32_t (&T)[8],
                                         uint4 r, uint4 s) {
  const uint32_t R[8] = {r.x, r.y, r.z, r.w, s.x, s.y, s.z, s.w};
  lt = 0u;
  eq = ~0u;
#pragma unroll
  for (int w = 7; w >= 0; --w) {
    lt = (~R[w] & (T[w] | lt)) | (T[w] & lt);
    eq &= ~(R[w] ^ T[w]);
  }
}

// Philox outputs j and j + 1 (j = 0 or 2) at counter (g, sw, p, .) of one
// group and key.  The two calls share the products of p and of round 1's x,
// and round 1's other product depends on the group alone: 33 of the 40
// multiplies of two calls are left.  The words that do not change within a
// launch lie in shared memory (philox_consts), loaded once per period.
struct PhiloxPair {
  uint32_t a[2], b[2], k00, c, k12, K0[7], K1[7];
};
constexpr int kPhiloxWords = 28;  // a, b of j = 0..3, k00, c, k12, 1 unused, K0[3..9], 1, K1[3..9], 1
__device__ void philox_consts(uint32_t* out, uint32_t g, uint32_t k0, uint32_t k1) {
  const uint32_t W0 = 0x9E3779B9u, W1 = 0xBB67AE85u;
  const uint64_t p0 = (uint64_t)0xD2511F53u * g;
#pragma unroll
  for (uint32_t j = 0; j < 4u; ++j) {
    const uint64_t q1 = (uint64_t)0xCD9E8D57u * ((uint32_t)(p0 >> 32) ^ j ^ k1);
    out[2 * (j & 2u) + (j & 1u)] = (uint32_t)(q1 >> 32) ^ (k0 + W0);          // a_j
    out[2 * (j & 2u) + 2 + (j & 1u)] = (uint32_t)q1 ^ (k0 + 2u * W0);         // b_j
  }
  out[8] = k0;
  out[9] = (uint32_t)p0 ^ (k1 + W1);
  out[10] = k1 + 2u * W1;
  out[11] = 0u;
#pragma unroll
  for (uint32_t r = 3; r < 10u; ++r) {
    out[12 + r - 3] = k0 + r * W0;
    out[20 + r - 3] = k1 + r * W1;
  }
}
__device__ __forceinline__ void philox_pair(const PhiloxPair& P, uint32_t sw, uint32_t p, uint4& ra,
                                            uint4& rb) {
  const uint64_t p1 = (uint64_t)0xCD9E8D57u * p;
  const uint64_t s0 = (uint64_t)0xD2511F53u * ((uint32_t)(p1 >> 32) ^ sw ^ P.k00);
  const uint64_t s1 = (uint64_t)0xCD9E8D57u * ((uint32_t)(s0 >> 32) ^ P.c);
  uint4 o[2];
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const uint64_t q0 = (uint64_t)0xD2511F53u * (P.a[j] ^ (uint32_t)p1);
    uint4 c = make_uint4((uint32_t)(s1 >> 32) ^ P.b[j], (uint32_t)s1,
                         (uint32_t)(q0 >> 32) ^ (uint32_t)s0 ^ P.k12, (uint32_t)q0);
#pragma unroll
    for (int r = 0; r < 7; ++r) {
      const uint64_t u0 = (uint64_t)0xD2511F53u * c.x;
      const uint64_t u1 = (uint64_t)0xCD9E8D57u * c.z;
      c = make_uint4((uint32_t)(u1 >> 32) ^ c.y ^ P.K0[r], (uint32_t)u1,
                     (uint32_t)(u0 >> 32) ^ c.w ^ P.K1[r], (uint32_t)u0);
    }
    o[j] = c;
  }
  ra = o[0];
  rb = o[1];
}

// A value the compiler keeps in a register: addresses that depend on the
// model's sizes are otherwise recomputed from them at every use, on the
// uniform datapath, which takes issue slots like any other instruction (a
// quarter of the kernel's).
__device__ __forceinline__ uint32_t keep(uint32_t x) {
  uint32_t y;
  asm volatile("mov.u32 %0, %1;" : "=r"(y) : "r"(x));
  return y;
}

// New word of a p-bit from its links' demands and its two comparison words.
__device__ __forceinline__ uint32_t redraw(uint32_t r0, uint32_t r1, uint32_t r2, uint32_t M2,
                                           uint2 ab) {
  const uint32_t neg = (r0 & r1) | (r2 & (r0 | r1));
  const uint32_t sel = ~(r0 ^ r1) & (~(r1 ^ r2) | M2);
  return neg ^ ((sel & ab.x) | (~sel & ab.y));
}

// A launch is one kernel: the CTA that is the last to have read the sweep
// index (counted in ctas_done) advances it for the next launch.
__device__ void advance_sweeps(WsHeader* hdr, uint32_t sweep0, uint32_t n_sweeps) {
  if (threadIdx.x + 1u == blockDim.x && atomicAdd(&hdr->ctas_done, 1u) == gridDim.x - 1u) {
    hdr->ctas_done = 0u;
    hdr->sweep0 = sweep0 + n_sweeps;
  }
}

// MULTI: some colour class is larger than the consumers.  ADV: the CTA counts
// itself among those that have read the sweep index.
template <int NC, bool MULTI, bool ADV, bool WGT>
__device__ void run_group_plain(const RunModelDev& rm_g, uint32_t g, uint32_t sweep0,
                                uint32_t n_sweeps, PlainShape sh, uint32_t* smem, WsHeader* hdr) {
  const RunModelDev rm = rm_g;
  const ModelDev& md = rm_g.md;  // (the run entry's copy: one dependent load less)
  // (a value read from lane 0 is known to be warp-uniform: branches and
  // loops on it need no convergence code)
  auto uni = [](auto x) { return __shfl_sync(0xffffffffu, x, 0); };
  const int n = uni(md.n), d = uni(md.d), nw = uni(md.nw);
  const int npb = n * d;
  const int tid = threadIdx.x, T = blockDim.x;
  const int lane = tid & 31, nwarps = T >> 5, warp = uni(tid >> 5);
  const int cw = sh.cons >> 5;
  const int iw = image_words(n, d);
  // sweeps of a period (the sizes in shared memory stay within those of a
  // long launch's period)
  const int ps = plain_launch_period(npb, sh.units, n_sweeps);
  // units (p-bit updates) of a full period, padded to whole tasks: the
  // padding's words are made like the others and never read
  const int punits = (ps * npb + 63) & ~63;

  // ---- shared memory (plain_smem_bytes)
  uint32_t* W = smem;
  // snapshots of the sweeps of two periods, in pairs: word w of sweep i at
  // pair i / 2, [w][i mod 2], so that one load reads a word of both sweeps
  uint32_t* snap = W + iw;
  const int psp = (ps + 1) & ~1;  // sweeps of a period, whole pairs
  // consumer entries in colour order, addresses in the shared window: link
  // pairs 0 and 1; link pair 2, the p-bit's own word, ~0 where it has 2 links
  uint4* sent = reinterpret_cast<uint4*>(snap + 2 * psp * iw);
  uint2* ring = reinterpret_cast<uint2*>(sent + 2 * npb);  // 3 periods of (A, B) words
  // record lists (byte offsets within a pair of snapshots), each padded to whole warps
  // with the ZERO word: links {own, a, b}, then phases {a, b} of weight 1,
  // 2 and 4
  const int npad = (npb + 31) & ~31;
  uint2* svio = ring + 3 * punits;
  uint32_t* sph = reinterpret_cast<uint32_t*>(svio + npad);
  // units of a period: p | m << 12 | sweep of the period << 16 | [m odd] <<
  // 30 | [m > 0] << 31
  uint32_t* sinfo = sph + npad + 96;
  uint32_t* sphx = sinfo + punits;      // philox_consts
  // bits 31..16 of the thresholds tA and tB as masks by link count (rows of
  // 36 words: 16 and 16, no bank conflicts between rows)
  uint32_t* stm = sphx + kPhiloxWords;
  uint32_t* cnt = stm + 144;  // 3 task counters
  uint32_t* smask = cnt + 4;  // 2 periods: the undecided units of each 32
  uint32_t* after = smask + 2 * (punits >> 5);
  // general-gate runs: acceptance thresholds and {p, always-mask} of the
  // coupled p-bits, per p-bit (colour order) the addresses of its coupled
  // neighbours and the offset of its acceptance words, gate phases with the
  // offsets of their words, and two periods of acceptance words (per sweep
  // one entry a coupled p-bit and a last one that accepts everything)
  const bool wgt_m = WGT && rm.cpl != nullptr;
  const int ncp = wgt_m ? uni(md.n_cp) : 0, nug = wgt_m ? uni(md.n_ug) : 0;
  uint4* sthr = reinterpret_cast<uint4*>(after);
  uint2* scp = reinterpret_cast<uint2*>(sthr + ncp);
  uint4* snb = reinterpret_cast<uint4*>(scp + ((ncp + 1) & ~1));
  uint4* suph = snb + npb;
  uint32_t* suof = reinterpret_cast<uint32_t*>(suph + nug);
  uint4* sacc = reinterpret_cast<uint4*>(suof + ((nug + 3) & ~3));
  if (WGT) after = reinterpret_cast<uint32_t*>(sacc + 2 * ps * (ncp + 1));
  const uint32_t hist_words = wgt_m ? (rm.bins * 10u + 3u) & ~3u : rm.bins * 8u;
  uint32_t* shist = rm.hist_smem ? after : nullptr;

  // ---- load the group image and the tables
  const uint32_t w_addr = (uint32_t)__cvta_generic_to_shared(W);
  const uint32_t* gstate = rm.state + (size_t)g * npb;
#pragma unroll 1
  for (int i = tid; i < iw; i += T) {
    uint32_t v;
    if (i < n) v = ((md.beta >> i) & 1u) ? ~0u : 0u;  // clamped input layer
    else if (i < (d + 1) * n) v = gstate[i - n];
    else v = (i == zero_idx(n, d)) ? 0u : ~0u;
    W[i] = v;
  }
  // the snapshots' words that no sweep writes: the input layer, ZERO, ONES
#pragma unroll 1
  for (int k = tid; k < (n + 2) * psp; k += T) {
    const int s = k / (n + 2), i = k - s * (n + 2);
    const uint32_t v = i < n ? (((md.beta >> i) & 1u) ? ~0u : 0u) : (i == n ? 0u : ~0u);
    reinterpret_cast<uint2*>(snap)[s * iw + (i < n ? i : i + d * n)] = make_uint2(v, v);
  }
  if (shist) {
#pragma unroll 1
    for (uint32_t i = tid; i < hist_words; i += T) shist[i] = 0u;
  }
  const uint32_t thr0 = md.thr[0], thr1 = md.thr[1], thr2 = md.thr[2], thr3 = md.thr[3];
  const uint32_t k0 = rm.seed_lo, k1 = rm.seed_hi;
  const uint32_t gglob = g + rm.group0;
  if (tid < 4) cnt[tid] = 0u;
  if (tid == T - 1) philox_consts(sphx, gglob, k0, k1);
#pragma unroll 1
  for (int i = tid; i < 128; i += T) {
    const int m = i >> 5, j = i & 15;
    const uint32_t t = (i & 16) ? thr_b(m, thr0, thr1) : thr_a(m, thr0, thr1, thr2, thr3);
    stm[m * 36 + (i & 31)] = (uint32_t)((int32_t)(t << j) >> 31);
  }
  const uint32_t zoff = 8u * (uint32_t)zero_idx(n, d);
  // record lists: lengths from the model (never more than there are p-bits)
  int n_rec[4];
#pragma unroll
  for (int l = 0; l < 4; ++l) n_rec[l] = min(max(uni(md.n_rec[l]), 0), npb);
  const int n_vio = n_rec[0], n_ph1 = (n_rec[1] + 31) & ~31;
  const int n_ph2 = min((n_rec[2] + 31) & ~31, npad + 64 - n_ph1);
  const int n_ph4 = min(n_rec[3], npad + 96 - n_ph1 - n_ph2);
  {  // the lists' padding
    const uint32_t zz = zoff | zoff << 16;
    if (n_vio + tid < npad) svio[n_vio + tid] = make_uint2(zz, zoff);
    if (n_rec[1] + tid < n_ph1) sph[n_rec[1] + tid] = zz;
    if (n_rec[2] + tid < n_ph2) sph[n_ph1 + n_rec[2] + tid] = zz;
    if (tid < 32 && n_ph1 + n_ph2 + n_ph4 + tid < npad + 96) sph[n_ph1 + n_ph2 + n_ph4 + tid] = zz;
  }
#pragma unroll 1
  for (int i = tid; i < npb; i += T) {
    Desc D = rm.desc[i];
    const Rec R = rm.rec[i];
    bool ok = D.dst >= n && D.dst < nw;
#pragma unroll
    for (int l = 0; l < 3; ++l) ok = ok && D.a[l] < nw && D.b[l] < nw;
    // Toffoli and table p-bits: sweep_kernel; coupled ones: general-gate runs
    if (D.mflag & (wgt_m ? 0x30 : 0x38)) ok = false;
    if (!ok) {  // never write through a bad index: the entry redraws the scratch word
      set_status(hdr, PB_EINVAL);
      D.dst = (uint16_t)nw;
      D.mflag = 0;
#pragma unroll
      for (int l = 0; l < 3; ++l) D.a[l] = D.b[l] = (uint16_t)zero_idx(n, d);
    }
    // three-link form: m=0: 0,0,0  m=1: r0,r0,0  m=2: r0,r1,0  m=3: r0,r1,r2
    const int m = D.mflag & 3;
    if (m == 1) { D.a[1] = D.a[0]; D.b[1] = D.b[0]; }
    auto at = [&](uint32_t w) { return w_addr + 4u * w; };
    sent[i] = make_uint4(at(D.a[0]), at(D.b[0]), at(D.a[1]), at(D.b[1]));
    sent[npb + i] = make_uint4(at(D.a[2]), at(D.b[2]), at(D.dst), m == 2 ? ~0u : 0u);
    if constexpr (WGT) {
      uint4 nb = make_uint4(at(D.dst), at(D.dst), 16u * (uint32_t)ncp, 0u);
      if (ok && wgt_m) {
        const uint32_t p = (uint32_t)(D.dst - n);
        const Cpl C = rm.cpl[p];
        const uint32_t a = C.flags >> 8;
        if (C.flags & 1u) {
          if (C.win >= nw || C.wout >= nw || a >= (uint32_t)ncp) {
            set_status(hdr, PB_EINVAL);
          } else {
            nb = make_uint4(at(C.win), at(C.wout), 16u * a, 1u);
            sthr[a] = make_uint4(C.A[0], C.A[1], C.A[2], C.A[3]);
            scp[a] = make_uint2(p, C.amask);
          }
        }
      }
      snb[i] = nb;
    }
    const uint32_t x = (uint32_t)(D.dst - n) | (uint32_t)m << 12 | (uint32_t)(m & 1) << 30 |
                       (m ? 1u << 31 : 0u);
#pragma unroll 1
    for (int u = i, k = 0; u < punits; u += npb, ++k) sinfo[u] = x | (uint32_t)k << 16;
    // record terms, at their slots in the lists (pb_compile)
    const int kv = R.slot, kp = R.w >> 3, w = R.w & 7;
    if (R.vd >= nw || R.va >= nw || R.vb >= nw || R.pa >= nw || R.pb >= nw ||
        (kv != 0xFFFF && kv >= n_vio) || (w && kp >= (w == 1 ? n_rec[1] : w == 2 ? n_rec[2] : n_ph4))) {
      set_status(hdr, PB_EINVAL);
    } else {
      if (kv != 0xFFFF) svio[kv] = make_uint2(8u * R.vd | (8u * R.va) << 16, 8u * R.vb);
      if (w) sph[(w == 1 ? 0 : w == 2 ? n_ph1 : n_ph1 + n_ph2) + kp] = 8u * R.pa | (8u * R.pb) << 16;
    }
  }
  if constexpr (WGT) {
#pragma unroll 1
    for (int i = tid; i < nug; i += T) {
      const UPh U = rm.uph[i];
      const bool ok = U.wout < nw && U.win < nw;
      if (!ok) set_status(hdr, PB_EINVAL);
      suph[i] = ok ? make_uint4(U.ph[0], U.ph[1], U.ph[2], U.ph[3]) : make_uint4(0u, 0u, 0u, 0u);
      suof[i] = ok ? 8u * U.wout | (8u * U.win) << 16 : zoff | zoff << 16;
    }
#pragma unroll 1
    for (int i = tid; i < 2 * ps; i += T) sacc[i * (ncp + 1) + ncp] = make_uint4(~0u, ~0u, ~0u, ~0u);
  }
  __syncthreads();
  if (ADV) advance_sweeps(hdr, sweep0, n_sweeps);

  const uint32_t batch = g % rm.n_batches;
  // planes 0..7 of thr1 (and of thr2 and thr3, <= thr1) hold no one bit
  const bool z1 = uni(thr1) < (1u << 24);
  const uint32_t n_periods = (n_sweeps + (uint32_t)ps - 1u) / (uint32_t)ps;
  auto sweeps_of = [&](uint32_t q) {
    const uint32_t left = n_sweeps - q * (uint32_t)ps;
    return left < (uint32_t)ps ? left : (uint32_t)ps;
  };
  // The launch's Philox words of outputs j, j + 1.
  const uint32_t sphx_addr = keep((uint32_t)__cvta_generic_to_shared(sphx));
  const uint32_t stm_addr = keep((uint32_t)__cvta_generic_to_shared(stm));
  auto load_keys = [&](PhiloxPair& P, uint32_t j) {
    const uint4 ab = lds4(sphx_addr + 8u * j);
    P.a[0] = ab.x; P.a[1] = ab.y; P.b[0] = ab.z; P.b[1] = ab.w;
    const uint4 h = lds4(sphx_addr + 32u);
    P.k00 = h.x; P.c = h.y; P.k12 = h.z;
    const uint4 x = lds4(sphx_addr + 48u), y = lds4(sphx_addr + 64u), z = lds4(sphx_addr + 80u),
                w = lds4(sphx_addr + 96u);
    P.K0[0] = x.x; P.K0[1] = x.y; P.K0[2] = x.z; P.K0[3] = x.w;
    P.K0[4] = y.x; P.K0[5] = y.y; P.K0[6] = y.z;
    P.K1[0] = z.x; P.K1[1] = z.y; P.K1[2] = z.z; P.K1[3] = z.w;
    P.K1[4] = w.x; P.K1[5] = w.y; P.K1[6] = w.z;
  };
  // Eight masks of a threshold: link count m, h = 0 (tA) or 1 (tB), planes
  // 8 o .. 8 o + 7.
  auto load_masks = [&](uint32_t (&Tm)[8], uint32_t m, uint32_t h, uint32_t o) {
    const uint32_t at = stm_addr + 144u * m + 64u * h + 32u * o;
    const uint4 x = lds4(at), y = lds4(at + 16u);
    Tm[0] = x.x; Tm[1] = x.y; Tm[2] = x.z; Tm[3] = x.w;
    Tm[4] = y.x; Tm[5] = y.y; Tm[6] = y.z; Tm[7] = y.w;
  };

  const uint32_t ring_addr = keep((uint32_t)__cvta_generic_to_shared(ring));
  const uint32_t sent_addr = keep((uint32_t)__cvta_generic_to_shared(sent));
  const uint32_t sinfo_addr = keep((uint32_t)__cvta_generic_to_shared(sinfo) + 4u * (uint32_t)lane);

  // Words of the 64 units from 64 c on of a period whose first sweep is sw0,
  // from planes 0..7 (unit idx: p-bit idx mod npb, in colour order, of the
  // period's sweep idx / npb), two units a lane so that four Philox chains
  // interleave.  When the thresholds' top bits are zero (z1: J above 5.5)
  // the equal lanes are those that drew eight zeros and no lane is below:
  // the word itself holds the equal lanes.  Otherwise the partial comparison
  // is stored and redone by finish_units.
  // (words: shared address of the period's words; masks: of its masks)
  auto start_units = [&](const PhiloxPair& P, uint32_t sw0, uint32_t c, uint32_t words,
                         uint32_t masks) {
    const uint32_t xa = sinfo_addr + 256u * c;
    const uint32_t X[2] = {lds(xa), lds(xa + 128u)};
    words += 512u * c + 8u * (uint32_t)lane;
    uint4 RR[2][2];
#pragma unroll
    for (int h = 0; h < 2; ++h)
      philox_pair(P, sw0 + ((X[h] >> 16) & 0x1Fu), X[h] & 0xFFFu, RR[h][0], RR[h][1]);
#pragma unroll
    for (uint32_t h = 0; h < 2u; ++h) {
      const uint32_t x = X[h];
      const uint4 R0 = RR[h][0], R1 = RR[h][1];
      const uint32_t linked = (uint32_t)((int32_t)x >> 31), odd = (uint32_t)((int32_t)(x << 1) >> 31);
      const uint32_t b0 = ~R0.x;  // [u < 2^31]
      uint2 ab;
      uint32_t open;
      if (z1) {
        const uint32_t Z = ~(R0.x | R0.y | R0.z | R0.w | R1.x | R1.y | R1.z | R1.w);
        ab.x = (linked & Z) | (~linked & b0);
        ab.y = (odd & Z) | (~odd & b0);
        open = linked & Z;
      } else {
        uint32_t Tm[8], eqA, eqB;
        const uint32_t m = (x >> 12) & 3u;
        load_masks(Tm, m, 0u, 0u);
        compare8(ab.x, eqA, Tm, R0, R1);
        load_masks(Tm, m, 1u, 0u);
        compare8(ab.y, eqB, Tm, R0, R1);
        // (t0 = 2^31 is decided by plane 0)
        open = (linked & eqA) | (odd & eqB);
      }
      asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(words + 256u * h), "r"(ab.x), "r"(ab.y)
                   : "memory");
      const unsigned mask = __ballot_sync(0xffffffffu, open != 0u);
      if (lane == 0) sts(masks + 8u * c + 4u * h, mask);
    }
  };
  // The undecided units among the 256 from 256 f on of period q (ns: its
  // units / 32): 32 of them to a pass, planes 8..15, then the rest while a
  // lane is undecided.
  auto finish_units = [&](uint32_t q, uint32_t f, uint32_t ns) {
    PhiloxPair P;
    const uint32_t c0 = 8u * f + (uint32_t)lane;
    const uint32_t mk = lane < 8 && c0 < ns ? smask[(q & 1u) * (uint32_t)(punits >> 5) + c0] : 0u;
    uint32_t incl = (uint32_t)__popc(mk);  // running count over the lanes' masks
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    const uint32_t total = __shfl_sync(0xffffffffu, incl, 7);
#pragma unroll 1
    for (uint32_t e0 = 0; e0 < total; e0 += 32u) {
      const uint32_t e = e0 + (uint32_t)lane;
      // the mask holding the e-th undecided unit, and its bit
      uint32_t j = __shfl_sync(0xffffffffu, incl, 3) <= e ? 4u : 0u;
      j += __shfl_sync(0xffffffffu, incl, (int)j + 1) <= e ? 2u : 0u;
      j += __shfl_sync(0xffffffffu, incl, (int)j) <= e ? 1u : 0u;
      uint32_t w = __shfl_sync(0xffffffffu, mk, (int)j);
      uint32_t r = e - (__shfl_sync(0xffffffffu, incl, (int)j) - (uint32_t)__popc(w)), bit = 0u;
#pragma unroll
      for (uint32_t h = 16u; h > 0u; h >>= 1) {
        const uint32_t c = (uint32_t)__popc(w & ((1u << h) - 1u));
        if (r >= c) { r -= c; w >>= h; bit += h; }
      }
      if (e < total) {
        const uint32_t idx = 32u * (8u * f + j) + bit;
        const uint32_t x = sinfo[idx], p = x & 0xFFFu;
        const int m = (int)((x >> 12) & 3u);
        const uint32_t sw = sweep0 + q * (uint32_t)ps + ((x >> 16) & 0x1Fu);
        uint2* slot = &ring[(q % 3u) * (uint32_t)punits + idx];
        uint32_t ltA = 0u, eqA, ltB, eqB, l8, e8, Tm[8];
        if (z1) {
          const uint2 ab = *slot;
          eqA = ab.x;
          ltB = (m & 1) ? 0u : ab.y;
          eqB = (m & 1) ? ab.y : 0u;
        } else {
          uint4 R0, R1;
          load_keys(P, 0u);
          philox_pair(P, sw, p, R0, R1);
          load_masks(Tm, (uint32_t)m, 0u, 0u);
          compare8(ltA, eqA, Tm, R0, R1);
          load_masks(Tm, (uint32_t)m, 1u, 0u);
          compare8(ltB, eqB, Tm, R0, R1);
          if (!(m & 1)) eqB = 0u;
        }
        uint4 R2, R3;
        load_keys(P, 2u);
        philox_pair(P, sw, p, R2, R3);
        load_masks(Tm, (uint32_t)m, 0u, 1u);
        compare8(l8, e8, Tm, R2, R3);
        ltA |= eqA & l8;
        eqA &= e8;
        load_masks(Tm, (uint32_t)m, 1u, 1u);
        compare8(l8, e8, Tm, R2, R3);
        ltB |= eqB & l8;
        eqB &= e8;
        const uint32_t tA = thr_a(m, thr0, thr1, thr2, thr3), tB = thr_b(m, thr0, thr1);
#pragma unroll 1
        for (uint32_t grp = 4; grp < 8u && (eqA | eqB) != 0u; ++grp) {
          const uint4 rr = philox_cold(make_uint4(gglob, sw, p, grp), k0, k1);
          compare_planes(ltA, eqA, tA, rr, grp);
          compare_planes(ltB, eqB, tB, rr, grp);
        }
        *slot = make_uint2(ltA, ltB);
      }
      __syncwarp();
    }
  };

  // General-gate runs: the acceptance words of 32 units from 32 c on of period
  // q (unit: coupled p-bit idx mod ncp of the period's sweep idx / ncp).  A
  // proposed flip of a lane in category e (e_in + 2 e_out, its disagreement
  // with the coupled neighbours) stands where word e has the lane: always, or
  // where the tag-6 uniform is below A[e].  Nearly every warp holds a lane
  // that 8 planes leave undecided, so 16 are compared at once.
  auto accept_units = [&](const PhiloxPair& P, uint32_t q, uint32_t c, uint32_t units) {
    const uint32_t idx = 32u * c + (uint32_t)lane;
    if (WGT && idx < units) {
      const uint32_t i = idx / (uint32_t)max(ncp, 1), a = idx - i * (uint32_t)ncp;
      const uint2 cp = scp[a];
      const uint4 A4 = sthr[a];
      const uint32_t A[4] = {A4.x, A4.y, A4.z, A4.w};
      const uint32_t sw = sweep0 + q * (uint32_t)ps + i, p = cp.x | (kTagCouple << 16);
      uint32_t lt[4], eq[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        lt[e] = (cp.y >> e) & 1u ? ~0u : 0u;
        eq[e] = ~lt[e];
      }
      auto compare = [&](uint4 r, uint32_t grp) {
#pragma unroll
        for (int e = 0; e < 4; ++e) compare_planes(lt[e], eq[e], A[e], r, grp);
      };
      uint4 R0, R1;
      philox_pair(P, sw, p, R0, R1);
      compare(R0, 0u);
      compare(R1, 1u);
      PhiloxPair P2;
      load_keys(P2, 2u);
      philox_pair(P2, sw, p, R0, R1);
      compare(R0, 2u);
      compare(R1, 3u);
#pragma unroll 1
      for (uint32_t grp = 4; grp < 8u && (eq[0] | eq[1] | eq[2] | eq[3]) != 0u; ++grp)
        compare(philox_cold(make_uint4(gglob, sw, p, grp), k0, k1), grp);
      sacc[((q & 1u) * (uint32_t)ps + i) * (uint32_t)(ncp + 1) + a] = make_uint4(lt[0], lt[1], lt[2], lt[3]);
    }
    __syncwarp();
  };

  int col_lo[NC + 1];
#pragma unroll
  for (int c = 0; c <= NC; ++c) col_lo[c] = uni(md.col_off[c]);

  uint32_t n_valid = 0u, n_samples = 0u;  // (32 chains x 2^26 sweeps at most)
  // smallest and largest recorded output (a run with few bins records few
  // of its samples)
  const uint32_t a_lo = rm.n_alphas ? rm.alpha_sorted[0] : 0u;
  const uint32_t a_hi = rm.n_alphas ? rm.alpha_sorted[rm.n_alphas - 1] : ~0u;
  const uint32_t svio_addr = keep((uint32_t)__cvta_generic_to_shared(svio) + 8u * (uint32_t)lane);
  const uint32_t sph_addr = keep((uint32_t)__cvta_generic_to_shared(sph) + 4u * (uint32_t)lane);
  const uint32_t last_off = keep(8u * (uint32_t)(d * n));
  const uint32_t iw4 = keep(4u * (uint32_t)iw);

  // Records (Fig. 2 Step 3) of the pair of sweeps sw, sw + 1 whose snapshots
  // start at shared address S (ns: the sweeps that exist).  The lanes take
  // the record terms in turn; the per-lane phase sums (three bit planes, mod
  // 8) of the two sweeps are reduced together, each half of the lanes taking
  // one of them.  Both sweeps cost little more than one: a term's entry and
  // its address arithmetic are shared, and the two dependent chains overlap.
  auto record = [&](uint32_t S, uint32_t sw, uint32_t ns) {
    uint32_t viol[2] = {0u, 0u}, f0[2] = {0u, 0u}, f1[2] = {0u, 0u}, f2[2] = {0u, 0u};
    auto ldv = [](uint32_t a, uint32_t (&v)[2]) {
      const uint2 x = lds2(a);
      v[0] = x.x;
      v[1] = x.y;
    };
    const uint32_t SS = S | (S << 16);  // offsets are added in pairs (no carry: below 64 KB)
    uint32_t ea = svio_addr;
#pragma unroll 2
    for (int k = 0; k < n_vio; k += 32, ea += 256u) {
      const uint2 e = lds2(ea);
      const uint32_t e0 = e.x + SS;
      uint32_t x[2], y[2], z[2];
      ldv(e0 & 0xFFFFu, x);
      ldv(e0 >> 16, y);
      ldv(e.y + S, z);
#pragma unroll
      for (int s = 0; s < 2; ++s) viol[s] |= x[s] ^ y[s] ^ z[s];
    }
    ea = sph_addr;
    auto terms = [&](uint32_t (&x)[2]) {  // the next entries' products
      const uint32_t e = lds(ea) + SS;
      uint32_t y[2];
      ldv(e & 0xFFFFu, x);
      ldv(e >> 16, y);
#pragma unroll
      for (int s = 0; s < 2; ++s) x[s] &= y[s];
      ea += 128u;
    };
#pragma unroll 1
    for (int k = 0; k < n_ph1; k += 32) {
      uint32_t x[2];
      terms(x);
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        const uint32_t c0 = f0[s] & x[s];
        f0[s] ^= x[s];
        f2[s] ^= f1[s] & c0;
        f1[s] ^= c0;
      }
    }
#pragma unroll 1
    for (int k = 0; k < n_ph2; k += 32) {
      uint32_t x[2];
      terms(x);
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        f2[s] ^= f1[s] & x[s];
        f1[s] ^= x[s];
      }
    }
#pragma unroll 2
    for (int k = 0; k < n_ph4; k += 32) {
      uint32_t x[2];
      terms(x);
#pragma unroll
      for (int s = 0; s < 2; ++s) f2[s] ^= x[s];
    }
#pragma unroll
    for (int s = 0; s < 2; ++s) viol[s] = __reduce_or_sync(0xffffffffu, viol[s]);
    {  // the lower half of the lanes keeps sweep 0, the upper sweep 1
      const bool hi = lane >= 16;
      const uint32_t o0 = __shfl_xor_sync(0xffffffffu, hi ? f0[0] : f0[1], 16);
      const uint32_t o1 = __shfl_xor_sync(0xffffffffu, hi ? f1[0] : f1[1], 16);
      const uint32_t o2 = __shfl_xor_sync(0xffffffffu, hi ? f2[0] : f2[1], 16);
      if (hi) { f0[0] = f0[1]; f1[0] = f1[1]; f2[0] = f2[1]; }
      add3(f0[0], f1[0], f2[0], o0, o1, o2);
    }
#pragma unroll
    for (int off = 8; off > 0; off >>= 1) {
      const uint32_t o0 = __shfl_xor_sync(0xffffffffu, f0[0], off);
      const uint32_t o1 = __shfl_xor_sync(0xffffffffu, f1[0], off);
      const uint32_t o2 = __shfl_xor_sync(0xffffffffu, f2[0], off);
      add3(f0[0], f1[0], f2[0], o0, o1, o2);
    }
    auto recorded = [&](uint32_t t) {
      return t >= rm.burn_in && (rm.record_every == 1u || (t - rm.burn_in) % rm.record_every == 0u);
    };
    if constexpr (WGT) {
      // the general gates' phases (2^-32 turn) of the lane's own chain
      uint32_t phi[2] = {0u, 0u};
#pragma unroll 4
      for (int i = 0; i < nug; ++i) {
        const uint4 ph = suph[i];
        const uint32_t e = suof[i] + SS;
        uint32_t wo[2], wi[2];
        ldv(e & 0xFFFFu, wo);
        ldv(e >> 16, wi);
#pragma unroll
        for (int s = 0; s < 2; ++s) {
          const bool y = (wo[s] >> lane) & 1u, x = (wi[s] >> lane) & 1u;
          const uint32_t a0 = y ? ph.z : ph.x, a1 = y ? ph.w : ph.y;
          phi[s] += x ? a1 : a0;
        }
      }
      uint32_t row[2];
      ldv(S + last_off + 8u * (uint32_t)(lane < n ? lane : 0), row);
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        if ((uint32_t)s >= ns) break;
        Recorder rec;
        rec.viol = viol[s];
        rec.f0 = __shfl_sync(0xffffffffu, f0[0], 16 * s);
        rec.f1 = __shfl_sync(0xffffffffu, f1[0], 16 * s);
        rec.f2 = __shfl_sync(0xffffffffu, f2[0], 16 * s);
        rec.lastw = lane < n ? row[s] : 0u;
        rec.phi = phi[s];
        if (!recorded(sw + (uint32_t)s)) continue;
        unsigned long long nv = 0ull, nsm = 0ull;
        rec.bin<true>(rm, g, batch, lane, shist, nv, nsm);
        n_valid += (uint32_t)nv;
        n_samples += (uint32_t)nsm;
      }
    } else {
    // lanes 16 s + r now hold sweep s; as rows 0..2 of a transpose: the planes
    const int r = lane & 15;
    const uint32_t plane = r == 0 ? f0[0] : (r == 1 ? f1[0] : f2[0]);
    // lane = chain within the group; alpha bit q = bit `lane` of word q of
    // the last layer
    const Transpose tr(lane);
    uint32_t row[2];
    const bool one = n <= 29;  // one transpose: rows 0..2 the planes, then the layer
    const int q = one ? lane - 3 : lane;
    ldv(S + last_off + 8u * (uint32_t)(q >= 0 && q < n ? q : 0), row);
    const bool active = g * 32u + (uint32_t)lane < rm.chains;
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      if ((uint32_t)s >= ns) break;
      const uint32_t t = sw + (uint32_t)s;
      if (!recorded(t)) continue;
      const uint32_t pl = __shfl_sync(0xffffffffu, plane, 16 * s + (lane & 3));
      uint32_t word = q >= 0 && q < n ? row[s] : 0u;
      uint32_t alpha, phase;
      if (one) {
        word = tr(lane < 3 ? pl : word, lane);
        alpha = word >> 3;
        phase = word & 7u;
      } else {
        alpha = tr(word, lane);
        phase = tr(lane < 3 ? pl : 0u, lane) & 7u;
      }
      const bool valid = active && !((viol[s] >> lane) & 1u);
      if (valid && alpha >= a_lo && alpha <= a_hi) {
        int bin = -1;
        if (rm.n_alphas == 0) {
          bin = (int)alpha;
        } else {
          int lo = 0, hi = rm.n_alphas - 1;
          while (lo <= hi) {
            const int mid = (lo + hi) >> 1;
            const uint32_t v = rm.alpha_sorted[mid];
            if (v == alpha) { bin = rm.alpha_slot[mid]; break; }
            if (v < alpha) lo = mid + 1; else hi = mid - 1;
          }
        }
        if (bin >= 0) {
          if (shist) atomicAdd(&shist[(uint32_t)bin * 8u + phase], 1u);
          else atomicAdd(&rm.hist[((size_t)batch * rm.bins + (uint32_t)bin) * 8u + phase], 1ull);
        }
      }
      n_valid += (uint32_t)__popc(__ballot_sync(0xffffffffu, valid));
      n_samples += (uint32_t)__popc(__ballot_sync(0xffffffffu, active));
    }
    }
  };

  // ---- periods: two to fill the pipeline, then period t is redrawn in
  // iteration t + 2 while t + 1 is finished and t + 2 started, and recorded
  // in iteration t + 3.  While it fills, every warp works.
  const uint32_t iters = n_sweeps > 0u ? n_periods + 3u : 0u;
#pragma unroll 1
  for (uint32_t it = 0; it < iters; ++it) {
    const uint32_t t = it - 2u;
    const bool fill = it < 2u;
    if (fill || warp >= cw) {
      // tasks of this iteration, longest first: finish period it - 1 (after its
      // acceptance words in a general-gate run), record
      // period it - 3, start period it; the first of a warp is its own, the
      // next come from a counter
      const uint32_t fq = it - 1u, rq = it - 3u, sq = it;
      const uint32_t w = (uint32_t)(fill ? warp : warp - cw);
      const uint32_t nw_t = (uint32_t)(fill ? nwarps : nwarps - cw);
      const uint32_t fs = fq < n_periods ? (sweeps_of(fq) * (uint32_t)npb + 31u) >> 5 : 0u;
      const uint32_t ss = sq < n_periods ? (sweeps_of(sq) * (uint32_t)npb + 63u) >> 6 : 0u;
      const uint32_t au = WGT && fq < n_periods ? sweeps_of(fq) * (uint32_t)ncp : 0u, na = (au + 31u) >> 5;
      const uint32_t nf = ((fs + 7u) >> 3) + na, nr = rq < n_periods ? (sweeps_of(rq) + 1u) >> 1 : 0u;
      uint32_t* counter = cnt + it % 3u;
      const uint32_t words = keep(ring_addr + 8u * (sq % 3u) * (uint32_t)punits);
      const uint32_t masks = keep((uint32_t)__cvta_generic_to_shared(smask) + 4u * (sq & 1u) * (uint32_t)(punits >> 5));
      PhiloxPair P;
      load_keys(P, 0u);
      if (w == 0u && lane == 0) cnt[(it + 1u) % 3u] = 0u;  // last used in iteration it - 2
#pragma unroll 1
      for (uint32_t k = w; k < nf + nr + ss;) {
        uint32_t nx = 0u;
        if (lane == 0) nx = atomicAdd(counter, 1u);
        if (WGT && k < na) {
          accept_units(P, fq, k, au);
        } else if (k < nf) {
          finish_units(fq, k - na, fs);
        } else if (k < nf + nr) {
          const uint32_t i = (k - nf) << 1, sw = sweep0 + rq * (uint32_t)ps + i;
          const uint32_t S = w_addr + iw4 * (1u + (rq & 1u) * (uint32_t)psp + i);
          record(S, sw, sweeps_of(rq) - i);
        } else {
          start_units(P, sweep0 + sq * (uint32_t)ps, k - nf - nr, words, masks);
        }
        k = nw_t + __shfl_sync(0xffffffffu, nx, 0);
      }
    } else if (t < n_periods) {
      {
        // the thread's first p-bit of each class: a consumer without one
        // redraws the scratch word from ZERO links
        uint32_t la[NC][3], lb[NC][3], da[NC], M2[NC];
        [[maybe_unused]] uint32_t wi[NC], wo[NC], ao[NC], cpm = 0u;  // coupled neighbours, words; classes
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          const int i = col_lo[c] + tid;
          const bool has = i < col_lo[c + 1];
          const uint32_t ea = sent_addr + 16u * (uint32_t)(has ? i : 0);
          const uint4 x = lds4(ea), y = lds4(ea + 16u * (uint32_t)npb);
          const uint32_t z = w_addr + 4u * (uint32_t)zero_idx(n, d);
          la[c][0] = has ? x.x : z;
          lb[c][0] = has ? x.y : z;
          la[c][1] = has ? x.z : z;
          lb[c][1] = has ? x.w : z;
          la[c][2] = has ? y.x : z;
          lb[c][2] = has ? y.y : z;
          da[c] = has ? y.z : w_addr + 4u * (uint32_t)nw;
          M2[c] = y.w;
          if constexpr (WGT) {
            const uint4 nb = snb[has ? i : 0];
            wi[c] = has ? nb.x : da[c];
            wo[c] = has ? nb.y : da[c];
            ao[c] = has ? nb.z : 16u * (uint32_t)ncp;
            cpm |= __any_sync(0xffffffffu, has && nb.w) ? 1u << c : 0u;
          }
        }
        const uint32_t cnt_t = sweeps_of(t);
        // (A, B) of this thread's unit of class 0, sweep 0 of the period
        [[maybe_unused]] uint32_t acc = (uint32_t)__cvta_generic_to_shared(sacc) +
                                        16u * (t & 1u) * (uint32_t)(ps * (ncp + 1));
        // Metropolis acceptance of a coupled p-bit's proposal v: its current
        // word at d, its neighbours' at i and o, its acceptance words at a
        auto accept = [&](uint32_t v, uint32_t d, uint32_t i, uint32_t o, uint32_t a) {
          const uint32_t old = lds(d), e1 = old ^ lds(i), e2 = old ^ lds(o);
          const uint4 w = lds4(a);
          const uint32_t lo = (e1 & w.y) | (~e1 & w.x), hi = (e1 & w.w) | (~e1 & w.z);
          return old ^ ((old ^ v) & ((e2 & hi) | (~e2 & lo)));
        };
        uint32_t ab_addr = ring_addr + 8u * ((t % 3u) * (uint32_t)punits + (uint32_t)tid);
        // snapshot of word address a: 2 a + so
        const uint32_t sbase = w_addr + 4u * (uint32_t)(iw * (1 + (int)(t & 1u) * psp)) - 2u * w_addr;
        // classes in which this warp has p-bits, and its units' words
        uint32_t act = 0u, abo[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          act |= warp * 32 < col_lo[c + 1] - col_lo[c] ? 1u << c : 0u;
          abo[c] = keep(8u * (uint32_t)col_lo[c]);
        }
        act = keep(act);
        const uint32_t npb8 = keep(8u * (uint32_t)npb);
        uint2 ab = make_uint2(0u, 0u);
        if (act & 1u) ab = lds2(ab_addr);
#pragma unroll 1
        for (uint32_t i = 0; i < cnt_t; ++i) {
          const uint32_t next = i + 1u < cnt_t ? npb8 : 0u;
          const uint32_t so = sbase + (i & ~1u) * iw4 + 4u * (i & 1u);
          auto step = [&](auto cc) {
            constexpr int C = decltype(cc)::value;
            if (act & (1u << C)) {
              const uint32_t r0 = lds(la[C][0]) ^ lds(lb[C][0]);
              const uint32_t r1 = lds(la[C][1]) ^ lds(lb[C][1]);
              const uint32_t r2 = lds(la[C][2]) ^ lds(lb[C][2]);
              uint32_t v = redraw(r0, r1, r2, M2[C], ab);
              if constexpr (WGT)
                if (cpm & (1u << C)) v = accept(v, da[C], wi[C], wo[C], acc + ao[C]);
              sts(da[C], v);
              sts(2u * da[C] + so, v);
              if constexpr (MULTI) {  // further p-bits of a class larger than the consumers
#pragma unroll 1
                for (int lo = col_lo[C], K = col_lo[C + 1] - lo, k = tid + sh.cons; k < K; k += sh.cons) {
                  const uint32_t ea = sent_addr + 16u * (uint32_t)(lo + k);
                  const uint4 x = lds4(ea), y = lds4(ea + 16u * (uint32_t)npb);
                  const uint2 ab2 = lds2(ab_addr + 8u * (uint32_t)(lo + k - tid));
                  const uint32_t s0 = lds(x.x) ^ lds(x.y);
                  const uint32_t s1 = lds(x.z) ^ lds(x.w);
                  const uint32_t s2 = lds(y.x) ^ lds(y.y);
                  uint32_t v2 = redraw(s0, s1, s2, y.w, ab2);
                  if constexpr (WGT) {
                    const uint4 nb = snb[lo + k];
                    if (nb.w) v2 = accept(v2, y.z, nb.x, nb.y, acc + nb.z);
                  }
                  sts(y.z, v2);
                  sts(2u * y.z + so, v2);
                }
              }
            }
            // the next step's words, loaded ahead of the barrier (a lane past
            // its class reads another unit's: unused; the allocation has room
            // for the 31 words past the last)
            constexpr int CN = (C + 1) % NC;
            if (act & (1u << CN)) ab = lds2(ab_addr + (CN ? abo[CN] : next));
            if (cw > 1) bar_sync_first(1u, (uint32_t)sh.cons);
            else __syncwarp();
          };
          step(std::integral_constant<int, 0>{});
          step(std::integral_constant<int, 1>{});
          if constexpr (NC > 2) step(std::integral_constant<int, 2>{});
          if constexpr (NC > 3) step(std::integral_constant<int, 3>{});
          ab_addr += npb8;
          if constexpr (WGT) acc += 16u * (uint32_t)(ncp + 1);
        }
      }
    }
    __syncthreads();
  }

  // ---- write the group image back, add the counts of this launch
  uint32_t* out = rm.state + (size_t)g * npb;
#pragma unroll 1
  for (int i = tid; i < npb; i += T) out[i] = W[n + i];
  if (WGT && shist && wgt_m) {  // (re, im, comp re, comp im) doubles per bin, then u32 counts
    const double* sd = reinterpret_cast<const double*>(shist);
#pragma unroll 1
    for (uint32_t i = tid; i < rm.bins; i += T) {
      const uint32_t cn = shist[8u * rm.bins + i];
      if (!cn) continue;
      unsigned long long* c = rm.hist + ((size_t)batch * rm.bins + i) * 8u;
      double* cd = reinterpret_cast<double*>(c);
      atomic_add_comp(&cd[0], &cd[3], sd[4u * i], sd[4u * i + 2u]);
      atomic_add_comp(&cd[1], &cd[4], sd[4u * i + 1u], sd[4u * i + 3u]);
      atomicAdd(c + 2, (unsigned long long)cn);
    }
  } else if (shist) {
    unsigned long long* gh = rm.hist + (size_t)batch * rm.bins * 8u;
#pragma unroll 1
    for (uint32_t i = tid; i < rm.bins * 8u; i += T)
      if (shist[i]) atomicAdd(&gh[i], (unsigned long long)shist[i]);
  }
  if (lane == 0) {
    if (n_valid) atomicAdd(&rm_g.valid[batch], (unsigned long long)n_valid);
    if (n_samples) atomicAdd(&rm_g.samples[batch], (unsigned long long)n_samples);
  }
  __syncthreads();
}

// One CTA per chain group of every model of the run (flat group index).
template <int NC, bool MULTI, bool WGT>
__global__ void __launch_bounds__(WGT ? kSweepThreadsWgt : kSweepThreadsPlain) sweep_plain_kernel(
    const RunModelDev* __restrict__ rm, int n_models, uint32_t n_sweeps, PlainShape sh,
    WsHeader* hdr) {
  extern __shared__ __align__(16) uint32_t smem[];
  const uint32_t sweep0 = *(volatile uint32_t*)&hdr->sweep0;
  const uint32_t flat = blockIdx.x;
  const RunModelDev& r = rm[find_model(rm, n_models, flat)];
  const uint32_t g = flat - r.group_base;
  if (g >= r.groups) return;  // (never: the grid is the runs' groups)
  run_group_plain<NC, MULTI, true, WGT>(r, g, sweep0, n_sweeps, sh, smem, hdr);
}

// Persistent form: a fixed grid pops (model, group) items from a
// cost-ordered work list with one atomic counter.  No CTA waits on another.
template <int NC, bool MULTI>
__global__ void __launch_bounds__(kSweepThreadsPlain) sweep_plain_persistent_kernel(
    const RunModelDev* __restrict__ rm, int n_models, const uint32_t* __restrict__ work,
    uint32_t n_work, uint32_t n_sweeps, PlainShape sh, WsHeader* hdr) {
  extern __shared__ __align__(16) uint32_t smem[];
  const uint32_t sweep0 = *(volatile uint32_t*)&hdr->sweep0;
  __shared__ uint32_t item;
  for (;;) {
    if (threadIdx.x == 0) item = atomicAdd(&hdr->work_next, 1u);
    __syncthreads();
    const uint32_t it = item;
    __syncthreads();
    if (it >= n_work) break;
    const uint32_t flat = work[it];
    const RunModelDev& r = rm[find_model(rm, n_models, flat)];
    const uint32_t g = flat - r.group_base;
    if (g < r.groups) run_group_plain<NC, MULTI, false, false>(r, g, sweep0, n_sweeps, sh, smem, hdr);
  }
  // the last CTA to leave also clears the work counter
  if (threadIdx.x == 0 && atomicAdd(&hdr->ctas_done, 1u) == gridDim.x - 1u) {
    hdr->ctas_done = 0u;
    hdr->work_next = 0u;
    hdr->sweep0 = sweep0 + n_sweeps;
  }
}

}  // namespace

// Calls f(NC, MULTI): NC colour steps (2..4), MULTI where some class is larger
// than the consumers.
template <class F>
static void plain_dispatch(int nc, bool multi, F f) {
  auto by_multi = [&](auto c) {
    if (multi) f(c, std::true_type{});
    else f(c, std::false_type{});
  };
  if (nc <= 2) by_multi(std::integral_constant<int, 2>{});
  else if (nc == 3) by_multi(std::integral_constant<int, 3>{});
  else by_multi(std::integral_constant<int, 4>{});
}

cudaError_t launch_sweeps_plain(const RunModelDev* d_rm, int n_models, uint32_t total_groups,
                                uint32_t n_sweeps, int cons, int prod, int units, int max_col, int nc,
                                bool wgt, size_t smem_bytes, WsHeader* hdr, cudaStream_t st) {
  const PlainShape sh{cons, prod / 32 + 1, units};
  const int threads = cons + 32 * sh.work;
  plain_dispatch(nc, max_col > cons, [&](auto c, auto m) {
    constexpr int NC = decltype(c)::value;
    constexpr bool M = decltype(m)::value;
    if (wgt) sweep_plain_kernel<NC, M, true><<<total_groups, threads, smem_bytes, st>>>(d_rm, n_models, n_sweeps, sh, hdr);
    else sweep_plain_kernel<NC, M, false><<<total_groups, threads, smem_bytes, st>>>(d_rm, n_models, n_sweeps, sh, hdr);
  });
  return cudaGetLastError();
}

cudaError_t launch_sweeps_plain_persistent(const RunModelDev* d_rm, int n_models,
                                           const uint32_t* d_work, uint32_t n_work,
                                           uint32_t n_sweeps, int cons, int prod, int units,
                                           int max_col, int nc, int grid, size_t smem_bytes, WsHeader* hdr,
                                           cudaStream_t st) {
  const PlainShape sh{cons, prod / 32 + 1, units};
  const int threads = cons + 32 * sh.work;
  plain_dispatch(nc, max_col > cons, [&](auto c, auto m) {
    sweep_plain_persistent_kernel<decltype(c)::value, decltype(m)::value>
        <<<grid, threads, smem_bytes, st>>>(d_rm, n_models, d_work, n_work, n_sweeps, sh, hdr);
  });
  return cudaGetLastError();
}

// Opt the kernels into large dynamic shared memory (once per run, outside
// any stream capture).
cudaError_t sweep_plain_prepare() {
  cudaError_t e = cudaSuccess;
  auto opt = [&](auto kern) {
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSweepSmemMax);
  };
  for (int nc = 2; nc <= 4; ++nc)
    for (int multi = 0; multi < 2; ++multi)
      plain_dispatch(nc, multi != 0, [&](auto c, auto m) {
        opt(sweep_plain_kernel<decltype(c)::value, decltype(m)::value, false>);
        opt(sweep_plain_kernel<decltype(c)::value, decltype(m)::value, true>);
        opt(sweep_plain_persistent_kernel<decltype(c)::value, decltype(m)::value>);
      });
  return e;
}

int sweep_plain_blocks_per_sm(int max_col, int cons, int nc, int threads, size_t smem) {
  int blocks = 0;
  cudaError_t e = cudaSuccess;
  plain_dispatch(nc, max_col > cons, [&](auto c, auto m) {
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
        &blocks, sweep_plain_persistent_kernel<decltype(c)::value, decltype(m)::value>, threads, smem);
  });
  return e == cudaSuccess ? blocks : 1;
}

}  // namespace pb
