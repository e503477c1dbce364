// Device helpers shared by the sweep kernels.
#pragma once
#include <cuda_runtime.h>

#include "pb_internal.h"
#include "philox.cuh"

namespace pb {

// Barrier `id` over the first `threads` threads of the CTA (whole warps).
__device__ __forceinline__ void bar_sync_first(uint32_t id, uint32_t threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// Out-of-line Philox for the rarely taken paths (keeps the hot loop small).
static __device__ __noinline__ uint4 philox_cold(uint4 c, uint32_t k0, uint32_t k1) {
  return philox4x32_10(c, k0, k1);
}

// Threshold pair of a p-bit with m links: tA for the lanes in `sel` (all
// links agree), tB for the others (see the consumer table set-up).
__device__ __forceinline__ uint32_t thr_a(int m, uint32_t t0, uint32_t t1, uint32_t t2, uint32_t t3) {
  return m == 0 ? t0 : (m == 1 ? t1 : (m == 2 ? t2 : t3));
}
__device__ __forceinline__ uint32_t thr_b(int m, uint32_t t0, uint32_t t1) {
  return (m == 0 || m == 2) ? t0 : t1;
}

__device__ __forceinline__ void add3(uint32_t& f0, uint32_t& f1, uint32_t& f2, uint32_t x0,
                                     uint32_t x1, uint32_t x2) {
  const uint32_t c0 = f0 & x0;
  f0 ^= x0;
  const uint32_t t = f1 ^ x1;
  const uint32_t c1 = (f1 & x1) | (c0 & t);
  f1 = t ^ c0;
  f2 ^= x2 ^ c1;
}

__device__ __forceinline__ int find_model(const RunModelDev* rm, int n_models, uint32_t flat) {
  int lo = 0, hi = n_models - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (rm[mid].group_base <= flat) lo = mid; else hi = mid - 1;
  }
  return lo;
}

__device__ __forceinline__ void set_status(WsHeader* hdr, int code) {
  if (hdr) atomicCAS(&hdr->status, 0u, (uint32_t)code);
}

// Words of a shared-memory group image: the (d+1) n layer words, ZERO, ONES
// and one scratch word (the store target of consumers without a p-bit in a
// colour class), rounded up to 16 bytes.
__host__ __device__ inline int image_words(int n, int d) { return (n_words(n, d) + 1 + 3) & ~3; }

// Initial chains of group g: a valid path with random H outputs (tag-1
// stream), every other bit its deterministic value, layer by layer.  The whole
// CTA; W: n_words of shared memory; itab per p-bit: 0xFFFFFFFF = H, else
// a | b << 16.
static __device__ void init_group(const RunModelDev& r, const ModelDev& md, uint32_t g,
                                  const uint32_t* __restrict__ itab, uint32_t* W, WsHeader* hdr) {
  const int n = md.n, d = md.d, nw = md.nw;
  for (int i = threadIdx.x; i < nw; i += blockDim.x) {
    uint32_t v = 0u;
    if (i < n) v = ((md.beta >> i) & 1u) ? ~0u : 0u;
    else if (i == ones_idx(n, d)) v = ~0u;
    W[i] = v;
  }
  __syncthreads();
  for (int k = 1; k <= d; ++k) {
    for (int q = threadIdx.x; q < n; q += blockDim.x) {
      const int p = (k - 1) * n + q;
      const uint32_t e = itab[p];
      uint32_t v;
      if (e == 0xFFFFFFFFu) {
        v = philox4x32_10(make_uint4(g + r.group0, 0u, (uint32_t)p | (kTagInit << 16), 0u),
                          r.seed_lo, r.seed_hi).x;
      } else if (e == 0xFFFFFFFEu) {  // Toffoli target: its own general link
        const GLink* G = r.glk ? r.glk + p : nullptr;
        if (!G || G->a[0] >= nw || G->b[0] >= nw || G->c[0] >= nw) { set_status(hdr, PB_EINVAL); v = 0u; }
        else v = W[G->a[0]] ^ (W[G->b[0]] & W[G->c[0]]);
      } else {
        const uint32_t a = e & 0xFFFFu, b = e >> 16;
        if ((int)a >= nw || (int)b >= nw) { set_status(hdr, PB_EINVAL); v = 0u; }
        else v = W[a] ^ W[b];
      }
      W[k * n + q] = v;
    }
    __syncthreads();
  }
  uint32_t* out = r.state + (size_t)g * n * d;
  for (int i = threadIdx.x; i < n * d; i += blockDim.x) out[i] = W[n + i];
}

// 32 x 32 bit transpose across a warp: on entry lane r holds row r; on
// return lane c holds column c (bit r = bit c of row r).  Five butterfly
// steps, each swapping the off-diagonal blocks of the current block size.
__device__ __forceinline__ uint32_t warp_transpose32(uint32_t x, int lane) {
  const uint32_t masks[5] = {0x0000FFFFu, 0x00FF00FFu, 0x0F0F0F0Fu, 0x33333333u, 0x55555555u};
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    const int j = 16 >> k;
    const uint32_t M = masks[k];
    const uint32_t y = __shfl_xor_sync(0xffffffffu, x, j);
    x = (lane & j) ? ((x & ~M) | ((y & ~M) >> j)) : ((x & M) | ((y & M) << j));
  }
  return x;
}

// Shared-window loads and stores (addresses as 32-bit words).
__device__ __forceinline__ uint32_t lds(uint32_t a) {
  uint32_t x;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(x) : "r"(a));
  return x;
}
__device__ __forceinline__ uint2 lds2(uint32_t a) {
  uint2 x;
  asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(x.x), "=r"(x.y) : "r"(a));
  return x;
}
__device__ __forceinline__ uint4 lds4(uint32_t a) {
  uint4 x;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(x.x), "=r"(x.y), "=r"(x.z), "=r"(x.w) : "r"(a));
  return x;
}
__device__ __forceinline__ void sts(uint32_t a, uint32_t v) {
  asm volatile("st.shared.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}

// 32 x 32 bit transpose with the lane's masks held in registers: a step is
// one shuffle, one rotation and one select.
struct Transpose {
  uint32_t m[5];
  __device__ explicit Transpose(int lane) {
    const uint32_t masks[5] = {0x0000FFFFu, 0x00FF00FFu, 0x0F0F0F0Fu, 0x33333333u, 0x55555555u};
#pragma unroll
    for (int k = 0; k < 5; ++k) m[k] = (lane & (16 >> k)) ? ~masks[k] : masks[k];
  }
  // lane r holds row r; returns column `lane` (bit r = bit `lane` of row r)
  __device__ uint32_t operator()(uint32_t x, int lane) const {
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      const int j = 16 >> k;
      const uint32_t y = __shfl_xor_sync(0xffffffffu, x, j);
      const uint32_t r = __funnelshift_l(y, y, (lane & j) ? 32 - j : j);
      x = (x & m[k]) | (r & ~m[k]);
    }
    return x;
  }
};

// Compensated FP64 accumulation of the phase sums: *s += x by an atomic add,
// whose old value gives the exact rounding error of fl(old + x) (Knuth's
// two-sum), and that error (plus `carry`, a compensation brought along) is
// added to the compensation word *c.  The sum is *s + *c; the rounding of the
// big partial sums no longer accumulates over the samples.
__device__ __forceinline__ void atomic_add_comp(double* s, double* c, double x, double carry = 0.0) {
  const double old = atomicAdd(s, x);
  const double nw = old + x;
  const double bp = nw - old;
  const double err = (old - (nw - bp)) + (x - bp) + carry;
  if (err != 0.0) atomicAdd(c, err);
}

// Record of one sweep (Fig. 2 Step 3), computed by the recorder warp from a
// snapshot of the sweep's final state while the stage warps run the next
// sweep, pipelined over the colour stages: read() gathers, for a range of
// p-bits, the violation word and the phase (three bit planes, mod 8);
// reduce() combines the lanes and takes the last layer; bin() adds one count
// per valid chain to (end state alpha, phase class).
struct Recorder {
  uint32_t viol = 0u, f0 = 0u, f1 = 0u, f2 = 0u, lastw = 0u;
  uint32_t phi = 0u;  // general gates: this lane's chain's phase, 2^-32 turn

  __device__ void clear() { viol = f0 = f1 = f2 = phi = 0u; }

  // Two-qubit tables lo..hi-1: each adds its entry's phase for the lane's
  // chain, and a zero entry marks the chain's path invalid.
  __device__ void read_t(const uint32_t* S, const TRec* tr, int lo, int hi, int lane) {
    bool bad = false;
#pragma unroll 1
    for (int i = lo; i < hi; ++i) {
      const TRec& R = tr[i];
      const uint32_t idx = ((S[R.wx0] >> lane) & 1u) | (((S[R.wx1] >> lane) & 1u) << 1) |
                           (((S[R.wy0] >> lane) & 1u) << 2) | (((S[R.wy1] >> lane) & 1u) << 3);
      phi += R.ph[idx];
      bad = bad || ((R.zmask >> idx) & 1u);
    }
    viol |= __ballot_sync(0xffffffffu, bad);
  }

  // Phases of general gates lo..hi-1 for the lane's own chain, eight gates
  // per batch with every load of a batch issued before the first use.
  __device__ void read_u(const uint32_t* S, const UPh* uph, int lo, int hi, int lane) {
    int i = lo;
#pragma unroll 1
    for (; i + 8 <= hi; i += 8) {
      uint4 ph[8];
      uint32_t ww[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        ph[j] = *reinterpret_cast<const uint4*>(uph[i + j].ph);
        ww[j] = *reinterpret_cast<const uint32_t*>(&uph[i + j].wout);  // wout | win << 16
      }
      uint32_t y[8], x[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        y[j] = (S[ww[j] & 0xFFFFu] >> lane) & 1u;
        x[j] = (S[ww[j] >> 16] >> lane) & 1u;
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const uint32_t a0 = y[j] ? ph[j].z : ph[j].x, a1 = y[j] ? ph[j].w : ph[j].y;
        phi += x[j] ? a1 : a0;
      }
    }
#pragma unroll 1
    for (; i < hi; ++i) {
      const UPh U = uph[i];
      const uint32_t y = (S[U.wout] >> lane) & 1u, x = (S[U.win] >> lane) & 1u;
      const uint32_t a0 = y ? U.ph[2] : U.ph[0], a1 = y ? U.ph[3] : U.ph[1];
      phi += x ? a1 : a0;
    }
  }

  // ANDV: general-gate runs, where a Toffoli target's term is
  // W[vd] ^ W[va] ^ (W[vb] & W[vc]) (vc = ONES elsewhere).
  template <bool ANDV = false>
  __device__ void read(const uint32_t* S, const Rec* srec, int lo, int hi, int lane) {
#pragma unroll 2
    for (int i = lo + lane; i < hi; i += 32) {
      const Rec R = srec[i];
      if constexpr (ANDV) viol |= S[R.vd] ^ S[R.va] ^ (S[R.vb] & S[R.vc]);
      else viol |= S[R.vd] ^ S[R.va] ^ S[R.vb];
      const uint32_t x = S[R.pa] & S[R.pb];
      add3(f0, f1, f2, (R.w & 1) ? x : 0u, (R.w & 2) ? x : 0u, (R.w & 4) ? x : 0u);
    }
  }

  __device__ void reduce(const uint32_t* S, int n, int d, int lane) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      const uint32_t ov = __shfl_xor_sync(0xffffffffu, viol, off);
      const uint32_t o0 = __shfl_xor_sync(0xffffffffu, f0, off);
      const uint32_t o1 = __shfl_xor_sync(0xffffffffu, f1, off);
      const uint32_t o2 = __shfl_xor_sync(0xffffffffu, f2, off);
      viol |= ov;
      add3(f0, f1, f2, o0, o1, o2);
    }
    lastw = lane < n ? S[d * n + lane] : 0u;
  }

  // The phasor of this lane's record: the general gates' phases plus the
  // phase class (2^29 per pi/4), in FP32 (FP64 issues far slower on this
  // part): the angle rounds to 24 bits (<= pi 2^-24 rad) and sincospif adds
  // about one ulp, so each term is within 3e-7 of e^{i angle}.
  __device__ void phasor(uint32_t phase, double& cs, double& sn) const {
    const uint32_t ang = phi + (phase << 29);
    float snf, csf;
    sincospif((float)(int32_t)ang * 0x1p-31f, &snf, &csf);
    cs = (double)csf;
    sn = (double)snf;
  }

  // Few bins (<= 8): all lanes would hit a handful of FP64 counters, so the
  // warp sums each distinct bin's terms with shuffles and one lane adds them
  // (whole warp, convergent).
  __device__ void bin_few(const RunModelDev& rm, uint32_t batch, int lane, uint32_t* shist,
                          int bin) {
    const uint32_t phase = ((f0 >> lane) & 1u) | (((f1 >> lane) & 1u) << 1) |
                           (((f2 >> lane) & 1u) << 2);
    double cs, sn;
    phasor(phase, cs, sn);
    const bool has = bin >= 0;
    unsigned pending = __ballot_sync(0xffffffffu, has);
    while (pending) {
      const int leader = __ffs((int)pending) - 1;
      const int b = __shfl_sync(0xffffffffu, bin, leader);
      const bool mine = has && bin == b;
      const unsigned m = __ballot_sync(0xffffffffu, mine);
      double r = mine ? cs : 0.0, q = mine ? sn : 0.0;
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) {
        r += __shfl_xor_sync(0xffffffffu, r, off);
        q += __shfl_xor_sync(0xffffffffu, q, off);
      }
      if (lane == leader) {
        if (shist) {
          double* sd = reinterpret_cast<double*>(shist) + 4u * (uint32_t)b;
          atomic_add_comp(&sd[0], &sd[2], r);
          atomic_add_comp(&sd[1], &sd[3], q);
          atomicAdd(&shist[8u * rm.bins + (uint32_t)b], (uint32_t)__popc(m));
        } else {
          unsigned long long* c = rm.hist + ((size_t)batch * rm.bins + (uint32_t)b) * 8u;
          double* cd = reinterpret_cast<double*>(c);
          atomic_add_comp(&cd[0], &cd[3], r);
          atomic_add_comp(&cd[1], &cd[4], q);
          atomicAdd(c + 2, (unsigned long long)__popc(m));
        }
      }
      pending &= ~m;
    }
  }

  // WGT: models with general gates (rm.cpl set) add e^{i 2 pi phase} in FP64
  // (re, im, count per bin) instead of one count per phase class.
  template <bool WGT>
  __device__ void bin(const RunModelDev& rm, uint32_t g, uint32_t batch, int lane, uint32_t* shist,
                      unsigned long long& n_valid, unsigned long long& n_samples) {
    // lane = chain within the group; alpha bit q = bit `lane` of layer-d word q
    const uint32_t chain = g * 32u + (uint32_t)lane;
    const bool active = chain < rm.chains;
    const bool valid = active && !((viol >> lane) & 1u);
    const uint32_t alpha = warp_transpose32(lastw, lane);
    const uint32_t phase = ((f0 >> lane) & 1u) | (((f1 >> lane) & 1u) << 1) |
                           (((f2 >> lane) & 1u) << 2);
    int bin = -1;
    if (valid) {
      const int na = rm.n_alphas;
      if (na == 0) {
        bin = (int)alpha;
      } else {
        int lo = 0, hi = na - 1;
        while (lo <= hi) {
          const int mid = (lo + hi) >> 1;
          const uint32_t v = rm.alpha_sorted[mid];
          if (v == alpha) { bin = rm.alpha_slot[mid]; break; }
          if (v < alpha) lo = mid + 1; else hi = mid - 1;
        }
      }
    }
    if constexpr (WGT) {
      if (rm.cpl != nullptr && rm.bins <= 8u) {  // whole warp here: see bin_few
        bin_few(rm, batch, lane, shist, bin);
        bin = -1;
      }
    }
    if (bin >= 0) {
      bool done = false;
      if constexpr (WGT) {
        if (rm.cpl != nullptr) {
          double cs, sn;
          phasor(phase, cs, sn);
          if (shist) {
            double* sd = reinterpret_cast<double*>(shist) + 4u * (uint32_t)bin;
            atomic_add_comp(&sd[0], &sd[2], cs);
            atomic_add_comp(&sd[1], &sd[3], sn);
            atomicAdd(&shist[8u * rm.bins + (uint32_t)bin], 1u);
          } else {
            unsigned long long* c = rm.hist + ((size_t)batch * rm.bins + (uint32_t)bin) * 8u;
            double* cd = reinterpret_cast<double*>(c);
            atomic_add_comp(&cd[0], &cd[3], cs);
            atomic_add_comp(&cd[1], &cd[4], sn);
            atomicAdd(c + 2, 1ull);
          }
          done = true;
        }
      }
      if (!done) {
        if (shist) atomicAdd(&shist[(uint32_t)bin * 8u + phase], 1u);
        else atomicAdd(&rm.hist[((size_t)batch * rm.bins + (uint32_t)bin) * 8u + phase], 1ull);
      }
    }
    n_valid += __popc(__ballot_sync(0xffffffffu, valid));
    n_samples += __popc(__ballot_sync(0xffffffffu, active));
  }
};

}  // namespace pb
