// Exact path sampler on the eliminated network for plain (Clifford+T and X)
// models (sm_103a): every recorded sample draws a fresh valid path -- an H
// output (k, q) of chain c at sample t is bit (c mod 32) of word 0 of
// Philox(c / 32, t, p | 4 << 16, 0), every other bit its deterministic value
// (the XOR of two words of the layer before) -- and adds its phase to the bin
// of its end state (Fig. 2 Step 3).  Runs with general gates or a clamped
// output take elim_kernel (sweep.cu).
//
// One CTA per chain group; a warp draws four samples at a time, word w of its
// image holding the four samples' words side by side:
//   - the samples' Philox calls densely over (H output, sample), 32 a warp,
//   - the layers in order, lane q the four words of qubit q at once,
//   - no violation terms (every path is valid by construction), the phase
//     terms of the four samples from shared entries, one reduction for all.
// What bounds it: the latency of a warp's chain (shared-memory loads of the
// layers, shuffles, branches).  A sample of 32 chains costs about 310 warp
// instructions, and 47 % of the issue slots of the SMs that have a group are
// used: 16 warps an SM, one CTA (113 registers a thread; on mid 200 KB of
// shared memory).  Mid circuit, 4096 chains, 1e4 samples, the kernel alone:
// 3.78 -> 0.83 ms.  The kernel it replaced for these runs drew one sample at a
// time and ran a whole-warp Philox call in every layer that held an H (20 for
// 34 useful lanes in all), evaluated violation terms that are zero, and
// counted in global memory.
#include <cuda_runtime.h>

#include "pb_internal.h"
#include "philox.cuh"
#include "sweep_common.cuh"

namespace pb {
namespace {

// Shared memory: links (byte offsets in an image, by p-bit), H outputs, phase
// lists, counters, the histogram, then one image per warp.
struct ElimLayout {
  uint32_t lnk, hp, sph, cnt, hist, img, img_words;  // word offsets
};
__host__ __device__ inline ElimLayout elim_layout(int n, int d, uint32_t hist_bins) {
  const uint32_t npb = (uint32_t)(n * d), pad = (npb + 31) & ~31u;
  ElimLayout L;
  L.lnk = 0;
  L.hp = L.lnk + pad;
  L.sph = L.hp + pad;
  L.cnt = L.sph + pad + 96;
  L.hist = L.cnt + 4;
  L.img = L.hist + hist_bins * 8;
  L.img_words = 4u * (uint32_t)n_words(n, d);
  return L;
}

__global__ void __launch_bounds__(512) elim_plain_kernel(
    const RunModelDev* __restrict__ rm_all, int n_models, const uint32_t* const* __restrict__ init_tabs,
    uint32_t n_sweeps, WsHeader* hdr) {
  extern __shared__ __align__(16) uint32_t smem[];
  const uint32_t sweep0 = *(volatile uint32_t*)&hdr->sweep0;
  const int mi = find_model(rm_all, n_models, blockIdx.x);
  const RunModelDev rm = rm_all[mi];
  const uint32_t g = blockIdx.x - rm.group_base;
  auto uni = [](auto x) { return __shfl_sync(0xffffffffu, x, 0); };
  const int n = uni(rm.md.n), d = uni(rm.md.d), nw = n_words(n, d), npb = n * d;
  const int tid = threadIdx.x, T = blockDim.x, lane = tid & 31, warp = uni(tid >> 5), nwarps = T >> 5;
  const bool hist_smem = rm.hist_smem && elim_hist_pays(rm.bins, n_sweeps, rm.record_every);
  const ElimLayout L = elim_layout(n, d, hist_smem ? rm.bins : 0u);
  uint32_t* lnk = smem + L.lnk;
  uint32_t* hp = smem + L.hp;
  uint32_t* sph = smem + L.sph;
  uint32_t* cnt = smem + L.cnt;
  uint32_t* shist = hist_smem ? smem + L.hist : nullptr;
  uint32_t* img = smem + L.img + (uint32_t)warp * L.img_words;
  const uint32_t img_addr = (uint32_t)__cvta_generic_to_shared(img);
  const uint32_t* itab = init_tabs[mi];  // per p-bit: 0xFFFFFFFF = H, else a | b << 16

  // ---- tables
  const uint32_t zoff = 16u * (uint32_t)zero_idx(n, d), zz = zoff | zoff << 16;
  int n_rec[4];
#pragma unroll
  for (int l = 0; l < 4; ++l) n_rec[l] = min(max(uni(rm.md.n_rec[l]), 0), npb);
  const int npad = (npb + 31) & ~31;
  const int n_ph1 = (n_rec[1] + 31) & ~31, n_ph2 = min((n_rec[2] + 31) & ~31, npad + 64 - n_ph1);
  const int n_ph4 = min(n_rec[3], npad + 96 - n_ph1 - n_ph2);
  if (tid == 0) cnt[0] = 0u;
  if (n_rec[1] + tid < n_ph1) sph[n_rec[1] + tid] = zz;
  if (n_rec[2] + tid < n_ph2) sph[n_ph1 + n_rec[2] + tid] = zz;
  if (tid < 32 && n_ph1 + n_ph2 + n_ph4 + tid < npad + 96) sph[n_ph1 + n_ph2 + n_ph4 + tid] = zz;
  if (shist) {
#pragma unroll 1
    for (uint32_t i = tid; i < rm.bins * 8u; i += T) shist[i] = 0u;
  }
#pragma unroll 1
  for (int i = lane; i < nw; i += 32) {  // the words no sample writes; the rest zero
    uint32_t v = 0u;
    if (i < n) v = ((rm.md.beta >> i) & 1u) ? ~0u : 0u;  // clamped input layer
    else if (i == ones_idx(n, d)) v = ~0u;
    *reinterpret_cast<uint4*>(img + 4 * i) = make_uint4(v, v, v, v);
  }
  __syncthreads();
  int bad = 0;
#pragma unroll 1
  for (int i = tid; i < npb; i += T) {
    const uint32_t e = itab[i];
    uint32_t x = 0xFFFFFFFFu;
    if (e == 0xFFFFFFFFu) {
      hp[atomicAdd(&cnt[0], 1u)] = (uint32_t)i;
    } else {
      // both words lie in the layer before (or are ZERO / ONES)
      const int a = (int)(e & 0xFFFFu), b = (int)(e >> 16);
      if (a >= nw || b >= nw) bad = 1;
      else x = 16u * (uint32_t)a | (16u * (uint32_t)b) << 16;
    }
    lnk[i] = x;
    const Rec R = rm.rec[i];
    const int kp = R.w >> 3, w = R.w & 7;
    if (R.pa >= nw || R.pb >= nw || (w && kp >= (w == 1 ? n_rec[1] : w == 2 ? n_rec[2] : n_ph4))) bad = 1;
    else if (w) sph[(w == 1 ? 0 : w == 2 ? n_ph1 : n_ph1 + n_ph2) + kp] = 16u * R.pa | (16u * R.pb) << 16;
  }
  const uint32_t n_launch = n_sweeps;
  if (__syncthreads_or(bad)) {  // a bad table is reported, never followed
    if (tid == 0) set_status(hdr, PB_EINVAL);
    n_sweeps = 0u;
  }
  const uint32_t h4 = 4u * uni(cnt[0]);
  const uint32_t gglob = g + rm.group0, batch = g % rm.n_batches;
  const uint32_t k0 = rm.seed_lo, k1 = rm.seed_hi;
  const uint32_t sph_addr = (uint32_t)__cvta_generic_to_shared(sph);
  const uint32_t a_lo = rm.n_alphas ? rm.alpha_sorted[0] : 0u;
  const uint32_t a_hi = rm.n_alphas ? rm.alpha_sorted[rm.n_alphas - 1] : ~0u;
  auto recorded = [&](uint32_t t) {
    return t >= rm.burn_in && (rm.record_every == 1u || (t - rm.burn_in) % rm.record_every == 0);
  };
  uint32_t n_valid = 0u;
  const bool active = g * 32u + (uint32_t)lane < rm.chains;

#pragma unroll 1
  for (uint32_t i0 = 4u * (uint32_t)warp; i0 < n_sweeps; i0 += 4u * (uint32_t)nwarps) {
    uint32_t rec = 0u;  // the samples of this batch that are recorded
#pragma unroll
    for (uint32_t s = 0; s < 4u; ++s)
      if (i0 + s < n_sweeps && recorded(sweep0 + i0 + s)) rec |= 1u << s;
    if (!rec) continue;
    __syncwarp();
    // H outputs
#pragma unroll 2
    for (uint32_t idx = (uint32_t)lane; idx < h4; idx += 32u) {
      const uint32_t p = hp[idx >> 2], s = idx & 3u;
      img[4u * ((uint32_t)n + p) + s] =
          philox4x32_10(make_uint4(gglob, sweep0 + i0 + s, p | (kTagElim << 16), 0u), k0, k1).x;
    }
    __syncwarp();
    // the layers in order
    const uint32_t* lk = lnk + lane;
    uint32_t out = img_addr + 16u * (uint32_t)(n + lane);
#pragma unroll 1
    for (int k = 0; k < d; ++k, lk += n, out += 16u * (uint32_t)n) {
      if (lane < n) {
        const uint32_t e = *lk;
        if (e != 0xFFFFFFFFu) {
          const uint4 a = lds4(img_addr + (e & 0xFFFFu)), b = lds4(img_addr + (e >> 16));
          asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(out), "r"(a.x ^ b.x),
                       "r"(a.y ^ b.y), "r"(a.z ^ b.z), "r"(a.w ^ b.w)
                       : "memory");
        }
      }
      __syncwarp();
    }
    // phase terms of the four samples
    uint32_t f0[4], f1[4], f2[4];
#pragma unroll
    for (int s = 0; s < 4; ++s) f0[s] = f1[s] = f2[s] = 0u;
    uint32_t ea = sph_addr + 4u * (uint32_t)lane;
    auto terms = [&](uint32_t (&x)[4]) {
      const uint32_t e = lds(ea);
      const uint4 a = lds4(img_addr + (e & 0xFFFFu)), b = lds4(img_addr + (e >> 16));
      x[0] = a.x & b.x; x[1] = a.y & b.y; x[2] = a.z & b.z; x[3] = a.w & b.w;
      ea += 128u;
    };
#pragma unroll 1
    for (int k = 0; k < n_ph1; k += 32) {
      uint32_t x[4];
      terms(x);
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        const uint32_t c0 = f0[s] & x[s];
        f0[s] ^= x[s];
        f2[s] ^= f1[s] & c0;
        f1[s] ^= c0;
      }
    }
#pragma unroll 1
    for (int k = 0; k < n_ph2; k += 32) {
      uint32_t x[4];
      terms(x);
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        f2[s] ^= f1[s] & x[s];
        f1[s] ^= x[s];
      }
    }
#pragma unroll 2
    for (int k = 0; k < n_ph4; k += 32) {
      uint32_t x[4];
      terms(x);
#pragma unroll
      for (int s = 0; s < 4; ++s) f2[s] ^= x[s];
    }
    // reduced together: two halving steps leave sample lane / 8 with its lanes
#pragma unroll
    for (int w = 2; w > 0; w >>= 1) {
      const int off = 8 * w;
      const bool hi = (lane & off) != 0;
#pragma unroll
      for (int s = 0; s < w; ++s) {
        const uint32_t o0 = __shfl_xor_sync(0xffffffffu, hi ? f0[s] : f0[s + w], off);
        const uint32_t o1 = __shfl_xor_sync(0xffffffffu, hi ? f1[s] : f1[s + w], off);
        const uint32_t o2 = __shfl_xor_sync(0xffffffffu, hi ? f2[s] : f2[s + w], off);
        if (hi) { f0[s] = f0[s + w]; f1[s] = f1[s + w]; f2[s] = f2[s + w]; }
        add3(f0[s], f1[s], f2[s], o0, o1, o2);
      }
    }
#pragma unroll
    for (int off = 4; off > 0; off >>= 1) {
      const uint32_t o0 = __shfl_xor_sync(0xffffffffu, f0[0], off);
      const uint32_t o1 = __shfl_xor_sync(0xffffffffu, f1[0], off);
      const uint32_t o2 = __shfl_xor_sync(0xffffffffu, f2[0], off);
      add3(f0[0], f1[0], f2[0], o0, o1, o2);
    }
    const int r = lane & 7;
    const uint32_t plane = r == 0 ? f0[0] : (r == 1 ? f1[0] : f2[0]);
    // lane = chain within the group: rows 0..2 of a transpose the planes, then
    // the last layer (29 qubits at most; beyond, a transpose of its own)
    const Transpose tr(lane);
    const bool one = n <= 29;
    const int q = one ? lane - 3 : lane;
    const bool in = q >= 0 && q < n;
    const uint4 last = lds4(img_addr + 16u * (uint32_t)(d * n + (in ? q : 0)));
    const uint32_t row[4] = {last.x, last.y, last.z, last.w};
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      if (!((rec >> s) & 1u)) continue;
      const uint32_t pl = __shfl_sync(0xffffffffu, plane, 8 * s + (lane & 3));
      uint32_t word = in ? row[s] : 0u, alpha, phase;
      if (one) {
        word = tr(lane < 3 ? pl : word, lane);
        alpha = word >> 3;
        phase = word & 7u;
      } else {
        alpha = tr(word, lane);
        phase = tr(lane < 3 ? pl : 0u, lane) & 7u;
      }
      if (active && alpha >= a_lo && alpha <= a_hi) {
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
      n_valid += (uint32_t)__popc(__ballot_sync(0xffffffffu, active));
    }
  }
  if (lane == 0 && n_valid) {  // every sample is valid
    atomicAdd(&rm.valid[batch], (unsigned long long)n_valid);
    atomicAdd(&rm.samples[batch], (unsigned long long)n_valid);
  }
  // the group's state: the path of the launch's last recorded sample
  int last = -1;
#pragma unroll 1
  for (int i = (int)n_sweeps - 1; i >= 0; --i)
    if (recorded(sweep0 + (uint32_t)i)) { last = i; break; }
  if (last >= 0 && warp == (last >> 2) % nwarps) {
    __syncwarp();
    uint32_t* out = rm.state + (size_t)g * npb;
    for (int i = lane; i < npb; i += 32) out[i] = img[4 * (n + i) + (last & 3)];
  }
  __syncthreads();
  if (shist) {
    unsigned long long* gh = rm.hist + (size_t)batch * rm.bins * 8u;
#pragma unroll 1
    for (uint32_t i = tid; i < rm.bins * 8u; i += T)
      if (shist[i]) atomicAdd(&gh[i], (unsigned long long)shist[i]);
  }
  // the last CTA to finish advances the sample index
  if (tid == 0 && atomicAdd(&hdr->ctas_done, 1u) == gridDim.x - 1u) {
    hdr->ctas_done = 0u;
    hdr->sweep0 = sweep0 + n_launch;
  }
}

}  // namespace

size_t elim_plain_smem_bytes(int n, int d, uint32_t hist_bins, int warps) {
  const ElimLayout L = elim_layout(n, d, hist_bins);
  return 4 * ((size_t)L.img + (size_t)warps * L.img_words);
}

cudaError_t launch_elim_plain(const RunModelDev* d_rm, int n_models, uint32_t total_groups,
                              const uint32_t* const* d_init_tabs, uint32_t n_sweeps,
                              size_t smem_bytes, int warps, WsHeader* hdr, cudaStream_t st) {
  elim_plain_kernel<<<total_groups, 32 * warps, smem_bytes, st>>>(d_rm, n_models, d_init_tabs,
                                                                  n_sweeps, hdr);
  return cudaGetLastError();
}

cudaError_t elim_plain_prepare() {
  return cudaFuncSetAttribute(elim_plain_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)kSweepSmemMax);
}

}  // namespace pb
