// BF16 tensor-core GEMM on tcgen05 (sm_103a) and the small kernels around
// it that the learned proposal's MLP needs (forward, backward, Adam).
//
// gemm_tile: D[M x N] = epilogue(alpha * A[M x K] * B[N x K]^T), A and B bf16
// row-major with K contiguous ("TN"), accumulation in fp32 in TMEM.  One CTA
// computes a TM x BN tile (TM 64 or 128, BN <= 256): K passes
// through shared memory in chunks of 128 (canonical K-major layout) in up to
// four stages filled by cp.async while earlier chunks multiply; one thread
// issues the MMAs of a chunk and commits them to the stage's mbarrier, all
// threads wait (bounded) before the stage is filled again, and the warps read
// their TMEM lanes for the epilogue.  What bounds it at the network's sizes
// (256 x 256 weights, 4096 rows) is latency, not rate: a launch of a few
// hundred tiles with one to 32 chunks each.  Small tiles where the rows
// leave SMs idle, and the stages, are for that: the weight gradients (K =
// 4096 rows) took 64 chunks one after the other, load, multiply, wait, 350 of
// a training step's 583 us.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "pb_internal.h"
#include "philox.cuh"
#include "tc_gemm.cuh"

#include <algorithm>
#include <cmath>
#include <new>
#include <vector>

namespace pb {

enum : int {
  kEpiRelu = 1,     // max(x, 0)
  kEpiOutBf16 = 2,  // store bf16 (else fp32)
  kEpiAccum = 4,    // fp32 output: D += x
  kEpiMask = 8,     // x *= (mask[row, col] > 0)   (ReLU derivative)
  kEpiBce = 16,     // fp32 logits: also the cross-entropy's gradient and terms
  kEpiPublic = kEpiRelu | kEpiOutBf16 | kEpiAccum | kEpiMask,  // flags of pb_gemm_bf16
};

struct GemmArgs {
  const __nv_bfloat16* A;
  const __nv_bfloat16* B;
  void* D;
  const float* bias;  // per output column, may be null
  const __nv_bfloat16* mask;
  int lda, ldb, ldd, ldm;
  int M, N, K;
  int flags;
  float alpha;
  uint32_t* status;  // set to PB_ETIMEOUT when a bounded wait expires
  __nv_bfloat16* Dt;  // when set: the result transposed, bf16 [N x ldt]
  int ldt;
  // kEpiBce (fp32 logits, N = npad >= n): the gradient of the binary cross-
  // entropy against target [M x n], dY = (sigmoid(l) - t) / M, bf16 in D2 and
  // Dt, and the loss terms (fp32 [M x n])
  const float* target;
  __nv_bfloat16* D2;
  float* terms;
  int n;
  int tm, bn;  // tile (gemm_tiles)
};

constexpr int kGemmK = 128;  // K elements of a stage (the copies in gemm_tile cover 16 columns of 8)
constexpr size_t kGemmSmemMax = 200 * 1024;
__host__ __device__ inline size_t gemm_stage_bytes(int tm, int bn) {
  return (size_t)(tm + bn) * kGemmK * 2;
}
__host__ __device__ inline int gemm_stages(int tm, int bn) {
  return 4 * gemm_stage_bytes(tm, bn) <= kGemmSmemMax ? 4 : 2;
}
// Tile: 128 rows and N rounded up to 16, at most 256, narrowed step by step to
// 64 x 32 while the tiles would leave most of the 152 SMs idle.  A result that
// lies over an operand (in_place) keeps at least 64 columns a tile: with one
// tile across N, a CTA has read all it needs of the rows that it writes (M <=
// 128 too: all of B), which smaller tiles would lose.
inline void gemm_tiles(GemmArgs& g, bool in_place) {
  int bn = ((g.N + 15) / 16) * 16, tm = 128;
  if (bn > 256) bn = 256;
  auto tiles = [&] { return ((g.M + tm - 1) / tm) * ((g.N + bn - 1) / bn); };
  if (bn > 128 && tiles() < 120) bn = 128;
  if (bn > 64 && tiles() < 120) bn = 64;
  if (!in_place && tiles() < 120) tm = 64;
  if (!in_place && bn > 32 && tiles() < 120) bn = 32;
  g.tm = tm;
  g.bn = bn;
}
__host__ __device__ inline uint32_t tmem_cols(int bn) {
  uint32_t c = 32;
  while ((int)c < bn) c <<= 1;
  return c;
}

// dY element and loss term of one logit (rows B).
__device__ __forceinline__ float bce_grad(float l, float t, int B) {
  return (1.f / (1.f + __expf(-l)) - t) / (float)B;
}
__device__ __forceinline__ float bce_term(float l, float t, int B) {
  return (fmaxf(l, 0.f) + log1pf(__expf(-fabsf(l))) - t * l) / (float)B;
}

// One tile (m0, n0) by a CTA of nine warps: eight copy and do the epilogue (two
// to a quadrant of TMEM lanes, each with half of the columns), the ninth
// issues the MMAs; S stages of dynamic shared memory at sm.  F: the flags, or
// -1 to read them from g; CTM, CBN: the tile, or 0 to read it from g.
constexpr int kGemmThreads = 288;
template <int S, int F, int CTM = 0, int CBN = 0>
__device__ __forceinline__ void gemm_tile(const GemmArgs& g, int m0, int n0, uint8_t* sm,
                                          uint64_t* mbar, uint32_t* tmem_base) {
  const int TM = CTM ? CTM : g.tm, BN = CBN ? CBN : g.bn;
  const uint32_t a_bytes = (uint32_t)TM * kGemmK * 2, stage = (uint32_t)gemm_stage_bytes(TM, BN);
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const uint32_t ncols = tmem_cols(BN);
  const int flags = F >= 0 ? F : g.flags;

  if (warp == 0) tc::tmem_alloc(tmem_base, ncols);
  if (tid == 0) {
    for (int s = 0; s < S; ++s) tc::mbar_init(&mbar[s], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // chunk c (K elements 128 c ..) into its stage: two 64-wide halves, each in
  // the canonical layout.  A thread copies one 8-element column of every
  // second 8-row group, so that its addresses only advance by constants (a
  // copy costs a handful of instructions, which is what paces a tile with few
  // warps); a warp copies 8 rows x 4 columns: 64-byte pieces of the rows, and
  // in shared memory 128-byte core matrices without bank conflicts.
  const int nch = (g.K + kGemmK - 1) / kGemmK;
  const int lr = (warp >> 2) * 8 + (lane & 7), lk = ((warp & 3) * 4 + (lane >> 3)) * 8;
  const uint32_t lo = tc::smem_u32(sm) + tc::chunk_offset(lr, lk & 63);
  const __nv_bfloat16* pa = g.A + (size_t)(m0 + lr) * g.lda + lk;
  const __nv_bfloat16* pb = g.B + (size_t)(n0 + lr) * g.ldb + lk;
  const bool whole = m0 + TM <= g.M && n0 + BN <= g.N;
  auto load = [&](int c) {
    if (c < nch) {
      uint32_t d = lo + (uint32_t)(c % S) * stage + (uint32_t)(lk >> 6) * (uint32_t)TM * 128u;
      uint32_t e = lo + (uint32_t)(c % S) * stage + a_bytes + (uint32_t)(lk >> 6) * (uint32_t)BN * 128u;
      const __nv_bfloat16 *q = pa, *w = pb;
      if (whole && (c + 1) * kGemmK <= g.K) {
#pragma unroll 4
        for (int r = 0; r < TM; r += 16, d += 2048u, q += (size_t)16 * g.lda) tc::cp_async16(d, q, 16u);
#pragma unroll 4
        for (int r = 0; r < BN; r += 16, e += 2048u, w += (size_t)16 * g.ldb)
          tc::cp_async16(e, w, 16u);
      } else {
        const bool kin = c * kGemmK + lk < g.K;
        const int ra = kin ? g.M - m0 - lr : 0, rb = kin ? g.N - n0 - lr : 0;  // rows left
#pragma unroll 1
        for (int r = 0; r < TM; r += 16, d += 2048u, q += (size_t)16 * g.lda)
          tc::cp_async16(d, r < ra ? (const void*)q : (const void*)g.A, r < ra ? 16u : 0u);
#pragma unroll 1
        for (int r = 0; r < BN; r += 16, e += 2048u, w += (size_t)16 * g.ldb)
          tc::cp_async16(e, r < rb ? (const void*)w : (const void*)g.B, r < rb ? 16u : 0u);
      }
      pa += kGemmK;
      pb += kGemmK;
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  // chunks loaded ahead; with four stages the MMAs of the previous chunk may
  // still run while the next ones are issued
  constexpr int A = S >= 4 ? S - 2 : S - 1;
  const bool copier = warp < 8;
  if (copier) {
#pragma unroll
    for (int c = 0; c < A; ++c) load(c);
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tbase = *tmem_base;
  const uint32_t idesc = tc::idesc_bf16_f32(TM, BN);
  bool ok = true;
  auto done = [&](int c) { return tc::mbar_wait(&mbar[c % S], (uint32_t)(c / S) & 1u); };

  for (int c = 0; c < nch; ++c) {
    if (copier) {
      asm volatile("cp.async.wait_group %0;" ::"n"(A - 1) : "memory");
      tc::fence_proxy_async_smem();
    }
    // publishes chunk c, and that the MMAs of chunk c + A - S are done; one
    // decision for the whole CTA (the loop has barriers)
    ok = __syncthreads_and(ok) != 0;
    if (!ok) break;
    if (copier) {
      load(c + A);  // into the stage of chunk c + A - S
    } else if (lane == 0) {
      tc::fence_after_sync();
      const uint32_t a0 = tc::smem_u32(sm) + (uint32_t)(c % S) * stage;
      // descriptors advance by constants (16-byte units): a K-step covers two
      // 8-wide K columns (LBO apart), four steps a 64-wide half
      uint64_t ad = tc::smem_desc(a0, tc::kLBO, tc::kSBO);
      uint64_t bd = tc::smem_desc(a0 + a_bytes, tc::kLBO, tc::kSBO);
      const int steps = min(kGemmK / 16, (g.K - c * kGemmK + 15) / 16);
      if (steps == kGemmK / 16) {
#pragma unroll
        for (int s = 0; s < kGemmK / 16; ++s)
          tc::mma_bf16(tbase, ad + (uint32_t)((s >> 2) * TM * 8 + (s & 3) * 16),
                       bd + (uint32_t)((s >> 2) * BN * 8 + (s & 3) * 16), idesc, (c > 0) || (s > 0));
      } else {
#pragma unroll 1
        for (int s = 0; s < steps; ++s)
          tc::mma_bf16(tbase, ad + (uint32_t)((s >> 2) * TM * 8 + (s & 3) * 16),
                       bd + (uint32_t)((s >> 2) * BN * 8 + (s & 3) * 16), idesc, (c > 0) || (s > 0));
      }
      tc::mma_commit(&mbar[c % S]);
      // before the next barrier: the stage that the copies after it fill
      const int p = c + 1 + A - S;
      if (p >= 0) ok = done(p);
    }
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  if (ok) ok = done(nch - 1);
  ok = __syncthreads_and(ok) != 0;
  if (!ok && tid == kGemmThreads - 32) {
    if (g.status) atomicCAS(g.status, 0u, (uint32_t)PB_ETIMEOUT);
    done(nch - 1);  // let MMAs in flight drain (bounded)
  }
  tc::fence_after_sync();

  if (ok && copier) {
    // accumulator rows: TM = 128: TMEM lane = row; TM = 64: row r at lane
    // 32 (r / 16) + r % 16
    const int quad = warp & 3;
    const int row = m0 + (TM == 128 ? quad * 32 + lane : quad * 16 + lane);
    const bool live = row < g.M && (TM == 128 || lane < 16);
    for (int c0 = (warp >> 2) * 16; c0 < BN; c0 += 32) {
      float v[16];
      tc::tmem_ld16(tbase + ((uint32_t)(quad * 32) << 16) + (uint32_t)c0, v);
      if (!live) continue;
      const int col0 = n0 + c0;
      const bool full = col0 + 16 <= g.N;
      __align__(16) __nv_bfloat16 mk[16];
      if ((flags & kEpiMask) && full && (g.ldm & 7) == 0 && ((uintptr_t)g.mask & 15) == 0) {
        const uint4* src = reinterpret_cast<const uint4*>(g.mask + (size_t)row * g.ldm + col0);
        reinterpret_cast<uint4*>(mk)[0] = src[0];
        reinterpret_cast<uint4*>(mk)[1] = src[1];
      } else if (flags & kEpiMask) {
#pragma unroll
        for (int i = 0; i < 16; ++i)
          mk[i] = col0 + i < g.N ? g.mask[(size_t)row * g.ldm + col0 + i] : __float2bfloat16(0.f);
      }
      float bs[16];
      const bool bias = g.bias != nullptr;
      if (bias && full && ((uintptr_t)(g.bias + col0) & 15) == 0) {
#pragma unroll
        for (int i = 0; i < 16; i += 4) {
          const float4 x = *reinterpret_cast<const float4*>(g.bias + col0 + i);
          bs[i] = x.x; bs[i + 1] = x.y; bs[i + 2] = x.z; bs[i + 3] = x.w;
        }
      } else if (bias) {
#pragma unroll
        for (int i = 0; i < 16; ++i) bs[i] = col0 + i < g.N ? g.bias[col0 + i] : 0.f;
      }
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const int col = col0 + i;
        if (col >= g.N) continue;
        float x = g.alpha * v[i];
        if (bias) x += bs[i];
        if (flags & kEpiRelu) x = fmaxf(x, 0.f);
        if (flags & kEpiMask) x = (__bfloat162float(mk[i]) > 0.f) ? x : 0.f;
        v[i] = x;
      }
      if (flags & kEpiBce) {
        __align__(16) __nv_bfloat16 gb[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const int col = col0 + i;
          float d = 0.f;
          if (col < g.n) {
            const float t = g.target[(size_t)row * g.n + col];
            d = bce_grad(v[i], t, g.M);
            g.terms[(size_t)row * g.n + col] = bce_term(v[i], t, g.M);
          }
          gb[i] = __float2bfloat16(d);
          if (col < g.N) g.Dt[(size_t)col * g.ldt + row] = gb[i];
        }
        // (rows of npad elements, a multiple of 16)
        uint4* dst = reinterpret_cast<uint4*>(g.D2 + (size_t)row * g.N + col0);
        dst[0] = reinterpret_cast<const uint4*>(gb)[0];
        dst[1] = reinterpret_cast<const uint4*>(gb)[1];
      }
      if (flags & kEpiOutBf16) {
        __align__(16) __nv_bfloat16 o[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) o[i] = __float2bfloat16(v[i]);
        __nv_bfloat16* d = reinterpret_cast<__nv_bfloat16*>(g.D);
        if (d) {
          d += (size_t)row * g.ldd + col0;
          if (full && (g.ldd & 7) == 0 && ((uintptr_t)g.D & 15) == 0) {
            reinterpret_cast<uint4*>(d)[0] = reinterpret_cast<const uint4*>(o)[0];
            reinterpret_cast<uint4*>(d)[1] = reinterpret_cast<const uint4*>(o)[1];
          } else {
#pragma unroll
            for (int i = 0; i < 16; ++i)
              if (col0 + i < g.N) d[i] = o[i];
          }
        }
        if (g.Dt) {
#pragma unroll
          for (int i = 0; i < 16; ++i)
            if (col0 + i < g.N) g.Dt[(size_t)(col0 + i) * g.ldt + row] = o[i];
        }
      } else {
        float* d = reinterpret_cast<float*>(g.D) + (size_t)row * g.ldd + col0;
        if (full && !(flags & kEpiAccum) && (g.ldd & 3) == 0 && ((uintptr_t)g.D & 15) == 0) {
#pragma unroll
          for (int i = 0; i < 16; i += 4)
            *reinterpret_cast<float4*>(d + i) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
        } else {
#pragma unroll
          for (int i = 0; i < 16; ++i)
            if (col0 + i < g.N) d[i] = (flags & kEpiAccum) ? d[i] + v[i] : v[i];
        }
      }
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tbase, ncols);
}

template <int S, int F>
__global__ void __launch_bounds__(kGemmThreads) gemm_bf16_tn_kernel(GemmArgs g) {
  extern __shared__ __align__(1024) uint8_t sm[];
  __shared__ uint64_t mbar[S];
  __shared__ uint32_t tmem_base;
  gemm_tile<S, F>(g, blockIdx.x * g.tm, blockIdx.y * g.bn, sm, mbar, &tmem_base);
}

// The kernel for a tile and flags: four stages where they fit (the network's
// own layers, by their flags), else two.
typedef void (*GemmKernel)(GemmArgs);
inline GemmKernel gemm_kernel(const GemmArgs& g) {
  if (gemm_stages(g.tm, g.bn) != 4) return gemm_bf16_tn_kernel<2, -1>;
  switch (g.flags) {
    case kEpiRelu | kEpiOutBf16: return gemm_bf16_tn_kernel<4, kEpiRelu | kEpiOutBf16>;
    case kEpiMask | kEpiOutBf16: return gemm_bf16_tn_kernel<4, kEpiMask | kEpiOutBf16>;
    case kEpiBce: return gemm_bf16_tn_kernel<4, kEpiBce>;
    default: return gemm_bf16_tn_kernel<4, -1>;
  }
}

// One-time set-up outside any stream capture (shared-memory opt-in).
cudaError_t mlp_fused_prepare();
cudaError_t grads_prepare();
cudaError_t mlp_prepare() {
  const cudaFuncAttribute a = cudaFuncAttributeMaxDynamicSharedMemorySize;
  cudaError_t e = cudaSuccess;
  for (GemmKernel k : {(GemmKernel)gemm_bf16_tn_kernel<2, -1>, (GemmKernel)gemm_bf16_tn_kernel<4, -1>,
                       (GemmKernel)gemm_bf16_tn_kernel<4, kEpiRelu | kEpiOutBf16>,
                       (GemmKernel)gemm_bf16_tn_kernel<4, kEpiMask | kEpiOutBf16>,
                       (GemmKernel)gemm_bf16_tn_kernel<4, kEpiBce>})
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, a, (int)kGemmSmemMax);
  if (e == cudaSuccess) e = grads_prepare();
  return e == cudaSuccess ? mlp_fused_prepare() : e;
}

// g with its tile chosen; the kernel opted in (mlp_prepare).
cudaError_t launch_gemm_tiled(const GemmArgs& g, cudaStream_t st) {
  dim3 grid((g.M + g.tm - 1) / g.tm, (g.N + g.bn - 1) / g.bn);
  const size_t smem = (size_t)gemm_stages(g.tm, g.bn) * gemm_stage_bytes(g.tm, g.bn);
  gemm_kernel(g)<<<grid, kGemmThreads, smem, st>>>(g);
  return cudaGetLastError();
}
cudaError_t launch_gemm_bf16(GemmArgs g, cudaStream_t st) {
  gemm_tiles(g, false);
  return launch_gemm_tiled(g, st);
}

}  // namespace pb

namespace pb {

// Self-test of the bounded wait every tensor-core kernel here uses: one
// thread initialises a one-arrival mbarrier, arrives on it or not, and
// waits for its first phase with tc::mbar_wait(max_iters).  A wait that runs
// out records PB_ETIMEOUT in the status word the way the GEMM and fused
// kernels do; nothing else (no MMA, no copy, no tensor memory) is in flight.
__device__ uint32_t g_selftest_status;

__global__ void selftest_wait_kernel(int arrive, uint32_t max_iters) {
  __shared__ __align__(8) uint64_t mbar;
  if (threadIdx.x != 0) return;
  tc::mbar_init(&mbar, 1u);
  if (arrive) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc::smem_u32(&mbar)) : "memory");
  }
  const bool ok = tc::mbar_wait(&mbar, 0u, max_iters);
  if (!ok) atomicCAS(&g_selftest_status, 0u, (uint32_t)PB_ETIMEOUT);
  asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(tc::smem_u32(&mbar)) : "memory");
}

}  // namespace pb

using namespace pb;

extern "C" PB_API int pb_gemm_bf16(const void* dA, int lda, const void* dB, int ldb, void* dD,
                                   int ldd, const float* dbias, const void* dmask, int ldm, int M,
                                   int N, int K, int flags, float alpha, uintptr_t stream) {
  if (!dA || !dB || !dD || M <= 0 || N <= 0 || K <= 0) return PB_EINVAL;
  if ((K % 8) || (lda % 8) || (ldb % 8) || lda < K || ldb < K || ldd < N) return PB_EINVAL;
  if (((uintptr_t)dA & 15) || ((uintptr_t)dB & 15)) return PB_EINVAL;
  if ((flags & kEpiMask) && (!dmask || ldm < N)) return PB_EINVAL;
  flags &= kEpiPublic;  // (kEpiBce would write through pointers that this call does not have)
  GemmArgs g{};
  g.A = static_cast<const __nv_bfloat16*>(dA);
  g.B = static_cast<const __nv_bfloat16*>(dB);
  g.D = dD;
  g.bias = dbias;
  g.mask = static_cast<const __nv_bfloat16*>(dmask);
  g.lda = lda;
  g.ldb = ldb;
  g.ldd = ldd;
  g.ldm = ldm;
  g.M = M;
  g.N = N;
  g.K = K;
  g.flags = flags;
  g.alpha = alpha;
  g.status = nullptr;
  const uintptr_t d0 = (uintptr_t)dD, d1 = d0 + ((size_t)(M - 1) * ldd + N) * (flags & kEpiOutBf16 ? 2 : 4);
  auto over = [&](const void* p, int rows, int ld) {
    const uintptr_t x = (uintptr_t)p;
    return x < d1 && d0 < x + ((size_t)(rows - 1) * ld + K) * 2;
  };
  gemm_tiles(g, over(dA, M, lda) || over(dB, N, ldb));
  // opt in the one kernel that runs (all of the network's on every call cost
  // 3 us: a 128 x 128 x 128 call 12.2 -> 9.3 us, host bound)
  if (cudaFuncSetAttribute(gemm_kernel(g), cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)kGemmSmemMax) != cudaSuccess)
    return PB_ECUDA;
  return launch_gemm_tiled(g, reinterpret_cast<cudaStream_t>(stream)) == cudaSuccess ? PB_OK : PB_ECUDA;
}

// ===========================================================================
// The proposal network q(s_j | s_{j-1}, j): K_in -> H -> H -> n, ReLU, BF16
// tensor-core GEMMs with fp32 accumulation, fp32 master weights and Adam.
// ===========================================================================
namespace pb {

// Parameter block (fp32, flat): W1 [H x kin], b1 [H], W2 [H x H], b2 [H],
// W3 [npad x H] (rows >= n stay zero), b3 [npad].
struct MlpOffsets {
  size_t W1, b1, W2, b2, W3, b3, total;
};
inline MlpOffsets mlp_offsets(int kin, int H, int npad) {
  MlpOffsets o;
  size_t p = 0;
  o.W1 = p; p += (size_t)H * kin;
  o.b1 = p; p += H;
  o.W2 = p; p += (size_t)H * H;
  o.b2 = p; p += H;
  o.W3 = p; p += (size_t)npad * H;
  o.b3 = p; p += npad;
  o.total = p;
  return o;
}

__global__ void transpose_bf16_kernel(const __nv_bfloat16* __restrict__ src, int R, int C,
                                      __nv_bfloat16* __restrict__ dst) {
  __shared__ __nv_bfloat16 tile[32][33];
  const int c0 = blockIdx.x * 32, r0 = blockIdx.y * 32;
  for (int i = threadIdx.y; i < 32; i += 8) {
    const int r = r0 + i, c = c0 + threadIdx.x;
    if (r < R && c < C) tile[i][threadIdx.x] = src[(size_t)r * C + c];
  }
  __syncthreads();
  for (int i = threadIdx.y; i < 32; i += 8) {
    const int c = c0 + i, r = r0 + threadIdx.x;
    if (r < R && c < C) dst[(size_t)c * R + r] = tile[threadIdx.x][i];
  }
}

cudaError_t transpose_bf16(const __nv_bfloat16* src, int R, int C, __nv_bfloat16* dst,
                           cudaStream_t st) {
  dim3 grid((C + 31) / 32, (R + 31) / 32), block(32, 8);
  transpose_bf16_kernel<<<grid, block, 0, st>>>(src, R, C, dst);
  return cudaGetLastError();
}

// Every parameter's bf16 copies from one fp32 weight (index i of the flat
// block): the row-major copy, the transpose the backward pass reads, and the
// canonical K-major image the fused kernels load: core matrices of 8 rows x
// 8 elements (128 bytes), K-adjacent ones 128 bytes apart, 8-row groups
// 16 K bytes apart (W2 in K-chunks of 64).
struct Bf16Views {
  __nv_bfloat16 *W1, *W2, *W3, *W2t, *W3t, *W1p, *W2p, *W3p;
  int kin, H, npad;
};
__device__ __forceinline__ uint32_t canonical_index(int r, int c, int K) {
  return (uint32_t)((r >> 3) * (K * 8) + (c >> 3) * 64 + (r & 7) * 8 + (c & 7));
}
__device__ __forceinline__ void write_bf16(const Bf16Views& b, uint32_t i, float w) {
  const uint32_t n1 = (uint32_t)(b.H * b.kin), n2 = (uint32_t)(b.H * b.H), n3 = (uint32_t)(b.npad * b.H);
  const uint32_t H = (uint32_t)b.H;
  const __nv_bfloat16 v = __float2bfloat16(w);
  if (i < n1) {  // W1 [H x kin]
    b.W1[i] = v;
    const uint32_t r = i / (uint32_t)b.kin;
    b.W1p[canonical_index((int)r, (int)(i - r * (uint32_t)b.kin), b.kin)] = v;
    return;
  }
  i -= n1;
  if (i < H) return;  // b1
  i -= H;
  if (i < n2) {  // W2 [H x H]
    b.W2[i] = v;
    const uint32_t r = i / H, c = i - r * H;
    b.W2t[c * H + r] = v;
    const uint32_t k0 = c & ~63u;
    b.W2p[H * k0 + canonical_index((int)r, (int)(c - k0), (int)min(64u, H - k0))] = v;
    return;
  }
  i -= n2;
  if (i < H) return;  // b2
  i -= H;
  if (i < n3) {  // W3 [npad x H]
    b.W3[i] = v;
    const uint32_t r = i / H, c = i - r * H;
    b.W3t[c * (uint32_t)b.npad + r] = v;
    b.W3p[canonical_index((int)r, (int)c, b.H)] = v;
  }
}
__global__ void refresh_bf16_kernel(const float* __restrict__ w, uint32_t count, Bf16Views b) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < count) write_bf16(b, i, w[i]);
}

// The weight gradients of one backward pass in one launch: tiles of gW2, gW1
// and gW3 (each a sum over the rows, K = rows), then the bias gradients (one
// warp per row of dZ2t / dZ1t), the n columns of db3 and the loss.  Every sum
// is taken in a fixed order, so that a training run is reproducible bit for
// bit.
struct GradArgs {
  GemmArgs w[3];        // gW2, gW1, gW3
  int tiles[3], mt[3];  // tiles of each, tiles along M
  const __nv_bfloat16 *dZ2t, *dZ1t;
  float *db2, *db1, *db3, *loss;
  const float *logits, *target, *terms;
  int H, B, n, npad;
};
constexpr int kGradStages = 4;
constexpr int kGradTm = 64, kGradBn = 16;  // 20 KB a stage

// out[j] = sum_b M[j][b] (bf16 rows, fp32 sums), one warp per row.
__device__ __forceinline__ void rowsum_bf16(const __nv_bfloat16* __restrict__ row, int C, int lane,
                                            float* __restrict__ out) {
  float s = 0.f;
#pragma unroll 8
  for (int c = lane; c < C; c += 32) s += __bfloat162float(row[c]);
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  if (lane == 0) *out = s;
}

__global__ void __launch_bounds__(kGemmThreads) grads_kernel(GradArgs a) {
  extern __shared__ __align__(1024) uint8_t sm[];
  __shared__ uint64_t mbar[kGradStages];
  __shared__ uint32_t tmem_base;
  __shared__ float part[256];
  int b = blockIdx.x;
  const int tid = threadIdx.x;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    if (b < a.tiles[k]) {
      gemm_tile<kGradStages, 0, kGradTm, kGradBn>(a.w[k], (b % a.mt[k]) * kGradTm,
                                                  (b / a.mt[k]) * kGradBn, sm, mbar, &tmem_base);
      return;
    }
    b -= a.tiles[k];
  }
  constexpr int kRows = 8;
  if (tid >= 256) return;  // (the ninth warp: MMAs only)
  const int rs = (a.H + kRows - 1) / kRows;  // bias rows, one warp each
  if (b < 2 * rs) {
    const int row = (b < rs ? b : b - rs) * kRows + (tid >> 5);
    if (row < a.H)
      rowsum_bf16((b < rs ? a.dZ2t : a.dZ1t) + (size_t)row * a.B, a.B, tid & 31,
                  (b < rs ? a.db2 : a.db1) + row);
    return;
  }
  // 256 strided partial sums and a tree: db3[c] (fp32 gradients), or the loss
  const int c = b - 2 * rs;
  float acc = 0.f;
  if (c < a.n) {
#pragma unroll 4
    for (int r = tid; r < a.B; r += 256)
      acc += bce_grad(a.logits[(size_t)r * a.npad + c], a.target[(size_t)r * a.n + c], a.B);
  } else {
#pragma unroll 8
    for (int i = tid; i < a.B * a.n; i += 256) acc += a.terms[i];
  }
  part[tid] = acc;
  __syncthreads();
  for (int s = 128; s > 0; s >>= 1) {
    if (tid < s) part[tid] += part[tid + s];
    __syncthreads();
  }
  if (tid == 0) *(c < a.n ? a.db3 + c : a.loss) = part[0];
}
cudaError_t grads_prepare() {
  return cudaFuncSetAttribute(grads_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)(kGradStages * gemm_stage_bytes(kGradTm, kGradBn)));
}

// One Adam step, the bf16 copies with it; the padded rows of W3 / b3 (flat
// indices in [z0, z1) and [z2, z3)) stay zero.
__global__ void adam_kernel(float* __restrict__ w, const float* __restrict__ g, float* __restrict__ m,
                            float* __restrict__ v, uint32_t count, float lr, float b1, float b2,
                            float eps, float c1, float c2, uint32_t z0, uint32_t z1, uint32_t z2,
                            uint32_t z3, Bf16Views b) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  const float gi = g[i];
  const float mi = b1 * m[i] + (1.f - b1) * gi;
  const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  float x = w[i];
  x -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  if ((i >= z0 && i < z1) || (i >= z2 && i < z3)) x = 0.f;
  w[i] = x;
  write_bf16(b, i, x);
}

}  // namespace pb

namespace {

struct MlpLayout {
  size_t w, m, v, g, W1, W2, W3, W2t, W3t, W1p, W2p, W3p, X, Xt, H1, H1t, H2, H2t, dY, dYt, dZ2,
      dZ2t, dZ1t, logits, target, terms, loss, status, total;
};

MlpLayout mlp_layout(int kin, int H, int npad, int B) {
  const pb::MlpOffsets o = pb::mlp_offsets(kin, H, npad);
  MlpLayout L{};
  size_t p = 0;
  auto take = [&](size_t bytes) {
    p = (p + 255) & ~(size_t)255;
    size_t at = p;
    p += bytes;
    return at;
  };
  L.w = take(o.total * 4);
  L.m = take(o.total * 4);
  L.v = take(o.total * 4);
  L.g = take(o.total * 4);
  L.W1 = take((size_t)H * kin * 2);
  L.W2 = take((size_t)H * H * 2);
  L.W3 = take((size_t)npad * H * 2);
  L.W2t = take((size_t)H * H * 2);
  L.W3t = take((size_t)H * npad * 2);
  L.W1p = take((size_t)H * kin * 2);
  L.W2p = take((size_t)H * H * 2);
  L.W3p = take((size_t)npad * H * 2);
  L.X = take((size_t)B * kin * 2);
  L.Xt = take((size_t)B * kin * 2);
  L.H1 = take((size_t)B * H * 2);
  L.H1t = take((size_t)B * H * 2);
  L.H2 = take((size_t)B * H * 2);
  L.H2t = take((size_t)B * H * 2);
  L.dY = take((size_t)B * npad * 2);
  L.dYt = take((size_t)B * npad * 2);
  L.dZ2 = take((size_t)B * H * 2);
  L.dZ2t = take((size_t)B * H * 2);
  L.dZ1t = take((size_t)B * H * 2);
  L.logits = take((size_t)B * npad * 4);
  L.target = take((size_t)B * npad * 4);
  L.terms = take((size_t)B * npad * 4);
  L.loss = take(256);
  L.status = take(16);
  L.total = (p + 255) & ~(size_t)255;
  return L;
}

int mlp_dims(int n, int d, int hidden, int batch, int* kin, int* npad) {
  if (n < 1 || n > 32 || d < 1 || d > 64) return PB_ERANGE;
  if (hidden < 16 || hidden > 256 || hidden % 16) return PB_ERANGE;
  if (batch < 128 || batch % 128) return PB_ERANGE;
  *kin = ((n + d + 15) / 16) * 16;
  *npad = ((n + 15) / 16) * 16;
  return PB_OK;
}

// D = epi(A[M x K] B[N x K]^T) of this network (and its transpose, bf16
// [N x M], when Dt is set).
pb::GemmArgs mm(const pb_mlp* p, const __nv_bfloat16* A, int lda, const __nv_bfloat16* B, int ldb,
                void* D, int ldd, int M, int N, int K, int flags, const float* bias = nullptr,
                const __nv_bfloat16* mask = nullptr, __nv_bfloat16* Dt = nullptr) {
  pb::GemmArgs g{};
  g.A = A;
  g.B = B;
  g.D = D;
  g.bias = bias;
  g.mask = mask;
  g.lda = lda;
  g.ldb = ldb;
  g.ldd = ldd;
  g.ldm = ldd;
  g.M = M;
  g.N = N;
  g.K = K;
  g.flags = flags;
  g.alpha = 1.f;
  g.status = p->status;
  g.Dt = Dt;
  g.ldt = M;
  return g;
}

pb::Bf16Views bf16_views(const pb_mlp* p) {
  return {p->W1, p->W2, p->W3, p->W2t, p->W3t, p->W1p, p->W2p, p->W3p, p->kin, p->H, p->npad};
}

// bf16 copies of the fp32 master weights.
cudaError_t refresh_bf16(pb_mlp* p) {
  const unsigned c = (unsigned)p->n_params;
  pb::refresh_bf16_kernel<<<(c + 255) / 256, 256, 0, p->st>>>(p->w, c, bf16_views(p));
  return cudaGetLastError();
}

// Forward of `rows` inputs already in p->X: H1, H2 (bf16), logits (fp32).
// train: also what the backward pass needs -- the transposes of H1 and H2,
// the gradient of the logits against p->target and the loss terms.
cudaError_t mlp_fwd(pb_mlp* p, int rows, bool train) {
  cudaError_t e;
  const int flags = pb::kEpiRelu | pb::kEpiOutBf16, H = p->H;
  if ((e = pb::launch_gemm_bf16(mm(p, p->X, p->kin, p->W1, p->kin, p->H1, H, rows, H, p->kin, flags,
                                   p->w + p->off_b1, nullptr, train ? p->H1t : nullptr),
                                p->st)) != cudaSuccess)
    return e;
  if ((e = pb::launch_gemm_bf16(mm(p, p->H1, H, p->W2, H, p->H2, H, rows, H, H, flags,
                                   p->w + p->off_b2, nullptr, train ? p->H2t : nullptr),
                                p->st)) != cudaSuccess)
    return e;
  pb::GemmArgs g = mm(p, p->H2, H, p->W3, H, p->logits, p->npad, rows, p->npad, H,
                      train ? pb::kEpiBce : 0, p->w + p->off_b3, nullptr, p->dYt);
  g.target = p->target;
  g.D2 = p->dY;
  g.terms = p->terms;
  g.n = p->n;
  return pb::launch_gemm_bf16(g, p->st);
}

// Backward of the mean BCE over `rows` after mlp_fwd(.., train): gradients
// into p->g, loss into p->loss[0].  p->Xt holds the inputs' transpose.
cudaError_t mlp_bwd(pb_mlp* p, int rows) {
  cudaError_t e;
  const int B = rows, H = p->H;
  const int flags = pb::kEpiMask | pb::kEpiOutBf16;
  // dZ2 = (dY W3) * [H2 > 0], dZ1 = (dZ2 W2) * [H1 > 0] (its transpose only)
  if ((e = pb::launch_gemm_bf16(mm(p, p->dY, p->npad, p->W3t, p->npad, p->dZ2, H, B, H, p->npad, flags,
                                   nullptr, p->H2, p->dZ2t), p->st)) != cudaSuccess ||
      (e = pb::launch_gemm_bf16(mm(p, p->dZ2, H, p->W2t, H, nullptr, H, B, H, H, flags, nullptr, p->H1,
                                   p->dZ1t), p->st)) != cudaSuccess)
    return e;
  // gW2 = dZ2^T H1, gW1 = dZ1^T X, gW3 = dY^T H2, the bias gradients, the loss
  pb::GradArgs a{};
  a.w[0] = mm(p, p->dZ2t, B, p->H1t, B, p->g + p->off_W2, H, H, H, B, 0);
  a.w[1] = mm(p, p->dZ1t, B, p->Xt, B, p->g + p->off_W1, p->kin, H, p->kin, B, 0);
  a.w[2] = mm(p, p->dYt, B, p->H2t, B, p->g + p->off_W3, H, p->npad, H, B, 0);
  int total = 0;
  for (int k = 0; k < 3; ++k) {
    pb::GemmArgs& g = a.w[k];
    g.tm = pb::kGradTm;
    g.bn = pb::kGradBn;
    a.mt[k] = (g.M + g.tm - 1) / g.tm;
    a.tiles[k] = a.mt[k] * ((g.N + g.bn - 1) / g.bn);
    total += a.tiles[k];
  }
  a.dZ2t = p->dZ2t;
  a.dZ1t = p->dZ1t;
  a.db2 = p->g + p->off_b2;
  a.db1 = p->g + p->off_b1;
  a.db3 = p->g + p->off_b3;
  a.loss = p->loss;
  a.logits = p->logits;
  a.target = p->target;
  a.terms = p->terms;
  a.H = H;
  a.B = B;
  a.n = p->n;
  a.npad = p->npad;
  total += 2 * ((H + 7) / 8) + p->n + 1;
  pb::grads_kernel<<<total, pb::kGemmThreads, pb::kGradStages * pb::gemm_stage_bytes(pb::kGradTm, pb::kGradBn),
                     p->st>>>(a);
  return cudaGetLastError();
}

}  // namespace

namespace pb {
cudaError_t mlp_forward_rows(pb_mlp* p, int rows) { return mlp_fwd(p, rows, false); }
cudaError_t mlp_gradient_rows(pb_mlp* p, int rows) {
  const cudaError_t e = mlp_fwd(p, rows, true);
  return e == cudaSuccess ? mlp_bwd(p, rows) : e;
}
cudaError_t mlp_adam_step(pb_mlp* p, float lr) {
  p->step += 1;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - std::pow(b1, (float)p->step), c2 = 1.f - std::pow(b2, (float)p->step);
  const uint32_t c = (uint32_t)p->n_params, H = (uint32_t)p->H;
  const uint32_t w3 = (uint32_t)p->off_W3, b3 = (uint32_t)p->off_b3, n = (uint32_t)p->n, np = (uint32_t)p->npad;
  adam_kernel<<<(c + 255) / 256, 256, 0, p->st>>>(p->w, p->g, p->m, p->v, c, lr, b1, b2, 1e-8f, c1, c2,
                                                 w3 + n * H, w3 + np * H, b3 + n, b3 + np,
                                                 bf16_views(p));
  return cudaGetLastError();
}
}  // namespace pb

extern "C" {

PB_API int pb_mlp_workspace_bytes(int n, int d, int hidden, int batch, size_t* bytes) {
  if (!bytes) return PB_EINVAL;
  int kin, npad;
  int rc = mlp_dims(n, d, hidden, batch, &kin, &npad);
  if (rc != PB_OK) return rc;
  *bytes = mlp_layout(kin, hidden, npad, batch).total;
  return PB_OK;
}

PB_API int pb_mlp_create(int n, int d, int hidden, int batch, uint64_t seed, void* d_ws,
                         size_t ws_bytes, uintptr_t stream, pb_mlp** out) {
  if (!out) return PB_EINVAL;
  *out = nullptr;
  int kin, npad;
  int rc = mlp_dims(n, d, hidden, batch, &kin, &npad);
  if (rc != PB_OK) return rc;
  if (!d_ws || ((uintptr_t)d_ws & 255)) return PB_EINVAL;
  const MlpLayout L = mlp_layout(kin, hidden, npad, batch);
  if (ws_bytes < L.total) return PB_ERANGE;
  pb_mlp* p = new (std::nothrow) pb_mlp;
  if (!p) return PB_ENOMEM;
  p->n = n; p->d = d; p->H = hidden; p->kin = kin; p->npad = npad; p->batch = batch;
  p->st = reinterpret_cast<cudaStream_t>(stream);
  p->ws = static_cast<char*>(d_ws);
  p->ws_bytes = ws_bytes;
  {
    const pb::MlpOffsets o = pb::mlp_offsets(kin, hidden, npad);
    p->off_W1 = o.W1; p->off_b1 = o.b1; p->off_W2 = o.W2; p->off_b2 = o.b2;
    p->off_W3 = o.W3; p->off_b3 = o.b3; p->n_params = o.total;
  }
  char* b = p->ws;
  p->w = (float*)(b + L.w); p->m = (float*)(b + L.m); p->v = (float*)(b + L.v); p->g = (float*)(b + L.g);
  p->W1 = (__nv_bfloat16*)(b + L.W1); p->W2 = (__nv_bfloat16*)(b + L.W2); p->W3 = (__nv_bfloat16*)(b + L.W3);
  p->W2t = (__nv_bfloat16*)(b + L.W2t); p->W3t = (__nv_bfloat16*)(b + L.W3t);
  p->W1p = (__nv_bfloat16*)(b + L.W1p); p->W2p = (__nv_bfloat16*)(b + L.W2p);
  p->W3p = (__nv_bfloat16*)(b + L.W3p);
  p->X = (__nv_bfloat16*)(b + L.X); p->Xt = (__nv_bfloat16*)(b + L.Xt);
  p->H1 = (__nv_bfloat16*)(b + L.H1); p->H1t = (__nv_bfloat16*)(b + L.H1t);
  p->H2 = (__nv_bfloat16*)(b + L.H2); p->H2t = (__nv_bfloat16*)(b + L.H2t);
  p->dY = (__nv_bfloat16*)(b + L.dY); p->dYt = (__nv_bfloat16*)(b + L.dYt);
  p->dZ2 = (__nv_bfloat16*)(b + L.dZ2); p->dZ2t = (__nv_bfloat16*)(b + L.dZ2t);
  p->dZ1t = (__nv_bfloat16*)(b + L.dZ1t);
  p->logits = (float*)(b + L.logits); p->target = (float*)(b + L.target); p->loss = (float*)(b + L.loss);
  p->terms = (float*)(b + L.terms);
  p->status = (uint32_t*)(b + L.status);
  // Initial weights: uniform(-1/sqrt(fan_in), 1/sqrt(fan_in)) from SplitMix64(seed), biases 0.
  std::vector<float> w(p->n_params, 0.f);
  uint64_t s = seed;
  auto next = [&]() {
    s += 0x9E3779B97F4A7C15ull;
    uint64_t z = s;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
  };
  auto fill = [&](size_t o, int rows, int cols, int fan_in, int live_rows, int live_cols) {
    const float a = 1.f / std::sqrt((float)fan_in);
    for (int r = 0; r < rows; ++r)
      for (int c = 0; c < cols; ++c) {
        const float u = (float)((next() >> 11) * (1.0 / 9007199254740992.0));
        w[o + (size_t)r * cols + c] = (r < live_rows && c < live_cols) ? (2.f * u - 1.f) * a : 0.f;
      }
  };
  fill(p->off_W1, hidden, kin, n + d, hidden, n + d);
  fill(p->off_W2, hidden, hidden, hidden, hidden, hidden);
  fill(p->off_W3, npad, hidden, hidden, n, hidden);
  if (pb::mlp_prepare() != cudaSuccess || cudaMemsetAsync(p->ws, 0, L.total, p->st) != cudaSuccess ||
      cudaMemcpyAsync(p->w, w.data(), w.size() * 4, cudaMemcpyHostToDevice, p->st) != cudaSuccess ||
      refresh_bf16(p) != cudaSuccess || cudaStreamSynchronize(p->st) != cudaSuccess) {
    delete p;
    return PB_ECUDA;
  }
  *out = p;
  return PB_OK;
}

PB_API int pb_selftest_wait(int arrive, uint32_t max_iters, int* status) {
  if (!status || max_iters == 0u || max_iters > (1u << 20)) return PB_EINVAL;
  const uint32_t zero = 0u;
  uint32_t v = 0u;
  if (cudaMemcpyToSymbol(pb::g_selftest_status, &zero, 4) != cudaSuccess) return PB_ECUDA;
  pb::selftest_wait_kernel<<<1, 32>>>(arrive ? 1 : 0, max_iters);
  if (cudaGetLastError() != cudaSuccess || cudaDeviceSynchronize() != cudaSuccess ||
      cudaMemcpyFromSymbol(&v, pb::g_selftest_status, 4) != cudaSuccess)
    return PB_ECUDA;
  *status = (int)v;
  return PB_OK;
}

PB_API int pb_mlp_status(pb_mlp* p, int clear, int* status) {
  if (!p || !status) return PB_EINVAL;
  uint32_t v = 0u;
  if (cudaStreamSynchronize(p->st) != cudaSuccess ||
      cudaMemcpy(&v, p->status, 4, cudaMemcpyDeviceToHost) != cudaSuccess)
    return PB_ECUDA;
  *status = (int)v;
  if (clear && v != 0u && cudaMemset(p->status, 0, 4) != cudaSuccess) return PB_ECUDA;
  return PB_OK;
}

PB_API int pb_mlp_info(const pb_mlp* p, int* dims /* n, d, hidden, k_in, batch, n_params */) {
  if (!p || !dims) return PB_EINVAL;
  dims[0] = p->n; dims[1] = p->d; dims[2] = p->H; dims[3] = p->kin; dims[4] = p->batch;
  dims[5] = (int)p->n_params;
  return PB_OK;
}

// get != 0: copy the fp32 master parameters to host (flat W1, b1, W2, b2,
// W3 [npad x H], b3 [npad]); get == 0: load them from host and refresh the
// bf16 copies.  Synchronous.
PB_API int pb_mlp_params(pb_mlp* p, float* host, int get) {
  if (!p || !host) return PB_EINVAL;
  if (cudaStreamSynchronize(p->st) != cudaSuccess) return PB_ECUDA;
  if (get) return cudaMemcpy(host, p->w, p->n_params * 4, cudaMemcpyDeviceToHost) == cudaSuccess ? PB_OK : PB_ECUDA;
  if (cudaMemcpy(p->w, host, p->n_params * 4, cudaMemcpyHostToDevice) != cudaSuccess) return PB_ECUDA;
  if (refresh_bf16(p) != cudaSuccess) return PB_ECUDA;
  return cudaStreamSynchronize(p->st) == cudaSuccess ? PB_OK : PB_ECUDA;
}

PB_API int pb_mlp_grads(pb_mlp* p, float* host) {
  if (!p || !host) return PB_EINVAL;
  if (cudaStreamSynchronize(p->st) != cudaSuccess) return PB_ECUDA;
  return cudaMemcpy(host, p->g, p->n_params * 4, cudaMemcpyDeviceToHost) == cudaSuccess ? PB_OK : PB_ECUDA;
}

// Forward of rows inputs (device bf16 [rows x k_in]) into device fp32
// logits [rows x n] (rows <= batch).
PB_API int pb_mlp_forward(pb_mlp* p, const void* d_x, int rows, float* d_logits) {
  if (!p || !d_x || !d_logits || rows <= 0 || rows > p->batch) return PB_EINVAL;
  if (cudaMemcpyAsync(p->X, d_x, (size_t)rows * p->kin * 2, cudaMemcpyDeviceToDevice, p->st) != cudaSuccess)
    return PB_ECUDA;
  if (mlp_fwd(p, rows, false) != cudaSuccess) return PB_ECUDA;
  if (cudaMemcpy2DAsync(d_logits, (size_t)p->n * 4, p->logits, (size_t)p->npad * 4, (size_t)p->n * 4,
                        rows, cudaMemcpyDeviceToDevice, p->st) != cudaSuccess)
    return PB_ECUDA;
  return PB_OK;
}

// Gradients of the mean BCE of rows (inputs bf16 [rows x k_in], targets fp32
// 0/1 [rows x n]) into the internal gradient block (pb_mlp_grads reads it);
// d_loss (device fp32, may be NULL) receives the loss.  rows: multiple of
// 8, <= batch.
PB_API int pb_mlp_backward(pb_mlp* p, const void* d_x, const float* d_target, int rows, float* d_loss) {
  if (!p || !d_x || !d_target || rows <= 0 || rows > p->batch || rows % 8) return PB_EINVAL;
  if (cudaMemcpyAsync(p->X, d_x, (size_t)rows * p->kin * 2, cudaMemcpyDeviceToDevice, p->st) != cudaSuccess ||
      cudaMemcpyAsync(p->target, d_target, (size_t)rows * p->n * 4, cudaMemcpyDeviceToDevice, p->st) != cudaSuccess)
    return PB_ECUDA;
  if (pb::transpose_bf16(p->X, rows, p->kin, p->Xt, p->st) != cudaSuccess ||
      pb::mlp_gradient_rows(p, rows) != cudaSuccess)
    return PB_ECUDA;
  if (d_loss && cudaMemcpyAsync(d_loss, p->loss, 4, cudaMemcpyDeviceToDevice, p->st) != cudaSuccess)
    return PB_ECUDA;
  return PB_OK;
}

// One Adam step (beta1 0.9, beta2 0.999, eps 1e-8) with the current gradients.
PB_API int pb_mlp_adam(pb_mlp* p, float lr) {
  if (!p || !(lr > 0.f)) return PB_EINVAL;
  return pb::mlp_adam_step(p, lr) == cudaSuccess ? PB_OK : PB_ECUDA;
}

PB_API void pb_mlp_free(pb_mlp* p) {
  if (!p) return;
  cudaStreamSynchronize(p->st);
  delete p;
}

}  // extern "C"

// ===========================================================================
// Fused forward of the whole network for inference: one CTA of 4 warps per
// 128 rows; x, the hidden activations and the weights (W2 streamed in
// K-chunks of 64, double-buffered) stay in shared memory, the accumulators in
// TMEM (256 columns, reused by the three layers).
// ===========================================================================
namespace pb {

// Modes of the fused kernel:
//   kFusedLogits  rows of x from global memory -> logits to global memory;
//   kFusedLogQ    rows (chain c, layer j of k .. d) built from the
//                 per-chain words P -> lq[c d + j-1] = log q(P[c][j-1] | x);
//   kFusedSample  rows (chain c, layer j) built from P (j == k) or Pn (j > k)
//                 -> s'_j drawn from q into Pn[c][j-1], lqf[c] += log q(s'_j | x).
enum : int { kFusedLogits = 0, kFusedLogQ = 1, kFusedSample = 2 };

struct FusedArgs {
  const __nv_bfloat16* X;  // [rows x kin] (kFusedLogits)
  const __nv_bfloat16 *W1p, *W2p, *W3p;  // canonical images (W2 in K-chunks of 64)
  const float *b1, *b2, *b3;
  float* logits;  // [rows x npad] (kFusedLogits)
  int rows, kin, H, npad;
  uint32_t* status;
  // per-chain modes
  const uint32_t* P;
  uint32_t* Pn;
  float* lq;
  float* lqf;
  const uint32_t* move_dev;
  const int* k_dev;  // per-chain modes: when set, the suffix start k is read here
                     // (kFusedLogQ: layers k .. d, in the 128-row kernel layer
                     // k + blockIdx.y; kFusedSample: j = k, jlast = d) and CTAs
                     // without a layer leave at once
  uint32_t beta, k0, k1, group0;
  int n, d, k, j, jlast;  // kFusedSample: layers j .. jlast, one after the other
  // shared-memory layout (byte offsets; fused_layout) and W2 chunk buffers
  uint32_t offH, offW1, offW3, offB, offWb, chunk_bytes;
  int nb;
};

// Dynamic shared memory of the fused kernel, sized per network: the x tile
// (128 x kin), the h tile (128 x H), W1, W3 and the biases resident for the
// whole launch, and nb buffers for the K-chunks of W2 (64 columns each)
// streamed in by bulk copies; nb is as large as the space allows.
constexpr size_t kFusedSmemMax = 222 * 1024;  // with the kernel's static shared memory (< 5 KB)

inline size_t round_kb(size_t b) { return (b + 1023) & ~(size_t)1023; }

// Fills the layout fields of `a`; returns the dynamic shared-memory size (0
// when not even two chunk buffers fit).
inline size_t fused_layout(FusedArgs& a) {
  const size_t X = round_kb((size_t)128 * a.kin * 2), Hs = round_kb((size_t)128 * a.H * 2);
  const size_t W1 = round_kb((size_t)a.H * a.kin * 2), W3 = round_kb((size_t)a.npad * a.H * 2);
  const size_t B = round_kb((size_t)(2 * a.H + a.npad) * 4);
  const int nchunks = (a.H + 63) / 64;
  const size_t chunk = round_kb((size_t)a.H * std::min(64, a.H) * 2);
  a.offH = (uint32_t)X;
  a.offW1 = (uint32_t)(X + Hs);
  a.offW3 = (uint32_t)(X + Hs + W1);
  a.offB = (uint32_t)(X + Hs + W1 + W3);
  a.offWb = (uint32_t)(X + Hs + W1 + W3 + B);
  a.chunk_bytes = (uint32_t)chunk;
  const size_t fixed = a.offWb;
  if (fixed + std::min(2, nchunks) * chunk > kFusedSmemMax) return 0;
  a.nb = (int)std::min<size_t>((size_t)nchunks, (kFusedSmemMax - fixed) / chunk);
  return fixed + (size_t)a.nb * chunk;
}

// Rows [r0, r0+nrows) x K of a row-major bf16 matrix into the canonical
// K-major layout at `dst` (8-row groups SBO = K * 16 bytes apart).
// The copies are asynchronous (cp.async, zero-filled past rmax); the caller
// waits with tc::cp_async_wait_all() before the data is used.
__device__ __forceinline__ void stage_rows(uint8_t* dst, const __nv_bfloat16* src, int ld, int r0,
                                           int nrows, int rmax, int k0, int K, int tid, int nthr) {
  const int vecs = K / 8;
  for (int v = tid; v < nrows * vecs; v += nthr) {
    const int r = v / vecs, c = v % vecs, row = r0 + r;
    const bool in = row < rmax;
    tc::cp_async16(dst + (r >> 3) * (K * 16) + c * 128 + (r & 7) * 16,
                   in ? (const void*)(src + (size_t)row * ld + k0 + c * 8) : (const void*)src,
                   in ? 16u : 0u);
  }
}

// Elements [8 c_lo, 8 c_hi) of row r of the x tile (canonical layout, SBO =
// kin * 16): x = [2 prev - 1 (n), onehot(j-1) (d), 0...], written as bf16
// bit patterns (1.0 = 0x3F80, -1.0 = 0xBF80).
__device__ __forceinline__ void build_x_part(uint8_t* sX, int kin, int n, int r, uint32_t prev,
                                             int j, int c_lo, int c_hi) {
  uint8_t* base = sX + (r >> 3) * (kin * 16) + (r & 7) * 16;
  auto elem = [&](int i) -> uint32_t {
    if (i < n) return ((prev >> i) & 1u) ? 0x3F80u : 0xBF80u;
    return i == n + j - 1 ? 0x3F80u : 0u;
  };
  for (int c = c_lo; c < c_hi; ++c) {
    uint4 w;
    if (8 * c + 8 <= n) {  // bits only: -1.0 with the sign flipped where set
      const uint32_t b = prev >> (8 * c);
      auto pair = [&](int k) {
        return 0xBF80BF80u ^ ((b << (15 - 2 * k)) & 0x8000u) ^ ((b << (30 - 2 * k)) & 0x80000000u);
      };
      *reinterpret_cast<uint4*>(base + c * 128) = make_uint4(pair(0), pair(1), pair(2), pair(3));
      continue;
    }
    w.x = elem(8 * c) | (elem(8 * c + 1) << 16);
    w.y = elem(8 * c + 2) | (elem(8 * c + 3) << 16);
    w.z = elem(8 * c + 4) | (elem(8 * c + 5) << 16);
    w.w = elem(8 * c + 6) | (elem(8 * c + 7) << 16);
    *reinterpret_cast<uint4*>(base + c * 128) = w;
  }
}

// log(1 + e^{-|l|}), the shared part of log sigma(l) and log sigma(-l):
// log sigma(+-l) = -(max(-+l, 0) + softplus_tail(l)).  Both fused modes that
// evaluate log q use this one expression, so a proposal's log q computed
// while it is drawn equals the one computed later for the same path.
__device__ __forceinline__ float softplus_tail(float l) { return __logf(1.f + __expf(-fabsf(l))); }

// Threads per row of the fused kernel: warps w, w + 4, ... share TMEM lane
// quadrant w % 4 (rows 32 (w % 4) ..) and split each row's work.
constexpr int kFusedParts = 4;
constexpr int kFusedThreads = 128 * kFusedParts;

template <int MODE>
__global__ void __launch_bounds__(kFusedThreads) mlp_fused_kernel(FusedArgs a) {
  extern __shared__ __align__(1024) uint8_t sm[];
  // mbarriers: wbar = W1 and W3 delivered; lbar[b] = the W2 chunk in buffer
  // b delivered; cbar[b] = the MMAs reading buffer b done (committed only
  // when the buffer is refilled within the same GEMM); done = all MMAs of
  // the current GEMM done (every thread waits once per GEMM); drain = all
  // MMAs done (after a failed wait only)
  constexpr int kMaxNb = 4;
  __shared__ uint64_t bars[2 + 2 * kMaxNb + 1];
  __shared__ uint32_t tmem_base;
  // the parts of a row exchange their bits and log q terms here
  __shared__ uint32_t xw[kFusedParts][128];
  __shared__ float xq[kFusedParts][128];
  uint64_t* wbar = &bars[0];
  uint64_t* done = &bars[1];
  uint64_t* drain = &bars[2];
  uint64_t* lbar = &bars[3];
  uint64_t* cbar = &bars[3 + kMaxNb];
  uint8_t* sX = sm;
  uint8_t* sH = sm + a.offH;
  uint8_t* sW1 = sm + a.offW1;
  uint8_t* sW3 = sm + a.offW3;
  float* sB = reinterpret_cast<float*>(sm + a.offB);  // b1 [H], b2 [H], b3 [npad]
  uint8_t* sWb = sm + a.offWb;                           // nb chunk buffers
  // warp w reads TMEM lanes 32 (w & 3) .. +31 (its rows) and handles part
  // w >> 2 (of kFusedParts) of the columns, x elements and bits of those rows
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int quad = warp & 3, part = warp >> 2;
  const int rl = quad * 32 + lane;  // row within the tile
  const int r0 = blockIdx.x * 128;
  const int H = a.H, kin = a.kin, npad = a.npad, nb = min(a.nb, kMaxNb);
  const int nchunks = (H + 63) / 64;
  auto chunk_k = [&](int c) { return (c == nchunks - 1 && (H % 64)) ? (H % 64) : 64; };
  const int kk = (MODE != kFusedLogits && a.k_dev) ? *a.k_dev : a.k;
  const int jfirst = MODE == kFusedLogQ ? kk + (int)blockIdx.y : (a.k_dev ? kk : a.j);
  const int jend = MODE == kFusedSample ? (a.k_dev ? a.d : a.jlast) : jfirst;
  if (MODE != kFusedLogits && (jfirst < 1 || jfirst > a.d)) return;  // whole CTA: no layer here

  if (warp == 0) tc::tmem_alloc(&tmem_base, 256);
  if (tid == 0) {
    for (int i = 0; i < 2 + 2 * kMaxNb + 1; ++i) tc::mbar_init(&bars[i], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int i = tid; i < H; i += kFusedThreads) {
    sB[i] = a.b1[i];
    sB[H + i] = a.b2[i];
  }
  for (int i = tid; i < npad; i += kFusedThreads) sB[2 * H + i] = a.b3[i];
  __syncthreads();  // TMEM address, barriers and biases visible
  const uint32_t tb = tmem_base;
  bool ok = true;
  uint32_t dph = 0u;  // parity of `done` (every thread)
  // thread 0: parities and the copies still to be waited for
  uint32_t wph = 0u, lph[kMaxNb] = {0u, 0u, 0u, 0u}, cph[kMaxNb] = {0u, 0u, 0u, 0u};
  bool lpend[kMaxNb] = {false, false, false, false};
  // After a failed wait the thread skips further waits and work but keeps
  // the same sequence of CTA barriers as the others.
  auto wait_on = [&](uint64_t* bar, uint32_t& ph) {
    if (!ok) return;
    ok = tc::mbar_wait(bar, ph);
    if (ok) ph ^= 1u;
  };
  // K-chunk c of W2 into buffer b (thread 0; the buffer is free)
  auto load_chunk = [&](int c, int b) {
    const uint32_t bytes = (uint32_t)(H * chunk_k(c) * 2);
    tc::mbar_expect_tx(&lbar[b], bytes);
    tc::bulk_load(sWb + (size_t)b * a.chunk_bytes, a.W2p + (size_t)H * c * 64, bytes, &lbar[b]);
    lpend[b] = true;
  };
  // the first min(nb, nchunks) chunks of the next GEMM over W2
  auto prefetch_w2 = [&]() {
    for (int c = 0; c < nb && c < nchunks; ++c) load_chunk(c, c);
  };
  if (tid == 0) {
    const uint32_t w1 = (uint32_t)(H * kin * 2), w3 = (uint32_t)(npad * H * 2);
    tc::mbar_expect_tx(wbar, w1 + w3);
    tc::bulk_load(sW1, a.W1p, w1, wbar);
    tc::bulk_load(sW3, a.W3p, w3, wbar);
    prefetch_w2();
  }
  const uint32_t taddr_row = tb + ((uint32_t)(quad * 32) << 16);
  const int row = r0 + rl;
  // generic-proxy shared writes of all threads visible to the tensor core
  auto publish = [&]() {
    tc::fence_proxy_async_smem();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
  };
  auto wait_done = [&]() {
    wait_on(done, dph);
    tc::fence_after_sync();
  };
  // h = relu(D + b) in bf16, into sH (canonical, K = H): this thread's row,
  // the part's share of the 8-column groups; one 64-column TMEM read covers
  // it (a share is at most 64 columns and starts at most at column 192)
  const int ngrp = H / 8;
  const int hc_lo = 8 * (part * ngrp / kFusedParts), hc_hi = 8 * ((part + 1) * ngrp / kFusedParts);
  auto epilogue_to_h = [&](const float* bias) {
    uint8_t* base = sH + (rl >> 3) * (H * 16) + (rl & 7) * 16;
    for (int c0 = hc_lo; c0 < hc_hi; c0 += 64) {
      float v[64];
      tc::tmem_ld64(taddr_row + (uint32_t)c0, v);
#pragma unroll
      for (int g = 0; g < 8; ++g) {
        if (c0 + 8 * g < hc_hi) {
          const float4 bl = *reinterpret_cast<const float4*>(bias + c0 + 8 * g);
          const float4 bh = *reinterpret_cast<const float4*>(bias + c0 + 8 * g + 4);
          const float bv[8] = {bl.x, bl.y, bl.z, bl.w, bh.x, bh.y, bh.z, bh.w};
          __align__(16) __nv_bfloat162 hb[4];
#pragma unroll
          for (int i = 0; i < 4; ++i)
            hb[i] = __floats2bfloat162_rn(fmaxf(v[8 * g + 2 * i] + bv[2 * i], 0.f),
                                          fmaxf(v[8 * g + 2 * i + 1] + bv[2 * i + 1], 0.f));
          *reinterpret_cast<uint4*>(base + ((c0 >> 3) + g) * 128) = *reinterpret_cast<uint4*>(hb);
        }
      }
    }
  };

  // per-chain modes: this thread's chain, its previous layer word and the
  // running log q of the proposal
  const int chain = row;
  uint32_t prev = a.beta;
  if (MODE != kFusedLogits && chain < a.rows && jfirst > 1)
    prev = a.P[(size_t)chain * a.d + (jfirst - 2)];
  float lq_acc = 0.f;

  for (int jl = jfirst; jl <= jend; ++jl) {
    // ---- x tile (row = chain r0 + r at layer jl, or a staged input row)
    if (MODE == kFusedLogits) {
      stage_rows(sX, a.X, kin, r0, 128, a.rows, 0, kin, tid, kFusedThreads);
      tc::cp_async_wait_all();
    } else {
      build_x_part(sX, kin, a.n, rl, prev, jl, part * (kin / 8) / kFusedParts,
                   (part + 1) * (kin / 8) / kFusedParts);
    }
    publish();

    // ---- layer 1: D = x W1^T
    if (tid == 0) {
      if (jl == jfirst) wait_on(wbar, wph);
      if (ok) {
        const uint32_t ax = tc::smem_u32(sX), bw = tc::smem_u32(sW1);
        const uint32_t idesc = tc::idesc_bf16_f32(128, H);
        for (int s = 0; s < kin / 16; ++s)
          tc::mma_bf16(tb, tc::smem_desc(ax + s * 256, 128, kin * 16),
                       tc::smem_desc(bw + s * 256, 128, kin * 16), idesc, s > 0);
      }
      tc::mma_commit(done);
    }
    wait_done();
    if (ok) epilogue_to_h(sB);
    publish();

    // ---- layer 2: D = h W2^T over the K-chunks of W2 (chunk c in buffer
    // c % nb); chunk c + nb - 1 is fetched once the MMAs of chunk c - 1 are done
    if (tid == 0) {
      for (int c = 0; c < nchunks; ++c) {
        const int b = c % nb;
        wait_on(&lbar[b], lph[b]);
        if (!ok) continue;
        lpend[b] = false;
        const int kc = chunk_k(c);
        const uint32_t ah = tc::smem_u32(sH) + c * 8 * 128;
        const uint32_t bw = tc::smem_u32(sWb + (size_t)b * a.chunk_bytes);
        const uint32_t idesc = tc::idesc_bf16_f32(128, H);
        for (int s = 0; s < kc / 16; ++s)
          tc::mma_bf16(tb, tc::smem_desc(ah + s * 256, 128, H * 16),
                       tc::smem_desc(bw + s * 256, 128, kc * 16), idesc, (c > 0) || (s > 0));
        if (c + nb < nchunks) tc::mma_commit(&cbar[b]);  // buffer b is refilled below
        if (c >= 1 && c - 1 + nb < nchunks) {
          const int bp = (c - 1) % nb;
          wait_on(&cbar[bp], cph[bp]);
          if (ok) load_chunk(c - 1 + nb, bp);
        }
      }
      tc::mma_commit(done);
    }
    wait_done();
    // every W2 buffer is free: thread 0 fetches the next layer's first chunks
    if (tid == 0 && ok && jl < jend) prefetch_w2();
    if (ok) epilogue_to_h(sB + H);
    publish();

    // ---- layer 3: D = h W3^T
    if (tid == 0) {
      if (ok) {
        const uint32_t ah = tc::smem_u32(sH), bw = tc::smem_u32(sW3);
        const uint32_t idesc = tc::idesc_bf16_f32(128, npad);
        for (int s = 0; s < H / 16; ++s)
          tc::mma_bf16(tb, tc::smem_desc(ah + s * 256, 128, H * 16),
                       tc::smem_desc(bw + s * 256, 128, H * 16), idesc, s > 0);
      }
      tc::mma_commit(done);
    }
    wait_done();
    // logits of this thread's row (npad is 16 or 32); the row's bits are
    // split between the two halves by Philox output (4 bits each):
    // part p takes bits 4 g .. 4 g + 3 for the g with g % kFusedParts == p
    uint32_t word = 0u;
    float sq = 0.f;
    if (ok) {
      float l[32];
      if (npad > 16) {
        tc::tmem_ld32(taddr_row, l);
      } else {
        float v[16];
        tc::tmem_ld16(taddr_row, v);
#pragma unroll
        for (int i = 0; i < 16; ++i) l[i] = v[i];
#pragma unroll
        for (int i = 16; i < 32; ++i) l[i] = 0.f;
      }
      const float* b3 = sB + 2 * H;
#pragma unroll
      for (int i = 0; i < 32; ++i) l[i] += i < npad ? b3[i] : 0.f;
      if (row < a.rows) {
        if (MODE == kFusedLogits) {
          if (part == 0) {
#pragma unroll
            for (int i = 0; i < 32; ++i)
              if (i < npad) a.logits[(size_t)row * npad + i] = l[i];
          }
        } else if (MODE == kFusedLogQ) {
          // log q of the current layer word: sum_q log sigma(+-l_q)
          const uint32_t bits = a.P[(size_t)row * a.d + (jl - 1)];
#pragma unroll
          for (int qb = 0; qb < 32; ++qb) {
            if (qb < a.n && (qb >> 2) % kFusedParts == part) {
              const float z = ((bits >> qb) & 1u) ? -l[qb] : l[qb];
              sq -= fmaxf(z, 0.f) + softplus_tail(l[qb]);
            }
          }
        } else {
          // draw s'_j bit by bit: u < sigmoid(l_q), u from Philox (chain,
          // move, (j-1) | tag 2 << 16, q/4)
          const uint32_t move = *a.move_dev;
          const uint32_t gc = a.group0 * 32u + (uint32_t)row;
          uint4 u4 = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
          for (int qb = 0; qb < 32; ++qb) {
            if (qb < a.n && (qb >> 2) % kFusedParts == part) {
              if ((qb & 3) == 0)
                u4 = philox4x32_10(make_uint4(gc, move, (uint32_t)(jl - 1) | (kTagMH << 16),
                                              (uint32_t)(qb >> 2)), a.k0, a.k1);
              const uint32_t u = (qb & 3) == 0 ? u4.x : (qb & 3) == 1 ? u4.y : (qb & 3) == 2 ? u4.z : u4.w;
              const float e = __expf(-fabsf(l[qb]));
              const float r = __fdividef(1.f, 1.f + e);
              const float p1 = l[qb] >= 0.f ? r : e * r;  // sigma(l)
              const float uf = ((float)(u >> 8) + 0.5f) * (1.f / 16777216.f);
              const uint32_t bit = uf < p1 ? 1u : 0u;
              word |= bit << qb;
              const float z = bit ? -l[qb] : l[qb];
              sq -= fmaxf(z, 0.f) + softplus_tail(l[qb]);
            }
          }
        }
      }
    }
    if (MODE != kFusedLogits) {
      xw[part][rl] = word;
      xq[part][rl] = sq;
    }
    // the TMEM reads of this layer are complete before the next layer's
    // MMAs, and the halves' bits are exchanged
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (MODE != kFusedLogits && ok && row < a.rows) {
      float sql = 0.f;
      uint32_t wrd = 0u;
#pragma unroll
      for (int q = 0; q < kFusedParts; ++q) {
        sql += xq[q][rl];
        wrd |= xw[q][rl];
      }
      if (MODE == kFusedLogQ) {
        if (part == 0) a.lq[(size_t)row * a.d + (jl - 1)] = sql;
      } else {
        prev = wrd;
        if (part == 0) a.Pn[(size_t)row * a.d + (jl - 1)] = prev;
        lq_acc += sql;
      }
    }
  }  // layers
  if (MODE == kFusedSample && ok && row < a.rows && part == 0) a.lqf[row] += lq_acc;
  if (!__syncthreads_and(ok)) {
    if (tid == 0) {
      if (a.status) atomicCAS(a.status, 0u, (uint32_t)PB_ETIMEOUT);
      // let MMAs and copies still in flight drain (bounded waits) before the
      // accumulator and the shared memory are given up
      tc::mma_commit(drain);
      tc::mbar_wait(drain, 0u);
      for (int b = 0; b < kMaxNb; ++b)
        if (lpend[b]) tc::mbar_wait(&lbar[b], lph[b]);
      if (wph == 0u) tc::mbar_wait(wbar, wph);
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tb, 256);
}

template __global__ void mlp_fused_kernel<kFusedLogits>(FusedArgs);
template __global__ void mlp_fused_kernel<kFusedLogQ>(FusedArgs);
template __global__ void mlp_fused_kernel<kFusedSample>(FusedArgs);

// ===========================================================================
// The per-chain modes with 64-row tiles: twice the CTAs of the 128-row
// kernel, and with half the rows the x and h tiles shrink enough that W1,
// W2 and W3 all stay in shared memory for the whole launch (one bulk copy
// each at the start; no W2 chunks streamed per layer).  MMAs are M = 64
// (idesc M field 4): row r of an accumulator sits in TMEM lane
// 32 (r / 16) + r % 16, so warp w (lane quadrant q = w % 4) holds rows
// 16 q .. 16 q + 15; its epilogue reads them with the 16x256b shape (thread
// t: rows t / 4 and 8 + t / 4 of the 16, columns 2 (t % 4) and the next, of
// each 8-column block), and the four warps of a quadrant split the hidden
// columns.  The logits of row 16 q + i are read by lane i < 16 of warp q
// (32x32b shape), which draws or scores the row's bits as the 128-row
// kernel does.  Same modes, arguments and results (the accumulation order
// of the tensor cores may differ in the last bit).
// ===========================================================================
constexpr int kTile64 = 64;

// Dynamic shared memory of the 64-row kernel: x (64 x kin), h (64 x H),
// W1, the whole W2 image, W3 and the biases; 0 when they do not fit.
inline size_t fused64_layout(FusedArgs& a) {
  const size_t X = round_kb((size_t)kTile64 * a.kin * 2), Hs = round_kb((size_t)kTile64 * a.H * 2);
  const size_t W1 = round_kb((size_t)a.H * a.kin * 2), W2 = round_kb((size_t)a.H * a.H * 2);
  const size_t W3 = round_kb((size_t)a.npad * a.H * 2);
  const size_t B = round_kb((size_t)(2 * a.H + a.npad) * 4);
  a.offH = (uint32_t)X;
  a.offW1 = (uint32_t)(X + Hs);
  a.offWb = (uint32_t)(X + Hs + W1);  // W2, chunk c at + c * H * 64 * 2
  a.offW3 = (uint32_t)(X + Hs + W1 + W2);
  a.offB = (uint32_t)(X + Hs + W1 + W2 + W3);
  a.chunk_bytes = (uint32_t)(a.H * 64 * 2);
  a.nb = 0;
  const size_t total = X + Hs + W1 + W2 + W3 + B;
  if (a.H % 64 != 0 || total > kFusedSmemMax) return 0;
  return total;
}

// 16 lanes x 256 bits (8 fp32 columns) of the warp's TMEM lane quadrant, 8
// blocks of 8 columns (addresses taddr + 8 j), one completion wait: v[4 j +
// 0, 1] = rows t / 4, columns 8 j + 2 (t % 4) + {0, 1}; v[4 j + 2, 3] = row
// 8 + t / 4, the same columns.
__device__ __forceinline__ void tmem_ld_16x256b_x8(uint32_t taddr, float (&v)[32]) {
  uint32_t r[32];
#pragma unroll
  for (int j = 0; j < 8; ++j)
    asm volatile("tcgen05.ld.sync.aligned.16x256b.x1.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[4 * j]), "=r"(r[4 * j + 1]), "=r"(r[4 * j + 2]), "=r"(r[4 * j + 3])
                 : "r"(taddr + 8u * (uint32_t)j)
                 : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

template <int MODE>
__global__ void __launch_bounds__(kFusedThreads) mlp_move64_kernel(FusedArgs a) {
  static_assert(MODE == kFusedLogQ || MODE == kFusedSample, "per-chain modes only");
  extern __shared__ __align__(1024) uint8_t sm[];
  __shared__ uint64_t bars[3];  // weights delivered, MMAs of a GEMM done, drain
  __shared__ uint32_t tmem_base;
  __shared__ uint32_t wrd[kTile64];  // drawn words of the layer, by row
  // the four parts of a row exchange their bits and log q terms here
  __shared__ uint32_t xw[kFusedParts][kTile64];
  __shared__ float xq[kFusedParts][kTile64];
  uint64_t* wbar = &bars[0];
  uint64_t* done = &bars[1];
  uint64_t* drain = &bars[2];
  uint8_t* sX = sm;
  uint8_t* sH = sm + a.offH;
  uint8_t* sW1 = sm + a.offW1;
  uint8_t* sW2 = sm + a.offWb;
  uint8_t* sW3 = sm + a.offW3;
  float* sB = reinterpret_cast<float*>(sm + a.offB);  // b1 [H], b2 [H], b3 [npad]
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int quad = warp & 3, part = warp >> 2;
  const int H = a.H, kin = a.kin, npad = a.npad;
  const int kk = a.k_dev ? *a.k_dev : a.k;
  // kFusedLogQ: an even share of the (tile, layer) pairs, tile by tile, so
  // that the weights are loaded once for all of them; kFusedSample: one tile,
  // the suffix layer after layer
  int jfirst = a.k_dev ? kk : a.j, jend = a.k_dev ? a.d : a.jlast, tile = blockIdx.x;
  long long pair = 0, pair_end = 0;
  if (MODE == kFusedLogQ) {
    const long long pairs = (long long)((a.rows + kTile64 - 1) / kTile64) * (a.d - kk + 1);
    pair = (long long)blockIdx.x * pairs / gridDim.x;
    pair_end = ((long long)blockIdx.x + 1) * pairs / gridDim.x;
    if (kk < 1 || pair >= pair_end) return;  // whole CTA: no pair here
  } else if (jfirst < 1 || jfirst > a.d) {
    return;  // whole CTA: no layer here
  }

  if (warp == 0) tc::tmem_alloc(&tmem_base, 256);
  if (tid == 0) {
    for (int i = 0; i < 3; ++i) tc::mbar_init(&bars[i], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int i = tid; i < H; i += kFusedThreads) {
    sB[i] = a.b1[i];
    sB[H + i] = a.b2[i];
  }
  for (int i = tid; i < npad; i += kFusedThreads) sB[2 * H + i] = a.b3[i];
  __syncthreads();  // TMEM address, barriers and biases visible
  const uint32_t tb = tmem_base;
  if (tid == 0) {
    const uint32_t w1 = (uint32_t)(H * kin * 2), w2 = (uint32_t)(H * H * 2), w3 = (uint32_t)(npad * H * 2);
    tc::mbar_expect_tx(wbar, w1 + w2 + w3);
    tc::bulk_load(sW1, a.W1p, w1, wbar);
    tc::bulk_load(sW2, a.W2p, w2, wbar);
    tc::bulk_load(sW3, a.W3p, w3, wbar);
  }
  bool ok = true, weights = false;
  uint32_t dph = 0u;
  // A wait whose outcome the whole CTA shares (every thread takes the same
  // branches and barriers after it).
  auto wait_all = [&](uint64_t* bar, uint32_t ph) {
    const bool w = ok && tc::mbar_wait(bar, ph);
    ok = __syncthreads_and(w) != 0;
    tc::fence_after_sync();
  };
  auto publish = [&]() {
    tc::fence_proxy_async_smem();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
  };
  // h = relu(D + bias) in bf16 into sH (canonical, K = H): warp (quad,
  // part) converts rows 16 quad .. + 15, columns 64 part .. + 63
  const uint32_t tq = tb + ((uint32_t)(quad * 32) << 16);
  auto epilogue = [&](const float* bias) {
    const int ra = 16 * quad + (lane >> 2), rb = ra + 8;
    uint8_t* ha = sH + (ra >> 3) * (H * 16) + (ra & 7) * 16;
    uint8_t* hb = sH + (rb >> 3) * (H * 16) + (rb & 7) * 16;
    for (int c0 = 64 * part; c0 < H; c0 += 256) {
      float v[32];
      tmem_ld_16x256b_x8(tq + (uint32_t)c0, v);
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int c = c0 + 8 * j + 2 * (lane & 3);
        const float b0 = bias[c], b1 = bias[c + 1];
        const __nv_bfloat162 xa = __floats2bfloat162_rn(fmaxf(v[4 * j] + b0, 0.f), fmaxf(v[4 * j + 1] + b1, 0.f));
        const __nv_bfloat162 xb = __floats2bfloat162_rn(fmaxf(v[4 * j + 2] + b0, 0.f), fmaxf(v[4 * j + 3] + b1, 0.f));
        const int off = (c >> 3) * 128 + (c & 7) * 2;
        *reinterpret_cast<__nv_bfloat162*>(ha + off) = xa;
        *reinterpret_cast<__nv_bfloat162*>(hb + off) = xb;
      }
    }
  };

  // this thread's row for the logits: lanes < 16 of every warp
  const int srow = 16 * quad + lane;  // row within the tile (lanes < 16)
  const int groups = (a.n + 3) / 4;  // 4-bit groups of a layer's bits (n <= 32: at most 8)
  const uint32_t move = MODE == kFusedSample ? *a.move_dev : 0u;
  // this thread's first piece (row, 16 bytes of 8 elements) of an x tile and
  // the step to its next one
  const int pieces = kin / 8;
  const int xr0 = tid / pieces, xc0 = tid % pieces, xdr = kFusedThreads / pieces, xdc = kFusedThreads % pieces;
  bool first = true;  // (the whole CTA's)
  do {  // tiles (kFusedSample: one)
  if (MODE == kFusedLogQ) {
    const int S = a.d - kk + 1;
    tile = (int)(pair / S);
    jfirst = kk + (int)(pair - (long long)tile * S);
    jend = (int)min((long long)a.d, jfirst + (pair_end - pair) - 1);
    pair += jend - jfirst + 1;
  }
  const int r0 = tile * kTile64;
  const int chain = r0 + srow;
  const bool live = lane < 16 && chain < a.rows;
  float lq_acc = 0.f;
  const uint32_t gc = a.group0 * 32u + (uint32_t)chain;
  // the previous-layer word of every row of the tile, for the x builders
  for (int r = tid; r < kTile64; r += kFusedThreads) {
    const int c = r0 + r;
    wrd[r] = (c < a.rows && jfirst > 1) ? a.P[(size_t)c * a.d + (jfirst - 2)] : a.beta;
  }
  __syncthreads();

  for (int jl = jfirst; jl <= jend; ++jl) {
    // ---- x tile: 64 rows x kin, 16-byte pieces of 8 elements
    for (int r = xr0, c = xc0; r < kTile64; r += xdr, c += xdc) {
      if (c >= pieces) {
        c -= pieces;
        if (++r >= kTile64) break;
      }
      build_x_part(sX, kin, a.n, r, wrd[r], jl, c, c + 1);
    }
    publish();
    // ---- layer 1: D = x W1^T
    if (tid == 0 && ok) {
      if (!weights) {
        weights = tc::mbar_wait(wbar, 0u);
        if (!weights) ok = false;
      }
      if (ok) {
        const uint32_t ax = tc::smem_u32(sX), bw = tc::smem_u32(sW1);
        const uint32_t idesc = tc::idesc_bf16_f32(kTile64, H);
        for (int s = 0; s < kin / 16; ++s)
          tc::mma_bf16(tb, tc::smem_desc(ax + s * 256, 128, kin * 16),
                       tc::smem_desc(bw + s * 256, 128, kin * 16), idesc, s > 0);
        tc::mma_commit(done);
      }
    }
    if (first) ok = __syncthreads_and(ok) != 0;  // thread 0's weight wait, shared
    first = false;
    wait_all(done, dph);
    dph ^= 1u;
    if (ok) epilogue(sB);
    publish();
    // ---- layer 2: D = h W2^T, W2 resident (K-chunk c of 64 at c H 128 bytes)
    if (tid == 0 && ok) {
      const uint32_t idesc = tc::idesc_bf16_f32(kTile64, H);
      const uint32_t ah = tc::smem_u32(sH), bw = tc::smem_u32(sW2);
      for (int c = 0; c < H / 64; ++c)
        for (int s = 0; s < 4; ++s)
          tc::mma_bf16(tb, tc::smem_desc(ah + c * 8 * 128 + s * 256, 128, H * 16),
                       tc::smem_desc(bw + c * a.chunk_bytes + s * 256, 128, 64 * 16), idesc,
                       (c > 0) || (s > 0));
      tc::mma_commit(done);
    }
    // while the tensor cores run layer 2: this thread's inputs to the logits
    // step (the draw's Philox outputs for groups part and part + 4, or the
    // current word), which depend on nothing the MMAs produce
    uint4 upre[2] = {make_uint4(0u, 0u, 0u, 0u), make_uint4(0u, 0u, 0u, 0u)};
    uint32_t bits = 0u;
    if (live) {
      if (MODE == kFusedSample) {
#pragma unroll
        for (int t = 0; t < 2; ++t) {
          const int g = part + kFusedParts * t;
          if (g < groups)
            upre[t] = philox4x32_10(make_uint4(gc, move, (uint32_t)(jl - 1) | (kTagMH << 16), (uint32_t)g),
                                    a.k0, a.k1);
        }
      } else {
        bits = a.P[(size_t)chain * a.d + (jl - 1)];
      }
    }
    wait_all(done, dph);
    dph ^= 1u;
    if (ok) epilogue(sB + H);
    publish();
    // ---- layer 3: D = h W3^T
    if (tid == 0 && ok) {
      const uint32_t ah = tc::smem_u32(sH), bw = tc::smem_u32(sW3);
      const uint32_t idesc = tc::idesc_bf16_f32(kTile64, npad);
      for (int s = 0; s < H / 16; ++s)
        tc::mma_bf16(tb, tc::smem_desc(ah + s * 256, 128, H * 16),
                     tc::smem_desc(bw + s * 256, 128, H * 16), idesc, s > 0);
      tc::mma_commit(done);
    }
    wait_all(done, dph);
    dph ^= 1u;
    // ---- logits: the four parts of a quadrant split each row's bits by
    // Philox output (part p takes the 4-bit groups g = p, p + 4, ...): lane
    // i < 16 of warp (quad, part) scores row 16 quad + i, logit columns
    // 4 g .. 4 g + 3; log q of the current word, or the draw
    uint32_t wpart = 0u;
    float qpart = 0.f;
    if (ok) {
      const float* b3 = sB + 2 * H;
#pragma unroll
      for (int t = 0; t < 2; ++t) {  // groups part, part + 4 (warp-uniform)
        const int g = part + kFusedParts * t;
        if (g >= groups) break;
        float la[4];
        tc::tmem_ld4(tq + 4u * (uint32_t)g, la);
        if (!live) continue;
        const uint4 u4 = upre[t];
        const uint32_t U[4] = {u4.x, u4.y, u4.z, u4.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int qb = 4 * g + i;
          if (qb >= a.n) break;
          const float l = la[i] + b3[qb];
          uint32_t bit;
          if (MODE == kFusedLogQ) {
            bit = (bits >> qb) & 1u;
          } else {
            const float e = __expf(-fabsf(l));
            const float r = __fdividef(1.f, 1.f + e);
            const float p1 = l >= 0.f ? r : e * r;  // sigma(l)
            const float uf = ((float)(U[i] >> 8) + 0.5f) * (1.f / 16777216.f);
            bit = uf < p1 ? 1u : 0u;
          }
          wpart |= bit << qb;
          const float z = bit ? -l : l;
          qpart -= fmaxf(z, 0.f) + softplus_tail(l);
        }
      }
    }
    if (live) {
      xw[part][srow] = wpart;
      xq[part][srow] = qpart;
    }
    // the TMEM reads of this layer are complete before the next layer's
    // MMAs; the parts' bits and log q terms are exchanged
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (ok && live && part == 0) {
      uint32_t word = 0u;
      float sq = 0.f;
#pragma unroll
      for (int q = 0; q < kFusedParts; ++q) {
        word |= xw[q][srow];
        sq += xq[q][srow];
      }
      if (MODE == kFusedLogQ) {
        a.lq[(size_t)chain * a.d + (jl - 1)] = sq;
        wrd[srow] = word;  // the current word: the next layer's input
      } else {
        wrd[srow] = word;
        a.Pn[(size_t)chain * a.d + (jl - 1)] = word;
        lq_acc += sq;
      }
    }
    __syncthreads();  // the drawn words are visible to the next x tile
  }  // layers
  if (MODE == kFusedSample && ok && live && part == 0) a.lqf[chain] += lq_acc;
  } while (MODE == kFusedLogQ && pair < pair_end);
  if (!ok && tid == 0) {
    if (a.status) atomicCAS(a.status, 0u, (uint32_t)PB_ETIMEOUT);
    // let MMAs and copies in flight drain (bounded) before TMEM and shared
    // memory are given up
    tc::mma_commit(drain);
    tc::mbar_wait(drain, 0u);
    if (!weights) tc::mbar_wait(wbar, 0u);
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tb, 256);
}

template __global__ void mlp_move64_kernel<kFusedLogQ>(FusedArgs);
template __global__ void mlp_move64_kernel<kFusedSample>(FusedArgs);

static FusedArgs fused_args(pb_mlp* p, int rows) {
  FusedArgs a{};
  a.jlast = 0;
  a.W1p = p->W1p;
  a.W2p = p->W2p;
  a.W3p = p->W3p;
  a.b1 = p->w + p->off_b1;
  a.b2 = p->w + p->off_b2;
  a.b3 = p->w + p->off_b3;
  a.rows = rows;
  a.kin = p->kin;
  a.H = p->H;
  a.npad = p->npad;
  a.n = p->n;
  a.d = p->d;
  a.status = p->status;
  return a;
}

// log q of the current suffix layers k..d of all chains (one launch).
cudaError_t mlp_fused_logq(pb_mlp* p, const uint32_t* P, uint32_t beta, int chains, int k, float* lq,
                           cudaStream_t st) {
  FusedArgs a = fused_args(p, chains);
  a.P = P;
  a.beta = beta;
  a.k = k;
  a.lq = lq;
  dim3 grid((chains + 127) / 128, p->d - k + 1);
  const size_t smem = fused_layout(a);
  if (smem == 0) return cudaErrorInvalidValue;
  mlp_fused_kernel<kFusedLogQ><<<grid, kFusedThreads, smem, st>>>(a);
  return cudaGetLastError();
}

// The same with the suffix start read from k_dev on the device, so that one
// captured graph serves every k: even shares of the suffix's (tile, layer)
// pairs for the 64-row kernel; for the 128-row kernel a grid over all d layers,
// whose CTAs past the suffix leave at once.
cudaError_t mlp_fused_logq_dev(pb_mlp* p, const uint32_t* P, uint32_t beta, int chains,
                               const int* k_dev, float* lq, cudaStream_t st) {
  FusedArgs a = fused_args(p, chains);
  a.P = P;
  a.beta = beta;
  a.k = 1;
  a.k_dev = k_dev;
  a.lq = lq;
  if (const size_t smem64 = fused64_layout(a)) {  // 64-row tiles, weights resident
    // CTAs: the SMs that the draw beside it (a CTA a tile, as long as a
    // tile's whole suffix) leaves free, where these finish before it does; two
    // a tile when the tiles fill the GPU (one evened the SMs' loads less: 1.23
    // ms a move of 65,536 chains against 1.21); every SM's worth between the
    // two.  A CTA for each (tile, layer) loaded 200 KB of weights and set up
    // tensor memory for one layer's work (200 moves and sweeps of 4096 chains:
    // 17.3 -> 16.9 ms, with the x tiles' shorter code 16.8)
    const int tiles = (chains + kTile64 - 1) / kTile64;
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int ctas = 2 * tiles <= sms ? sms - tiles : std::max(sms, 2 * tiles);
    mlp_move64_kernel<kFusedLogQ><<<ctas, kFusedThreads, smem64, st>>>(a);
    return cudaGetLastError();
  }
  dim3 grid((chains + 127) / 128, p->d);
  const size_t smem = fused_layout(a);
  if (smem == 0) return cudaErrorInvalidValue;
  mlp_fused_kernel<kFusedLogQ><<<grid, kFusedThreads, smem, st>>>(a);
  return cudaGetLastError();
}

// Layers j .. jlast of the proposal for all chains (one launch; each CTA
// carries its 128 chains through the layers in turn).
cudaError_t mlp_fused_sample(pb_mlp* p, const uint32_t* P, uint32_t* Pn, uint32_t beta, int chains,
                             int k, int j, int jlast, float* lqf, uint32_t k0, uint32_t k1,
                             const uint32_t* move_dev, uint32_t group0, cudaStream_t st) {
  FusedArgs a = fused_args(p, chains);
  a.P = P;
  a.Pn = Pn;
  a.beta = beta;
  a.k = k;
  a.j = j;
  a.jlast = jlast;
  a.lqf = lqf;
  a.k0 = k0;
  a.k1 = k1;
  a.move_dev = move_dev;
  a.group0 = group0;
  const size_t smem = fused_layout(a);
  if (smem == 0) return cudaErrorInvalidValue;
  mlp_fused_kernel<kFusedSample><<<(chains + 127) / 128, kFusedThreads, smem, st>>>(a);
  return cudaGetLastError();
}

// Layers k .. d of the proposal, k read from k_dev on the device.
cudaError_t mlp_fused_sample_dev(pb_mlp* p, const uint32_t* P, uint32_t* Pn, uint32_t beta,
                                 int chains, const int* k_dev, float* lqf, uint32_t k0, uint32_t k1,
                                 const uint32_t* move_dev, uint32_t group0, cudaStream_t st) {
  FusedArgs a = fused_args(p, chains);
  a.P = P;
  a.Pn = Pn;
  a.beta = beta;
  a.k = 1;
  a.j = 1;
  a.jlast = p->d;
  a.k_dev = k_dev;
  a.lqf = lqf;
  a.k0 = k0;
  a.k1 = k1;
  a.move_dev = move_dev;
  a.group0 = group0;
  if (const size_t smem64 = fused64_layout(a)) {  // 64-row tiles, weights resident
    mlp_move64_kernel<kFusedSample><<<(chains + kTile64 - 1) / kTile64, kFusedThreads, smem64, st>>>(a);
    return cudaGetLastError();
  }
  const size_t smem = fused_layout(a);
  if (smem == 0) return cudaErrorInvalidValue;
  mlp_fused_kernel<kFusedSample><<<(chains + 127) / 128, kFusedThreads, smem, st>>>(a);
  return cudaGetLastError();
}

cudaError_t mlp_forward_fused(pb_mlp* p, int rows) {
  FusedArgs a{};
  a.X = p->X;
  a.W1p = p->W1p;
  a.W2p = p->W2p;
  a.W3p = p->W3p;
  a.b1 = p->w + p->off_b1;
  a.b2 = p->w + p->off_b2;
  a.b3 = p->w + p->off_b3;
  a.logits = p->logits;
  a.rows = rows;
  a.kin = p->kin;
  a.H = p->H;
  a.npad = p->npad;
  a.status = p->status;
  a.n = p->n;
  const size_t smem = fused_layout(a);
  if (smem == 0) return cudaErrorInvalidValue;
  mlp_fused_kernel<kFusedLogits><<<(rows + 127) / 128, kFusedThreads, smem, p->st>>>(a);
  return cudaGetLastError();
}

cudaError_t mlp_fused_prepare() {
  cudaError_t e = cudaFuncSetAttribute(mlp_fused_kernel<kFusedLogits>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFusedSmemMax);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(mlp_fused_kernel<kFusedLogQ>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kFusedSmemMax);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(mlp_fused_kernel<kFusedSample>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFusedSmemMax);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(mlp_move64_kernel<kFusedLogQ>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)kFusedSmemMax);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(mlp_move64_kernel<kFusedSample>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFusedSmemMax);
  return e;
}

}  // namespace pb

extern "C" PB_API int pb_mlp_forward_fused(pb_mlp* p, const void* d_x, int rows, float* d_logits) {
  if (!p || !d_x || !d_logits || rows <= 0 || rows > p->batch) return PB_EINVAL;
  if (p->kin > 96 || p->npad > 32) return PB_ERANGE;
  if (cudaMemcpyAsync(p->X, d_x, (size_t)rows * p->kin * 2, cudaMemcpyDeviceToDevice, p->st) != cudaSuccess)
    return PB_ECUDA;
  if (pb::mlp_forward_fused(p, rows) != cudaSuccess) return PB_ECUDA;
  if (cudaMemcpy2DAsync(d_logits, (size_t)p->n * 4, p->logits, (size_t)p->npad * 4, (size_t)p->n * 4,
                        rows, cudaMemcpyDeviceToDevice, p->st) != cudaSuccess)
    return PB_ECUDA;
  return PB_OK;
}
