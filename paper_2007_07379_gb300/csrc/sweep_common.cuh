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

}  // namespace pb
