// Small device helpers shared by the RPQ kernels.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace rpq {

typedef unsigned long long u64;
typedef unsigned int u32;

constexpr u32 FULL_MASK = 0xffffffffu;
constexpr u32 NO_SOURCE = 0xffffffffu;

__device__ __forceinline__ u32 lane_id() { return threadIdx.x & 31; }

__device__ __forceinline__ u32 lanemask_lt() {
  u32 m;
  asm volatile("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}

__device__ __forceinline__ u64 globaltimer_ns() {
  u64 t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// SplitMix64 output for state x (Steele, Lea and Flood, OOPSLA 2014): add the
// golden-ratio increment, then the variant-13 64-bit finalizer.
__host__ __device__ __forceinline__ u64 splitmix64(u64 x) {
  u64 z = x + 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// splitmix64(src << 32 | y) for many y < 2^31 (vertex ids) of one src.  Adding
// the increment never carries out of the low half there (its low half is below
// 2^31), so the high half of the first stage, its share of the first multiply
// and the bits it shifts into the low half depend on src alone: 20 integer
// operations per row instead of 26.  The digest passes are bound by them.
struct RowHash {
  u32 k;  // high half << 2
  u32 c;  // the high half's share of the first product's high half
  __device__ __forceinline__ explicit RowHash(u32 src) {
    const u32 hi = src + 0x9E3779B9u;
    k = hi << 2;
    c = (hi ^ (hi >> 30)) * 0x1CE4E5B9u;
  }
  __device__ __forceinline__ u64 operator()(u32 y) const {
    const u32 lo = y + 0x7F4A7C15u;
    const u32 l1 = lo ^ (lo >> 30) ^ k;
    u64 z = (u64)l1 * 0x1CE4E5B9u + ((u64)(l1 * 0xBF58476Du + c) << 32);
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
  }
};

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL_MASK, v, o);
  return v;
}

__device__ __forceinline__ u64 warp_xor(u64 v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v ^= __shfl_xor_sync(FULL_MASK, v, o);
  return v;
}

}  // namespace rpq
