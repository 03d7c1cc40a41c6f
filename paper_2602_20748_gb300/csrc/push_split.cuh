// How a top-down level is split over the warps, for the bit-sliced and the
// batched engine.
#pragma once

#include "device_common.cuh"
#include "rpq_internal.h"

namespace rpq {

// Reserves up to `chunks` spill records with one atomic add and returns how
// many of them fit below `cap` (their first index in *at).  Records below
// the capacity are always written by their reserver, so the spill phase,
// which reads min(count, cap) records, never reads one nobody wrote; the
// chunks that do not fit are processed in place.
__device__ __forceinline__ unsigned spill_reserve(unsigned long long *count, unsigned chunks, unsigned long long cap,
                                                  unsigned long long *at) {
  const unsigned long long first = atomicAdd(count, (unsigned long long)chunks);
  *at = first;
  if (first >= cap) return 0;
  return (unsigned)min((unsigned long long)chunks, cap - first);
}

// Chunk length of a top-down level whose frontier has mf out-edges: long rows
// are cut so that every warp gets about eight chunks, from SPILL_EDGES_MIN to
// SPILL_EDGES edges, up to 16 times longer where the records would not fit half
// of the queue (rows that find it full stay whole with one warp).  One chunk per warp
// left the last warp of a level at five times the first one's time; a fixed
// 1,024 left a level of 36,830 edges from a hundred entries to the four warps
// that held them.
__device__ __forceinline__ u32 spill_chunk(u64 mf, u64 n_warps, u64 cap) {
  u64 s = SPILL_EDGES_MIN;
  while (s < SPILL_EDGES && s * n_warps * 8 < mf) s <<= 1;
  while (s * cap < 2 * mf && s < SPILL_EDGES * 16) s <<= 1;
  return (u32)s;
}

// Entries a warp takes at a time: 32 while every warp gets some, of at most
// 4,096 edges on average, and in a level of more than 256 edges per warp while
// it gets four grabs; fewer otherwise, down to one.
__device__ __forceinline__ u32 push_grab(u64 n_cur, u64 mf, u64 n_warps) {
  const u64 grabs = mf > n_warps * 256 ? 4 : 1;
  u32 e = 32;
  while (e > 1 && (n_cur < n_warps * e * grabs || mf * e > 4096 * n_cur)) e >>= 1;
  return e;
}

// List slots a warp reserves at a time in a top-down level of mf edges: below
// PUSH_EXACT edges the appends are few enough for an atomic each, and the
// lists stay free of unused slots, which the next level would read.
constexpr u64 PUSH_EXACT = 1ull << 16;

__device__ __forceinline__ u64 grid_warp() { return ((u64)blockIdx.x * blockDim.x + threadIdx.x) >> 5; }
__device__ __forceinline__ u64 grid_warps() { return ((u64)gridDim.x * blockDim.x) >> 5; }

// Work items of a phase, `step` consecutive ones at a time: a warp's first
// item is its own (warp * step), the next ones come from the phase's cursor.
// Phases with fewer items than warps touch no cursor: the 4,864 warps of a
// full grid asking one counter for nothing took 8-10 us.
// next_item: the first item of the warp's next grab (warp-uniform, all lanes
// call it).
__device__ __forceinline__ u64 next_item(unsigned long long *cursor, u64 n_warps, u32 step) {
  u64 t = 0;
  if (lane_id() == 0) t = atomicAdd(cursor, (unsigned long long)step);
  return n_warps * step + __shfl_sync(FULL_MASK, t, 0);
}

}  // namespace rpq
