// Grid-wide barrier of the persistent (cooperative) launches.
//
// What bounds it: a chain of round trips to L2 and the fences around them.
// Blocks arrive on one counter that only grows and wait on a flag on a line of
// its own, which the last block to arrive writes: nobody polls the line that
// takes the atomics, nothing is reset, and the error word is read once, by the
// releasing block, instead of by every waiting block on every poll.  608
// blocks (4 per SM) doing nothing else pass it in 1.7 us; a counter that is
// reset and a generation word beside it, polled together with the error word,
// took 3.6 us, and arriving in groups of 32 at a root counter 2.1 us.
#pragma once

#include "device_common.cuh"
#include "rpq_internal.h"

namespace rpq {

// Barrier number `epoch` (1, 2, ...: each block counts its own calls, which
// every block of the launch makes alike) of a launch whose control block was
// zero at its start.  Waits are bounded by limit_ns; on expiry the error word
// is set and the block returns false.  An error recorded by any block before
// the barrier makes it return false in every block: the releasing block hands
// the error out with the epoch, so all threads of the grid take the same
// branch.  before(): run by thread 0 when the block's other threads have
// arrived, before the block does.
template <typename F>
__device__ __forceinline__ bool grid_sync(BfsCtl *c, unsigned nblocks, unsigned &epoch, u64 limit_ns, F before) {
  __shared__ unsigned s_go;
  epoch++;
  __syncthreads();
  if (threadIdx.x == 0) {
    volatile unsigned *flag = &c->bar_flag;
    const unsigned want = epoch << 1;  // counter and epoch may wrap: compared for equality only
    unsigned go;
    before();
    __threadfence();
    if (atomicAdd(&c->bar_count, 1u) + 1u == epoch * nblocks) {
      __threadfence();
      go = want | (*(volatile unsigned *)&c->err ? 1u : 0u);
      *flag = go;
    } else {
      const u64 t0 = globaltimer_ns();
      unsigned spins = 0;
      while (((go = *flag) & ~1u) != want) {
        // the first polls are back to back; a longer wait (an uneven phase)
        // leaves the memory system to the blocks still working
        if (++spins > 8) __nanosleep(100);
        if ((spins & 63u) != 0) continue;
        // another block gave up waiting, or this wait is over its limit
        if (*(volatile unsigned *)&c->err == (unsigned)(-RPQ_ERR_TIMEOUT)) break;
        if (globaltimer_ns() - t0 > limit_ns) {
          atomicCAS(&c->err, 0u, (unsigned)(-RPQ_ERR_TIMEOUT));
          break;
        }
      }
      if ((go & ~1u) != want) go = 1;
      __threadfence();
    }
    s_go = go;  // the next call writes it only after its first __syncthreads
  }
  __syncthreads();
  return (s_go & 1u) == 0;
}

__device__ __forceinline__ bool grid_sync(BfsCtl *c, unsigned nblocks, unsigned &epoch, u64 limit_ns) {
  return grid_sync(c, nblocks, epoch, limit_ns, [] {});
}

}  // namespace rpq
