// Teams of blocks of a cooperative launch, and the barrier of a team.
#pragma once

#include <cuda_runtime.h>

namespace irtps {

// The blocks that work on one solve: all of a plain launch, or the range of a
// batched launch that belongs to one object (bid = block index within it).
struct Team {
  int bid, nblk;
};
__device__ __forceinline__ Team whole_grid() { return Team{(int)blockIdx.x, (int)gridDim.x}; }

#ifndef IRTPS_BARRIER_SLEEP_NS
#define IRTPS_BARRIER_SLEEP_NS 64
#endif
constexpr unsigned kBarrierSleepNs = IRTPS_BARRIER_SLEEP_NS;  // back-off between barrier polls

// Barrier of the nblk blocks of a team in a cooperative launch (all blocks
// co-resident).  Thread 0 of each block arrives on a counter; the last one resets it and advances the
// generation word the others poll.  Every poll loop is bounded: on running out it
// raises the error flag, and all blocks leave the solve at the next check.
__device__ __forceinline__ void grid_barrier(unsigned *count, volatile unsigned *gen, int *err, int nblk) {
  __syncthreads();
  if (threadIdx.x == 0 && !*(volatile int *)err) {  // after a failure every barrier is a no-op
    const unsigned g0 = *gen;
    __threadfence();
    if (atomicAdd(count, 1u) == (unsigned)nblk - 1u) {
      *count = 0u;
      __threadfence();
      atomicAdd((unsigned *)gen, 1u);
    } else {
      unsigned long long polls = 0;
      while (*gen == g0) {
        if (++polls > (1ull << 24)) {
          atomicExch(err, 1);
          break;
        }
        if (kBarrierSleepNs > 0) __nanosleep(kBarrierSleepNs);
      }
    }
    __threadfence();
  }
  __syncthreads();
}

}  // namespace irtps
