// Grid-wide barrier for cooperative launches (all blocks co-resident, which the runtime
// guarantees or refuses the launch). Thread 0 of each block arrives on a counter that starts
// at zero with the launch (red.release, after a block barrier: it publishes the block's
// writes) and polls it, a bounded number of times, until every block has arrived (ld.acquire:
// the other blocks' writes are visible to this block's later plain, coherent loads). A wait
// that gives up sets ERR_TIMEOUT and returns false: the caller returns, and the other blocks
// then time out at the same barrier, so a launch always ends. About 2,000 cycles on GB300
// where no block is late; the earlier form (a fenced atomic, a reset by the last block, polls
// with 64 ns sleeps) took 3,000 to 4,000.
#pragma once
#include "sph_kernels.h"

namespace sph {

constexpr unsigned kBarrierSpinLimit = 1u << 21;   // polls of half a microsecond: about a second

// target: the arrivals of the barriers so far, zero at the launch's start (thread 0's copy is
// the one used).
__device__ __forceinline__ bool grid_barrier(unsigned* count, unsigned& target, Global* g) {
  __shared__ int ok;
  __syncthreads();
  target += gridDim.x;
  if (threadIdx.x == 0) {
    ok = 1;
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;\n" ::"l"(count) : "memory");
    unsigned spins = 0, seen;
    while (true) {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];\n" : "=r"(seen) : "l"(count) : "memory");
      if ((int)(seen - target) >= 0) break;
      if (++spins > kBarrierSpinLimit) {
        atomicOr(&g->err, ERR_TIMEOUT);
        ok = 0;
        break;
      }
    }
  }
  __syncthreads();
  return ok != 0;
}

}  // namespace sph
