// Grid-wide barrier for a co-resident (cooperative) grid, with a bounded wait.
#pragma once

#include <cuda_runtime.h>

namespace pf {

// bar[0] counts arrivals, bar[1] is the generation, bar[2] the error flag.  A
// block that waits longer than `limit` clock cycles sets the flag and reports
// failure.
__device__ inline bool grid_barrier(unsigned* bar, long long limit) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    ok = 1;
    volatile unsigned* vgen = bar + 1;
    const unsigned gen = *vgen;
    __threadfence();
    const unsigned arrived = atomicAdd(bar, 1u);
    if (arrived == gridDim.x - 1) {
      bar[0] = 0;
      __threadfence();
      atomicAdd(bar + 1, 1u);
    } else {
      const long long t0 = clock64();
      while (*vgen == gen) {
        if (clock64() - t0 > limit) {
          atomicExch(bar + 2, 1u);
          ok = 0;
          break;
        }
      }
    }
    __threadfence();
  }
  __syncthreads();
  return ok != 0;
}

}  // namespace pf
