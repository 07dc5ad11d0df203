// The bounded grid barrier of the persistent batch kernel.
#pragma once

namespace dgnn {

constexpr long long kBarrierCycles = 2000000000LL;   // about a second

// Barrier of `blocks` co-resident blocks.  Every block's thread 0 counts its arrival (bar[0]);
// the last to arrive resets the count and advances the generation (bar[1]), the others wait for
// the new generation.  Writes before the barrier are visible after it (fences around the
// count).  Returns false in every thread of a block whose wait expired.
__device__ __forceinline__ bool grid_barrier_bounded(unsigned* bar, unsigned blocks) {
  __syncthreads();
  int expired = 0;
  if (threadIdx.x == 0) {
    volatile unsigned* gen = bar + 1;
    const unsigned g = *gen;
    __threadfence();
    if (atomicAdd(bar, 1u) == blocks - 1) {
      atomicExch(bar, 0u);
      __threadfence();
      atomicAdd(bar + 1, 1u);
    } else {
      const long long t0 = clock64();
      while (*gen == g) {
        if (clock64() - t0 > kBarrierCycles) {
          expired = 1;
          break;
        }
      }
    }
    __threadfence();
  }
  return __syncthreads_or(expired) == 0;
}

}  // namespace dgnn
