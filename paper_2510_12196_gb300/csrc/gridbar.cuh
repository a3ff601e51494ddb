// The bounded barrier of the cooperative kernels.
#pragma once

#include "common.cuh"

namespace gm {

// Grid barrier state (zero-initialised; count returns to 0 after each use).
struct GridBar {
  unsigned int count;
  unsigned int gen;
  unsigned int err;  // set when a wait gave up
  unsigned int pad;
};
constexpr unsigned long long kBarWaitNs = 1000000000ULL;  // a wait gives up after one second
constexpr unsigned kBarSpinLimit = 1u << 26;               // and after this many polls in any case

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

struct GridSync {
  GridBar* bar;
  unsigned int* flag;  // shared memory of the calling block
  unsigned int need;   // arrivals that release the barrier (gridDim.x)
  // Every block arrives once; the last one resets the count and advances the
  // generation the others poll.  Fences order each block's phase writes
  // before its arrival and the following reads after the release.  A wait
  // that exceeds the limit marks the barrier failed; the blocks then leave
  // the kernel at their next barrier and the host reports the failure.
  __device__ __forceinline__ void sync() const {
    __syncthreads();
    if (threadIdx.x == 0) {
      const unsigned g0 = *(volatile unsigned*)&bar->gen;
      __threadfence();
      if (atomicAdd(&bar->count, 1u) == need - 1) {
        bar->count = 0;
        __threadfence();
        atomicAdd(&bar->gen, 1u);
      } else {
        unsigned spins = 0;
        const unsigned long long t0 = global_ns();
        while (*(volatile unsigned*)&bar->gen == g0) {
          if (++spins > kBarSpinLimit || global_ns() - t0 > kBarWaitNs || *(volatile unsigned*)&bar->err) {
            atomicOr(&bar->err, 1u);
            break;
          }
          __nanosleep(64);
        }
      }
      __threadfence();
      *flag = *(volatile unsigned*)&bar->err;
    }
    __syncthreads();
    if (*(volatile unsigned*)flag) asm volatile("exit;");
  }
};

}  // namespace gm
