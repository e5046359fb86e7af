// Barrier over the blocks of a cooperative launch, with a bounded wait.
#pragma once

#include <stdint.h>

#include "tc_ptx.cuh"

namespace polar {
namespace {

// The barrier's words in device memory; both zero between launches (the last block to leave resets them).
struct GridBarWords {
  unsigned int count, left;
};

struct GridBarrier {
  GridBarWords* w;
  volatile int* abort_flag;   // in shared memory, zero at the start
  unsigned int target;        // arrivals the next sync waits for
  uint64_t limit_ns;          // bound of a wait: longer than any block's work between two barriers

  __device__ __forceinline__ GridBarrier(GridBarWords* words, int* abort, uint64_t limit = 2 * WAIT_LIMIT_NS)
      : w(words), abort_flag(abort), target(0), limit_ns(limit) {}

  // Every block's global writes before it are visible after it. False when the wait expired or the block had
  // aborted before. Must be reached by all threads of the block.
  __device__ __forceinline__ bool sync() {
    __syncthreads();
    target += gridDim.x;
    if (threadIdx.x == 0 && !*abort_flag && gridDim.x > 1) {
      asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&w->count) : "memory");
      const uint64_t t0 = gtime();
      for (uint32_t i = 1;; ++i) {
        unsigned int v;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&w->count) : "memory");
        if ((int)(v - target) >= 0) break;   // arrivals count on past 2^32 in a very long loop
        if ((i & 63u) == 0 && gtime() - t0 > limit_ns) {
          *abort_flag = 1;
          break;
        }
      }
    }
    __syncthreads();
    return !*abort_flag;
  }

  // After the block's last sync: the last block out clears the words for the next launch.
  __device__ __forceinline__ void leave() {
    if (threadIdx.x == 0 && w) {   // no words: a launch without barriers
      __threadfence();
      if (atomicAdd(&w->left, 1u) == gridDim.x - 1) {
        w->count = 0;
        w->left = 0;
      }
    }
  }
};

}  // namespace
}  // namespace polar
