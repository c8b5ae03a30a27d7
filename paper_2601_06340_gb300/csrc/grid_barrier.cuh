// Barrier over the CTAs of one cooperative launch (FP64 and 3D marches).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace bpm {

// A counter, zero at launch, that every CTA raises once per barrier (compared
// by its distance from the target, so it may wrap), with a bounded wait: `later`
// polls of 0.2 us (one CTA) to about 0.6 us (all SMs polling), one second at most,
// and `first` polls, 14 to 40 seconds, for the launch's first barrier, which may
// have to wait for other kernels to leave the SMs that the last CTAs need.  After
// an expired wait the CTA raises and waits no more, so the others' waits expire
// too and the launch ends.  1.13 us on GB300 between 8 to 152 CTAs.
struct GridBarrier {
  unsigned* counter;
  int* s_dead;                // shared: a wait of this CTA expired
  uint32_t target = 0;
  int polls, later;
  bool dead = false;
  __device__ __forceinline__ GridBarrier(unsigned* c, int* s, int first = 1 << 26,
                                         int later_polls = 1 << 21)
      : counter(c), s_dead(s), polls(first), later(later_polls) {
    if (threadIdx.x == 0) *s = 0;
  }
  __device__ __forceinline__ void sync() {
    target += gridDim.x;
    __syncthreads();
    if (threadIdx.x == 0 && !dead) {
      asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(counter) : "memory");
      uint32_t v = 0;
      int n = 0;
      do {
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(counter) : "memory");
      } while (int32_t(v - target) < 0 && ++n < polls);
      if (int32_t(v - target) < 0) *s_dead = 1;
    }
    __syncthreads();
    if (*s_dead) dead = true;
    polls = later;
  }
};

}  // namespace bpm
