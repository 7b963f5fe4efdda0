// Barriers in shared memory (mbarrier) of the convolution kernels, and the bounded wait on them.
#pragma once

#include <stdint.h>

namespace lbm_nn {

// Polls of a wait.  One suspends the thread until the phase completes, but for no more than 4.0 us (measured with 1 to 32
// warps an SM, although the hint allows 20), so a wait gives up after 2.1 s: ten times the longest one of a sound launch,
// the four million positions of the weight gradient's longest segment.  A bound on the clock instead made the loop longer
// and a forward pass on one image 2 % slower.
constexpr int kWaitPolls = 1 << 19;

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// bounded wait for the completion of phase `parity` of an mbarrier; false when it gave up
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
  uint32_t done = 0;
  for (int it = 0; it < kWaitPolls && !done; ++it)
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(bar), "r"(parity), "r"(20000)
        : "memory");
  return done != 0;
}

}  // namespace lbm_nn
