// The one loop behind every wait on an mbarrier (sm_100a).
//
// The bound is a time, in cycles of the SM.  A count of polls is no bound: a failed mbarrier.try_wait comes back after 4 us on a
// barrier that nothing touches, and after 27 ns on one that others arrive at without completing its phase (measured), so 2^18 polls
// are anything from 7 ms to a second.  The cycle counter because it is one instruction: with the global timer behind every failed
// poll, or with 256 polls and then the timer and the abort flag, the loops around the waits get slower (inverted-residual stack on
// 32 images 310 us with counted polls, 335 and 348 so, 312 with the cycle counter; 1024-token encoder 791, 806, 813, 790).
#pragma once
#include <cstdint>

namespace dnnf {

constexpr uint32_t kWaitLimitCycles = 1u << 31;    // 1.1 s at 1965 MHz (the counter wraps after twice that)

__device__ __forceinline__ uint32_t sm_cycles() { uint32_t t; asm volatile("mov.u32 %0, %%clock;" : "=r"(t)); return t; }

// True once `poll` is; false, with the CTA's abort flag set, when the limit has passed.
template <class Poll>
__device__ __forceinline__ bool bounded_wait(Poll poll, volatile int* abort_flag, uint32_t limit_cycles = kWaitLimitCycles) {
  const uint32_t start = sm_cycles();
#pragma unroll 1
  do { if (poll()) return true; } while (sm_cycles() - start < limit_cycles);
  *abort_flag = 1;
  return false;
}

}  // namespace dnnf
