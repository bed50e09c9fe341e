// Issue of asynchronous instructions (TMA requests, tcgen05.mma, commits) from one lane of a converged warp (sm_100a).
//
// These instructions take their descriptors, coordinates and barrier addresses from uniform registers.  In a loop that
// sits under `if (lane == 0)` the compiler has to move every operand there, instruction by instruction, in front of each
// of them; a role loop that ALL lanes of a warp walk with identical values, with only the issuing instructions under
// elect.sync, keeps them there.  Measured in a bare ring (one producer, one issuer, a wait, four 128 x N x 16 MMAs and a
// commit per k-tile; B row-major): 582 -> 382 cycles per k-tile at N = 128, 581 -> 365 at N = 64, 750 -> 514 (the
// tensor pipe's own time) at N = 256; the producer alone 536 -> 366 cycles per k-tile of three requests.
#pragma once
#include <cstdint>

namespace dnnf {

// True in exactly one lane of a converged warp.  Has to stand right at the branch around the instructions to issue.
__device__ __forceinline__ bool elect_one() {
  uint32_t pred;
  asm volatile("{\n.reg .pred p;\nelect.sync _|p, 0xffffffff;\nselp.u32 %0, 1, 0, p;\n}" : "=r"(pred));
  return pred != 0;
}
// The warp's index, known to be the same in all its lanes.
__device__ __forceinline__ int uniform_warp() { return __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0); }

}  // namespace dnnf
