// Bit-matrix helpers shared by the kernels that turn columns into words.
#pragma once

#include <cstdint>

namespace tpir {

// Transposes the 32 x 32 bit matrix of a warp (lane i's word = row i): lane j
// gets bit j of every lane, lane i's at bit i.  Five exchanges of s x s blocks:
// s = 16 and 8 by byte selection, s = 4, 2, 1 by a rotation and a mask.
struct WarpTranspose {
  uint32_t sel16, sel8, keep4, keep2, keep1, rot4, rot2, rot1;
  // (the lane is read here, not passed in, so that a caller short of registers
  // can form the object anew where it needs it)
  __device__ __forceinline__ WarpTranspose() {
    uint32_t lane;
    asm volatile("mov.u32 %0, %%laneid;" : "=r"(lane));
    sel16 = lane & 16u ? 0x3276u : 0x5410u;
    sel8 = lane & 8u ? 0x3715u : 0x6240u;
    keep4 = lane & 4u ? 0xF0F0F0F0u : 0x0F0F0F0Fu;
    keep2 = lane & 2u ? 0xCCCCCCCCu : 0x33333333u;
    keep1 = lane & 1u ? 0xAAAAAAAAu : 0x55555555u;
    rot4 = lane & 4u ? 28u : 4u;
    rot2 = lane & 2u ? 30u : 2u;
    rot1 = lane & 1u ? 31u : 1u;
  }
  static __device__ __forceinline__ uint32_t step(uint32_t x, uint32_t s, uint32_t keep, uint32_t rot) {
    const uint32_t y = __shfl_xor_sync(0xFFFFFFFFu, x, s);
    return (x & keep) | (__funnelshift_l(y, y, rot) & ~keep);
  }
  __device__ __forceinline__ uint32_t operator()(uint32_t x) const {
    x = __byte_perm(x, __shfl_xor_sync(0xFFFFFFFFu, x, 16), sel16);
    x = __byte_perm(x, __shfl_xor_sync(0xFFFFFFFFu, x, 8), sel8);
    x = step(x, 4, keep4, rot4);
    x = step(x, 2, keep2, rot2);
    return step(x, 1, keep1, rot1);
  }
};

}  // namespace tpir
