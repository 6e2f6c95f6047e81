// 32 x 32 bit transpose across a warp.
#pragma once

#include <stdint.h>

namespace ccm {

// operator(): lane i's word holds bit j = a[i][j]; afterwards lane j's word
// holds bit i = a[i][j].  Five exchanges: blocks of 16, 8, 4, 2, 1 swap their
// off-diagonal halves.  The lane's selectors are kept in registers.
struct BitTranspose {
  uint32_t sel16, sel8, keep4, keep2, keep1, rot4, rot2, rot1;
  __device__ __forceinline__ explicit BitTranspose(int lane) {
    sel16 = (lane & 16) ? 0x3276u : 0x5410u;
    sel8 = (lane & 8) ? 0x3715u : 0x6240u;
    keep4 = (lane & 4) ? 0xf0f0f0f0u : 0x0f0f0f0fu;
    keep2 = (lane & 2) ? 0xccccccccu : 0x33333333u;
    keep1 = (lane & 1) ? 0xaaaaaaaau : 0x55555555u;
    rot4 = (lane & 4) ? 28u : 4u;
    rot2 = (lane & 2) ? 30u : 2u;
    rot1 = (lane & 1) ? 31u : 1u;
  }
  __device__ __forceinline__ uint32_t operator()(uint32_t x) const {
    x = __byte_perm(x, __shfl_xor_sync(0xffffffffu, x, 16), sel16);
    x = __byte_perm(x, __shfl_xor_sync(0xffffffffu, x, 8), sel8);
    uint32_t y = __shfl_xor_sync(0xffffffffu, x, 4);
    x = (x & keep4) | (__funnelshift_l(y, y, rot4) & ~keep4);
    y = __shfl_xor_sync(0xffffffffu, x, 2);
    x = (x & keep2) | (__funnelshift_l(y, y, rot2) & ~keep2);
    y = __shfl_xor_sync(0xffffffffu, x, 1);
    return (x & keep1) | (__funnelshift_l(y, y, rot1) & ~keep1);
  }
};

}  // namespace ccm
