// What the rows of keys do not exceed (HeadBound), gathered by the kernels that write or look at them.
#pragma once
#include "common.h"
#include "ptx.cuh"

namespace fastar {

// The sum of the squares of eight bf16 numbers.
__device__ __forceinline__ float square_sum8(const uint4& v, float s) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int e = 0; e < 4; ++e)
    asm("{.reg .b16 l, h; mov.b32 {l, h}, %1; fma.rn.f32.bf16 %0, l, l, %0; fma.rn.f32.bf16 %0, h, h, %0;}" : "+f"(s) : "r"(w[e]));
  return s;
}
// Raises a bound to the words of a warp, with one atomic.  `had` is the bound as it was read before; hardly a warp has more.
__device__ __forceinline__ void raise_bound_warp(uint32_t* bound, uint32_t had, uint32_t word) {
  word = __reduce_max_sync(0xffffffffu, word);
  if ((threadIdx.x & 31) == 0 && word > had) atomicMax(bound, word);
}

}  // namespace fastar
