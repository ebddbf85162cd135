// Norms of rows, by the kernels that bound logits.
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
}  // namespace fastar
