// What the rows of keys and values do not exceed (HeadBound), gathered by the kernels that write or look at them.
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
// The largest magnitude of eight bf16 numbers, as the word of a float; infinity where one is no number.
__device__ __forceinline__ uint32_t largest8(const uint4& v) {
  const uint32_t m = __vmaxu2(__vmaxu2(v.x & 0x7FFF7FFFu, v.y & 0x7FFF7FFFu), __vmaxu2(v.z & 0x7FFF7FFFu, v.w & 0x7FFF7FFFu));
  return min(max(m << 16, m & 0xFFFF0000u), 0x7F800000u);
}
// Raises a bound to a thread's word.  `had` is the bound as it was read before; hardly a thread has more.
__device__ __forceinline__ void raise_bound(uint32_t* bound, uint32_t had, uint32_t word) {
  if (word > had) atomicMax(bound, word);
}
// The same by a whole warp, with one atomic.
__device__ __forceinline__ void raise_bound_warp(uint32_t* bound, uint32_t had, uint32_t word) {
  word = __reduce_max_sync(0xffffffffu, word);
  if ((threadIdx.x & 31) == 0 && word > had) atomicMax(bound, word);
}

}  // namespace fastar
