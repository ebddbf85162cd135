// Per row keep the k largest entries (S4: block scores, C2: prompt relevance), used by the kernels of update_kernels.cu and, for the
// prompt, at the end of the relevance kernel.
#pragma once
#include "common.h"
#include "ptx.cuh"

namespace fastar {

// S4 / C2: per row keep the k largest entries (ties -> lower index), listed ascending.
// One warp per row, the row in registers (entry 32 i + lane).  The k-th largest key is found bit by bit, from the highest bit in which the
// row's keys differ: one count over the row per bit, a dozen instructions per 32 entries, no barrier; the entries above it and the first of
// those equal to it are then listed in index order by ballots.  Latency-bound (a few thousand dependent instructions), and the time
// follows the registers a lane holds, whatever part of them the row fills: 2.5 us with 4, 3.9 with 16, 6.1 with 36, 8.9 with 64 (8 heads x
// 32 rows of block scores; 1 024 prompt tokens 8.8 with 36, 19.8 with 64).  Hence steps: 4, 16 and 64 are a factor of four apart, 8 halves
// the second (220 blocks of 12 heads 5.6 -> 4.5 us, 128 of 8 4.4 -> 3.5), and 36 divides the widest of them so that 131 072 keys in 128-slot
// blocks, or 1 024 prompt tokens, with an eighth to spare, are on the cheap side.  Measured against a 256-thread bitonic sort of (key,
// index): 256 rows of 1056 32.0 -> 7.2 us, 3400 rows of 512 78 -> 9.2 us, 444 rows of 256 7.6 -> 4.4 us, 36 rows of 512 prompt tokens 8.4 ->
// 6.5 us.
struct TopkArgs {
  void* src;                       // PROMPT: ordered-uint relevance (zeros are put back); else block scores as floats
  const float* src_hi;             // high digits of weighted scores, or nullptr
  int64_t src_head_stride;
  int src_row_stride, rows;
  const int32_t* len;              // [H] live slots, len_div per entry; nullptr: n_fixed entries
  int len_div, n_fixed, keep;
  int32_t* out;
  int64_t out_head_stride;
  int out_row_stride, out_fill;
  int32_t* nsel;
  int force_first, force_last;
  int* status;
};
TopkArgs block_topk_args(const CacheView& c, int nqb, int keep, int force_sink, int force_recent);      // update_kernels.cu

// One row by one warp.
template <bool PROMPT, int NV>
__device__ __forceinline__ void topk_row(const TopkArgs& a, int h, int row) {
  const int lane = threadIdx.x & 31;
  const int n = a.len ? (a.len[h] + a.len_div - 1) / a.len_div : a.n_fixed;
  const int k = min(a.keep, n);
  const int64_t so = static_cast<int64_t>(h) * a.src_head_stride + static_cast<int64_t>(row) * a.src_row_stride;
  // Keys are unsigned integers: the order-preserving image of a float (prompt relevance), or a block's collision
  // count, lo + 256 * hi when the histograms are weighted (both parts are exact integers in fp32, their sum below
  // 2^26).  Forced entries (the first force_first and the last force_last of the row) get bit 30 and so rank before
  // all others, in their own score order.
  uint32_t v[NV], hi = 0u, lo = 0xFFFFFFFFu;
  const int last = max(n - 1, 0);
#pragma unroll
  for (int q = 0; q < NV; ++q) v[q] = __ldcg(static_cast<const uint32_t*>(a.src) + so + min(32 * q + lane, last));   // all in flight at once
  if (!PROMPT) {
#pragma unroll
    for (int q = 0; q < NV; ++q) v[q] = static_cast<uint32_t>(__uint_as_float(v[q]));
    if (a.src_hi) {
#pragma unroll
      for (int q = 0; q < NV; ++q) v[q] += 256u * static_cast<uint32_t>(a.src_hi[so + min(32 * q + lane, last)]);
    }
    if (a.force_first > 0 || a.force_last > 0) {
#pragma unroll
      for (int q = 0; q < NV; ++q)
        if (32 * q + lane < a.force_first || 32 * q + lane >= n - a.force_last) v[q] |= 1u << 30;
    }
  }
#pragma unroll
  for (int q = 0; q < NV; ++q) {
    const bool in = 32 * q + lane < n;
    lo = min(lo, in ? v[q] : 0xFFFFFFFFu);
    v[q] = in ? v[q] : 0u;
    hi = max(hi, v[q]);
  }
  if (PROMPT) {                    // the next call's maxima start from zero
#pragma unroll
    for (int q = 0; q < NV; ++q)
      if (32 * q + lane < n) static_cast<uint32_t*>(a.src)[so + 32 * q + lane] = 0u;
  }
  hi = __reduce_max_sync(0xffffffffu, hi);
  lo = __reduce_min_sync(0xffffffffu, lo);
  // t: the largest value that at least k keys reach, or a lower one that no other key reaches.  Entries past the row are 0 and every candidate is above 0.
  const int bits = 32 - __clz(hi ^ lo);
  uint32_t t = bits >= 32 ? 0u : hi & ~((1u << bits) - 1u);
  for (int bit = bits - 1; bit >= 0; --bit) {
    const uint32_t cand = t | (1u << bit);
    int cnt[4] = {0, 0, 0, 0};
#pragma unroll
    for (int q = 0; q < NV; ++q) cnt[q & 3] += v[q] >= cand ? 1 : 0;
    const int reach = static_cast<int>(__reduce_add_sync(0xffffffffu, (cnt[0] + cnt[1]) + (cnt[2] + cnt[3])));
    if (reach >= k) t = cand;
    if (reach == k) break;                 // the k keys are told apart from the others: the lower bits do not matter
  }
  int above = 0;
#pragma unroll
  for (int q = 0; q < NV; ++q) above += v[q] > t ? 1 : 0;
  int equal_left = k - static_cast<int>(__reduce_add_sync(0xffffffffu, above));   // how many of the keys equal to t are kept
  int32_t* orow = a.out + static_cast<int64_t>(h) * a.out_head_stride + static_cast<int64_t>(row) * a.out_row_stride;
  const uint32_t below = (1u << lane) - 1u;
  int run = 0;
#pragma unroll
  for (int q = 0; q < NV; ++q) {
    const int i = 32 * q + lane;
    const bool eq = i < n && v[q] == t;
    const uint32_t eq_mask = __ballot_sync(0xffffffffu, eq);
    const bool take = i < n && (v[q] > t || (eq && __popc(eq_mask & below) < equal_left));
    const uint32_t mask = __ballot_sync(0xffffffffu, take);
    if (take) orow[FASTAR_IDX(run + __popc(mask & below), k, a.status)] = i;
    run += __popc(mask);
    equal_left -= __popc(eq_mask);
  }
  for (int i = k + lane; i < a.out_fill; i += 32) orow[i] = -1;
  if (a.nsel && row == 0 && lane == 0) a.nsel[h] = k;
}

}  // namespace fastar
