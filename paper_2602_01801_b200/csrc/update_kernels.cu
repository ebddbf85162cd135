// HBM-bound and integer kernels of the step (plain CUDA: coalesced vector access, warp shuffles,
// shared-memory sorts and scans):
//   S1  sign-random-projection codes (+ 1/|x|)               paper Section 5.1 (LSH)
//   T2  threshold, T3 grouping plan, T4 compaction / append / eviction plan   Section 5.2
//   T3/T4 commit lives in commit_kernel.cu
//   S2  per-block bucket histograms, S4 / C2 top-k with ties to the lower index   Sections 5.3, 5.4
#include "common.h"
#include "ptx.cuh"
#include "bound.cuh"
#include "topk.cuh"

#include <type_traits>

namespace fastar {

// ---------------------------------------------------------------------------------------------
// block-wide helpers (blockDim.x a multiple of 32, at most 1024)
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ int block_sum(int v, int* red) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  v = __reduce_add_sync(0xffffffffu, v);
  __syncthreads();
  if (lane == 0) red[warp] = v;
  __syncthreads();
  return __reduce_add_sync(0xffffffffu, lane < nw ? red[lane] : 0);
}
__device__ __forceinline__ int block_max(int v, int* red) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  v = __reduce_max_sync(0xffffffffu, v);
  __syncthreads();
  if (lane == 0) red[warp] = v;
  __syncthreads();
  return __reduce_max_sync(0xffffffffu, red[lane < nw ? lane : 0]);
}
// exclusive scan of one value per thread; *total receives the block sum
__device__ __forceinline__ int block_exscan(int v, int* red, int* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  int inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += t;
  }
  __syncthreads();
  if (lane == 31) red[warp] = inc;
  __syncthreads();
  const int x = lane < nw ? red[lane] : 0;
  const int base = static_cast<int>(__reduce_add_sync(0xffffffffu, lane < warp ? x : 0));
  *total = static_cast<int>(__reduce_add_sync(0xffffffffu, x));
  return base + inc - v;
}
__device__ __forceinline__ void bitonic_sort_smem(unsigned long long* keys, int np2) {
  for (int k = 2; k <= np2; k <<= 1) {
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int t = threadIdx.x; t < (np2 >> 1); t += blockDim.x) {
        const int i = ((t & ~(j - 1)) << 1) | (t & (j - 1));   // j is a power of two
        const bool up = (i & k) == 0;
        const unsigned long long a = keys[i], b = keys[i + j];
        if ((a > b) == up) { keys[i] = b; keys[i + j] = a; }
      }
      __syncthreads();
    }
  }
}

// ---------------------------------------------------------------------------------------------
// fp32 -> bf16 entry conversion (strided sources, contiguous destinations): up to three tensors of a call in one launch, one per
// blockIdx.z (a small call is a chain of launches; one per tensor made six of a step's 21).
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ void convert_rows(const ConvertArgs::Tensor& x, int h, int D, int64_t thread, int64_t threads) {
  const int64_t per_head = static_cast<int64_t>(x.n) * D / 4;
  for (int64_t q = thread; q < per_head; q += threads) {
    const int64_t e = q * 4;
    const int row = static_cast<int>(e / D), col = static_cast<int>(e % D);
    const float4 v = *reinterpret_cast<const float4*>(x.src + h * x.hs + row * x.ts + col);
    uint2 o;
    o.x = pack_bf16x2(v.x, v.y);
    o.y = pack_bf16x2(v.z, v.w);
    *reinterpret_cast<uint2*>(x.dst + (static_cast<int64_t>(h) * x.n + row) * D + col) = o;
  }
}
// The rows of all heads by all threads of a launch, four loads of each under way.  (Head by head, each from the first thread on, the heads
// followed one another and most threads had none.  Hash and conversion, d = 128, by two launches, so, now: 40 heads x 64 rows 9.4, 17.8, 6.3 us;
// 40 x 600 32, 33.5, 13.5; 12 x 4680 66, 33, 25; 1 x 256 6.5, 6.6, 6.0.)
template <int D>
__device__ __forceinline__ void convert_heads(const ConvertArgs::Tensor& x, int H, int thread, int threads) {
  constexpr int B = 4;
  const int total = H * x.n * (D / 4);               // below 2^25
  for (int q0 = thread; q0 < total; q0 += B * threads) {
    float4 v[B];
#pragma unroll
    for (int b = 0; b < B; ++b) {
      const int q = q0 + b * threads, row = q / (D / 4), h = row / x.n;
      if (q < total) v[b] = *reinterpret_cast<const float4*>(x.src + h * x.hs + (row - h * x.n) * x.ts + q % (D / 4) * 4);
    }
#pragma unroll
    for (int b = 0; b < B; ++b) {
      const int q = q0 + b * threads;
      if (q < total) *reinterpret_cast<uint2*>(x.dst + static_cast<int64_t>(q) * 4) = make_uint2(pack_bf16x2(v[b].x, v[b].y), pack_bf16x2(v[b].z, v[b].w));
    }
  }
}
__global__ void convert_kernel(const ConvertArgs a, int D) {
  chain_wait();
  convert_rows(a.t[blockIdx.z], blockIdx.y, D, blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x, static_cast<int64_t>(gridDim.x) * blockDim.x);
}
int launch_convert_f32_to_bf16(const ConvertArgs& a, int H, int D, cudaStream_t st) {
  int64_t want = 0;
  for (int i = 0; i < a.count; ++i) {
    const int64_t blocks = (static_cast<int64_t>(a.t[i].n) * D / 4 + 255) / 256;
    want = blocks > want ? blocks : want;
  }
  if (want == 0) return 0;
  launch_chained(convert_kernel, dim3(static_cast<int>(want < 1024 ? want : 1024), H, a.count), 256, 0, st, a, D);
  return cudaGetLastError() == cudaSuccess ? 1 : FASTAR_ERR_CUDA;
}

// Eight counters as bf16: all of them (SHIFT < 0: exact up to 256), or one of their two 8-bit digits.
template <int SHIFT>
__device__ __forceinline__ uint4 pack_counts(const int (&v)[8]) {
  uint32_t w[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const int lo = SHIFT < 0 ? v[2 * e] : (v[2 * e] >> (SHIFT < 0 ? 0 : SHIFT)) & 255, hi = SHIFT < 0 ? v[2 * e + 1] : (v[2 * e + 1] >> (SHIFT < 0 ? 0 : SHIFT)) & 255;
    w[e] = pack_bf16x2(static_cast<float>(lo), static_cast<float>(hi));
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}

// ---------------------------------------------------------------------------------------------
// S1: codes (and reciprocal norms).
// ---------------------------------------------------------------------------------------------
// X[n x D] . R^T[D x 32] is a skinny contraction (N = 32) bound by reading X once, so it runs on warp-level
// mma.sync (m16n8k16, bf16 in, fp32 accumulate) with R held in registers: one warp = 16 rows per pass, no shared
// memory, ~100 instructions per 16 rows.  The next group's rows are fetched as this one's are used up (40 x 10800 rows, 110 MB,
// 17 us at the measured bandwidth: 48 -> 39 us; 12 x 4680 9.9 -> 8.9).  Fragment layout (g = lane / 4, t = lane % 4):
//   A: a0 = X[g][2t..], a1 = X[g+8][2t..], a2 = X[g][2t+8..], a3 = X[g+8][2t+8..]   (bf16 pairs)
//   B: b0 = R[n = 8*nt + g][2t..], b1 = R[n][2t+8..];   C: c0,c1 = row g, cols 2t,2t+1;  c2,c3 = row g+8.
// ROWS > 0 (the query side of S2 in the same launch: 12 x 4680 rows 9.2 + 2.7 -> 10.2 us, 2 x 600 4.1 + 2.3 -> 4.4): blocks of 64 or 128 rows,
// whose bucket histograms the CTA writes.  With four of eight warps idle for blocks of 64, 40 x 10800 rows took 45 us, with two blocks a pass 37
// (d = 64 29 -> 22); with a launch of their own for the histograms 33 (26).  Blocks of 128: 34 (21) us, 31 (24) with that launch.
// F32: the rows are fp32 (conv.t[0]); the kernel rounds them on their way, writes them where the kernels behind it read them, and converts
// conv's other tensors too (an update's values): one head x 256 rows, d = 64, 2.2 + 3.4 -> 4.7 us and a launch less for the host.
struct BlockHist {
  __nv_bfloat16* hist;         // [H][max_qb][hist_cols]
  int max_qb, hist_cols;
};
template <int D, int ROWS, bool F32>
__global__ void __launch_bounds__(256, 2) prep_kernel(const __nv_bfloat16* __restrict__ x, int H, int n, int64_t hs, int64_t ts,
                                                   const __nv_bfloat16* __restrict__ lsh, int T, int B,
                                                   uint32_t* __restrict__ code_out, float* __restrict__ rnorm_out,
                                                   int64_t out_stride, UpdateScratch clear, BlockHist bh, const ConvertArgs conv) {
  constexpr bool BLOCKS = ROWS > 0;
  constexpr int per_block = BLOCKS ? ROWS / 16 : 1, blocks_a_pass = BLOCKS ? 8 / per_block : 1;
  __shared__ __align__(16) int hist[BLOCKS ? 2 : 1][blocks_a_pass][BLOCKS ? 1024 : 4];      // [pass & 1][block of the pass]
  if (BLOCKS)
    for (int q = threadIdx.x; q < 2 * blocks_a_pass * 1024 / 4; q += 256) reinterpret_cast<int4*>(&hist[0][0][0])[q] = make_int4(0, 0, 0, 0);
  constexpr int KS = D / 16;
  constexpr int RP = D + 8;                    // padded row of the staged projection matrix (bank-conflict free)
  __shared__ __align__(16) __nv_bfloat16 r_s[32 * RP];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane >> 2, t = lane & 3;
  const int ncol = T * B;
  // the projection matrix goes through shared memory once per CTA (coalesced 128-bit loads), then into registers
  for (int q = threadIdx.x; q < 32 * (D / 8); q += blockDim.x) {
    const int col = q / (D / 8), ch = q % (D / 8);
    uint4 v = make_uint4(0, 0, 0, 0);
    if (col < ncol) v = *reinterpret_cast<const uint4*>(lsh + col * D + ch * 8);
    *reinterpret_cast<uint4*>(r_s + col * RP + ch * 8) = v;
  }
  // 16-row groups of all heads, dealt to the warps of a grid that fills the SMs once, eight to a CTA's pass
  // BLOCKS: groups are numbered through whole blocks, so that a pass has one block of 128 rows or two of 64.  The histograms of two passes
  // take turns: a thread that has written its columns of one clears them at once, and by the barrier of the next pass they are free.
  const int groups_per_head = BLOCKS ? (n + ROWS - 1) / ROWS * per_block : (n + 15) / 16;
  const int total_groups = groups_per_head * H;
  const int stride = static_cast<int>(gridDim.x) * 8;
  uint4 va[KS / 2], vb[KS / 2];
  using Source = std::conditional_t<F32, float, __nv_bfloat16>;
  const Source* src;
  if constexpr (F32) src = conv.t[0].src;
  else src = x;
  const Source *xa = src, *xb = src;                                   // this lane's rows of the group that is fetched
  __nv_bfloat16 *oa = nullptr, *ob = nullptr;                          // F32: and where they go
  auto rows = [&](int grp) {
    const int h = grp / groups_per_head;
    const int r0 = (grp - h * groups_per_head) * 16;
    const int ra = min(r0 + g, n - 1), rb = min(r0 + g + 8, n - 1);    // rows past the end repeat the last one
    const int64_t head = F32 ? conv.t[0].hs : hs, row = F32 ? conv.t[0].ts : ts;
    xa = src + h * head + ra * row + 8 * t;
    xb = src + h * head + rb * row + 8 * t;
    if constexpr (F32) {
      oa = conv.t[0].dst + (static_cast<int64_t>(h) * n + ra) * D + 8 * t;
      ob = conv.t[0].dst + (static_cast<int64_t>(h) * n + rb) * D + 8 * t;
    }
  };
  auto fetch = [&](int kk) {                                           // one 128-bit load per row and 32-wide k block, F32: two
    if constexpr (F32) {
      auto round8 = [](const float* p) {
        const float4 u = *reinterpret_cast<const float4*>(p), v = *reinterpret_cast<const float4*>(p + 4);
        return make_uint4(pack_bf16x2(u.x, u.y), pack_bf16x2(u.z, u.w), pack_bf16x2(v.x, v.y), pack_bf16x2(v.z, v.w));
      };
      va[kk] = round8(xa + 32 * kk);
      vb[kk] = round8(xb + 32 * kk);
      *reinterpret_cast<uint4*>(oa + 32 * kk) = va[kk];
      *reinterpret_cast<uint4*>(ob + 32 * kk) = vb[kk];
    } else {
      va[kk] = *reinterpret_cast<const uint4*>(xa + 32 * kk);
      vb[kk] = *reinterpret_cast<const uint4*>(xb + 32 * kk);
    }
  };
  const int first = blockIdx.x * 8 + warp;
  chain_wait();                                // (the projection matrix is written when the cache is created)
  if (first < total_groups) {
    rows(first);
#pragma unroll
    for (int kk = 0; kk < KS / 2; ++kk) fetch(kk);
  }
  const int64_t thread = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x, threads = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t q = thread; q < clear.n_best; q += threads) clear.best[q] = 0ull;
  for (int64_t q = thread; q < clear.n_cnt16; q += threads) clear.cnt[q] = make_uint4(0, 0, 0, 0);
  for (int64_t q = thread; q < clear.n_heads; q += threads) clear.n_match[q] = 0;
  __syncthreads();
  uint32_t bf[KS][4][2];
#pragma unroll
  for (int ks = 0; ks < KS; ++ks)
#pragma unroll
    for (int nt = 0; nt < 4; ++nt) {
      // The contraction index may be permuted freely as long as A and B agree: lane t of a quad reads 8
      // contiguous elements (one 128-bit load) per 32-wide k block, k = 32*(ks/2) + 8t + 4*(ks%2) + {0,1 | 2,3}.
      const int col = 8 * nt + g;
      const __nv_bfloat16* rp = r_s + col * RP + 32 * (ks >> 1) + 8 * t + 4 * (ks & 1);
      bf[ks][nt][0] = *reinterpret_cast<const uint32_t*>(rp);
      bf[ks][nt][1] = *reinterpret_cast<const uint32_t*>(rp + 2);
    }
  int buffer = 0;
  for (int grp = first; BLOCKS ? grp - warp < total_groups : grp < total_groups; grp += stride) {
    const int h = grp / groups_per_head;
    const int r0 = (grp - h * groups_per_head) * 16;
    const bool more = grp + stride < total_groups;
    if (more) rows(grp + stride);
    if (!BLOCKS || grp < total_groups) {         // (the last pass may have a block less)
      float acc[4][4];
#pragma unroll
      for (int nt = 0; nt < 4; ++nt)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[nt][e] = 0.f;
      float sqa = 0.f, sqb = 0.f;
#pragma unroll
      for (int ks = 0; ks < KS; ++ks) {
        const uint4 pa = va[ks >> 1], pb = vb[ks >> 1];
        const uint32_t a0 = (ks & 1) ? pa.z : pa.x, a2 = (ks & 1) ? pa.w : pa.y;
        const uint32_t a1 = (ks & 1) ? pb.z : pb.x, a3 = (ks & 1) ? pb.w : pb.y;
        {
          const float2 f0 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&a0));
          const float2 f2 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&a2));
          const float2 f1 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&a1));
          const float2 f3 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&a3));
          sqa = fmaf(f0.x, f0.x, fmaf(f0.y, f0.y, fmaf(f2.x, f2.x, fmaf(f2.y, f2.y, sqa))));
          sqb = fmaf(f1.x, f1.x, fmaf(f1.y, f1.y, fmaf(f3.x, f3.x, fmaf(f3.y, f3.y, sqb))));
        }
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
          asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                       : "+f"(acc[nt][0]), "+f"(acc[nt][1]), "+f"(acc[nt][2]), "+f"(acc[nt][3])
                       : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(bf[ks][nt][0]), "r"(bf[ks][nt][1]));
        if ((ks & 1) && more) fetch(ks >> 1);               // the registers are free: the next group's rows, in flight until its turn
      }
      // sign bits: this lane owns columns 8*nt + 2t, +1 of rows g and g+8; OR over the quad gives all 32 columns
      uint32_t ma = 0, mb = 0;
#pragma unroll
      for (int nt = 0; nt < 4; ++nt) {
        const int c0 = 8 * nt + 2 * t;
        ma |= (acc[nt][0] > 0.f ? 1u : 0u) << c0;
        ma |= (acc[nt][1] > 0.f ? 1u : 0u) << (c0 + 1);
        mb |= (acc[nt][2] > 0.f ? 1u : 0u) << c0;
        mb |= (acc[nt][3] > 0.f ? 1u : 0u) << (c0 + 1);
      }
#pragma unroll
      for (int o = 1; o <= 2; o <<= 1) {
        ma |= __shfl_xor_sync(0xffffffffu, ma, o);
        mb |= __shfl_xor_sync(0xffffffffu, mb, o);
        sqa += __shfl_xor_sync(0xffffffffu, sqa, o);
        sqb += __shfl_xor_sync(0xffffffffu, sqb, o);
      }
      uint32_t ca = 0, cb = 0;
      for (int tt = 0; tt < T; ++tt) {
        ca |= ((ma >> (tt * B)) & ((1u << B) - 1u)) << (8 * tt);
        cb |= ((mb >> (tt * B)) & ((1u << B) - 1u)) << (8 * tt);
      }
      if (BLOCKS && t < T) {                   // table t of rows g and g + 8
        int* counts = hist[buffer][warp / per_block] + (t << B);
        if (r0 + g < n) atomicAdd(counts + ((ca >> (8 * t)) & 0xFFu), 1);
        if (r0 + g + 8 < n) atomicAdd(counts + ((cb >> (8 * t)) & 0xFFu), 1);
      }
      if (t == 0) {
        if (r0 + g < n) {
          code_out[h * out_stride + r0 + g] = ca;
          if (rnorm_out) rnorm_out[h * out_stride + r0 + g] = sqa > 0.f ? 1.f / sqrtf(sqa) : 0.f;
        }
        if (r0 + g + 8 < n) {
          code_out[h * out_stride + r0 + g + 8] = cb;
          if (rnorm_out) rnorm_out[h * out_stride + r0 + g + 8] = sqb > 0.f ? 1.f / sqrtf(sqb) : 0.f;
        }
      }
    }
    if (BLOCKS) {
      __syncthreads();
      const int half = threadIdx.x >> 7, column = 8 * (threadIdx.x & 127), block = (grp - warp) / per_block + half;       // of all heads
      if (half < blocks_a_pass && block * per_block < total_groups && column < bh.hist_cols) {
        const int blocks = groups_per_head / per_block;
        int* counts = &hist[buffer][half][column];
        int v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) { v[e] = counts[e]; counts[e] = 0; }
        *reinterpret_cast<uint4*>(bh.hist + (static_cast<int64_t>(block / blocks) * bh.max_qb + block % blocks) * bh.hist_cols + column) = pack_counts<-1>(v);
      }
      buffer ^= 1;
    }
  }
  if constexpr (F32) {
    if (conv.count > 1) convert_heads<D>(conv.t[1], H, static_cast<int>(thread), static_cast<int>(threads));      // (by constants: an index puts the array on the stack)
    if (conv.count > 2) convert_heads<D>(conv.t[2], H, static_cast<int>(thread), static_cast<int>(threads));
  }
}
static int launch_prep_generic(const CacheView& c, const __nv_bfloat16* x, int n, int64_t hs, int64_t ts, uint32_t* code_out,
                               float* rnorm_out, int64_t out_stride, cudaStream_t st, const UpdateScratch& clear = UpdateScratch{},
                               const ConvertArgs& conv = ConvertArgs{}) {
  if (n <= 0) return 0;
  const int groups = ((n + 15) / 16) * c.H;                      // 16 rows per warp pass
  // CTAs for the rows (eight warps of 16 a pass) or for the zeros (32 KB each), whichever needs more: a few tokens against many heads
  // with long caches leave far more to clear than to hash (40 heads x 65536 slots, 1 to 16 tokens: an update of 81 us with CTAs for
  // the rows only, 50 with these).
  int64_t want = max(static_cast<int64_t>(groups + 7) / 8, (clear.n_best / 2 + clear.n_cnt16 + 2047) / 2048);
  if (conv.count > 1) want = max(want, static_cast<int64_t>(conv.count - 1) * c.H * n * c.D / 4 / 256);      // four numbers a thread
  const dim3 grid(static_cast<unsigned>(max(static_cast<int64_t>(1), min(want, static_cast<int64_t>(2 * 148)))));
  auto launch = [&](auto kernel) {
    launch_chained(kernel, grid, 256, 0, st, x, c.H, n, hs, ts, c.lsh, c.T, c.B, code_out, rnorm_out, out_stride, clear, BlockHist{}, conv);
  };
  if (c.D == 128) conv.count > 0 ? launch(prep_kernel<128, 0, true>) : launch(prep_kernel<128, 0, false>);
  else conv.count > 0 ? launch(prep_kernel<64, 0, true>) : launch(prep_kernel<64, 0, false>);
  return cudaGetLastError() == cudaSuccess ? 1 : FASTAR_ERR_CUDA;
}
// Codes of the queries and the bucket histograms of their blocks of block_q rows.
int launch_query_blocks(const CacheView& c, const __nv_bfloat16* q, int nq, int64_t hs, int64_t ts, int block_q, cudaStream_t st, const ConvertArgs& conv) {
  if (nq <= 0) return 0;
  const int64_t groups = static_cast<int64_t>((nq + block_q - 1) / block_q) * c.H * (block_q / 16);
  const int grid = static_cast<int>(min((groups + 7) / 8, static_cast<int64_t>(2 * 148)));
  auto launch = [&](auto kernel) {
    launch_chained(kernel, grid, 256, 0, st, q, c.H, nq, hs, ts, c.lsh, c.T, c.B, c.code_q_sa, nullptr, c.max_tokens, UpdateScratch{}, BlockHist{c.hq, c.max_qb, c.hist_cols}, conv);
  };
  if (conv.count > 0) {
    if (c.D == 128) block_q == 128 ? launch(prep_kernel<128, 128, true>) : launch(prep_kernel<128, 64, true>);
    else block_q == 128 ? launch(prep_kernel<64, 128, true>) : launch(prep_kernel<64, 64, true>);
  } else {
    if (c.D == 128) block_q == 128 ? launch(prep_kernel<128, 128, false>) : launch(prep_kernel<128, 64, false>);
    else block_q == 128 ? launch(prep_kernel<64, 128, false>) : launch(prep_kernel<64, 64, false>);
  }
  return cudaGetLastError() == cudaSuccess ? 1 : FASTAR_ERR_CUDA;
}
bool plan_is_fused(const CacheView& c, int n);
int plan_fused_smem(const CacheView& c, int n);
// The words that the search and the matching of an update accumulate into, as zeros (by a memset of their own they cost 4 us with its
// two gaps): those of the view's heads and no others, because the view may be a range of heads whose neighbours are at work.  The
// rows of `best` are max_tokens words of 8 bytes, so a range's first word may lie between two 16-byte boundaries.
UpdateScratch update_scratch(const CacheView& c, int n) {
  UpdateScratch z{};
  z.best = c.best;
  z.n_best = static_cast<int64_t>(c.H) * c.max_tokens;
  if (!plan_is_fused(c, n)) {                // the planner in one kernel counts in its shared memory
    z.cnt = reinterpret_cast<uint4*>(c.cnt);             // the capacity is a multiple of 128
    z.n_cnt16 = static_cast<int64_t>(c.H) * c.CAP / 4;
    z.n_match = c.n_match;
    z.n_heads = c.H;
  }
  return z;
}
// The first kernel of an update: codes and reciprocal norms of the new keys, and the zeros.
int launch_prep_update(const CacheView& c, const __nv_bfloat16* k_new, int n, int64_t hs, int64_t ts, cudaStream_t st, const ConvertArgs& conv) {
  return launch_prep_generic(c, k_new, n, hs, ts, c.code_new, c.rnorm_new, c.max_tokens, st, update_scratch(c, n), conv);
}
int launch_prep_codes_strided(const CacheView& c, const __nv_bfloat16* x, int n, int64_t hs, int64_t ts, uint32_t* code_out,
                              int64_t out_stride, cudaStream_t st) {
  return launch_prep_generic(c, x, n, hs, ts, code_out, nullptr, out_stride, st);
}

// ---------------------------------------------------------------------------------------------
// T2-T4 planning: one kernel where its counters fit a CTA's shared memory (plan_fused_kernel, plan_is_fused), else three; all work
// O(n + L), no sort:
//   match_count : decode the packed arg-max, threshold (T2), count the tokens matched to each slot
//   plan        : one CTA per head: scan the slot counts -> groups (touched slots) and their member
//                 ranges; scan the tokens -> unmatched tokens in token order; place them (append, then
//                 victims in (stamp, slot) order).  Validate, then commit.
//   scatter     : put each matched token into its group's member range
// Members of a group land in arbitrary order; the commit walks them in ascending token order, so the
// result does not depend on it.
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) match_count_kernel(const CacheView c, int n, float tau, const UpdateOut out) {
  chain_wait();
  const int h = blockIdx.y;
  const int64_t tb = static_cast<int64_t>(h) * c.max_tokens;
  int mine = 0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const unsigned long long b = c.best[tb + i];
    int j = -1;
    float s = 0.f;
    if (b != 0ull) {
      j = FASTAR_IDX(static_cast<int>(0xFFFFFFFFu - static_cast<uint32_t>(b & 0xFFFFFFFFull)), c.CAP, c.status);
      s = ordered_to_float(static_cast<uint32_t>(b >> 32));
    }
    const bool matched = j >= 0 && s >= tau;
    c.match[tb + i] = matched ? j : -1;
    c.sim[tb + i] = s;
    if (out.match) out.match[static_cast<int64_t>(h) * n + i] = matched ? j : -1;
    if (out.sim) out.sim[static_cast<int64_t>(h) * n + i] = s;
    if (matched) atomicAdd(c.cnt + static_cast<int64_t>(h) * c.CAP + j, 1);
    mine += matched ? 1 : 0;
  }
  if (c.pool_shared) {                       // the planner of every head needs every head's number of unmatched tokens
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mine += __shfl_xor_sync(0xFFFFFFFFu, mine, o);
    if ((threadIdx.x & 31) == 0 && mine > 0) atomicAdd(c.n_match + h, mine);
  }
}

// Eviction.  evictable = live, past the sink prefix, stamp < now, not touched by this update.  The oldest E go, ties by slot; what is
// looked for is the age (now - stamp) that at least E evictable slots reach, the greatest such.  False: there are fewer than E.
// untouched(j, free): whether slots j .. j + 15 are matched by no token; keys: room for the victims, up to a power of two.
template <class Untouched>
__device__ __forceinline__ bool choose_victims(const CacheView& c, int h, int L, int now, int E, unsigned long long* keys, int* red,
                                               int& evicted_tokens, const Untouched& untouched) {
  const int tid = threadIdx.x;
  const int64_t tb = static_cast<int64_t>(h) * c.max_tokens, sb = static_cast<int64_t>(h) * c.CAP;
  bool ok = true;
  // The 16 slots of pass p from j = 16 (1024 p + tid) on, read with 128-bit loads: their ages, 0 = not evictable.
  auto ages16 = [&](int j, int (&age)[16]) {
    if (j < L) {                                 // j is a multiple of 16 and the capacity a multiple of 128
      bool free[16];
      untouched(j, free);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int4 sp = *reinterpret_cast<const int4*>(c.stamp + sb + j + 4 * q);
        const int sq[4] = {sp.x, sp.y, sp.z, sp.w};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int s = j + 4 * q + u;
          age[4 * q + u] = (s < L && s >= c.n_sink && free[4 * q + u] && sq[u] < now) ? now - sq[u] : 0;
        }
      }
    } else {
#pragma unroll
      for (int u = 0; u < 16; ++u) age[u] = 0;
    }
  };
  // Up to 2 x 16384 slots a thread keeps its ages in registers, two to a word, so the search for the age and the compaction read
  // nothing again (12 heads x 32768 slots at capacity: 87 -> 44 us).  A third pass would be eight more of the 64 registers that 1 024
  // threads leave each, and two are all that fit (12 bytes spill already): longer caches, and ages above 16 bits, go through L2 in
  // every pass, as all did before.
  constexpr int kPasses = 2;
  uint32_t held[kPasses][8];
  int cand = 0, a_min = 0x7fffffff, a_max = 0;
  for (int j0 = 0, p = 0; j0 < L; j0 += 16 * blockDim.x, ++p) {
    int age[16];
    ages16(j0 + 16 * tid, age);
#pragma unroll
    for (int u = 0; u < 16; ++u)
      if (age[u] > 0) { ++cand; a_min = min(a_min, age[u]); a_max = max(a_max, age[u]); }
#pragma unroll
    for (int q = 0; q < kPasses; ++q)
      if (p == q)
#pragma unroll
        for (int u = 0; u < 8; ++u) held[q][u] = (static_cast<uint32_t>(age[2 * u]) & 0xFFFFu) | (static_cast<uint32_t>(age[2 * u + 1]) << 16);
  }
  cand = block_sum(cand, red);
  a_min = -block_max(-a_min, red);
  a_max = block_max(a_max, red);
  if (cand < E) ok = false;
  const bool in_regs = L <= kPasses * 16 * static_cast<int>(blockDim.x) && a_max <= 0xFFFF;
  auto for_each_pass = [&](auto&& body) {        // body(first slot, ages)
    int age[16];
    if (in_regs) {
#pragma unroll
      for (int p = 0; p < kPasses; ++p) {
        const int j0 = p * 16 * blockDim.x;
        if (j0 >= L) break;
#pragma unroll
        for (int u = 0; u < 8; ++u) { age[2 * u] = held[p][u] & 0xFFFFu; age[2 * u + 1] = held[p][u] >> 16; }
        body(j0 + 16 * tid, age);
      }
    } else {
      for (int j0 = 0; j0 < L; j0 += 16 * blockDim.x) {
        ages16(j0 + 16 * tid, age);
        body(j0 + 16 * tid, age);
      }
    }
  };
  auto reach = [&](int a) {                      // evictable slots of that age or older
    int cn = 0;
    for_each_pass([&](int, int (&age)[16]) {
#pragma unroll
      for (int u = 0; u < 16; ++u) cn += age[u] >= a ? 1 : 0;
    });
    return block_sum(cn, red);
  };
  if (ok) {
    int lo = a_min, hi = a_max;                  // all reach a_min
    while (lo < hi) {
      const int mid = lo + ((hi - lo + 1) >> 1);
      if (reach(mid) >= E) lo = mid; else hi = mid - 1;
    }
    const int a_star = lo;
    const int need_eq = E - reach(a_star + 1);
    // ordered compaction of the victims: all older slots, and the first need_eq slots of that age
    int eq_run = 0, out_run = 0;
    for_each_pass([&](int j, int (&age)[16]) {
      int my_eq = 0;
#pragma unroll
      for (int u = 0; u < 16; ++u) my_eq += age[u] == a_star ? 1 : 0;
      int tot_eq;
      int eq_rank = eq_run + block_exscan(my_eq, red, &tot_eq);
      int my_take = 0;
      unsigned take_mask = 0;
#pragma unroll
      for (int u = 0; u < 16; ++u) {
        const bool is_eq = age[u] == a_star;
        const bool take = age[u] > a_star || (is_eq && eq_rank < need_eq);
        eq_rank += is_eq ? 1 : 0;
        take_mask |= (take ? 1u : 0u) << u;
        my_take += take ? 1 : 0;
      }
      int tot_take;
      int pos = out_run + block_exscan(my_take, red, &tot_take);
#pragma unroll
      for (int u = 0; u < 16; ++u)
        if ((take_mask >> u) & 1u)
          keys[pos++] = (static_cast<unsigned long long>(static_cast<uint32_t>(now - age[u])) << 32) | static_cast<uint32_t>(j + u);
      eq_run += tot_eq;
      out_run += tot_take;
    });
    int e2 = 1;
    while (e2 < E) e2 <<= 1;
    for (int p = E + tid; p < e2; p += blockDim.x) keys[p] = ~0ull;
    __syncthreads();
    bitonic_sort_smem(keys, e2);
    int ev = 0;
    for (int k = tid; k < E; k += blockDim.x) {
      const int v = static_cast<int>(keys[k] & 0xFFFFFFFFull);
      c.victims[tb + k] = v;
      ev += c.count[sb + v];
    }
    evicted_tokens = block_sum(ev, red);
  }
  return ok;
}

__global__ void __launch_bounds__(1024) plan_kernel(const CacheView c, int n, int32_t* __restrict__ dest_out) {
  chain_wait();
  extern __shared__ unsigned long long keys[];   // victim sort buffer, only touched when evicting
  __shared__ int red[32];
  const int h = blockIdx.x, tid = threadIdx.x;
  const int64_t tb = static_cast<int64_t>(h) * c.max_tokens;
  const int64_t sb = static_cast<int64_t>(h) * c.CAP;
  const int64_t gb = static_cast<int64_t>(h) * (c.max_tokens + 1);
  const int L = c.len[h];
  const int now = *c.now;

  // groups: 16 consecutive slots per thread and pass (four 128-bit loads in flight; counts past the live length
  // are zero and the capacity is a multiple of 128, so whole vectors can be read up to the capacity).  The
  // numbers of groups and of members are scanned together, packed into one word (both stay below 2^16).
  int seg_run = 0, mem_run = 0;
  for (int j0 = 0; j0 < L; j0 += 16 * blockDim.x) {
    const int j = j0 + 16 * tid;
    int cn[16];
    if (j < c.CAP) {
      const int4* p = reinterpret_cast<const int4*>(c.cnt + sb + j);
      const int4 v0 = p[0], v1 = p[1], v2 = p[2], v3 = p[3];
      cn[0] = v0.x; cn[1] = v0.y; cn[2] = v0.z; cn[3] = v0.w;
      cn[4] = v1.x; cn[5] = v1.y; cn[6] = v1.z; cn[7] = v1.w;
      cn[8] = v2.x; cn[9] = v2.y; cn[10] = v2.z; cn[11] = v2.w;
      cn[12] = v3.x; cn[13] = v3.y; cn[14] = v3.z; cn[15] = v3.w;
    } else {
#pragma unroll
      for (int u = 0; u < 16; ++u) cn[u] = 0;
    }
    int my_seg = 0, my_mem = 0;
#pragma unroll
    for (int u = 0; u < 16; ++u) { my_seg += cn[u] > 0; my_mem += cn[u]; }
    int tot;
    const int ex = block_exscan((my_seg << 16) | my_mem, red, &tot);
    const int tot_seg = tot >> 16, tot_mem = tot & 0xFFFF;
    int seg = seg_run + (ex >> 16);
    int mem = mem_run + (ex & 0xFFFF);
#pragma unroll
    for (int u = 0; u < 16; ++u) {
      if (cn[u] > 0) {
        c.segslot[tb + seg] = j + u;
        c.segpos[gb + seg] = mem;
        c.cur[sb + j + u] = mem;
        ++seg;
        mem += cn[u];
      }
    }
    seg_run += tot_seg;
    mem_run += tot_mem;
  }
  const int n_seg = seg_run, M = mem_run;
  if (tid == 0) c.segpos[gb + n_seg] = M;

  // Slot limit of this head.  Shared page pool: the free pages go to the heads in head order, each asking for what its
  // unmatched tokens need up to the capacity.  Every head's planner repeats the same short scan over the heads before
  // it (lengths, matched counts and the pool's fill are only written by the kernels that follow), so the CTAs need no
  // exchange.  A head's pages are never returned, so a head holds ceil(length / page) of them.
  __shared__ int s_limit, s_grant, s_base;
  if (tid == 0) {
    int limit = c.CAP, grant = 0, base = 0;
    if (c.pool_shared) {
      int next = *c.next_free;
      for (int g = 0; g <= h; ++g) {
        const int Lg = c.len[g], Ug = n - c.n_match[g];
        const int held = (Lg + c.PT - 1) / c.PT;
        const int asked = (min(c.CAP, Lg + Ug) + c.PT - 1) / c.PT - held;
        const int got = min(asked, c.pool_pages - next);
        if (g == h) { grant = got; base = next; limit = min(c.CAP, (held + got) * c.PT); }
        next += got;
      }
    }
    s_limit = limit; s_grant = grant; s_base = base;
  }
  __syncthreads();
  const int limit = s_limit, grant = s_grant;
  if (grant > 0) {
    const int held = (L + c.PT - 1) / c.PT;
    for (int p = tid; p < grant; p += blockDim.x) c.page_table[static_cast<int64_t>(h) * c.CAPB + held + p] = s_base + p;
  }

  // Unmatched tokens in token order.  The first `limit - L` of them are appended; that needs no count of the others.
  const int room = limit - L;
  int u_run = 0;
  for (int i0 = 0; i0 < n; i0 += 4 * blockDim.x) {
    const int i = i0 + 4 * tid;
    int un[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) un[u] = (i + u < n && c.match[tb + i + u] < 0) ? 1 : 0;
    int tot;
    int k = u_run + block_exscan(un[0] + un[1] + un[2] + un[3], red, &tot);
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (un[u]) {
        c.ulist[tb + k] = i + u;
        if (k < room) {
          c.dest[tb + i + u] = L + k;
          if (dest_out) dest_out[static_cast<int64_t>(h) * n + i + u] = L + k;
        }
        ++k;
      }
    u_run += tot;
  }
  const int U = u_run;
  const int A = min(U, room);
  const int E = U - A;
  int ok = 1;
  int evicted_tokens = 0;
  if (E > 0) {
    ok = choose_victims(c, h, L, now, E, keys, red, evicted_tokens, [&](int j, bool (&free)[16]) {
      const int4* p = reinterpret_cast<const int4*>(c.cnt + sb + j);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int4 cn = p[q];
        free[4 * q] = cn.x == 0; free[4 * q + 1] = cn.y == 0; free[4 * q + 2] = cn.z == 0; free[4 * q + 3] = cn.w == 0;
      }
    }) ? 1 : 0;
  }
  __syncthreads();
  // destinations of the tokens that take a victim's slot (matched tokens get theirs in the scatter kernel)
  if (ok) {
    for (int k = A + tid; k < U; k += blockDim.x) {
      const int i = FASTAR_IDX(c.ulist[tb + k], n, c.status), d = FASTAR_IDX(c.victims[tb + k - A], c.CAP, c.status);
      c.dest[tb + i] = d;
      if (dest_out) dest_out[static_cast<int64_t>(h) * n + i] = d;
    }
  } else {
    for (int i = tid; i < n; i += blockDim.x) {
      c.dest[tb + i] = -1;
      if (dest_out) dest_out[static_cast<int64_t>(h) * n + i] = -1;
    }
    if (tid == 0) record_status(c.status, kErrCapacity);
  }
  if (tid == 0) {
    PlanRec pr;
    pr.ok = ok;
    pr.n_matched = M;
    pr.n_seg = n_seg;
    pr.n_unmatched = U;
    pr.n_append = ok ? A : 0;
    pr.n_evict = ok ? E : 0;
    pr.len_old = L;
    pr.len_new = ok ? L + A : L;
    pr.evicted_tokens = evicted_tokens;
    pr.pages_granted = grant;
    pr.pad[0] = pr.pad[1] = 0;
    c.plan[h] = pr;
  }
}

// The three steps in one CTA per head, for caches and calls whose counters fit its shared memory: what each slot is matched by is
// counted there (16 bits a slot), the counter's old value is a token's rank in its group, and the groups' starts replace the counters,
// so that neither counts nor positions go through memory, nothing has to be cleared for them and two launches are saved.  A thread's
// tokens (i = tid, tid + 1024, ... up to K of them) stay in its registers.  Bound by the latencies of a few dependent steps of one CTA.
template <int K>
__global__ void __launch_bounds__(1024) plan_fused_kernel(const CacheView c, int n, float tau, const UpdateOut out) {
  chain_wait();
  extern __shared__ unsigned long long plan_s[];       // [CAP / 4] counters, then the victim sort buffer
  __shared__ int red[32];
  __shared__ int fresh_s[K * 32];                      // unmatched tokens of (pass, warp), then of those before
  const int h = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t tb = static_cast<int64_t>(h) * c.max_tokens, gb = static_cast<int64_t>(h) * (c.max_tokens + 1), ob = static_cast<int64_t>(h) * n;
  uint32_t* cnt = reinterpret_cast<uint32_t*>(plan_s); // slots 2 q and 2 q + 1
  unsigned long long* keys = plan_s + c.CAP / 4;
  const int L = c.len[h], now = *c.now;
  unsigned long long best[K];
#pragma unroll
  for (int k = 0; k < K; ++k) best[k] = k * 1024 + tid < n ? c.best[tb + k * 1024 + tid] : 0ull;
  for (int q = tid; q < (L + 15) / 16 * 2; q += 1024) reinterpret_cast<uint4*>(cnt)[q] = make_uint4(0, 0, 0, 0);
  __syncthreads();

  // a token's slot and its rank among the slot's tokens (below 2^14), or kFresh
  constexpr uint32_t kFresh = 0xFFFFFFFFu;
  uint32_t place[K];
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int i = k * 1024 + tid;
    int j = -1;
    float s = 0.f;
    if (best[k] != 0ull) {
      j = FASTAR_IDX(static_cast<int>(0xFFFFFFFFu - static_cast<uint32_t>(best[k] & 0xFFFFFFFFull)), c.CAP, c.status);
      s = ordered_to_float(static_cast<uint32_t>(best[k] >> 32));
    }
    const bool matched = j >= 0 && s >= tau;
    place[k] = kFresh;
    if (i < n) {
      c.sim[tb + i] = s;
      if (out.match) out.match[ob + i] = matched ? j : -1;
      if (out.sim) out.sim[ob + i] = s;
      if (matched) place[k] = static_cast<uint32_t>(j) | ((atomicAdd(cnt + (j >> 1), 1u << (16 * (j & 1))) >> (16 * (j & 1))) & 0xFFFFu) << 16;
    }
    const uint32_t m = __ballot_sync(0xffffffffu, i < n && !matched);
    if (lane == 0) fresh_s[k * 32 + warp] = __popc(m);
  }
  __syncthreads();
  int U;
  const int fresh_before = block_exscan(tid < K * 32 ? fresh_s[tid] : 0, red, &U);
  if (tid < K * 32) fresh_s[tid] = fresh_before;

  // Groups, 16 consecutive slots per thread and pass; a touched slot's counter becomes 2^15 + the start of its members.  The tables are
  // put together in shared memory (slot and start in one word, where the victims come later) and leave in order: a scattered 4-byte store
  // takes an SM a cycle per lane, and there is one SM per head.
  uint32_t* table = reinterpret_cast<uint32_t*>(keys);
  uint16_t* slot16 = reinterpret_cast<uint16_t*>(cnt);
  int n_seg = 0, M = 0;
  for (int j0 = 0; j0 < L; j0 += 16 * 1024) {
    const int j = j0 + 16 * tid;
    uint32_t w[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    if (j < L) {
      const uint4 a = reinterpret_cast<const uint4*>(cnt + j / 2)[0], b = reinterpret_cast<const uint4*>(cnt + j / 2)[1];
      w[0] = a.x; w[1] = a.y; w[2] = a.z; w[3] = a.w; w[4] = b.x; w[5] = b.y; w[6] = b.z; w[7] = b.w;
    }
    uint32_t touched = 0;
    int my_mem = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      touched |= ((w[q] & 0xFFFFu) != 0 ? 1u : 0u) << (2 * q) | (w[q] >> 16 != 0 ? 2u : 0u) << (2 * q);
      my_mem += (w[q] & 0xFFFFu) + (w[q] >> 16);
    }
    int tot;
    const int ex = block_exscan((__popc(touched) << 16) | my_mem, red, &tot);
    int seg = n_seg + (ex >> 16), mem = M + (ex & 0xFFFF);
    for (; touched; touched &= touched - 1) {            // a few of the sixteen
      const int slot = j + __ffs(touched) - 1;
      const int members = slot16[slot];
      table[seg++] = static_cast<uint32_t>(slot) | static_cast<uint32_t>(mem) << 16;
      slot16[slot] = static_cast<uint16_t>(0x8000 | mem);
      mem += members;
    }
    n_seg += tot >> 16;
    M += tot & 0xFFFF;
  }
  __syncthreads();
  for (int q = tid; q < n_seg; q += 1024) {
    const uint32_t e = table[q];
    c.segslot[tb + q] = e & 0xFFFFu;
    c.segpos[gb + q] = e >> 16;
  }
  if (tid == 0) c.segpos[gb + n_seg] = M;
  __syncthreads();

  const int room = c.CAP - L, A = min(U, room), E = U - A;
  int evicted_tokens = 0;
  bool ok = true;
  if (E > 0)
    ok = choose_victims(c, h, L, now, E, keys, red, evicted_tokens, [&](int j, bool (&free)[16]) {
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const uint32_t w = cnt[j / 2 + q];
        free[2 * q] = (w & 0xFFFFu) == 0;
        free[2 * q + 1] = w >> 16 == 0;
      }
    });
  __syncthreads();

  // members into their groups' ranges (through shared memory, as above); unmatched tokens, in token order, appended or into the victims'
  // slots
  uint16_t* members = reinterpret_cast<uint16_t*>(keys);
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int i = k * 1024 + tid;
    const bool fresh = i < n && place[k] == kFresh;
    const uint32_t m = __ballot_sync(0xffffffffu, fresh);
    int d = -1;
    if (fresh) {
      const int r = fresh_s[k * 32 + warp] + __popc(m & ((1u << lane) - 1u));
      c.ulist[tb + r] = i;
      if (ok) d = r < A ? L + r : FASTAR_IDX(c.victims[tb + r - A], c.CAP, c.status);
    } else if (i < n && ok) {
      const int j = place[k] & 0xFFFFu;
      d = j;
      members[FASTAR_IDX(static_cast<int>((slot16[j] & 0x7FFFu) + (place[k] >> 16)), n, c.status)] = static_cast<uint16_t>(i);
    }
    if (i < n) {
      c.dest[tb + i] = d;
      if (out.dest) out.dest[ob + i] = d;
    }
  }
  __syncthreads();
  if (ok)
    for (int q = tid; q < M; q += 1024) c.order[tb + q] = members[q];
  if (tid == 0) {
    if (!ok) record_status(c.status, kErrCapacity);
    PlanRec pr;
    pr.ok = ok ? 1 : 0;
    pr.n_matched = M;
    pr.n_seg = n_seg;
    pr.n_unmatched = U;
    pr.n_append = ok ? A : 0;
    pr.n_evict = ok ? E : 0;
    pr.len_old = L;
    pr.len_new = ok ? L + A : L;
    pr.evicted_tokens = evicted_tokens;
    pr.pages_granted = 0;
    pr.pad[0] = pr.pad[1] = 0;
    c.plan[h] = pr;
  }
}

__global__ void __launch_bounds__(256) scatter_kernel(const CacheView c, int n, int32_t* __restrict__ dest_out) {
  chain_wait();
  const int h = blockIdx.y;
  if (!c.plan[h].ok) return;
  const int64_t tb = static_cast<int64_t>(h) * c.max_tokens;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const int j = c.match[tb + i];
    if (j >= 0) {
      const int pos = FASTAR_IDX(atomicAdd(c.cur + static_cast<int64_t>(h) * c.CAP + FASTAR_IDX(j, c.CAP, c.status), 1), n, c.status);
      c.order[tb + pos] = i;
      c.dest[tb + i] = j;
      if (dest_out) dest_out[static_cast<int64_t>(h) * n + i] = j;
    }
  }
}

// ---------------------------------------------------------------------------------------------
// Query-probe correspondence (Section 5.2: the corresponding token of a query is the cached key with the highest
// attention score): the similarity kernel ranked the cached keys by <q_i, k_j>; the merge decision is taken on the
// key similarity, so the packed word of token i becomes (cos(k_i, k_j*), j*) with the cosine in the same fp32
// form as the cosine search (dot * 1/|k_i| * 1/|k_j*|).  Half a warp per token, one 128-bit load per lane and row.
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) probe_cosine_kernel(const CacheView c, const __nv_bfloat16* __restrict__ k_new, int n,
                                                           int64_t hs, int64_t ts) {
  chain_wait();
  const int64_t rows = static_cast<int64_t>(c.H) * n;
  const unsigned hmask = 0xFFFFu << (threadIdx.x & 16);
  for (int64_t q = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; (q >> 4) < rows;
       q += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int e8 = static_cast<int>(q & 15);
    const int64_t rowid = q >> 4;
    const int h = static_cast<int>(rowid / n), i = static_cast<int>(rowid % n);
    const int64_t tb = static_cast<int64_t>(h) * c.max_tokens;
    const unsigned long long b = c.best[tb + i];
    if (b == 0ull) continue;                         // empty cache: nothing was ranked (same for all 16 lanes)
    const int j = FASTAR_IDX(static_cast<int>(0xFFFFFFFFu - static_cast<uint32_t>(b & 0xFFFFFFFFull)), c.CAP, c.status);
    float dot = 0.f;
    if (e8 * 8 < c.D) {
      const uint4 a = *reinterpret_cast<const uint4*>(k_new + h * hs + i * ts + e8 * 8);
      const uint4 kk = *reinterpret_cast<const uint4*>(c.pool_k + slot_row_offset(c, c.page_table + static_cast<int64_t>(h) * c.CAPB, j) + e8 * 8);
      const __nv_bfloat162* pa = reinterpret_cast<const __nv_bfloat162*>(&a);
      const __nv_bfloat162* pk = reinterpret_cast<const __nv_bfloat162*>(&kk);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float2 fa = __bfloat1622float2(pa[e]), fk = __bfloat1622float2(pk[e]);
        dot = fmaf(fa.x, fk.x, dot);
        dot = fmaf(fa.y, fk.y, dot);
      }
    }
#pragma unroll
    for (int o = 8; o >= 1; o >>= 1) dot += __shfl_xor_sync(hmask, dot, o);
    if (e8 == 0) {
      const float cosv = dot * c.rnorm[static_cast<int64_t>(h) * c.CAP + j] * c.rnorm_new[tb + i];
      c.best[tb + i] = (static_cast<unsigned long long>(float_to_ordered(cosv)) << 32) | (b & 0xFFFFFFFFull);
    }
  }
}

int launch_probe_cosine(const CacheView& c, const __nv_bfloat16* k_new, int n, int64_t hs, int64_t ts, cudaStream_t st) {
  const int64_t total = static_cast<int64_t>(c.H) * n * 16;
  const int grid = static_cast<int>((total + 255) / 256 < 148 * 8 ? (total + 255) / 256 : 148 * 8);
  launch_chained(probe_cosine_kernel, grid, 256, 0, st, c, k_new, n, hs, ts);
  return cudaGetLastError() == cudaSuccess ? 1 : FASTAR_ERR_CUDA;
}

template <int K>
static int launch_plan_fused(const CacheView& c, int n, float tau, const UpdateOut& out, int smem, cudaStream_t st) {
  const int cfg = ensure_dynamic_smem(reinterpret_cast<const void*>(plan_fused_kernel<K>), smem);
  if (cfg != FASTAR_OK) return cfg;
  launch_chained(plan_fused_kernel<K>, c.H, 1024, smem, st, c, n, tau, out);
  return cudaGetLastError() == cudaSuccess ? 1 : FASTAR_ERR_CUDA;
}

bool plan_is_fused(const CacheView& c, int n) {
  return !c.pool_shared && n <= 8192 && c.CAP <= 65536 && plan_fused_smem(c, n) <= 220 * 1024;
}
int plan_fused_smem(const CacheView& c, int n) {
  int room = 1;                              // victims, up to a power of two
  while (room < n) room <<= 1;
  return c.CAP * 2 + room * 8;
}

int launch_plan(const CacheView& c, int n, float tau, const UpdateOut& out, cudaStream_t st) {
  if (plan_is_fused(c, n)) {
    const int smem = plan_fused_smem(c, n);
    switch ((n + 1023) / 1024) {             // every pass over the tokens counts (12 x 4680 with 8 for 5: 14.8 us, with 5 12.0; seven run as eight)
      case 1: return launch_plan_fused<1>(c, n, tau, out, smem, st);
      case 2: return launch_plan_fused<2>(c, n, tau, out, smem, st);
      case 3: return launch_plan_fused<3>(c, n, tau, out, smem, st);
      case 4: return launch_plan_fused<4>(c, n, tau, out, smem, st);
      case 5: return launch_plan_fused<5>(c, n, tau, out, smem, st);
      case 6: return launch_plan_fused<6>(c, n, tau, out, smem, st);
      default: return launch_plan_fused<8>(c, n, tau, out, smem, st);
    }
  }
  const int cfg = ensure_dynamic_smem(reinterpret_cast<const void*>(plan_kernel), 16384 * 8);
  if (cfg != FASTAR_OK) return cfg;
  const dim3 grid((n + 255) / 256, c.H);
  launch_chained(match_count_kernel, grid, 256, 0, st, c, n, tau, out);
  launch_chained(plan_kernel, c.H, 1024, 16384 * 8, st, c, n, out.dest);
  launch_chained(scatter_kernel, grid, 256, 0, st, c, n, out.dest);
  return cudaGetLastError() == cudaSuccess ? 3 : FASTAR_ERR_CUDA;
}

// ---------------------------------------------------------------------------------------------
// S2 (key side) + end of an update: bucket histogram of every key block, new lengths, stats, clock.
// ---------------------------------------------------------------------------------------------
// One CTA of 128 threads per block: a slot per thread, then 16 bytes of the histogram per thread.  A block's row is 2 KB of bf16 for
// at most 128 codes, so what bounds it is writing the rows (40 heads x 512 blocks: 42 MB, 6.4 us) and the CTAs' starts; with 2-byte
// stores by 256 threads 39 -> 29 us, 12 heads x 256 blocks 6.8 -> 5.5.
// It has every live slot in hand, so the bounds of a block's keys and multiplicities come from here: exact, and gone with the slot that set them.
// (Bounds of a head that only rise, where keys and counts are written, would keep it out of the attention's flat items long after the eviction of
// a key far longer than the rest, and m would be bounded by all that ever matched.)  12 heads x 256 blocks 5.8 -> 6.3 us, 40 x 512 30 -> 35, of
// which the hash and the commit, which raised them, have lost 1.1 and 7; by atomics into one place per head it took 7.3 to 50.
// A key without a reciprocal norm: |k|^2 is zero (or below the smallest float), infinite or no number.
__device__ __forceinline__ bool key_is_zero(const __nv_bfloat16* k, int D) {
  float sq = 0.f;
#pragma unroll 1
  for (int e = 0; e < D; e += 8) sq = square_sum8(*reinterpret_cast<const uint4*>(k + e), sq);
  return sq <= 0.f;
}
__global__ void __launch_bounds__(128, 16) key_hist_kernel(const CacheView c, int use_plan, fastar_update_stats* stats_out,
                                                       int advance_clock) {
  chain_wait();
  extern __shared__ __align__(16) int hist[];          // hist_cols counters, a multiple of 64
  __shared__ uint3 bound_s[4];
  const int b = blockIdx.x, h = blockIdx.y;
  const int L = use_plan ? c.plan[h].len_new : c.len[h];
  for (int q = threadIdx.x; q < c.hist_cols / 4; q += blockDim.x) reinterpret_cast<int4*>(hist)[q] = make_int4(0, 0, 0, 0);
  __syncthreads();
  const int s0 = b * c.PT, s1 = min(L, s0 + c.PT);
  const int nb = 1 << c.B;
  float norm = 0.f, log2m = 0.f, joint = 0.f;          // the largest of the slots
  // weighted histograms (a selector option): a slot counts m times, as its merged tokens would; an entry saturates
  // at 65535 and is stored as two 8-bit digits, each exact in bf16, that S3 contracts separately
  for (int s = s0 + threadIdx.x; s < s1; s += blockDim.x) {
    const int64_t q = static_cast<int64_t>(h) * c.CAP + s;
    const uint32_t code = c.kcode[q];
    const float rn = c.rnorm[q];
    const int wgt = c.hist_weighted ? min(c.count[q], 65535) : 1;
    const float lm = c.log2m[q];
    float x = __fdividef(1.f, rn);
    if (rn == 0.f && key_is_zero(c.pool_k + slot_row_offset(c, c.page_table + static_cast<int64_t>(h) * c.CAPB, s), c.D)) x = 0.f;
    norm = fmaxf(norm, x);
    log2m = fmaxf(log2m, lm);
    joint = fmaxf(joint, fmaf(kJoint, x, lm));
    for (int t = 0; t < c.T; ++t) atomicAdd(&hist[t * nb + ((code >> (8 * t)) & 0xFFu)], wgt);
  }
  // (none is negative, so their words are in the floats' order)
  const uint32_t norm_w = __reduce_max_sync(0xffffffffu, __float_as_uint(norm)), log2m_w = __reduce_max_sync(0xffffffffu, __float_as_uint(log2m));
  const uint32_t joint_w = __reduce_max_sync(0xffffffffu, __float_as_uint(joint));
  if ((threadIdx.x & 31) == 0) bound_s[threadIdx.x >> 5] = make_uint3(norm_w, log2m_w, joint_w);
  __syncthreads();
  if (threadIdx.x == 0) {
    uint3 w = bound_s[0];
#pragma unroll
    for (int i = 1; i < 4; ++i) w = make_uint3(max(w.x, bound_s[i].x), max(w.y, bound_s[i].y), max(w.z, bound_s[i].z));
    c.bound[static_cast<int64_t>(h) * c.CAPB + b] = BlockBound{__uint_as_float(w.x), __uint_as_float(w.y), __uint_as_float(w.z), 0.f};
  }
  const int64_t ho = (static_cast<int64_t>(h) * c.CAPB + b) * c.hist_cols;
  for (int q = threadIdx.x; q < c.hist_cols / 8; q += blockDim.x) {
    int v[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = hist[8 * q + e];
    if (c.hist_weighted) {
#pragma unroll
      for (int e = 0; e < 8; ++e) v[e] = min(max(v[e], 0), 65535);       // max: a sum of saturated weights could wrap
      reinterpret_cast<uint4*>(c.hk_hi + ho)[q] = pack_counts<8>(v);
    }
    reinterpret_cast<uint4*>(c.hk + ho)[q] = c.hist_weighted ? pack_counts<0>(v) : pack_counts<-1>(v);
  }
  if (b == 0 && threadIdx.x == 0 && use_plan) {
    const PlanRec pr = c.plan[h];
    c.len[h] = pr.len_new;
    if (c.pool_shared && pr.pages_granted > 0) atomicAdd(c.next_free, pr.pages_granted);
    if (stats_out) {
      fastar_update_stats s;
      s.matched = pr.n_matched;
      s.touched = pr.n_seg;
      s.appended = pr.n_append;
      s.evicted_slots = pr.n_evict;
      s.evicted_tokens = pr.evicted_tokens;
      s.length = pr.len_new;
      s.ok = pr.ok;
      s.pages_granted = pr.pages_granted;
      stats_out[h] = s;
    }
    if (h == 0 && advance_clock) *c.now = *c.now + 1;
  }
}
int launch_finalize_hist(const CacheView& c, fastar_update_stats* stats_out, int advance_clock, cudaStream_t st) {
  launch_chained(key_hist_kernel, dim3(c.CAPB, c.H), 128, c.hist_cols * 4, st, c, advance_clock >= 0 ? 1 : 0, stats_out,
                                                                  advance_clock > 0 ? 1 : 0);
  return cudaGetLastError() == cudaSuccess ? 1 : FASTAR_ERR_CUDA;
}

// ---------------------------------------------------------------------------------------------
// An un-cached segment of an attention call: the biases of its rows, and what |k|^2 of its keys does not exceed, by kSegParts parts of the
// tokens of a head, which the attention puts together (so there is nothing to clear and no atomic).  Half a warp (a quarter at d = 64) has a row.
// The parts are CTAs of 64 threads, on the SMs that the block top-k leaves idle where there is one (12 heads x 4680 tokens, with the top-k 3.9 + 8.5 -> 9.0 us).
// ---------------------------------------------------------------------------------------------
template <int D>
__device__ __forceinline__ void segment_part(const CacheView& c, const SegArgs& s, int h, int part) {
  constexpr int LPR = D / 8, RPW = 32 / LPR, B = 4;    // lanes a row, rows a warp, rows of a thread that are under way
  __shared__ uint32_t bound;
  if (threadIdx.x == 0) bound = 0u;
  __syncthreads();
  const int sl = threadIdx.x % LPR, rpc = blockDim.x / LPR;
  for (int i = (h * kSegParts + part) * blockDim.x + threadIdx.x; i < s.total; i += c.H * kSegParts * blockDim.x) c.seg_bias[i] = i < s.ns ? 0.f : -INFINITY;
  const int r0 = static_cast<int>(static_cast<int64_t>(s.ns) * part / kSegParts), r1 = static_cast<int>(static_cast<int64_t>(s.ns) * (part + 1) / kSegParts);
  uint32_t most = 0;
  for (int rb = r0 + (threadIdx.x >> 5) * RPW; rb < r1; rb += B * rpc) {
    uint4 kr[B];
#pragma unroll
    for (int b = 0; b < B; ++b) {                      // past the end the last row again
      const int row = min(rb + b * rpc + static_cast<int>(threadIdx.x & 31) / LPR, r1 - 1);
      kr[b] = *reinterpret_cast<const uint4*>(s.k + h * s.hs + row * s.ts + sl * 8);
    }
#pragma unroll
    for (int b = 0; b < B; ++b) {
      float sq = square_sum8(kr[b], 0.f);
#pragma unroll
      for (int o = LPR / 2; o >= 1; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
      most = max(most, __float_as_uint(sq));
    }
  }
  most = __reduce_max_sync(0xffffffffu, most);
  if ((threadIdx.x & 31) == 0) atomicMax(&bound, most);
  __syncthreads();
  if (threadIdx.x == 0) c.seg_bound[h * kSegParts + part] = bound;
}
template <int D>
__global__ void __launch_bounds__(64) segment_kernel(const CacheView c, const SegArgs s) {
  chain_wait();
  segment_part<D>(c, s, blockIdx.y, blockIdx.x);
}
int launch_segment(const CacheView& c, const SegArgs& s, cudaStream_t st) {
  const dim3 grid(kSegParts, c.H);
  if (c.D == 128) launch_chained(segment_kernel<128>, grid, 64, 0, st, c, s);
  else launch_chained(segment_kernel<64>, grid, 64, 0, st, c, s);
  return cudaGetLastError() == cudaSuccess ? 1 : FASTAR_ERR_CUDA;
}

constexpr int kTopkWarps = 2;      // rows per CTA: few, so that a few hundred rows spread over all SMs
template <bool PROMPT, int NV>
__global__ void __launch_bounds__(32 * kTopkWarps) topk_kernel(const TopkArgs a) {
  chain_wait();
  const int row = blockIdx.x * kTopkWarps + (threadIdx.x >> 5);
  if (row < a.rows) topk_row<PROMPT, NV>(a, blockIdx.y, row);
}
// The same with the parts of a segment behind the rows' CTAs.
template <int NV, int D>
__global__ void __launch_bounds__(32 * kTopkWarps) topk_segment_kernel(const TopkArgs a, const CacheView c, const SegArgs s) {
  chain_wait();
  const int ctas = (a.rows + kTopkWarps - 1) / kTopkWarps, row = blockIdx.x * kTopkWarps + (threadIdx.x >> 5);
  if (static_cast<int>(blockIdx.x) >= ctas) segment_part<D>(c, s, blockIdx.y, blockIdx.x - ctas);
  else if (row < a.rows) topk_row<false, NV>(a, blockIdx.y, row);
}

template <bool PROMPT>
static int launch_topk(const TopkArgs& a, int columns, const CacheView& c, const SegArgs* seg, cudaStream_t st) {
  const int ctas = (a.rows + kTopkWarps - 1) / kTopkWarps, threads = 32 * kTopkWarps;
  auto launch = [&](auto width) {
    constexpr int NV = decltype(width)::value;
    if (PROMPT || !seg) launch_chained(topk_kernel<PROMPT, NV>, dim3(ctas, c.H), threads, 0, st, a);
    else if (c.D == 128) launch_chained(topk_segment_kernel<NV, 128>, dim3(ctas + kSegParts, c.H), threads, 0, st, a, c, *seg);
    else launch_chained(topk_segment_kernel<NV, 64>, dim3(ctas + kSegParts, c.H), threads, 0, st, a, c, *seg);
  };
  if (columns <= 128) launch(std::integral_constant<int, 4>{});
  else if (columns <= 256) launch(std::integral_constant<int, 8>{});
  else if (columns <= 512) launch(std::integral_constant<int, 16>{});
  else if (columns <= 1152) launch(std::integral_constant<int, 36>{});
  else if (columns <= 2048) launch(std::integral_constant<int, 64>{});
  else return FASTAR_ERR_UNSUPPORTED_SHAPE;          // the entry points refuse such rows
  return cudaGetLastError() == cudaSuccess ? 1 : FASTAR_ERR_CUDA;
}

TopkArgs block_topk_args(const CacheView& c, int nqb, int keep, int force_sink, int force_recent) {
  TopkArgs a{};
  a.src = c.scores;
  a.src_hi = c.hist_weighted ? c.scores_hi : nullptr;
  a.src_head_stride = a.out_head_stride = static_cast<int64_t>(c.max_qb) * c.CAPB;
  a.src_row_stride = a.out_row_stride = c.CAPB;
  a.rows = nqb;
  a.len = c.len;
  a.len_div = c.PT;
  a.keep = keep;
  a.out = c.sel;
  a.out_fill = min(keep, c.CAPB);
  a.nsel = c.nsel;
  a.force_first = force_sink;
  a.force_last = force_recent;
  a.status = c.status;
  return a;
}
int launch_topk_blocks(const CacheView& c, int nqb, int keep, int force_sink, int force_recent, const SegArgs* seg, cudaStream_t st) {
  return launch_topk<false>(block_topk_args(c, nqb, keep, force_sink, force_recent), c.CAPB, c, seg, st);
}
// ---------------------------------------------------------------------------------------------
// AnnCA with the LSH bucket rule (Section 5.3): a prompt token is kept for a frame iff, in at least one table, a
// query of the frame falls into its bucket.  One CTA per (frame, head): the buckets the frame's queries occupy are
// marked in a T x 256 bit map in shared memory, every prompt token tests its T buckets, and the kept tokens are
// written in ascending order (block scan) with their count.
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) bucket_select_kernel(const CacheView c, int nq, int frame_len, int np) {
  chain_wait();
  __shared__ uint32_t marks[4 * 8];
  __shared__ int red[32];
  const int f = blockIdx.x, h = blockIdx.y, tid = threadIdx.x;
  if (tid < 32) marks[tid] = 0u;
  __syncthreads();
  const uint32_t* qc = c.code_q_ca + static_cast<int64_t>(h) * c.max_tokens;
  const int i1 = min(nq, (f + 1) * frame_len);
  for (int i = f * frame_len + tid; i < i1; i += blockDim.x) {
    const uint32_t code = qc[i];
    for (int t = 0; t < c.T; ++t) {
      const uint32_t w = (code >> (8 * t)) & 0xFFu;
      atomicOr(&marks[t * 8 + (w >> 5)], 1u << (w & 31u));
    }
  }
  __syncthreads();
  const uint32_t* pc = c.code_p_ca + static_cast<int64_t>(h) * c.max_prompt;
  int32_t* out = c.selp + (static_cast<int64_t>(h) * c.max_frames + f) * c.max_prompt;
  int run = 0;
  for (int p0 = 0; p0 < np; p0 += blockDim.x) {
    const int p = p0 + tid;
    int take = 0;
    if (p < np) {
      const uint32_t code = pc[p];
      for (int t = 0; t < c.T; ++t) {
        const uint32_t w = (code >> (8 * t)) & 0xFFu;
        take |= static_cast<int>((marks[t * 8 + (w >> 5)] >> (w & 31u)) & 1u);
      }
    }
    int tot;
    const int pos = run + block_exscan(take, red, &tot);
    if (take) out[pos] = p;
    run += tot;
  }
  if (tid == 0) c.nselp[static_cast<int64_t>(h) * c.max_frames + f] = run;
}

int launch_bucket_select(const CacheView& c, int nq, int frame_len, int n_frames, int np, cudaStream_t st) {
  launch_chained(bucket_select_kernel, dim3(n_frames, c.H), 256, 0, st, c, nq, frame_len, np);
  return cudaGetLastError() == cudaSuccess ? 1 : FASTAR_ERR_CUDA;
}

TopkArgs prompt_topk_args(const CacheView& c, int n_frames, int np, int keep) {
  TopkArgs a{};
  a.src = c.rel;
  a.src_head_stride = a.out_head_stride = static_cast<int64_t>(c.max_frames) * c.max_prompt;
  a.src_row_stride = a.out_row_stride = c.max_prompt;
  a.rows = n_frames;
  a.n_fixed = np;
  a.keep = keep;
  a.out = c.selp;
  a.out_fill = min(keep, np);
  a.status = c.status;
  return a;
}
int launch_topk_prompt(const CacheView& c, int n_frames, int np, int keep, cudaStream_t st) {
  return launch_topk<true>(prompt_topk_args(c, n_frames, np, keep), np, c, nullptr, st);
}

// ---------------------------------------------------------------------------------------------
// reset / import helpers, output decoding
// ---------------------------------------------------------------------------------------------
__global__ void reset_meta_kernel(const CacheView c) {
  const int64_t total = static_cast<int64_t>(c.H) * c.CAP;
  for (int64_t q = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; q < total;
       q += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    c.count[q] = 0;
    c.stamp[q] = 0;
    c.log2m[q] = -INFINITY;
    c.rnorm[q] = 0.f;
    c.kcode[q] = 0;
    // one full set of pages per head: the identity; a shared pool: no page handed out yet (entries of pages a head
    // does not hold stay at page 0, a valid address that only masked-out slots ever read)
    if (q < static_cast<int64_t>(c.H) * c.CAPB) c.bound[q] = BlockBound{};
    if (q < static_cast<int64_t>(c.H) * c.CAPB) c.page_table[q] = c.pool_shared ? 0 : static_cast<int32_t>(q);
    if (q < c.H) c.len[q] = 0;
    if (q == 0) { *c.now = 0; *c.status = 0; *c.next_free = 0; }
  }
}
int launch_reset(const CacheView& c, cudaStream_t st) {
  const size_t pool = static_cast<size_t>(c.pool_pages) * c.PT * c.D * sizeof(__nv_bfloat16);
  if (cudaMemsetAsync(c.pool_k, 0, pool, st) != cudaSuccess) return FASTAR_ERR_CUDA;
  if (cudaMemsetAsync(c.pool_v, 0, pool, st) != cudaSuccess) return FASTAR_ERR_CUDA;
  if (cudaMemsetAsync(c.hk, 0, static_cast<size_t>(c.H) * c.CAPB * c.hist_cols * 2, st) != cudaSuccess) return FASTAR_ERR_CUDA;
  if (c.pool_k8 && cudaMemsetAsync(c.pool_k8, 0, static_cast<size_t>(c.pool_pages) * c.PT * 128, st) != cudaSuccess) return FASTAR_ERR_CUDA;
  reset_meta_kernel<<<296, 256, 0, st>>>(c);
  return cudaGetLastError() == cudaSuccess ? 1 : FASTAR_ERR_CUDA;
}

// after an import: clear dead slots, derive log2 m, keep counts of dead slots at 0
template <int D>
__global__ void import_fix_kernel(const CacheView c) {
  const int h = blockIdx.y;
  const int L = c.len[h];
  const int lane = threadIdx.x & 31;
  const int32_t* pt_h = c.page_table + static_cast<int64_t>(h) * c.CAPB;
  for (int s = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); s < c.CAP; s += gridDim.x * (blockDim.x >> 5)) {
    const int64_t q = static_cast<int64_t>(h) * c.CAP + s;
    if (s >= L) {
      const int64_t ro = slot_row_offset(c, pt_h, s);
      for (int e = lane * 2; e < D; e += 64) {
        *reinterpret_cast<uint32_t*>(c.pool_k + ro + e) = 0u;
        *reinterpret_cast<uint32_t*>(c.pool_v + ro + e) = 0u;
      }
      if (lane == 0) { c.count[q] = 0; c.stamp[q] = 0; c.log2m[q] = -INFINITY; c.rnorm[q] = 0.f; c.kcode[q] = 0; }
    } else if (lane == 0) {
      c.log2m[q] = log2f(static_cast<float>(max(1, c.count[q])));
    }
  }
}
int launch_import_derive(const CacheView& c, cudaStream_t st) {
  // codes and reciprocal norms of every slot (the pools are [H][CAP][D] under the identity page table)
  int r = launch_prep_generic(c, c.pool_k, c.CAP, static_cast<int64_t>(c.CAP) * c.D, c.D, c.kcode, c.rnorm, c.CAP, st);
  if (r < 0) return r;
  const dim3 grid(min((c.CAP + 7) / 8, 1024), c.H);
  if (c.D == 128) import_fix_kernel<128><<<grid, 256, 0, st>>>(c);
  else import_fix_kernel<64><<<grid, 256, 0, st>>>(c);
  if (cudaGetLastError() != cudaSuccess) return FASTAR_ERR_CUDA;
  int r3 = 0;
  if (c.pool_k8) {                                   // search codes of every slot from the imported keys
    r3 = c.sign_codes ? launch_sign_rows(c, c.kcode, c.CAP, c.CAP, c.pool_k8, c.CAP, st)
                      : launch_quantize_keys(c, c.pool_k, c.CAP, static_cast<int64_t>(c.CAP) * c.D, c.D, c.rnorm, c.CAP, c.pool_k8,
                                             c.CAP, st);
    if (r3 < 0) return r3;
  }
  int r2 = launch_finalize_hist(c, nullptr, -1, st);
  if (r2 < 0) return r2;
  return r + 1 + r2 + r3;
}

// ---------------------------------------------------------------------------------------------
// Self-test of the bounded waits: warp 0 waits on a barrier that never completes and gives up after `limit_ns`
// (status word <- time-out, abort flag set); warp 1 waits on a second dead barrier with the full limit and must be
// released by the abort flag.  `released` receives 1 when it was.  Nothing is in flight, so the CTA simply returns.
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(64) bounded_wait_selftest_kernel(int* status, unsigned long long limit_ns, int* released) {
  __shared__ __align__(8) unsigned long long bars[2];
  __shared__ int abort_word;
  volatile int* abort_flag = &abort_word;
  if (threadIdx.x == 0) {
    mbar_init(smem_u32(&bars[0]), 1);
    mbar_init(smem_u32(&bars[1]), 1);
    abort_word = 0;
    fence_mbar_init();
  }
  __syncthreads();
  const int warp = threadIdx.x >> 5;
  if (warp == 0) {
    const bool ok = mbar_wait(smem_u32(&bars[0]), 0, abort_flag, status, limit_ns);
    if (ok && threadIdx.x == 0) record_status(status, FASTAR_ERR_CUDA);      // cannot happen: nobody arrives
  } else {
    const bool ok = mbar_wait(smem_u32(&bars[1]), 0, abort_flag, nullptr);
    if (threadIdx.x == 32) *released = ok ? 0 : 1;
  }
}
int launch_bounded_wait_selftest(const CacheView& c, int limit_us, int* released, cudaStream_t st) {
  bounded_wait_selftest_kernel<<<1, 64, 0, st>>>(c.status, static_cast<unsigned long long>(limit_us) * 1000ull, released);
  return cudaGetLastError() == cudaSuccess ? 1 : FASTAR_ERR_CUDA;
}

__global__ void decode_rel_kernel(const CacheView c, int n_frames, int np, float scale, float* __restrict__ rel_out) {
  chain_wait();
  const int h = blockIdx.y;
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < n_frames * np; q += gridDim.x * blockDim.x) {
    const int f = q / np, p = q % np;
    rel_out[(static_cast<int64_t>(h) * n_frames + f) * np + p] =
        ordered_to_float(c.rel[(static_cast<int64_t>(h) * c.max_frames + f) * c.max_prompt + p]) * scale;
  }
}
int launch_decode_rel(const CacheView& c, int n_frames, int np, float scale, float* rel_out, cudaStream_t st) {
  launch_chained(decode_rel_kernel, dim3((n_frames * np + 255) / 256, c.H), 256, 0, st, c, n_frames, np, scale, rel_out);
  return cudaGetLastError() == cudaSuccess ? 1 : FASTAR_ERR_CUDA;
}

}  // namespace fastar
