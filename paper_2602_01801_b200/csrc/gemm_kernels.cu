// S3: bucket-collision scores HQ x HK^T (AnnSA block selection, Sections 5.1 / 5.4) on tcgen05 / TMEM / TMA.
//
// One CTA = one 128-row tile of HQ and a range of 64-row tiles of HK; D[128 x 64] fp32 lives in TMEM, double buffered so the
// epilogue of tile t overlaps the MMAs of tile t+1.  The product is small (37 x 220 x 1024 for a 12-head layer's head), so it is
// bound by the latency of sixteen dependent 64-column steps, and by how many SMs take part: 64 keys a tile and two CTAs per SM
// (128 keys and one CTA before: 10.9 -> 7.7 us; 32 x 1056 x 1024 of 8 heads 13.4 -> 9.4; 85 x 507 of 40 heads 35 -> 24).
// Warp roles: warps 0-7 epilogue (two threads per row / TMEM lane, one per 32-column half), warp 8 TMA
// producer, warp 9 TMEM allocation + MMA issue.  Operands are bf16, K-major, 128-byte swizzled.
#include "common.h"
#include "ptx.cuh"
#include "topk.cuh"


namespace fastar {

struct GemmArgs {
  int rows_a;              // valid rows of HQ per head (nqb)
  int nkc;                 // K chunks of 64
  TopkArgs top;            // RANK: the ranking of the rows
};

constexpr int kChunkBytes = 128 * 128;       // 128 rows x 64 bf16
constexpr int kTileN = 64;                   // rows of HK per tile
constexpr int kTmemCols = 2 * kTileN;
constexpr int kGemmThreads = 320;            // warps 0-7 epilogue, 8 TMA producer, 9 MMA issue
constexpr int kGemmProducerWarp = 8, kGemmMmaWarp = 9;

// Ring stages of a chunk of both operands.  A CTA's sixteen chunks are a chain of loads, so a grid of one CTA per SM at most takes all the
// shared memory for its ring: two round trips to L2 instead of four (48 CTAs 8.0 -> 7.5 us, 128 9.4 -> 8.3, 24 7.3 -> 6.85, 6 7.6 -> 7.45).  A
// larger grid has two CTAs per SM, each with half of the loads under way, and a few CTAs find L2 idle: they are slower with the long ring (four
// 6.4 -> 6.85, one that ranks 8.4 -> 8.7).
constexpr int kFewStages = 4, kManyStages = 9;
template <int NST>
struct GemmSmem {
  static constexpr int stage_bytes = kChunkBytes + kTileN * 128;
  static constexpr int bar_off = NST * stage_bytes;
  static constexpr int total = bar_off + 256;
};

// RANK: a head's key blocks fit one tile and its query blocks are few, so the CTA has whole rows and ranks them too (a launch less: 2 heads,
// 5 x 10 blocks 6.4 + 2.5 -> 7.8 us).
template <bool RANK, int NST>
__global__ void __launch_bounds__(kGemmThreads, 2)
gemm_kernel(const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_b, const CacheView c,
            const GemmArgs g) {
  using SM = GemmSmem<NST>;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const uint32_t sbase = smem_u32(smem_raw);
  uint8_t* sgen = smem_raw;
  if (sbase & 1023u) {                  // swizzled tiles need 1024-byte alignment; uniform for the CTA
    if (threadIdx.x == 0) record_status(c.status, FASTAR_ERR_CUDA);
    return;
  }
  const uint32_t ring_s = sbase;
  const uint32_t bar_s = sbase + SM::bar_off;
  // barrier slots (8 bytes each)
  const uint32_t bar_full = bar_s;                   // [NST]
  const uint32_t bar_empty = bar_s + 8 * NST;        // [NST]
  const uint32_t bar_tfull = bar_s + 16 * NST;       // [2]
  const uint32_t bar_tempty = bar_tfull + 16;        // [2]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(sgen + SM::bar_off + 16 * NST + 32);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(sgen + SM::bar_off + 16 * NST + 36);
  static_assert(16 * NST + 40 <= 256, "barrier area");

  const int warp = warp_index(), lane = threadIdx.x & 31;
  const int h = blockIdx.y;
  const int m0 = blockIdx.x * 128;
  if (threadIdx.x == 0) {
    for (int s = 0; s < NST; ++s) {
      mbar_init(bar_full + 8 * s, 1);
      mbar_init(bar_empty + 8 * s, 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(bar_tfull + 8 * b, 1);
      mbar_init(bar_tempty + 8 * b, 8);          // one arrival per epilogue warp
    }
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == kGemmProducerWarp && lane == 0) {
    tma_prefetch_desc(&tm_a);
    tma_prefetch_desc(&tm_b);
  }
  __syncthreads();
  if (warp == kGemmMmaWarp) {
    tmem_alloc(smem_u32(tmem_slot), kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  chain_wait();

  // ---- tile range of this CTA ----------------------------------------------------------------
  const int n_tiles = (((__shfl_sync(0xffffffffu, c.len[h], 0) + c.PT - 1) / c.PT) + kTileN - 1) / kTileN;
  const int per = (n_tiles + gridDim.z - 1) / gridDim.z;
  const int t0 = blockIdx.z * per;
  const int ntl = max(0, min(n_tiles, t0 + per) - t0);
  const int nkc = g.nkc;

  if (ntl > 0) {
    if (warp == kGemmProducerWarp) {
      // ------------------------------------------------------------------ TMA producer
      bool ok = true;
      int it = 0;
      if (lane == 0) {
        for (int tl = 0; tl < ntl && ok; ++tl) {
          const int t = t0 + tl;
          for (int kc = 0; kc < nkc; ++kc, ++it) {
            const int s = it % NST;
            const uint32_t ph = (it / NST) & 1;
            ok = mbar_wait<kIssueWaitHintNs>(bar_empty + 8 * s, ph ^ 1, abort_flag, c.status);
            if (!ok) break;
            const uint32_t st_s = ring_s + s * SM::stage_bytes;
            mbar_arrive_expect_tx(bar_full + 8 * s, SM::stage_bytes);
            tma_load_3d(st_s, &tm_a, bar_full + 8 * s, kc * 64, m0, h);
            tma_load_3d(st_s + kChunkBytes, &tm_b, bar_full + 8 * s, kc * 64, t * kTileN, h);
          }
        }
      }
      // drain: let the loads still in flight land before the CTA may exit.  Full barriers are consumed by the
      // MMA warp in order; waiting on the last ones is enough and cheap.  Bounded like every other wait.
      if (lane == 0)
        for (int k = max(0, it - NST); k < it; ++k) mbar_wait<kIssueWaitHintNs>(bar_full + 8 * (k % NST), (k / NST) & 1, abort_flag, c.status);
    } else if (warp == kGemmMmaWarp) {
      // ------------------------------------------------------------------ MMA issue
      {
        const uint32_t lead = elect_lane();
        constexpr uint32_t idesc = make_idesc_bf16(128, kTileN, 0);
        bool ok = true;
        int it = 0;
        for (int tl = 0; tl < ntl && ok; ++tl) {
          const int buf = tl & 1, bph = (tl >> 1) & 1;
          ok = mbar_wait_warp<kIssueWaitHintNs>(bar_tempty + 8 * buf, bph ^ 1, abort_flag, c.status);
          if (!ok) break;
          tc_fence_after();
          const uint32_t d_t = tmem + buf * kTileN;
          for (int kc = 0; kc < nkc; ++kc, ++it) {
            const int s = it % NST;
            ok = mbar_wait_warp<kIssueWaitHintNs>(bar_full + 8 * s, (it / NST) & 1, abort_flag, c.status);
            if (!ok) break;
            tc_fence_after();
            const uint32_t st_s = ring_s + s * SM::stage_bytes;
#pragma unroll
            for (int k4 = 0; k4 < 4; ++k4) {
              const uint64_t ad = make_smem_desc(st_s + k4 * 32, 16, 1024);
              const uint64_t bd = make_smem_desc(st_s + kChunkBytes + k4 * 32, 16, 1024);
              umma_ss(d_t, ad, bd, idesc, (kc | k4) != 0, lead);
            }
            umma_commit(bar_empty + 8 * s, lead);
          }
          if (ok) umma_commit(bar_tfull + 8 * buf, lead);
        }
      }
    } else {
      // ------------------------------------------------------------------ epilogue (256 threads)
      const int wg = warp >> 2;
      const int r = (warp & 3) * 32 + lane;         // A row inside the tile = TMEM lane
      const int row = m0 + r;
      const uint32_t lane_addr = static_cast<uint32_t>((warp & 3) * 32) << 16;
      bool ok = true;
      for (int tl = 0; tl < ntl && ok; ++tl) {
        const int t = t0 + tl;
        const int buf = tl & 1, bph = (tl >> 1) & 1;
        ok = __all_sync(0xffffffffu, mbar_wait(bar_tfull + 8 * buf, bph, abort_flag, c.status));
        if (!ok) break;                              // warp-uniform: TMEM loads are warp-collective
        tc_fence_after();
        uint32_t v[32];
        tmem_ld32(tmem + lane_addr + buf * kTileN + wg * 32, v);
        tmem_wait_ld();
        tc_fence_before();
        mbar_arrive_warp(bar_tempty + 8 * buf);      // the scores are in registers: release the accumulator
        if (row < g.rows_a) {
          const int col = t * kTileN + wg * 32;
          float* dst = c.scores + (static_cast<int64_t>(h) * c.max_qb + row) * c.CAPB + col;
          if ((c.CAPB & 3) == 0) {                   // rows start on 16-byte boundaries
#pragma unroll
            for (int j = 0; j < 32; j += 4)
              if (col + j < c.CAPB)
                *reinterpret_cast<float4*>(dst + j) = make_float4(__uint_as_float(v[j]), __uint_as_float(v[j + 1]), __uint_as_float(v[j + 2]), __uint_as_float(v[j + 3]));
          } else {
#pragma unroll
            for (int j = 0; j < 32; ++j)
              if (col + j < c.CAPB) dst[j] = __uint_as_float(v[j]);
          }
        }
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == kGemmMmaWarp) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
  if (RANK)
    for (int row = warp; row < g.rows_a; row += kGemmThreads / 32) topk_row<false, kTileN / 32>(g.top, h, row);
}

template <bool RANK, int NST>
static int launch_gemm_t(const CacheView& c, const CUtensorMap& tm_hq, const CUtensorMap& tm_hk, const GemmArgs& g, dim3 grid, cudaStream_t st) {
  const int cfg = ensure_dynamic_smem(reinterpret_cast<const void*>(gemm_kernel<RANK, NST>), GemmSmem<NST>::total);
  if (cfg != FASTAR_OK) return cfg;
  launch_chained(gemm_kernel<RANK, NST>, grid, kGemmThreads, GemmSmem<NST>::total, st, tm_hq, tm_hk, c, g);
  return cudaGetLastError() == cudaSuccess ? 1 : FASTAR_ERR_CUDA;
}
template <bool RANK>
static int launch_gemm(const CacheView& c, const CUtensorMap& tm_hq, const CUtensorMap& tm_hk, const GemmArgs& g, cudaStream_t st) {
  int dev = 0, sm_count = 148;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sm_count, cudaDevAttrMultiProcessorCount, dev);
  const dim3 grid((g.rows_a + 127) / 128, c.H, (c.CAPB + kTileN - 1) / kTileN);
  const int64_t ctas = static_cast<int64_t>(grid.x) * grid.y * grid.z;
  if constexpr (!RANK)
    if (ctas >= 6 && ctas <= sm_count) return launch_gemm_t<RANK, kManyStages>(c, tm_hq, tm_hk, g, grid, st);
  return launch_gemm_t<RANK, kFewStages>(c, tm_hq, tm_hk, g, grid, st);
}

int launch_s3_scores(const CacheView& c, const CUtensorMap& tm_hq, const CUtensorMap& tm_hk, int nqb, cudaStream_t st) {
  GemmArgs g{};
  g.rows_a = nqb;
  g.nkc = c.hist_cols / 64;
  return launch_gemm<false>(c, tm_hq, tm_hk, g, st);
}

// Scores and the kept blocks.  One launch where a head's blocks fit one tile and a warp has two rows at most; more rows would wait for one
// another in the few CTAs (a row is 1.5 us), and weighted histograms have two products to rank.
int launch_s3_topk(const CacheView& c, const CUtensorMap& tm_hq, const CUtensorMap& tm_hk, int nqb, int keep, int force_sink, int force_recent,
                   cudaStream_t st) {
  GemmArgs g{};
  g.rows_a = nqb;
  g.nkc = c.hist_cols / 64;
  g.top = block_topk_args(c, nqb, keep, force_sink, force_recent);
  return launch_gemm<true>(c, tm_hq, tm_hk, g, st);
}
bool s3_ranks(const CacheView& c, int nqb) { return c.CAPB <= kTileN && nqb <= 2 * (kGemmThreads / 32) && !c.hist_weighted; }

}  // namespace fastar
