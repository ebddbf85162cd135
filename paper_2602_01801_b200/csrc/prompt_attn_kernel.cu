// C3 for up to 64 kept prompt tokens per frame (AnnCA, Section 5.3): out = soft-max(q k^T / sqrt(d)) v over the kept tokens.
//
// One key tile, so there is no running maximum and nothing to rescale, and all query tiles of a (head, frame) attend to the same
// rows: a CTA gathers the kept K and V rows once and streams 128-row query tiles past them.  The (head, frame, query tile) units lie
// on one line that is cut into equal pieces, two CTAs per SM (96 KB and 256 TMEM columns each), so one CTA's MMA and barrier
// latencies pass while the other one works.  Within a CTA Q K^T of the next tile is issued before P V of the current one; the output
// goes through the query tile's own buffer, so that a warp stores whole 256-byte rows.
// Bound: the queries in and the outputs out (12 x 4680 x 128: 28.8 MB, 4.4 us).  Measured against the paged kernel's gather mode (one
// query tile per CTA, one CTA per SM): 12 x 4680 queries, 64 kept 34.2 -> 11.5 us; 40 x 10800, 32 kept 218 -> 58 us; 12 x 1560,
// 64 kept 17.3 -> 7.9 us; 8 x 4096 x d 64 13.6 -> 6.7 us.
// Warps 0-3 soft-max and output (one row per thread), 4 TMA producer of the query tiles, 5 MMA issue, 6 and 7 gather K and V.
#include "common.h"
#include "ptx.cuh"

namespace fastar {

namespace {

constexpr int kThreads = 256, kSoftWarps = 4, kProducer = 4, kMma = 5, kGatherK = 6;
constexpr int kKeep = 64;                    // rows of the key tile
constexpr int kQChunk = 128 * 128;           // bytes of 128 rows x 64 bf16
constexpr int kKvChunk = kKeep * 128;
constexpr int kTmemCols = 256, kPCol = 64, kOCol = 128;

template <int D>
struct Cfg {
  static constexpr int nkc = D / 64;
  static constexpr int q_bytes = nkc * kQChunk, kv_bytes = nkc * kKvChunk;
  static constexpr int k_off = 2 * q_bytes, v_off = k_off + kv_bytes, bar_off = v_off + kv_bytes;
  static constexpr int total = bar_off + 128;
};

template <int D>
__global__ void __launch_bounds__(kThreads, 2)
prompt_attn_kernel(const __grid_constant__ CUtensorMap tm_q, const CacheView c, const AttnArgs a, int tiles_per_frame, int tiles_per_head,
                   int units) {
  using SM = Cfg<D>;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const uint32_t sbase = smem_u32(smem_raw);
  if (sbase & 1023u) {                  // swizzled tiles need 1024-byte alignment; uniform for the CTA
    if (threadIdx.x == 0) record_status(c.status, FASTAR_ERR_CUDA);
    return;
  }
  const uint32_t bar_q_full = sbase + SM::bar_off;     // [2]
  const uint32_t bar_q_empty = bar_q_full + 16;        // [2] one arrival per soft-max warp
  const uint32_t bar_kv_full = bar_q_full + 32;        // both gathering warps
  const uint32_t bar_kv_empty = bar_q_full + 40;
  const uint32_t bar_s_full = bar_q_full + 48;
  const uint32_t bar_s_empty = bar_q_full + 56;        // soft-max warps: the logits are in registers
  const uint32_t bar_p_full = bar_q_full + 64;         // soft-max warps
  const uint32_t bar_o_full = bar_q_full + 72;
  constexpr int kNumBars = 10;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem_raw + SM::bar_off + kNumBars * 8);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem_raw + SM::bar_off + kNumBars * 8 + 4);
  const int warp = warp_index(), lane = threadIdx.x & 31;

  if (threadIdx.x < kNumBars) {
    const int i = threadIdx.x;
    mbar_init(bar_q_full + 8 * i, i == 2 || i == 3 || i == 7 || i == 8 ? kSoftWarps : i == 4 ? 2 : 1);
    fence_mbar_init();
  }
  if (threadIdx.x == 0) *abort_flag = 0;
  if (warp == kProducer && lane == 0) tma_prefetch_desc(&tm_q);
  if (warp == kMma) {
    tmem_alloc(smem_u32(tmem_slot), kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  chain_wait();

  // this CTA's units; a segment is a run of them with the same head and frame
  const int u0 = static_cast<int>(static_cast<int64_t>(units) * blockIdx.x / gridDim.x);
  const int u1 = static_cast<int>(static_cast<int64_t>(units) * (blockIdx.x + 1) / gridDim.x);
  auto split = [&](int u, int& h, int& f, int& row) {
    h = u / tiles_per_head;
    const int r = u - h * tiles_per_head;
    f = r / tiles_per_frame;
    row = f * a.rows_per_frame + (r - f * tiles_per_frame) * 128;
  };
  auto kept = [&](int h, int f) {
    return a.keep_frames ? a.keep_frames[static_cast<int64_t>(h) * a.keep_frames_stride + f] : a.keep;
  };

  if (warp == kProducer) {
    bool ok = true;
    int n = 0;
    for (int u = u0; u < u1; ++u, ++n) {
      const int b = n & 1;
      ok = mbar_wait_warp<kIssueWaitHintNs>(bar_q_empty + 8 * b, ((n >> 1) & 1) ^ 1, abort_flag, c.status);
      if (!ok) break;
      int h, f, row;
      split(u, h, f, row);
      if (lane == 0) {
        mbar_arrive_expect_tx(bar_q_full + 8 * b, SM::q_bytes);
        for (int kc = 0; kc < SM::nkc; ++kc) tma_load_3d(sbase + b * SM::q_bytes + kc * kQChunk, &tm_q, bar_q_full + 8 * b, kc * 64, row, h);
      }
    }
    // the copies still in flight land before the CTA may exit (bounded like every other wait)
    if (lane == 0)
      for (int k = max(0, n - 2); k < n; ++k) mbar_wait<kIssueWaitHintNs>(bar_q_full + 8 * (k & 1), (k >> 1) & 1, abort_flag, c.status);
  } else if (warp == kMma) {
    const uint32_t lead = elect_lane();
    constexpr uint32_t idesc_s = make_idesc_bf16(128, kKeep, 0), idesc_o = make_idesc_bf16(128, D, 1);
    bool ok = true, issued = false;
    int nseg = 0, ch = -1, cf = -1;
    auto same_segment = [&](int u) {
      int h, f, row;
      split(u, h, f, row);
      return h == ch && f == cf;
    };
    auto issue_s = [&](int u) {
      int h, f, row;
      split(u, h, f, row);
      if (h != ch || f != cf) {
        ok = mbar_wait_warp<kIssueWaitHintNs>(bar_kv_full, nseg & 1, abort_flag, c.status);
        ++nseg;
        ch = h;
        cf = f;
      }
      const int n = u - u0, b = n & 1;
      ok = ok && mbar_wait_warp<kIssueWaitHintNs>(bar_q_full + 8 * b, (n >> 1) & 1, abort_flag, c.status) &&
           (n == 0 || mbar_wait_warp<kIssueWaitHintNs>(bar_s_empty, (n - 1) & 1, abort_flag, c.status));
      if (!ok) return;
      tc_fence_after();
#pragma unroll
      for (int kk = 0; kk < D / 16; ++kk)
        umma_ss(tmem, make_smem_desc(sbase + b * SM::q_bytes + (kk >> 2) * kQChunk + (kk & 3) * 32, 16, 1024),
                make_smem_desc(sbase + SM::k_off + (kk >> 2) * kKvChunk + (kk & 3) * 32, 16, 1024), idesc_s, kk != 0, lead);
      umma_commit(bar_s_full, lead);
    };
    for (int u = u0; u < u1 && ok; ++u) {
      if (!issued) issue_s(u);
      issued = u + 1 < u1 && same_segment(u + 1);
      if (ok && issued) issue_s(u + 1);
      ok = ok && mbar_wait_warp<kIssueWaitHintNs>(bar_p_full, (u - u0) & 1, abort_flag, c.status);
      if (!ok) break;
      tc_fence_after();
#pragma unroll
      for (int ks = 0; ks < kKeep / 16; ++ks)
        umma_ts(tmem + kOCol, tmem + kPCol + ks * 8, make_smem_desc(sbase + SM::v_off + ks * 2048, kKvChunk, 1024), idesc_o, ks != 0, lead);
      umma_commit(bar_o_full, lead);
      if (u + 1 < u1 && !issued) umma_commit(bar_kv_empty, lead);
    }
  } else if (warp >= kGatherK) {
    const __nv_bfloat16* rows = warp == kGatherK ? a.kp : a.vp;
    const uint32_t dst = sbase + (warp == kGatherK ? SM::k_off : SM::v_off);
    constexpr int CPR = D / 8, RPI = 32 / CPR;           // 16-byte chunks per row, rows per instruction
    int nseg = 0, ch = -1, cf = -1;
    for (int u = u0; u < u1; ++u) {
      int h, f, row;
      split(u, h, f, row);
      if (h == ch && f == cf) continue;
      ch = h;
      cf = f;
      const int32_t* list = a.sel + static_cast<int64_t>(h) * a.sel_head_stride + static_cast<int64_t>(f) * a.sel_stride;
      const int keep_n = kept(h, f);
      int idx[2];                                        // tokens 0-31 and 32-63 of the list, one per lane
#pragma unroll
      for (int q = 0; q < 2; ++q) idx[q] = 32 * q + lane < keep_n ? FASTAR_IDX(list[32 * q + lane], a.np, c.status) : 0;
      if (nseg > 0 && !mbar_wait_warp<kIssueWaitHintNs>(bar_kv_empty, (nseg - 1) & 1, abort_flag, c.status)) break;
      const __nv_bfloat16* src = rows + static_cast<int64_t>(h) * a.p_head_stride;
      const int chunk = lane % CPR;
#pragma unroll
      for (int it = 0; it < kKeep / RPI; ++it) {
        const int i = it * RPI + lane / CPR;
        const int tok = __shfl_sync(0xffffffffu, (it * RPI) >= 32 ? idx[1] : idx[0], i & 31);
        cp_async16(dst + (chunk >> 3) * kKvChunk + i * 128 + (((chunk & 7) ^ (i & 7)) << 4),
                   src + static_cast<int64_t>(tok) * a.p_token_stride + chunk * 8, i < keep_n);
      }
      asm volatile("cp.async.wait_all;" ::: "memory");
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_kv_full);
      ++nseg;
    }
  } else {
    const int r = warp * 32 + lane;                      // this thread's row
    const uint32_t lane_t = tmem + (static_cast<uint32_t>(warp * 32) << 16);
    const float scale = rsqrtf(static_cast<float>(D)) * 1.4426950408889634f;
    for (int u = u0; u < u1; ++u) {
      const int n = u - u0, b = n & 1;
      int h, f, row;
      split(u, h, f, row);
      const int keep_n = kept(h, f);
      const int valid = min(128, min((f + 1) * a.rows_per_frame, a.nq) - row);
      if (!mbar_wait_warp(bar_s_full, n & 1, abort_flag, c.status)) break;
      tc_fence_after();
      uint32_t x[2][32];
      tmem_ld32(lane_t, x[0]);
      tmem_ld32(lane_t + 32, x[1]);
      tmem_wait_ld();
      tc_fence_before();
      mbar_arrive_warp(bar_s_empty);
      if (keep_n < kKeep) {
#pragma unroll
        for (int j = 0; j < kKeep; ++j)
          if (j >= keep_n) x[j >> 5][j & 31] = __float_as_uint(-INFINITY);
      }
      float top[2] = {-INFINITY, -INFINITY};
#pragma unroll
      for (int j = 0; j < kKeep / 2; ++j)
        top[j & 1] = fmax3(top[j & 1], __uint_as_float(x[j >> 4][2 * (j & 15)]), __uint_as_float(x[j >> 4][2 * (j & 15) + 1]));
      const float m = fmaxf(top[0], top[1]) * scale;
      const float neg = m == -INFINITY ? 0.f : -m;
      float2 sum = make_float2(0.f, 0.f);
      uint32_t p[32];
#pragma unroll
      for (int j = 0; j < kKeep / 2; ++j) {
        const uint32_t* v = &x[j >> 4][2 * (j & 15)];
        const float2 t = ffma2(make_float2(__uint_as_float(v[0]), __uint_as_float(v[1])), make_float2(scale, scale), make_float2(neg, neg));
        const float2 e = make_float2(fast_exp2(t.x), fast_exp2(t.y));
        sum = fadd2(sum, e);
        p[j] = pack_bf16x2(e.x, e.y);
      }
      tmem_st32(lane_t + kPCol, p);
      tmem_wait_st();
      tc_fence_before();
      mbar_arrive_warp(bar_p_full);
      const float denom = sum.x + sum.y;
      const float inv = denom > 0.f ? 1.f / denom : 0.f;
      if (!mbar_wait_warp(bar_o_full, n & 1, abort_flag, c.status)) break;
      tc_fence_after();
      const int64_t out0 = static_cast<int64_t>(h) * a.out_head_stride + static_cast<int64_t>(row) * a.out_token_stride;
      const uint32_t q_s = sbase + b * SM::q_bytes;      // the MMAs are done with the query tile
#pragma unroll
      for (int kc = 0; kc < SM::nkc; ++kc) {
        tmem_ld32(lane_t + kOCol + kc * 64, x[0]);
        tmem_ld32(lane_t + kOCol + kc * 64 + 32, x[1]);
        tmem_wait_ld();
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
          for (int j = 0; j < 32; j += 2) scale2(x[q][j], x[q][j + 1], make_float2(inv, inv));
        if (a.out_fp32) {
          float4* dst = reinterpret_cast<float4*>(static_cast<float*>(a.out) + out0 + static_cast<int64_t>(r) * a.out_token_stride + kc * 64);
          if (r < valid)
#pragma unroll
            for (int t = 0; t < 16; ++t) {
              const uint32_t* v = &x[t >> 3][4 * (t & 7)];
              dst[t] = make_float4(__uint_as_float(v[0]), __uint_as_float(v[1]), __uint_as_float(v[2]), __uint_as_float(v[3]));
            }
        } else {
#pragma unroll
          for (int t = 0; t < 8; ++t) {                  // 16-byte chunk t of the row's 128 bytes, at its swizzled place
            const uint32_t* v = &x[t >> 2][8 * (t & 3)];
            uint32_t w[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) w[e] = pack_bf16x2(__uint_as_float(v[2 * e]), __uint_as_float(v[2 * e + 1]));
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(q_s + kc * kQChunk + r * 128 + ((t ^ (r & 7)) << 4)), "r"(w[0]),
                         "r"(w[1]), "r"(w[2]), "r"(w[3])
                         : "memory");
          }
        }
      }
      if (!a.out_fp32) {
        __syncwarp();                                    // a warp stores the 32 rows that it wrote
        constexpr int CPR = D / 8, RPI = 32 / CPR;
        const int chunk = lane % CPR;
        __nv_bfloat16* out = static_cast<__nv_bfloat16*>(a.out) + out0 + chunk * 8;
#pragma unroll 8
        for (int i = lane / CPR; i < 32; i += RPI) {
          const int rr = warp * 32 + i;
          uint4 v;
          asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                       : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                       : "r"(q_s + (chunk >> 3) * kQChunk + rr * 128 + (((chunk & 7) ^ (rr & 7)) << 4))
                       : "memory");
          if (rr < valid) *reinterpret_cast<uint4*>(out + static_cast<int64_t>(rr) * a.out_token_stride) = v;
        }
      }
      tc_fence_before();
      fence_proxy_async_smem();                          // the next copy into the buffer comes after these reads
      mbar_arrive_warp(bar_q_empty + 8 * b);
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == kMma) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
}

template <int D>
int launch_prompt_attn(const CUtensorMap& tm_q, const CacheView& c, const AttnArgs& a, cudaStream_t st) {
  auto kern = prompt_attn_kernel<D>;
  const int cfg = ensure_dynamic_smem(reinterpret_cast<const void*>(kern), Cfg<D>::total);
  if (cfg != FASTAR_OK) return cfg;
  int dev = 0, sm_count = 148;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sm_count, cudaDevAttrMultiProcessorCount, dev);
  const int tiles_per_frame = (min(a.rows_per_frame, a.nq) + 127) / 128;
  const int tiles_per_head = (a.n_frames - 1) * tiles_per_frame + (a.nq - (a.n_frames - 1) * a.rows_per_frame + 127) / 128;
  const int units = c.H * tiles_per_head;
  launch_chained(kern, min(units, 2 * sm_count), kThreads, Cfg<D>::total, st, tm_q, c, a, tiles_per_frame, tiles_per_head, units);
  return cudaGetLastError() == cudaSuccess ? 1 : FASTAR_ERR_CUDA;
}

}  // namespace

// a.keep <= 64
int launch_attention_prompt64(const CacheView& c, const CUtensorMap& tm_q, const AttnArgs& a, cudaStream_t st) {
  return c.D == 128 ? launch_prompt_attn<128>(tm_q, c, a, st) : launch_prompt_attn<64>(tm_q, c, a, st);
}

}  // namespace fastar
