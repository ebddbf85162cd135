// C1: relevance of the prompt tokens (AnnCA, Section 5.3): rel[h][f][p] = max over the queries i of frame f of <q_i, k_p>, on the
// bf16 rows or on the 8-bit codes (then times |q_i| |k_p|).  The scores are never written to memory.
//
// The prompt keys are the rows (TMEM lanes) of the contraction and the queries its columns, so that the maximum runs along the
// columns, inside a thread: 16 values of a row per thread and accumulator half, eight instructions, and only when a frame ends do
// the four lanes that share a row meet (with the queries as rows every 32 columns cost a butterfly of 31 shuffles).  A CTA keeps up
// to four prompt tiles (512 tokens) in shared memory and streams query tiles past them, so a query row is read once per 512 prompt
// tokens; four accumulators of 128 columns let the MMAs run ahead of the epilogue.  The work, (head, prompt group, query tile)
// units on one line, is cut into equal pieces, one per CTA.  Bound: reading the queries (12 x 4680 x 128: 14.4 MB, 2.2 us) and 64
// cycles per 128 x 128 x 16 product (12 x 37 x 4 tiles: 3.2 us at 148 SMs and 1.9 GHz), plus a CTA's start and end.  Measured (queries as rows, two
// CTAs per SM, atomics per 32 columns and tile -> this): 12 heads x 4680 queries x 512 tokens 27.0 -> 16.3 us, of which 6 are the
// start and end of a CTA; 40 x 10800 x 512 169 -> 74 us; 12 x 1560 x 512 14.3 -> 10.6 us; 8-bit codes 12 x 4680 27.7 -> 16.2 us.
// Warps 0-15 epilogue, in two groups of eight that take the accumulators in turn (one tile is 1 900 cycles of barrier, TMEM and
// arithmetic latency for a group, so one group alone left the tensor cores idle two thirds of the time); a warp has prompt rows
// 32 (w & 3).. of a tile and query columns 64 (w >> 2 & 1)...  Warp 16 TMA producer, 17 MMA issue
// (18 and 19 only make up the warpgroup whose registers the epilogue takes over).
#include "common.h"
#include "ptx.cuh"
#include "topk.cuh"

namespace fastar {

TopkArgs prompt_topk_args(const CacheView& c, int n_frames, int np, int keep);      // update_kernels.cu

namespace {

constexpr int kThreads = 640, kEpiWarps = 16, kProducer = 16, kMma = 17;
constexpr int kEpiRegs = 112, kIssueRegs = 32;  // 512 x 112 + 128 x 32 = 640 x 96, the registers of the launch
constexpr int kChunk = 128 * 128;            // bytes of 128 rows x 64 bf16, or of 128 code rows
constexpr int kMaxGroup = 4;                 // prompt tiles of a CTA
constexpr int kBuffers = 4;                  // accumulators

struct RelArgs {
  int nq, np, frame_len;
  int group;               // prompt tiles per CTA
  int prompt_tiles, query_tiles, prompt_groups;
  int units;               // heads * prompt_groups * query_tiles
  const float* qn;         // CODE8: |q|, [H][max_tokens]
  const float* kn;         // CODE8: |k_p|, [H][max_prompt]
  TopkArgs top;            // NV > 0: the ranking of a head's rows
};

template <int NKC>
struct Cfg {
  static constexpr int stages = NKC == 2 ? 3 : 4;
  static constexpr int tile = NKC * kChunk;
  static constexpr int bars = 256;
  static int total(int group) { return group * tile + stages * tile + bars; }
};

// NKC: 128-byte chunks of a row (bf16: d / 64, codes: 1)
// NV > 0: the CTA that finishes a head ranks its frames' tokens too (topk_row with NV registers), which saves a launch (see c1_ranks).
template <int NKC, bool CODE8, int NV>
__global__ void __launch_bounds__(kThreads, 1)
relevance_kernel(const __grid_constant__ CUtensorMap tm_p, const __grid_constant__ CUtensorMap tm_q, const CacheView c, const RelArgs g) {
  using SM = Cfg<NKC>;
  constexpr int S = SM::stages;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const uint32_t sbase = smem_u32(smem_raw);
  if (sbase & 1023u) {                  // swizzled tiles need 1024-byte alignment; uniform for the CTA
    if (threadIdx.x == 0) record_status(c.status, FASTAR_ERR_CUDA);
    return;
  }
  const uint32_t p_s = sbase, ring_s = sbase + g.group * SM::tile;
  const int bar_off = (g.group + S) * SM::tile;
  const uint32_t bar_full = sbase + bar_off;           // [S]
  const uint32_t bar_empty = bar_full + 8 * S;         // [S]
  const uint32_t bar_tfull = bar_empty + 8 * S;        // [kBuffers]
  const uint32_t bar_tempty = bar_tfull + 8 * kBuffers;  // [kBuffers] one arrival per warp of a group
  const uint32_t bar_pfull = bar_tempty + 8 * kBuffers;
  const uint32_t bar_pempty = bar_pfull + 8;
  constexpr int kNumBars = 2 * S + 2 * kBuffers + 2;
  static_assert(kNumBars * 8 + 12 <= SM::bars, "barrier area");
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem_raw + bar_off + kNumBars * 8);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem_raw + bar_off + kNumBars * 8 + 4);
  volatile int* last_s = abort_flag + 1;
  const int warp = warp_index(), lane = threadIdx.x & 31;

  if (threadIdx.x < kNumBars) {
    const int i = static_cast<int>(threadIdx.x) - 2 * S - kBuffers;
    mbar_init(bar_full + 8 * threadIdx.x, i >= 0 && i < kBuffers ? kEpiWarps / 2 : 1);
    fence_mbar_init();
  }
  if (threadIdx.x == 0) *abort_flag = 0;
  if (warp == kProducer && lane == 0) {
    tma_prefetch_desc(&tm_p);
    tma_prefetch_desc(&tm_q);
  }
  if (warp == kMma) {
    tmem_alloc(smem_u32(tmem_slot), kBuffers * 128);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  chain_wait();

  // this CTA's units; a segment is a run of them with the same head and prompt group
  const int u0 = static_cast<int>(static_cast<int64_t>(g.units) * blockIdx.x / gridDim.x);
  const int u1 = static_cast<int>(static_cast<int64_t>(g.units) * (blockIdx.x + 1) / gridDim.x);
  auto tiles_of = [&](int seg) { return min(g.group, g.prompt_tiles - (seg % g.prompt_groups) * g.group); };

  if (warp >= kEpiWarps) {
    setmaxnreg_dec<kIssueRegs>();
    if (warp == kProducer) {
      bool ok = true;
      int it = 0, nseg = 0, cur = -1;
      for (int u = u0; u < u1 && ok; ++u, ++it) {
        const int seg = u / g.query_tiles, t = u % g.query_tiles, h = seg / g.prompt_groups;
        if (seg != cur) {
          if (nseg > 0) ok = mbar_wait_warp<kIssueWaitHintNs>(bar_pempty, (nseg - 1) & 1, abort_flag, c.status);
          if (!ok) break;
          cur = seg;
          ++nseg;
          if (lane == 0) {
            const int gt = tiles_of(seg), p0 = (seg % g.prompt_groups) * g.group;
            mbar_arrive_expect_tx(bar_pfull, gt * SM::tile);
            for (int i = 0; i < gt; ++i)
              for (int kc = 0; kc < NKC; ++kc) tma_load_3d(p_s + i * SM::tile + kc * kChunk, &tm_p, bar_pfull, kc * 64, (p0 + i) * 128, h);
          }
        }
        const int s = it % S;
        ok = mbar_wait_warp<kIssueWaitHintNs>(bar_empty + 8 * s, ((it / S) & 1) ^ 1, abort_flag, c.status);
        if (!ok) break;
        if (lane == 0) {
          mbar_arrive_expect_tx(bar_full + 8 * s, SM::tile);
          for (int kc = 0; kc < NKC; ++kc) tma_load_3d(ring_s + s * SM::tile + kc * kChunk, &tm_q, bar_full + 8 * s, kc * 64, t * 128, h);
        }
      }
      // the copies still in flight land before the CTA may exit (bounded like every other wait)
      if (lane == 0) {
        for (int k = max(0, it - S); k < it; ++k) mbar_wait<kIssueWaitHintNs>(bar_full + 8 * (k % S), (k / S) & 1, abort_flag, c.status);
        if (nseg > 0) mbar_wait<kIssueWaitHintNs>(bar_pfull, (nseg - 1) & 1, abort_flag, c.status);
      }
    } else if (warp == kMma) {
      const uint32_t lead = elect_lane();
      constexpr uint32_t idesc = CODE8 ? make_idesc_e4m3(128, 128) : make_idesc_bf16(128, 128, 0);
      bool ok = true;
      int it = 0, nseg = 0, cur = -1, acc = 0;
      for (int u = u0; u < u1 && ok; ++u, ++it) {
        const int seg = u / g.query_tiles;
        if (seg != cur) {
          ok = mbar_wait_warp<kIssueWaitHintNs>(bar_pfull, nseg & 1, abort_flag, c.status);
          if (!ok) break;
          cur = seg;
          ++nseg;
        }
        const int s = it % S, gt = tiles_of(seg);
        ok = mbar_wait_warp<kIssueWaitHintNs>(bar_full + 8 * s, (it / S) & 1, abort_flag, c.status);
        if (!ok) break;
        for (int i = 0; i < gt; ++i, ++acc) {
          const int b = acc % kBuffers;
          ok = mbar_wait_warp<kIssueWaitHintNs>(bar_tempty + 8 * b, ((acc / kBuffers) & 1) ^ 1, abort_flag, c.status);
          if (!ok) break;
          tc_fence_after();
#pragma unroll
          for (int k4 = 0; k4 < 4 * NKC; ++k4) {
            const uint32_t off = (k4 >> 2) * kChunk + (k4 & 3) * 32;
            const uint64_t ad = make_smem_desc(p_s + i * SM::tile + off, 16, 1024), bd = make_smem_desc(ring_s + s * SM::tile + off, 16, 1024);
            if (CODE8) umma_ss_f8(tmem + b * 128, ad, bd, idesc, k4 != 0, lead);
            else umma_ss(tmem + b * 128, ad, bd, idesc, k4 != 0, lead);
          }
          umma_commit(bar_tfull + 8 * b, lead);
        }
        if (!ok) break;
        umma_commit(bar_empty + 8 * s, lead);
        if (u + 1 < u1 && (u + 1) / g.query_tiles != seg) umma_commit(bar_pempty, lead);
      }
    }
  } else {
    setmaxnreg_inc<kEpiRegs>();
    // Thread: rows 16 hf + 8 e + lane / 4 of its warp's 32, value k = 2 hf + e; columns 8 i + 2 (lane & 3) + {0, 1} of its 64.
    const uint32_t lane_addr = static_cast<uint32_t>((warp & 3) * 32) << 16;
    const int half = (warp >> 2) & 1, grp = warp >> 3;
    // This group's prompt tiles: every second one, i = 2 s + grp; of a lone tile every second unit.
    float mx[kMaxGroup / 2][4];
#pragma unroll
    for (int s = 0; s < kMaxGroup / 2; ++s)
#pragma unroll
      for (int k = 0; k < 4; ++k) mx[s][k] = -INFINITY;
    auto tile_at = [&](int s, int gt) { return gt == 1 ? s : 2 * s + grp; };
    // frame f of segment seg is complete as far as this CTA goes: its maxima of prompt tile i
    auto flush = [&](float (&m)[4], int seg, int i, int f) {
      const int h = seg / g.prompt_groups;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        m[k] = fmaxf(m[k], __shfl_xor_sync(0xffffffffu, m[k], 1));
        m[k] = fmaxf(m[k], __shfl_xor_sync(0xffffffffu, m[k], 2));
      }
      const int k = lane & 3;                          // each lane of the quad reports one row
      const float v = k == 0 ? m[0] : k == 1 ? m[1] : k == 2 ? m[2] : m[3];
      const int p = ((seg % g.prompt_groups) * g.group + i) * 128 + (warp & 3) * 32 + 8 * k + (lane >> 2);
      if (p < g.np)
        atomicMax(c.rel + (static_cast<int64_t>(h) * c.max_frames + f) * c.max_prompt + p,
                  float_to_ordered(CODE8 ? v * g.kn[static_cast<int64_t>(h) * c.max_prompt + p] : v));
#pragma unroll
      for (int q = 0; q < 4; ++q) m[q] = -INFINITY;
    };
    auto flush_all = [&](int seg, int f) {
      const int gt = tiles_of(seg);
#pragma unroll
      for (int q = 0; q < kMaxGroup / 2; ++q)
        if (tile_at(q, gt) < gt) flush(mx[q], seg, tile_at(q, gt), f);
    };
    bool ok = true;
    int acc0 = 0, cur = -1, f_cur = -1;                // accumulators of the units before; f_cur: frame that mx belongs to, -1 none
    for (int u = u0; u < u1 && ok; ++u) {
      const int seg = u / g.query_tiles, t = u % g.query_tiles;
      if (seg != cur) {
        if (f_cur >= 0) flush_all(cur, f_cur);
        cur = seg;
        f_cur = -1;
      }
      const int gt = tiles_of(seg);
      const int c0 = t * 128 + half * 64, c1 = min(c0 + 64, g.nq);      // this warp's queries
      const int f_first = c0 / g.frame_len, f_last = (c1 - 1) / g.frame_len;
      bool any = false;
#pragma unroll
      for (int q = 0; q < kMaxGroup / 2; ++q) {
        const int i = tile_at(q, gt);
        if (i >= gt || (gt == 1 && ((u - u0) & 1) != grp) || !ok) continue;
        const int b = (acc0 + i) % kBuffers;
        float2 qn[8];
        if (CODE8) {
          const float* src = g.qn + static_cast<int64_t>(seg / g.prompt_groups) * c.max_tokens;
#pragma unroll
          for (int n = 0; n < 8; ++n) {
            const int j = c0 + 8 * n + 2 * (lane & 3);
            qn[n] = make_float2(j < g.nq ? src[j] : 0.f, j + 1 < g.nq ? src[j + 1] : 0.f);
          }
        }
        ok = mbar_wait_warp(bar_tfull + 8 * b, ((acc0 + i) / kBuffers) & 1, abort_flag, c.status);
        if (!ok) continue;                             // warp-uniform: TMEM loads are warp-collective
        tc_fence_after();
        uint32_t x[2][32];
        tmem_ld_frag(tmem + lane_addr + b * 128 + half * 64, x[0]);
        tmem_ld_frag(tmem + lane_addr + (16u << 16) + b * 128 + half * 64, x[1]);
        tmem_wait_ld();
        tc_fence_before();
        mbar_arrive_warp(bar_tempty + 8 * b);
        if (c0 >= c1) continue;                        // nothing but rows past the last query
        any = true;
        if (CODE8) {
#pragma unroll
          for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int j = 0; j < 8; ++j) scale2(x[k >> 1][4 * j + 2 * (k & 1)], x[k >> 1][4 * j + 2 * (k & 1) + 1], qn[j]);
        }
        int f = f_cur;
        for (int fr = f_first; fr <= f_last; ++fr) {
          if (fr != f) {
            if (f >= 0) flush(mx[q], seg, i, f);
            f = fr;
          }
          const int64_t end = static_cast<int64_t>(fr + 1) * g.frame_len;
          const int lo = max(fr * g.frame_len - c0, 0), hi = (end < c1 ? static_cast<int>(end) : c1) - c0;
          const bool whole = lo == 0 && hi == 64;
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            float y[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) y[j] = __uint_as_float(x[k >> 1][4 * (j >> 1) + 2 * (k & 1) + (j & 1)]);
            if (!whole) {
#pragma unroll
              for (int j = 0; j < 16; ++j) {
                const int col = 8 * (j >> 1) + 2 * (lane & 3) + (j & 1);
                y[j] = col >= lo && col < hi ? y[j] : -INFINITY;
              }
            }
            const float a0 = fmax3(y[0], y[1], y[2]), a1 = fmax3(y[3], y[4], y[5]), a2 = fmax3(y[6], y[7], y[8]);
            const float a3 = fmax3(y[9], y[10], y[11]), a4 = fmax3(y[12], y[13], y[14]);
            mx[q][k] = fmax3(fmax3(a0, a1, a2), fmax3(a3, a4, y[15]), mx[q][k]);
          }
        }
      }
      acc0 += gt;
      if (any) f_cur = f_last;
    }
    if (ok && f_cur >= 0) flush_all(cur, f_cur);
    if constexpr (NV > 0) {
      // A head's units are those of consecutive CTAs; each tells, after its last report, and the last one of a head has all maxima.  (Also
      // after a time-out, so that the counters go back to zero.)
      const int per_head = g.prompt_groups * g.query_tiles, h0 = u0 / per_head, h1 = (u1 - 1) / per_head;
      auto cta_of = [&](int u) { return static_cast<int>((static_cast<int64_t>(u + 1) * gridDim.x - 1) / g.units); };
      for (int h = h0; h <= h1; ++h) {
        named_barrier_sync(1, kEpiWarps * 32);
        if (threadIdx.x == 0) {
          const int ctas = cta_of((h + 1) * per_head - 1) - cta_of(h * per_head) + 1;
          const int last = atomic_add_acq_rel(c.rel_count + h, 1) == ctas - 1 ? 1 : 0;
          if (last) c.rel_count[h] = 0;
          *last_s = last;
        }
        named_barrier_sync(1, kEpiWarps * 32);
        if (*last_s)
          for (int row = warp; row < g.top.rows; row += kEpiWarps) topk_row<true, NV>(g.top, h, row);
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == kMma) {
    tc_fence_after();
    tmem_dealloc(tmem, kBuffers * 128);
  }
}

template <int NKC, bool CODE8, int NV>
int launch_relevance_t(const CUtensorMap& tm_p, const CUtensorMap& tm_q, const CacheView& c, RelArgs g, cudaStream_t st) {
  using SM = Cfg<NKC>;
  auto kern = relevance_kernel<NKC, CODE8, NV>;
  const int cfg = ensure_dynamic_smem(reinterpret_cast<const void*>(kern), SM::total(kMaxGroup));
  if (cfg != FASTAR_OK) return cfg;
  int dev = 0, sm_count = 148;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sm_count, cudaDevAttrMultiProcessorCount, dev);
  g.prompt_tiles = (g.np + 127) / 128;
  g.query_tiles = (g.nq + 127) / 128;
  // Prompt tiles per CTA: a unit of `group` tiles takes about group + 1/2 tile times (the query tile is fetched once), and the
  // longest piece counts.  Few units (a short prompt, one frame of one head) are spread over more CTAs with smaller groups.
  double best = 0;
  for (int n = kMaxGroup; n >= 1; n /= 2) {
    const int groups = (g.prompt_tiles + n - 1) / n;
    const int64_t units = static_cast<int64_t>(c.H) * groups * g.query_tiles;
    const double cost = static_cast<double>((units + sm_count - 1) / sm_count) * (min(n, g.prompt_tiles) + 0.5);
    if (n == kMaxGroup || cost < best) {
      best = cost;
      g.group = n;
      g.prompt_groups = groups;
      g.units = static_cast<int>(units);
    }
  }
  launch_chained(kern, min(g.units, sm_count), kThreads, SM::total(g.group), st, tm_p, tm_q, c, g);
  return cudaGetLastError() == cudaSuccess ? 1 : FASTAR_ERR_CUDA;
}

// keep = 0: the maxima only; else the kept tokens of every frame too, by the steps of launch_topk.
template <int NKC, bool CODE8>
int launch_relevance(const CUtensorMap& tm_p, const CUtensorMap& tm_q, const CacheView& c, RelArgs g, int keep, cudaStream_t st) {
  if (keep == 0) return launch_relevance_t<NKC, CODE8, 0>(tm_p, tm_q, c, g, st);
  g.top = prompt_topk_args(c, (g.nq + g.frame_len - 1) / g.frame_len, g.np, keep);
  if (g.np <= 128) return launch_relevance_t<NKC, CODE8, 4>(tm_p, tm_q, c, g, st);
  if (g.np <= 256) return launch_relevance_t<NKC, CODE8, 8>(tm_p, tm_q, c, g, st);
  return launch_relevance_t<NKC, CODE8, 16>(tm_p, tm_q, c, g, st);
}

}  // namespace

// Whether a head's frames are ranked by the CTA that finishes it.  On the device that is no gain: one CTA ranks a head, sixteen rows at a time,
// where the top-k has an SM for every two rows.  It pays where a call is short enough to be bound by its launches (one head, 640 queries, 512
// prompt tokens 17.1 -> 14.6 us a call, 2 x 1200 17.1 -> 14.9, 12 x 1200 and 256 tokens 17.3 -> 17.4), and there only for few rows, short ones
// (16 frames of 512 tokens 17.3 -> 18.6, 32 17.2 -> 18.7, one of 1 024 17.1 -> 19.2); 12 x 4680 queries 20.4 -> 23.2, 40 x 10800 and 1 024
// tokens 158 -> 168.  Beside kernels that fill the SMs (the host-tensor step) the size does not matter: between the two kernels the next one
// of the others takes the SMs, and with the top-k there are two such places (25 heads x 9 222 tokens, a host call 4 320 us, with the top-k
// 4 398).
bool c1_ranks(const CacheView& c, int nq, int n_frames, int np, bool beside) {
  return n_frames <= 8 && np <= 512 && (beside || static_cast<int64_t>(c.H) * ((nq + 127) / 128) <= 148);
}

// c.rel (zero before the call where it is used) receives the maxima as ordered integers.
int launch_c1_relevance(const CacheView& c, const CUtensorMap& tm_q, const CUtensorMap& tm_kp, int nq, int np, int frame_len,
                        int keep, cudaStream_t st) {
  RelArgs g{};
  g.nq = nq;
  g.np = np;
  g.frame_len = frame_len;
  return c.D == 128 ? launch_relevance<2, false>(tm_kp, tm_q, c, g, keep, st) : launch_relevance<1, false>(tm_kp, tm_q, c, g, keep, st);
}

// The same on the 8-bit codes of the directions: code(q) . code(k_p) * |q| * |k_p|; the caller decodes with 1 / (256 sqrt(d)).
int launch_c1_relevance_fp8(const CacheView& c, const CUtensorMap& tm_q8, const CUtensorMap& tm_kp8, const float* qn,
                            const float* kn, int nq, int np, int frame_len, int keep, cudaStream_t st) {
  RelArgs g{};
  g.nq = nq;
  g.np = np;
  g.frame_len = frame_len;
  g.qn = qn;
  g.kn = kn;
  return launch_relevance<1, true>(tm_kp8, tm_q8, c, g, keep, st);
}

}  // namespace fastar
