// Candidate-set attention on tcgen05 / TMEM (paper Section 5.1: attention over N(q); Lemma 1:
// logits shifted by log m, values are group means):
//   paged  : AnnSA's selected-block attention and the dense Eq. 1 baseline.  A query block attends
//            to the key blocks listed in `sel`; one key block = one cache page = one TMA box, looked
//            up through the page table.
//   gather : AnnCA's attention over the kept prompt tokens of the query's frame; rows of K_p / V_p
//            are gathered by index with 128-bit loads into the same swizzled tile layout.
//
// One CTA = 128 query rows (TMEM lanes).  The key tiles are dealt alternately to two soft-max groups (g = j & 1, four warps each):
// one group's exponentials overlap the other's loads, shifts and MMAs.
//   S_g = Q K_j^T                   tcgen05.mma, SMEM x SMEM -> TMEM
//   P_g = exp2(S_g*scale + log2 m - m)      registers -> bf16 -> TMEM
//   O  += P_g V_j                   tcgen05.mma, TMEM x SMEM: V is the MN-major operand straight from its [key][d] page
// What bounds it: 128 x 128 exponentials are 1 024 cycles of an SM's special-function units, the two MMAs of the tile another
// 1 024 of the tensor core, and all of them want the shared-memory read path, which the operand reads of an MMA take first (a
// barrier or a load answers after some 300 cycles meanwhile).  So little goes through shared memory, and nothing waits in line:
//   - P goes through tensor memory (with P in shared memory the MMAs of a tile saturate the read path), beside S and not over
//     it, so that Q K^T of a group's next tile runs while this one is in its exponentials;
//   - that leaves room for one O, so both groups use one running maximum per row.  The two warps that own the same rows hand it
//     to each other from tile to tile by named barriers: each looks at its tile only after the other has looked at the one before.
//     It is raised lazily, only when a logit exceeds it by more than 2^8; who raises it rescales O (P V of all earlier tiles
//     done, that of this tile waiting for its P);
//   - the soft-max warps hold a tile in the 16 x 256-bit fragment shape, four rows x 32 columns a thread: a thread reads 32
//     biases, not 128, and a warp still has its rows to itself;
//   - Q K^T and P V are issued by two warps, so that a barrier that one of them waits for does not hold back the other.
// TMEM columns: S[0], S[1], P[0], P[1], O (2 x 128 + 2 x 64 + 128 at d = 128).  K and V tiles share one TMA ring: K0 K1 K2 | K3 V0 | ...
// Measured (B200, kernel time; before = P in shared memory, a thread per row, one issuing thread): 12 heads, d = 128, 4 680 queries
// on 32 of 224 blocks 139.6 -> 121 us (0.60 of the measured bf16 peak); the same with the chunk's 4 680 keys beside 291 -> 242 us;
// 8 heads, 4 096 queries on all 16 384 keys 326 -> 275 us; d = 64, 64 of 1 024 blocks 161 -> 142 us.  A tile takes an SM 1 830
// cycles: a warp runs some 860 instructions per tile and two soft-max warps per scheduler do not cover their latencies.
// Warp roles: warps 0-3 soft-max group 0, 4-7 group 1, 8 producer (TMA or gather), 9 Q K^T, 10 P V, 11 none.
#include "common.h"
#include "ptx.cuh"

namespace fastar {

constexpr int kQChunk = 128 * 128;   // bytes of one 128-row x 64-column bf16 chunk
constexpr int kAttnThreads = 384;
constexpr int kSoftWarps = 8, kProducerWarp = 8, kQkWarp = 9, kPvWarp = 10;
// Registers a thread: 384 x 168 at launch, dealt anew by role (8 x 32 x 216 + 4 x 32 x 72 = 384 x 168)
constexpr int kSoftRegs = 216, kIssueRegs = 72;

template <int D, int BKT>
struct AttnSmem {
  static constexpr int q_bytes = (D / 64) * kQChunk;
  static constexpr int kv_bytes = (D / 64) * BKT * 128;          // one K or V tile
  static constexpr int RS = 160 * 1024 / kv_bytes > 12 ? 12 : 160 * 1024 / kv_bytes;   // ring stages
  // A bias row is overwritten by that of eight tiles later, whose key tile needs (at most twelve places earlier) the key tile two
  // later consumed, and so this tile's logits and biases read.
  static constexpr int NB = 8;
  static constexpr int q_off = 0;
  static constexpr int ring_off = q_off + q_bytes;
  static constexpr int bias_off = ring_off + RS * kv_bytes;
  static constexpr int xchg_off = bias_off + NB * BKT * 4;       // [2][128] (maximum, sum) of the two groups' rows
  static constexpr int max_off = xchg_off + 2048;                // [4][8][4] running maxima: warp of the group, lane / 4, row / 8
  static constexpr int bar_off = max_off + 512;
  static constexpr int total = bar_off + 512;
  static constexpr int p_col = 2 * BKT, o_col = 3 * BKT;         // TMEM columns (S at 0 and BKT)
  static constexpr int tmem_cols = 3 * BKT + D <= 256 ? 256 : 512;
};

// SEG (paged mode only): tiles of an un-cached K/V segment follow the cache tiles.
template <int D, int BKT, bool GATHER, bool SEG>
__global__ void __launch_bounds__(kAttnThreads, 1)
attn_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
            const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_sk,
            const __grid_constant__ CUtensorMap tm_sv, const CacheView c, const AttnArgs a) {
  using SM = AttnSmem<D, BKT>;
  constexpr int RS = SM::RS, NB = SM::NB;
  constexpr int HD = D / 2;             // output columns written by one thread in the epilogue
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const uint32_t sbase = smem_u32(smem_raw);
  uint8_t* sgen = smem_raw;
  if (sbase & 1023u) {                  // swizzled tiles need 1024-byte alignment; uniform for the CTA
    if (threadIdx.x == 0) record_status(c.status, FASTAR_ERR_CUDA);
    return;
  }
  const uint32_t q_s = sbase + SM::q_off;
  const uint32_t ring_s = sbase + SM::ring_off;
  float* bias_g = reinterpret_cast<float*>(sgen + SM::bias_off);
  const uint32_t bias_s = sbase + SM::bias_off;
  const uint32_t bar = sbase + SM::bar_off;
  const uint32_t bar_q_full = bar;
  const uint32_t bar_r_full = bar + 8;               // [RS]
  const uint32_t bar_r_empty = bar_r_full + 8 * RS;  // [RS]
  const uint32_t bar_s_full = bar_r_empty + 8 * RS;  // [2] the MMAs' commit, and the issuing warp once the biases are there
  const uint32_t bar_pv_done = bar_s_full + 16;      // [2]
  const uint32_t bar_s_empty = bar_pv_done + 16;     // [2] the warps of a group
  const uint32_t bar_p_full = bar_s_empty + 16;      // [2] the warps of a group
  const uint32_t bar_xchg = bar_p_full + 16;         // [1] the two groups meet here before the epilogue
  constexpr int kNumBars = 1 + 2 * RS + 9;
  static_assert(kNumBars * 8 + 8 <= 512, "barrier area");
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(sgen + SM::bar_off + kNumBars * 8);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(sgen + SM::bar_off + kNumBars * 8 + 4);

  const int warp = warp_index(), lane = threadIdx.x & 31;
  const int h = blockIdx.y;

  // ---- which rows ------------------------------------------------------------------------------
  const int q0 = GATHER ? static_cast<int>(blockIdx.z) * a.rows_per_frame + static_cast<int>(blockIdx.x) * 128
                        : static_cast<int>(blockIdx.x) * a.block_q;
  const int valid_rows = GATHER ? min(128, min(a.rows_per_frame - static_cast<int>(blockIdx.x) * 128, a.nq - q0))
                                : min(a.block_q, a.nq - q0);
  if (valid_rows <= 0) return;          // uniform for the CTA; nothing allocated yet

  // one thread per barrier
  if (threadIdx.x < kNumBars) {
    const int i = static_cast<int>(threadIdx.x) - (kNumBars - 9);         // s_full, pv_done, s_empty, p_full, xchg
    mbar_init(bar + 8 * threadIdx.x, i == 8 ? kSoftWarps : i >= 4 ? kSoftWarps / 2 : i == 0 || i == 1 ? 2 : 1);
    fence_mbar_init();
  }
  if (threadIdx.x == 0) *abort_flag = 0;
  if (warp == kProducerWarp && lane == 0) {
    tma_prefetch_desc(&tm_q);
    if (!GATHER) { tma_prefetch_desc(&tm_k); tma_prefetch_desc(&tm_v); }
    if (SEG) { tma_prefetch_desc(&tm_sk); tma_prefetch_desc(&tm_sv); }
  }
  if (warp == kPvWarp) {
    tmem_alloc(smem_u32(tmem_slot), SM::tmem_cols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  chain_wait();

  // ---- which key tiles (warp-uniform for the role loops) --------------------------------------
  int nt;
  int ntc = 0;                          // paged mode: tiles taken from the cache; tiles [ntc, nt) are segment tiles
  int keep_n = a.keep;                  // gather mode: kept prompt tokens of this CTA's frame
  const int L = GATHER ? 0 : __shfl_sync(0xffffffffu, c.len[h], 0);
  const int32_t* list = nullptr;
  if (!GATHER) {
    if (a.sel == nullptr) {
      ntc = (L + BKT - 1) / BKT;
    } else {
      ntc = __shfl_sync(0xffffffffu, a.nsel[h], 0);
      list = a.sel + static_cast<int64_t>(h) * a.sel_head_stride + static_cast<int64_t>(blockIdx.x) * a.sel_stride;
    }
    nt = ntc + (SEG ? a.seg_tiles : 0);
  } else {
    const int f = blockIdx.z;
    if (a.keep_frames) keep_n = __shfl_sync(0xffffffffu, a.keep_frames[static_cast<int64_t>(h) * a.keep_frames_stride + f], 0);
    nt = (keep_n + BKT - 1) / BKT;
    list = a.sel + static_cast<int64_t>(h) * a.sel_head_stride + static_cast<int64_t>(f) * a.sel_stride;
  }

  // Gather mode with a single key tile (the usual AnnCA case, keep <= BKT): all threads fetch the kept rows
  // of K_p and V_p at once, instead of leaving 2 x BKT x D x 2 bytes of 16-byte gathers to one warp.
  bool prefilled = false;
  if (GATHER && nt == 1) {
    constexpr int CPR = D / 8;                         // 16-byte chunks per row
    const __nv_bfloat16* kp_h = a.kp + static_cast<int64_t>(h) * a.p_head_stride;
    const __nv_bfloat16* vp_h = a.vp + static_cast<int64_t>(h) * a.p_head_stride;
    for (int q = threadIdx.x; q < 2 * BKT * CPR; q += blockDim.x) {
      const int which = q / (BKT * CPR), qq = q % (BKT * CPR);
      const int i = qq / CPR, ch = qq % CPR;
      uint4 val = make_uint4(0, 0, 0, 0);
      if (i < keep_n) {
        const int idx = FASTAR_IDX(list[i], a.np, c.status);
        val = *reinterpret_cast<const uint4*>((which ? vp_h : kp_h) + static_cast<int64_t>(idx) * a.p_token_stride + ch * 8);
      }
      const uint32_t off = which * SM::kv_bytes + (ch >> 3) * (BKT * 128) + i * 128 + (((ch & 7) ^ (i & 7)) << 4);
      asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(ring_s + off), "r"(val.x), "r"(val.y), "r"(val.z), "r"(val.w)
                   : "memory");
    }
    for (int i = threadIdx.x; i < BKT; i += blockDim.x) bias_g[i] = (i < keep_n) ? 0.f : -INFINITY;
    fence_proxy_async_smem();
    __syncthreads();
    if (threadIdx.x == 0) {
      mbar_arrive(bar_r_full);                         // K0 -> stage 0
      mbar_arrive(bar_r_full + 8);                     // V0 -> stage 1
    }
    prefilled = true;
  }

  // Places of K_j and V_j in the ring: K0 K1 K2 | K3 V0 | K4 V1 | ..., the order in which the MMAs get to them (Q K^T of a tile
  // starts when the logits two tiles before have left S, P V when that tile's exponentials are done, after one more Q K^T).
  auto place_k = [](int j) { return j + max(0, j - 3); };
  auto place_v = [nt](int j) { return j + min(nt, j + 4); };

  if (warp >= kSoftWarps) {
    setmaxnreg_dec<kIssueRegs>();
    if (warp == kProducerWarp) {
      // ================================================================ producer
      if (lane == 0 && nt > 0) {
        mbar_arrive_expect_tx(bar_q_full, SM::q_bytes);
        for (int kc = 0; kc < D / 64; ++kc) tma_load_3d(q_s + kc * kQChunk, &tm_q, bar_q_full, kc * 64, q0, h);
      }
      bool ok = true;
      int place = 0;
      auto each_tile = [&](auto&& load) {                // in ring order
        for (int j = 0; j < 3 && j < nt && ok; ++j) load(true, j);
        for (int j = 0; j < nt && ok; ++j) {
          if (j + 3 < nt) load(true, j + 3);
          if (ok) load(false, j);
        }
      };
      auto stage_free = [&](int st) {
        return mbar_wait_warp<kIssueWaitHintNs>(bar_r_empty + 8 * st, ((place / RS) & 1) ^ 1, abort_flag, c.status);
      };
      if (!GATHER) {
        // block ids and page ids of 32 tiles at a time, one coalesced load each; lane 0 issues the copies.  Two windows: the low
        // one holds the value tile in turn, key tiles (three ahead) may already need the next.
        const int32_t* pt_h = c.page_table + static_cast<int64_t>(h) * c.CAPB;
        const float* l2m_h = c.log2m + static_cast<int64_t>(h) * c.CAP;
        int blk_l = 0, page_l = 0, blk_n = 0, page_n = 0, base = 0;
        auto fetch = [&](int j0, int& blk, int& page) {
          const int jj = j0 + lane;
          if (jj < ntc) {
            blk = FASTAR_IDX(list ? list[jj] : jj, c.CAPB, c.status);
            page = FASTAR_IDX(pt_h[blk], c.pool_pages, c.status);
          } else if (SEG && jj < nt) {        // tile of the un-cached segment: its index, no page
            blk = jj - ntc;
            page = -1;
          }
        };
        fetch(0, blk_l, page_l);
        fetch(32, blk_n, page_n);
        each_tile([&](bool is_k, int j) {
          if (!is_k && j >= base + 32) {                          // value tiles enter the next window
            base += 32;
            blk_l = blk_n; page_l = page_n;
            fetch(base + 32, blk_n, page_n);
          }
          const bool hi = j >= base + 32;
          const int blk = __shfl_sync(0xffffffffu, hi ? blk_n : blk_l, j & 31);
          const int page = __shfl_sync(0xffffffffu, hi ? page_n : page_l, j & 31);
          const int st = place % RS;
          ok = stage_free(st);
          if (!ok) return;
          if (lane == 0) {
            const bool seg = SEG && page < 0;   // rows past the segment's end arrive as zeros and carry a -inf bias
            const CUtensorMap* tm = seg ? (is_k ? &tm_sk : &tm_sv) : (is_k ? &tm_k : &tm_v);
            mbar_arrive_expect_tx(bar_r_full + 8 * st, SM::kv_bytes + (is_k ? BKT * 4 : 0));
            for (int kc = 0; kc < D / 64; ++kc)
              tma_load_3d(ring_s + st * SM::kv_bytes + kc * BKT * 128, tm, bar_r_full + 8 * st, kc * 64, seg ? blk * BKT : 0,
                          seg ? h : page);
            if (is_k) {
              const int b8 = j % NB;
              const float* bias_src = seg ? a.seg_bias + static_cast<int64_t>(blk) * BKT : l2m_h + static_cast<int64_t>(blk) * BKT;
              bulk_load_1d(bias_s + b8 * BKT * 4, bias_src, BKT * 4, bar_r_full + 8 * st);
            }
          }
          ++place;
        });
        // what is still in flight must land before the CTA may exit (normally the MMAs have consumed all of it)
        if (lane == 0 && nt > 0) {
          mbar_wait(bar_q_full, 0, abort_flag, c.status);
          for (int k = max(0, place - RS); k < place; ++k) mbar_wait(bar_r_full + 8 * (k % RS), (k / RS) & 1, abort_flag, c.status);
        }
      } else {
        // gather rows of K_p / V_p by index: 16-byte chunks, written at their swizzled position
        constexpr int CPR = D / 8;                       // 16-byte chunks per row
        const __nv_bfloat16* kp_h = a.kp + static_cast<int64_t>(h) * a.p_head_stride;
        const __nv_bfloat16* vp_h = a.vp + static_cast<int64_t>(h) * a.p_head_stride;
        if (!prefilled)
          each_tile([&](bool is_k, int j) {
            const int st = place % RS;
            ok = stage_free(st);
            if (!ok) return;
            const __nv_bfloat16* src_h = is_k ? kp_h : vp_h;
            const uint32_t dst = ring_s + st * SM::kv_bytes;
            for (int q = lane; q < BKT * CPR; q += 32) {
              const int i = q / CPR, ch = q % CPR;
              const int tok = j * BKT + i;
              uint4 val = make_uint4(0, 0, 0, 0);
              if (tok < keep_n) {
                const int idx = FASTAR_IDX(list[tok], a.np, c.status);
                val = *reinterpret_cast<const uint4*>(src_h + static_cast<int64_t>(idx) * a.p_token_stride + ch * 8);
              }
              const uint32_t off = (ch >> 3) * (BKT * 128) + i * 128 + (((ch & 7) ^ (i & 7)) << 4);
              asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst + off), "r"(val.x), "r"(val.y), "r"(val.z),
                           "r"(val.w)
                           : "memory");
            }
            const int b8 = j % NB;
            if (is_k)
              for (int i = lane; i < BKT; i += 32) bias_g[b8 * BKT + i] = (j * BKT + i < keep_n) ? 0.f : -INFINITY;
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_r_full + 8 * st);
            ++place;
          });
        if (lane == 0 && nt > 0) mbar_wait(bar_q_full, 0, abort_flag, c.status);
      }
    } else if (warp == kQkWarp) {
      // ================================================================ S_g = Q K_j^T
      const uint32_t lead = elect_lane();
      constexpr uint32_t idesc = make_idesc_bf16(128, BKT, 0);
      bool ok = nt > 0 && mbar_wait_warp(bar_q_full, 0, abort_flag, c.status);
      for (int j = 0; j < nt && ok; ++j) {
        const int pl = place_k(j), st = pl % RS, g = j & 1;
        // S_g is free once its group holds the logits of its last tile in registers
        ok = mbar_wait_warp(bar_r_full + 8 * st, (pl / RS) & 1, abort_flag, c.status) &&
             (j < 2 || mbar_wait_warp(bar_s_empty + 8 * g, ((j >> 1) - 1) & 1, abort_flag, c.status));
        if (!ok) break;
        tc_fence_after();
        const uint32_t kt = ring_s + st * SM::kv_bytes;
#pragma unroll
        for (int kk = 0; kk < D / 16; ++kk) {
          const uint64_t ad = make_smem_desc(q_s + (kk >> 2) * kQChunk + (kk & 3) * 32, 16, 1024);
          const uint64_t bd = make_smem_desc(kt + (kk >> 2) * (BKT * 128) + (kk & 3) * 32, 16, 1024);
          umma_ss(tmem + g * BKT, ad, bd, idesc, kk != 0, lead);
        }
        umma_commit(bar_s_full + 8 * g, lead);
        umma_commit(bar_r_empty + 8 * st, lead);
        if (lead) mbar_arrive(bar_s_full + 8 * g);     // what this warp has seen land (the biases) is there for the waiting warps
      }
    } else if (warp == kPvWarp) {
      // ================================================================ O += P_g V_j
      const uint32_t lead = elect_lane();
      constexpr uint32_t idesc = make_idesc_bf16(128, D, 1);
      bool ok = true;
      for (int j = 0; j < nt && ok; ++j) {
        const int pl = place_v(j), st = pl % RS, g = j & 1;
        ok = mbar_wait_warp(bar_r_full + 8 * st, (pl / RS) & 1, abort_flag, c.status) &&
             mbar_wait_warp(bar_p_full + 8 * g, (j >> 1) & 1, abort_flag, c.status);
        if (!ok) break;
        tc_fence_after();
        const uint32_t vt = ring_s + st * SM::kv_bytes;
#pragma unroll
        for (int ks = 0; ks < BKT / 16; ++ks) {
          const uint64_t bd = make_smem_desc(vt + ks * 2048, BKT * 128, 1024);
          umma_ts(tmem + SM::o_col, tmem + SM::p_col + g * (BKT / 2) + ks * 8, bd, idesc, (j | ks) != 0, lead);
        }
        umma_commit(bar_pv_done + 8 * g, lead);
        umma_commit(bar_r_empty + 8 * st, lead);
      }
    }
  } else {
    // ================================================================== soft-max groups + epilogue (256 threads)
    setmaxnreg_inc<kSoftRegs>();
    constexpr int NH = BKT / 64;                        // 64-column halves
    const int g = warp >> 2;                            // soft-max group: key tiles j with (j & 1) == g
    const uint32_t lane_addr = static_cast<uint32_t>((warp & 3) * 32) << 16;
    const int rq = (warp & 3) * 32 + (lane >> 2);       // this thread's rows: rq + 8 q, q = 2 half + e
    const float scale = rsqrtf(static_cast<float>(D)) * 1.4426950408889634f;
    const uint32_t s_t = tmem + lane_addr + g * BKT, p_t = tmem + lane_addr + SM::p_col + g * (BKT / 2), o_t = tmem + lane_addr + SM::o_col;
    constexpr uint32_t kHalf = 16u << 16;               // the second sixteen lanes
    float2* xchg = reinterpret_cast<float2*>(sgen + SM::xchg_off);
    float m[4];
    float2 l[4];                                        // running maxima; sums over the even and the odd columns
#pragma unroll
    for (int q = 0; q < 4; ++q) { m[q] = -INFINITY; l[q] = make_float2(0.f, 0.f); }
    float4* max_s = reinterpret_cast<float4*>(sgen + SM::max_off) + (warp & 3) * 8 + (lane >> 2);
    // the barriers of the hand-over: this warp waits for its partner's look at the tile before, and tells of its own
    const uint32_t heard = 1 + (warp & 3) + 4 * g, told = 1 + (warp & 3) + 4 * (g ^ 1);
    // After a time-out a warp goes on to its last tile without waiting, so that its partner is never left at a named barrier.
    bool ok = true;
    const int n_mine = (nt - g + 1) >> 1;               // tiles of this group
    bool s_ready = false;
    for (int i = 0; i < n_mine; ++i) {
      const int j = 2 * i + g;
      if (j > 0) named_barrier_sync(heard, 64);
      float4 seen = j > 0 ? *max_s : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
      if (!s_ready) ok = ok && mbar_wait_warp(bar_s_full + 8 * g, i & 1, abort_flag, c.status);
      tc_fence_after();
      // the logits of this warp's rows: x[hf][ch][4 k + 2 e + c] is row 16 hf + 8 e + lane / 4, column 64 ch + 8 k + 2 (lane & 3) + c
      uint32_t x[2][NH][32];
#pragma unroll
      for (int hf = 0; hf < 2; ++hf)
#pragma unroll
        for (int ch = 0; ch < NH; ++ch)
          if (ok) tmem_ld_frag(s_t + hf * kHalf + ch * 64, x[hf][ch]);
      const float2* bp = reinterpret_cast<const float2*>(bias_g + (j % NB) * BKT + 2 * (lane & 3));
      float2 bias[8 * NH];
#pragma unroll
      for (int k = 0; k < 8 * NH; ++k) bias[k] = bp[4 * k];
      tmem_wait_ld();
      tc_fence_before();
      mbar_arrive_warp(bar_s_empty + 8 * g);           // logits and biases are in registers
      // (asked here, needed later: a barrier answers slowly while MMAs run)
      const bool p_free = i == 0 || mbar_test_wait(bar_pv_done + 8 * g, (i - 1) & 1);
      float mx[4];
#pragma unroll
      for (int hf = 0; hf < 2; ++hf)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          float top[2] = {-INFINITY, -INFINITY};
#pragma unroll
          for (int k = 0; k < 8 * NH; ++k) {
            uint32_t* v = &x[hf][k >> 3][4 * (k & 7) + 2 * e];
            const float2 t = ffma2(make_float2(__uint_as_float(v[0]), __uint_as_float(v[1])), make_float2(scale, scale), bias[k]);
            v[0] = __float_as_uint(t.x);
            v[1] = __float_as_uint(t.y);
            top[k & 1] = fmax3(top[k & 1], t.x, t.y);
          }
          mx[2 * hf + e] = fmaxf(top[0], top[1]);
        }
      const float cur[4] = {seen.x, seen.y, seen.z, seen.w};
      bool raise = false, behind = false;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        raise |= mx[q] > cur[q] + 8.f || (cur[q] == -INFINITY && mx[q] > -INFINITY);
        behind |= cur[q] != m[q];
      }
      if (__any_sync(0xffffffffu, raise || behind)) {
        float alpha[4];
        bool resc = false;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          // the same for the four threads of a row
          mx[q] = fmaxf(mx[q], __shfl_xor_sync(0xffffffffu, mx[q], 1));
          mx[q] = fmaxf(mx[q], __shfl_xor_sync(0xffffffffu, mx[q], 2));
          float top = cur[q];
          alpha[q] = 1.f;
          if (mx[q] > cur[q] + 8.f || (cur[q] == -INFINITY && mx[q] > -INFINITY)) {
            top = mx[q];
            alpha[q] = cur[q] == -INFINITY ? 0.f : fast_exp2(cur[q] - top);
            resc = j > 0;
          }
          // this thread's sum follows both the partner's raise and its own
          if (m[q] != top) {
            const float f = m[q] == -INFINITY ? 0.f : fast_exp2(m[q] - top);
            l[q].x *= f;
            l[q].y *= f;
          }
          m[q] = top;
        }
        if ((lane & 3) == 0) *max_s = make_float4(m[0], m[1], m[2], m[3]);
        if (__any_sync(0xffffffffu, resc)) {
          // O is relative to the old maxima: P V of the tile before must be in it, that of this tile follows its P
          ok = ok && mbar_wait_warp(bar_pv_done + 8 * (g ^ 1), ((j - 1) >> 1) & 1, abort_flag, c.status);
          tc_fence_after();
          if (ok)
#pragma unroll 1
            for (int cc = 0; cc < 2 * (D / 32); ++cc) {
              const int hf = cc & 1;
              const uint32_t o_c = o_t + hf * kHalf + (cc >> 1) * 32;
              const float a0 = hf ? alpha[2] : alpha[0], a1 = hf ? alpha[3] : alpha[1];
              uint32_t v[16];
              tmem_ld_frag16(o_c, v);
              tmem_wait_ld();
#pragma unroll
              for (int t = 0; t < 16; ++t) v[t] = __float_as_uint(__uint_as_float(v[t]) * ((t & 2) ? a1 : a0));
              tmem_st_frag16(o_c, v);
            }
        }
        __syncwarp();
      }
      if (j + 1 < nt) named_barrier_arrive(told, 64);
      // P_g is free once P V of the group's last tile has read it
      if (!__all_sync(0xffffffffu, p_free)) ok = ok && mbar_wait_warp(bar_pv_done + 8 * g, (i - 1) & 1, abort_flag, c.status);
      tc_fence_after();
      // exponentials -> bf16 P
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        float2 neg[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) neg[e].x = neg[e].y = m[2 * hf + e] == -INFINITY ? 0.f : -m[2 * hf + e];
#pragma unroll
        for (int ch = 0; ch < NH; ++ch) {
          uint32_t p[16];
#pragma unroll
          for (int k = 0; k < 8; ++k)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              const uint32_t* v = &x[hf][ch][4 * k + 2 * e];
              const float2 u = fadd2(make_float2(__uint_as_float(v[0]), __uint_as_float(v[1])), neg[e]);
              const float2 pr = make_float2(fast_exp2(u.x), fast_exp2(u.y));
              l[2 * hf + e] = fadd2(l[2 * hf + e], pr);
              p[2 * k + e] = pack_bf16x2(pr.x, pr.y);
            }
          if (ok) tmem_st_half_frag(p_t + hf * kHalf + ch * 32, p);
        }
      }
      s_ready = i + 1 < n_mine && mbar_test_wait(bar_s_full + 8 * g, (i + 1) & 1);
      tmem_wait_st();
      tc_fence_before();
      mbar_arrive_warp(bar_p_full + 8 * g);
      s_ready = __all_sync(0xffffffffu, s_ready);
    }
    // ---- the two groups meet: (m, l) of every row through shared memory ----
    if (nt > 0) ok = ok && mbar_wait_warp(bar_pv_done + 8 * ((nt - 1) & 1), ((nt - 1) >> 1) & 1, abort_flag, c.status);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float sum = l[q].x + l[q].y;
      sum += __shfl_xor_sync(0xffffffffu, sum, 1);
      sum += __shfl_xor_sync(0xffffffffu, sum, 2);
      if ((lane & 3) == 0) xchg[g * 128 + rq + 8 * q] = make_float2(m[q], sum);
    }
    mbar_arrive_warp(bar_xchg);
    ok = mbar_wait_warp(bar_xchg, 0, abort_flag, c.status) && ok;
    tc_fence_after();
    const int r = (warp & 3) * 32 + lane;         // from here on a thread owns one row, half of its columns
    const bool wr = r < valid_rows;               // loads are warp-collective, only the stores are per row
    if (ok) {
      // O is relative to the last maximum, which the group of the last tile knows; the other one may be a raise behind
      const float2 r0 = xchg[r], r1 = xchg[128 + r];
      const float m_all = fmaxf(r0.x, r1.x);
      const float a0 = (r0.x == -INFINITY) ? 0.f : fast_exp2(r0.x - m_all);
      const float a1 = (r1.x == -INFINITY) ? 0.f : fast_exp2(r1.x - m_all);
      const float denom = r0.y * a0 + r1.y * a1;
      const float inv = denom > 0.f ? 1.f / denom : 0.f;
      const int64_t off = static_cast<int64_t>(h) * a.out_head_stride + static_cast<int64_t>(q0 + r) * a.out_token_stride + g * HD;
#pragma unroll 1
      for (int cc = 0; cc < HD / 32; ++cc) {
        uint32_t v[32];
        if (nt > 0) {
          tmem_ld32(tmem + SM::o_col + lane_addr + g * HD + cc * 32, v);
          tmem_wait_ld();
        }
        float o[32];
#pragma unroll
        for (int t = 0; t < 32; ++t) o[t] = nt > 0 ? __uint_as_float(v[t]) * inv : 0.f;
        if (!wr) continue;
        if (a.out_fp32) {
          float4* dst = reinterpret_cast<float4*>(static_cast<float*>(a.out) + off + cc * 32);
#pragma unroll
          for (int t = 0; t < 8; ++t) dst[t] = make_float4(o[4 * t], o[4 * t + 1], o[4 * t + 2], o[4 * t + 3]);
        } else {
          uint4* dst = reinterpret_cast<uint4*>(static_cast<__nv_bfloat16*>(a.out) + off + cc * 32);
#pragma unroll
          for (int t = 0; t < 4; ++t)
            dst[t] = make_uint4(pack_bf16x2(o[8 * t], o[8 * t + 1]), pack_bf16x2(o[8 * t + 2], o[8 * t + 3]),
                                pack_bf16x2(o[8 * t + 4], o[8 * t + 5]), pack_bf16x2(o[8 * t + 6], o[8 * t + 7]));
        }
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == kPvWarp) {
    tc_fence_after();
    tmem_dealloc(tmem, SM::tmem_cols);
  }
}

template <int D, int BKT, bool GATHER, bool SEG>
static int launch_attn(const CUtensorMap& tq, const CUtensorMap& tk, const CUtensorMap& tv, const CUtensorMap& tsk,
                       const CUtensorMap& tsv, const CacheView& c, const AttnArgs& a, dim3 grid, cudaStream_t st) {
  using SM = AttnSmem<D, BKT>;
  auto kern = attn_kernel<D, BKT, GATHER, SEG>;
  const int cfg = ensure_dynamic_smem(reinterpret_cast<const void*>(kern), SM::total);
  if (cfg != FASTAR_OK) return cfg;
  launch_chained(kern, grid, kAttnThreads, SM::total, st, tq, tk, tv, tsk, tsv, c, a);
  return cudaGetLastError() == cudaSuccess ? 1 : FASTAR_ERR_CUDA;
}

// tm_seg_k / tm_seg_v: maps of the un-cached segment (box {64, page_tokens, 1}); nullptr when a.seg_tiles == 0.
int launch_attention_paged(const CacheView& c, const CUtensorMap& tm_q, const CUtensorMap& tm_pool_k,
                           const CUtensorMap& tm_pool_v, const CUtensorMap* tm_seg_k, const CUtensorMap* tm_seg_v,
                           const AttnArgs& a, cudaStream_t st) {
  if (a.seg_tiles > 0 && (!tm_seg_k || !tm_seg_v || !a.seg_bias)) return FASTAR_ERR_INVALID_ARG;
  const CUtensorMap& sk = a.seg_tiles > 0 ? *tm_seg_k : tm_q;      // never read without segment tiles
  const CUtensorMap& sv = a.seg_tiles > 0 ? *tm_seg_v : tm_q;
  const dim3 grid((a.nq + a.block_q - 1) / a.block_q, c.H, 1);
  if (c.D == 128 && c.PT == 128) return a.seg_tiles > 0 ? launch_attn<128, 128, false, true>(tm_q, tm_pool_k, tm_pool_v, sk, sv, c, a, grid, st)
                                                          : launch_attn<128, 128, false, false>(tm_q, tm_pool_k, tm_pool_v, sk, sv, c, a, grid, st);
  if (c.D == 128 && c.PT == 64) return a.seg_tiles > 0 ? launch_attn<128, 64, false, true>(tm_q, tm_pool_k, tm_pool_v, sk, sv, c, a, grid, st)
                                                          : launch_attn<128, 64, false, false>(tm_q, tm_pool_k, tm_pool_v, sk, sv, c, a, grid, st);
  if (c.D == 64 && c.PT == 128) return a.seg_tiles > 0 ? launch_attn<64, 128, false, true>(tm_q, tm_pool_k, tm_pool_v, sk, sv, c, a, grid, st)
                                                          : launch_attn<64, 128, false, false>(tm_q, tm_pool_k, tm_pool_v, sk, sv, c, a, grid, st);
  if (c.D == 64 && c.PT == 64) return a.seg_tiles > 0 ? launch_attn<64, 64, false, true>(tm_q, tm_pool_k, tm_pool_v, sk, sv, c, a, grid, st)
                                                          : launch_attn<64, 64, false, false>(tm_q, tm_pool_k, tm_pool_v, sk, sv, c, a, grid, st);
  return FASTAR_ERR_UNSUPPORTED_SHAPE;
}

int launch_attention_gather(const CacheView& c, const CUtensorMap& tm_q, const AttnArgs& a, cudaStream_t st) {
  // one key tile of 64: a kernel of its own, which keeps the tile and streams the queries (12 x 4680 queries, 64 kept: 34.2 -> 11.5 us)
  if (a.keep <= 64) return launch_attention_prompt64(c, tm_q, a, st);
  const dim3 grid((a.rows_per_frame + 127) / 128, c.H, a.n_frames);
  if (c.D == 128) return launch_attn<128, 128, true, false>(tm_q, tm_q, tm_q, tm_q, tm_q, c, a, grid, st);
  return launch_attn<64, 128, true, false>(tm_q, tm_q, tm_q, tm_q, tm_q, c, a, grid, st);
}

}  // namespace fastar
