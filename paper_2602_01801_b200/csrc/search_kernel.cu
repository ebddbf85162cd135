// TempCache's correspondence search (paper Section 5.2: the top-1 cached key of every new key) as one persistent kernel:
// scores of 256 new keys x 128 cached keys on tcgen05, row arg-max fused, the score matrix never leaves the SM.
//
// What bounds it is the shared-memory read path.  A 128 x 128 x 16 MMA with both operands in shared memory reads 8 KB in
// the 64 cycles it takes, all the path can deliver, and the MMAs have priority: eight of them take 573 cycles instead
// of 512 while the whole SM gets 32 128-bit loads through (the arg-max wants 1/|k_j| of every column: 128 such loads).
// With A in tensor memory the same eight MMAs take 513 cycles and 120 loads fit beside them.  Hence:
//   - the new keys are moved to tensor memory once per work segment (256 rows = two A tiles) and an MMA reads only the
//     cached keys from shared memory; a key tile is fetched once for both A tiles;
//   - scores are read from tensor memory in the 16 x 256-bit fragment shape: a thread holds 16 columns of four rows and
//     needs 16 factors for its 64 scores, not 64 (a 128-bit load that all lanes share still returns 512 bytes);
//   - the factors arrive by a bulk copy on the key tile's barrier (no staging by threads, no barrier of their own for the epilogue warps);
//   - two groups of eight epilogue warps, one per A tile, work half a tile period apart, so that the tensor-memory reads of
//     one overlap the arithmetic of the other; three accumulators rotate between them.
// Work is dealt by length, not by CTA: one CTA per SM, all (head, row unit, key tile) work on a line that is cut into
// equal pieces, so there is no last wave.  The line is walked in `waves` whose keys fit L2 together: the pieces
// of one wave lie in the same few heads, which the SMs then read from L2 instead of each streaming its own head.
// Pieces of the same rows meet in a 64-bit atomicMax on (ordered score, ~slot): ties go to the lowest slot.
//
// Measured (B200, kernel time, before = CTAs of 128 rows or CTA pairs with both operands in shared memory): 12 heads, d = 128,
// 4 680 new against 28 080 cached keys 370 -> 308 us (0.80 of the measured bf16 peak); 40 heads, 10 800 against 64 800: 5.78 ->
// 5.29 ms (1.36 PFLOP/s: the power limit holds the clock at 1.55 GHz there); 8 heads, d = 64, 4 096 against 16 384: 138 ->
// 103 us.  A key tile takes an SM 1 380-1 460 cycles, its 16 MMAs 1 025.  Since then: asking for scores, factors and maxima together 328 -> 303
// and 100 -> 93; the rows' maxima side by side 303 -> 293 and 93.4 -> 91.4; no slots for maxima that no match can come of 292 -> 293 and
// 91.9 -> 89.1, by the query probe (12 x 1560 on 14 040) 64.4 -> 62.8.  What was slower: working out scores only where a row's largest dot
// product times the largest factor of the columns reaches its maximum (308 and 106: some row of a warp's 32 does in most tiles), a tile's halves
// taking turns in the registers, loads a half ahead (322 and 103), asking for the next accumulator's barrier early (1 to 3 %).
#include "common.h"
#include "ptx.cuh"

namespace fastar {

namespace {

// what a score is: cosine (factor 1/|k_j|), or plain dot product (query probe)
enum { SCORE_COS = 0, SCORE_DOT = 1 };

constexpr int kThreads = 640;                 // warps 0-15 epilogue, 16 TMA producer, 17 TMEM allocation + MMA issue, 18-19 none
constexpr int kEpiWarps = 16, kProducer = 16, kMma = 17;
// Registers a thread: 640 x 96 at launch, dealt anew by role (16 x 32 x 104 + 4 x 32 x 64 = 640 x 96)
constexpr int kEpiRegs = 104, kIssueRegs = 64;
constexpr int kAccs = 3;                      // accumulators of 128 TMEM columns
constexpr int kAcol = kAccs * 128;            // first TMEM column of the A tiles
constexpr int kChunk = 128 * 128;             // 128 rows x 128 bytes, one swizzled box
constexpr int kMaxHeads = 1024;               // per launch (the tile counts of the heads are kept in shared memory)
constexpr int kWaveBytes = 96 << 20;          // keys that one wave touches (126 MB of L2)

// One segment: rows [256 u, 256 u + 256) of head h against key tiles [t0, t1).
struct Seg {
  int h, u, t0, t1;                           // h < 0: no more work
  int len, two;                               // live slots of the head; 1: both A tiles hold rows
};

template <int D, int SCORE>
struct Cfg {
  static constexpr int nkc = D / 64;                               // 128-byte chunks per row
  static constexpr int tile_bytes = nkc * kChunk;
  static constexpr int stages = 8 / nkc;                           // 128 KB of key tiles
  static constexpr int factors = 2 * stages;                       // ring of factor rows (see the producer)
  static constexpr int a_cols = nkc * 32;                          // TMEM columns of one A tile
  static constexpr int a_off = 0;                                  // staging of the two A tiles
  static constexpr int ring_off = 2 * tile_bytes;
  static constexpr int rn_off = ring_off + stages * tile_bytes;
  static constexpr int pre_off = rn_off + (SCORE == SCORE_COS ? factors * 512 : 0);
  static constexpr int len_off = pre_off + (kMaxHeads + 8) * 4;    // live slots of the heads
  static constexpr int row_off = len_off + kMaxHeads * 4;    // [3][256] running row maxima of the last segments
  static constexpr int seg_off = row_off + 3 * 256 * 4;            // [2] Seg
  static constexpr int bar_off = seg_off + 64;
  static constexpr int total = bar_off + 512;
};

// The scores of one accumulator that a thread holds: x[half][4 i + 2 e + c] is row 16 half + 8 e + lane / 4 of the warp's 32
// rows, column 8 i + 2 (lane & 3) + c of its 64.
struct Frag {
  uint32_t x[2][32];
};
template <int HALF, int E>
__device__ __forceinline__ float row_max(const Frag& f) {
  float m[5];
#pragma unroll
  for (int k = 0; k < 5; ++k) {                      // values 3 k .. 3 k + 2 of the row's sixteen
    float y[3];
#pragma unroll
    for (int q = 0; q < 3; ++q) y[q] = __uint_as_float(f.x[HALF][4 * ((3 * k + q) >> 1) + 2 * E + ((3 * k + q) & 1)]);
    m[k] = fmax3(y[0], y[1], y[2]);
  }
  return fmax3(fmax3(m[0], m[1], m[2]), fmaxf(m[3], m[4]), __uint_as_float(f.x[HALF][28 + 2 * E + 1]));
}
// The maximum cm of a thread's columns of one of its rows reaches what the row asks for: the slot of it is looked for, the lowest column.
// row_best: what a slot has to reach to matter, or the row's maximum over all threads that share it if that is more, in shared memory (-inf or
// positive), `seen` what was read of it; a maximum below it is another thread's to report, an equal one may be the lower slot.
template <int HALF, int E>
__device__ __forceinline__ void take_max(const Frag& f, float cm, int jb, int* row_best, float seen, float best, int& best_j) {
  if (cm > best && cm >= seen) {
    if (cm > 0.f) atomicMax(row_best, __float_as_int(cm));
    int idx[4];                                      // four short chains, the lowest columns in idx[0]
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      idx[k] = 64;
#pragma unroll
      for (int q = 4 * k + 3; q >= 4 * k; --q)
        idx[k] = (__uint_as_float(f.x[HALF][4 * (q >> 1) + 2 * E + (q & 1)]) == cm) ? 8 * (q >> 1) + (q & 1) : idx[k];
    }
    best_j = jb + min(min(idx[0], idx[1]), min(idx[2], idx[3]));
  }
}

// This CTA's segments.  pre[h] = key tiles of the heads before h.  The line counts a key tile once per row unit: the last unit
// of a head may hold one A tile only, but a key tile costs it as much (4680 rows: 0.90 against 0.92 us).
struct SegIter {
  const int* pre;
  int row_tiles, units, waves, wave, h, x, x1;
  int64_t total;
  __device__ __forceinline__ void init(const int* pre_s, int heads, int n, int64_t bytes_per_tile) {
    pre = pre_s;
    row_tiles = (n + 127) >> 7;
    const int tiles = pre[heads];
    units = (row_tiles + 1) >> 1;
    total = static_cast<int64_t>(tiles) * units;
    // enough waves for L2, but no piece under 16 tiles
    const int64_t want = (tiles * bytes_per_tile + kWaveBytes - 1) / kWaveBytes, most = total / (16 * static_cast<int64_t>(gridDim.x));
    waves = static_cast<int>(max(static_cast<int64_t>(1), min(want, most)));
    wave = -1;
    h = 0;
    x = x1 = 0;
  }
  __device__ __forceinline__ bool next(Seg& s) {
    while (true) {
      while (x >= x1) {
        if (++wave >= waves) return false;
        const int64_t pieces = static_cast<int64_t>(waves) * gridDim.x, i = static_cast<int64_t>(wave) * gridDim.x + blockIdx.x;
        x = static_cast<int>(total * i / pieces);
        x1 = static_cast<int>(total * (i + 1) / pieces);
      }
      while (x >= pre[h + 1] * units) ++h;              // x < total, so there is such a head
      const int tiles = pre[h + 1] - pre[h], off = x - pre[h] * units;
      s.h = h;
      s.u = off / tiles;
      s.two = row_tiles - 2 * s.u >= 2 ? 1 : 0;
      s.t0 = off - s.u * tiles;
      s.t1 = min(tiles, s.t0 + (x1 - x));
      x += s.t1 - s.t0;
      return true;
    }
  }
};

}  // namespace

template <int D, int SCORE>
__global__ void __launch_bounds__(kThreads, 1)
search_kernel(const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_b, const CacheView c, int n, int h0,
              int heads) {
  using SM = Cfg<D, SCORE>;
  constexpr int S = SM::stages, R = SM::factors;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const uint32_t sbase = smem_u32(smem_raw);
  if (sbase & 1023u) {                  // swizzled tiles need 1024-byte alignment; uniform for the CTA
    if (threadIdx.x == 0) record_status(c.status, FASTAR_ERR_CUDA);
    return;
  }
  const uint32_t a_s = sbase + SM::a_off, ring_s = sbase + SM::ring_off, rn_s = sbase + SM::rn_off, bar = sbase + SM::bar_off;
  int* pre = reinterpret_cast<int*>(smem_raw + SM::pre_off);
  int* len_s = reinterpret_cast<int*>(smem_raw + SM::len_off);
  const uint32_t bar_full = bar;                          // [S]
  const uint32_t bar_empty = bar_full + 8 * S;            // [S]
  const uint32_t bar_tfull = bar_empty + 8 * S;           // [kAccs] the MMAs' commit, and the issuing warp (the factors have landed)
  const uint32_t bar_tempty = bar_tfull + 8 * kAccs;      // [kAccs]
  const uint32_t bar_afull = bar_tempty + 8 * kAccs;      // [1] segment described, A tiles landed in the staging area
  const uint32_t bar_atm = bar_afull + 8;                 // [1] A tiles copied to tensor memory (staging free again)
  constexpr int kBars = 2 * S + 2 * kAccs + 2;
  static_assert(kBars * 8 + 8 <= 512, "barrier area");
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem_raw + SM::bar_off + kBars * 8);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem_raw + SM::bar_off + kBars * 8 + 4);

  const int warp = warp_index(), lane = threadIdx.x & 31;
  if (threadIdx.x < kBars) {
    const int b = threadIdx.x, te = 2 * S + kAccs;        // tempty collects a group's warps, atm all of them
    mbar_init(bar + 8 * b, b >= te && b < te + kAccs ? kEpiWarps / 2 : b == kBars - 1 ? kEpiWarps : b >= 2 * S && b < te ? 2 : 1);
    fence_mbar_init();
  }
  if (threadIdx.x == 0) *abort_flag = 0;
  if (warp == kMma) {
    tmem_alloc(smem_u32(tmem_slot), 512);
    tmem_relinquish();
  }
  if (warp == kProducer) {                                // prefix sum of the heads' key tiles
    if (lane == 0) {
      tma_prefetch_desc(&tm_a);
      tma_prefetch_desc(&tm_b);
      pre[0] = 0;
    }
    chain_wait();
    int run = 0;
    for (int b = 0; b < heads; b += 32) {
      const int len = b + lane < heads ? c.len[h0 + b + lane] : 0;
      if (b + lane < heads) len_s[b + lane] = len;
      int v = (len + 127) >> 7;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
      }
      if (b + lane < heads) pre[b + lane + 1] = run + v;
      run += __shfl_sync(0xffffffffu, v, 31);
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  chain_wait();
  Seg* seg_s = reinterpret_cast<Seg*>(smem_raw + SM::seg_off);

  if (warp >= kEpiWarps) {
    setmaxnreg_dec<kIssueRegs>();                  // one instruction for the whole warpgroup (18 and 19 have no other task)
    if (warp == kProducer) {
      // -------------------------------------------------------------------- TMA producer
      bool ok = true;
      int it = 0, nseg = 0;
      const int pages_per_tile = 128 / c.PT;                // 1 or 2
      SegIter iter;
      iter.init(pre, heads, n, SM::tile_bytes);
      Seg sg;
      for (bool more = true; more;) {
        more = iter.next(sg);
        // The others read segment nseg from slot nseg & 1.  Once every epilogue warp has taken segment nseg - 1 (it waits
        // for that here, the staging area must be free too) nobody needs segment nseg - 2 any more.
        if (nseg > 0) ok = mbar_wait_warp<kIssueWaitHintNs>(bar_atm, (nseg - 1) & 1, abort_flag, c.status);
        if (!ok) break;
        const int h = h0 + sg.h;
        if (lane == 0) {
          sg.len = more ? len_s[sg.h] : 0;
          if (!more) sg.h = -1;
          seg_s[nseg & 1] = sg;
          if (more) {
            const int na = sg.two ? 2 : 1;
            mbar_arrive_expect_tx(bar_afull, na * SM::tile_bytes);
            for (int a = 0; a < na; ++a)
              for (int kc = 0; kc < SM::nkc; ++kc)
                tma_load_3d(a_s + a * SM::tile_bytes + kc * kChunk, &tm_a, bar_afull, kc * 64, sg.u * 256 + a * 128, h);
          } else {
            mbar_arrive(bar_afull);
          }
        }
        ++nseg;
        if (!more) break;
        // page ids of 32 tiles with one coalesced load, so that no global load sits between two copies
        const int32_t* pt_h = c.page_table + static_cast<int64_t>(h) * c.CAPB;
        int pg0 = 0, pg1 = 0;
        for (int t = sg.t0; t < sg.t1; ++t, ++it) {
          const int q = (t - sg.t0) & 31;
          if (q == 0 && t + lane < sg.t1) {
            pg0 = FASTAR_IDX(pt_h[(t + lane) * pages_per_tile], c.pool_pages, c.status);
            pg1 = pages_per_tile == 2 ? FASTAR_IDX(pt_h[(t + lane) * pages_per_tile + 1], c.pool_pages, c.status) : 0;
          }
          const int page0 = __shfl_sync(0xffffffffu, pg0, q), page1 = __shfl_sync(0xffffffffu, pg1, q);
          const int st = it % S;
          ok = mbar_wait_warp<kIssueWaitHintNs>(bar_empty + 8 * st, ((it / S) & 1) ^ 1, abort_flag, c.status);
          if (!ok) break;
          if (lane == 0) {
            const uint32_t dst = ring_s + st * SM::tile_bytes;
            mbar_arrive_expect_tx(bar_full + 8 * st, SM::tile_bytes + (SCORE == SCORE_COS ? 512 : 0));
            for (int kc = 0; kc < SM::nkc; ++kc) {
              tma_load_3d(dst + kc * kChunk, &tm_b, bar_full + 8 * st, kc * 64, 0, page0);
              if (pages_per_tile == 2) tma_load_3d(dst + kc * kChunk + c.PT * 128, &tm_b, bar_full + 8 * st, kc * 64, 0, page1);
            }
            if (SCORE == SCORE_COS) {
              // Slot it % R was last read by the epilogue of tile it - R.  The key stage waited for above was freed by the
              // MMAs of tile it - S = it - R + S, which needed accumulators that both groups had read after they had
              // finished tile it - R + S - 4 at least, S >= 4.
              const int fr = it % R;
              bulk_load_1d(rn_s + fr * 512, c.rnorm + static_cast<int64_t>(h) * c.CAP + t * 128, 512, bar_full + 8 * st);
            }
          }
        }
        if (!ok) break;
      }
      // what is still in flight must land before the CTA may exit (normally all of it has: the MMAs consumed it)
      if (lane == 0) {
        for (int k = max(0, it - S); k < it; ++k) mbar_wait(bar_full + 8 * (k % S), (k / S) & 1, abort_flag, c.status);
        if (nseg > 0) mbar_wait(bar_afull, (nseg - 1) & 1, abort_flag, c.status);
      }
    } else if (warp == kMma) {
      // -------------------------------------------------------------------- MMA issue
      const uint32_t lead = elect_lane();
      constexpr uint32_t idesc = make_idesc_bf16(128, 128, 0);
      bool ok = true;
      int it = 0, b = 0, bph = 0;
      for (int nseg = 0;; ++nseg) {
        ok = mbar_wait_warp<kIssueWaitHintNs>(bar_atm, nseg & 1, abort_flag, c.status);
        if (!ok) break;
        const Seg sg = seg_s[nseg & 1];
        if (sg.h < 0) break;
        // A barrier answers after about a hundred cycles (the MMAs' operand reads come first on the shared-memory path), and
        // the tensor core holds only a few issued MMAs: the barriers of the next accumulator are asked in the middle of
        // the current one's MMAs, and waited for only when the answer was no.
        const int n_acc = (sg.t1 - sg.t0) * (sg.two ? 2 : 1);
        int a = 0;
        bool ready = false;
        for (int k = 0; k < n_acc; ++k) {
          const int st = it % S;
          if (!ready) {
            if (a == 0) ok = mbar_wait_warp<kIssueWaitHintNs>(bar_full + 8 * st, (it / S) & 1, abort_flag, c.status);
            if (ok) ok = mbar_wait_warp<kIssueWaitHintNs>(bar_tempty + 8 * b, bph ^ 1, abort_flag, c.status);
            if (!ok) break;
          }
          tc_fence_after();
          const uint32_t bt = ring_s + st * SM::tile_bytes, d = tmem + b * 128, at = tmem + kAcol + a * SM::a_cols;
          auto issue = [&](int k0) {
#pragma unroll
            for (int kk = k0; kk < k0 + SM::nkc * 2; ++kk) {
              const uint64_t bd = make_smem_desc(bt + (kk >> 2) * kChunk + (kk & 3) * 32, 16, 1024);
              umma_ts(d, at + kk * 8, bd, idesc, kk != 0, lead);
            }
          };
          issue(0);
          const uint32_t tfull = bar_tfull + 8 * b, empty = bar_empty + 8 * st;
          const bool last = a == sg.two;                   // last A tile of this key tile
          if (++b == kAccs) { b = 0; bph ^= 1; }
          if (last) ++it;
          a = last ? 0 : 1;
          ready = k + 1 < n_acc && mbar_test_wait(bar_tempty + 8 * b, bph ^ 1) &&
                  (!last || mbar_test_wait(bar_full + 8 * (it % S), (it / S) & 1));
          ready = __all_sync(0xffffffffu, ready);
          issue(SM::nkc * 2);
          umma_commit(tfull, lead);
          if (lead) mbar_arrive(tfull);                    // what this warp has seen land (the factors) is there for the waiting warps
          if (last) umma_commit(empty, lead);
        }
        if (!ok) break;
      }
    }
  } else {
    // -------------------------------------------------------------------- epilogue (512 threads)
    setmaxnreg_inc<kEpiRegs>();
    const int grp = warp >> 3;                     // A tile of this warp
    const int cg = (warp >> 2) & 1;                // columns 64 cg ... 64 cg + 63 of every tile
    const int r = (warp & 3) * 32 + lane;          // TMEM lane of the A copy
    const int rq = (warp & 3) * 32 + (lane >> 2);  // this thread's rows: rq, rq + 8, rq + 16, rq + 24
    const uint32_t lane_addr = static_cast<uint32_t>((warp & 3) * 32) << 16;
    bool ok = true;
    int it = 0;                                    // key tiles so far
    int b = grp, bph = 0;                          // this group's next accumulator, and its barriers' phase
    int* row_s = reinterpret_cast<int*>(smem_raw + SM::row_off);
    if (threadIdx.x < 256) row_s[threadIdx.x] = __float_as_int(-INFINITY);
    named_barrier_sync(1, kEpiWarps * 32);
    int slot3 = 0;                                 // segment number modulo 3
    bool skipped = false;
    for (int nseg = 0;; ++nseg) {
      // The A tiles go to tensor memory: a warp copies one 128-byte chunk of the rows of its lanes.  The MMAs that read the
      // previous one are complete (this group has seen its last accumulator of the segment before).
      ok = mbar_wait_warp(bar_afull, nseg & 1, abort_flag, c.status);
      if (!ok) break;
      const Seg sg = seg_s[nseg & 1];
      // The threads of a row share its running maximum, so that one looks for the column of a new maximum only when the row's
      // other columns do not beat it already.  Warps are at most one segment apart: three generations.
      int* best_s = row_s + slot3 * 256 + grp * 128 + ((warp & 3) * 8 + (lane >> 2)) * 4;      // a thread's four rows side by side
      slot3 = slot3 == 2 ? 0 : slot3 + 1;
      if (cg == 0) row_s[slot3 * 256 + grp * 128 + r] = __float_as_int(-INFINITY);
      if (sg.h < 0) {
        mbar_arrive_warp(bar_atm);
        break;
      }
      const int h = h0 + sg.h;
      const bool mine = grp == 0 || sg.two;
      {
        if (mine && cg < SM::nkc) {
          uint32_t regs[32];
          const uint32_t src = a_s + grp * SM::tile_bytes + cg * kChunk + r * 128;
#pragma unroll
          for (int ch = 0; ch < 8; ++ch)
            asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                         : "=r"(regs[4 * ch]), "=r"(regs[4 * ch + 1]), "=r"(regs[4 * ch + 2]), "=r"(regs[4 * ch + 3])
                         : "r"(src + ((ch ^ (r & 7)) << 4))
                         : "memory");
          tmem_st32(tmem + lane_addr + kAcol + grp * SM::a_cols + cg * 32, regs);
          tmem_wait_st();
        }
        tc_fence_before();
        mbar_arrive_warp(bar_atm);
      }
      // A group that sat a segment out may be ahead of the accumulators by more than one phase of their barriers: it waits until
      // the other group has come here too (all accumulators of the segments before are complete then).
      if (skipped && mine) ok = mbar_wait_warp(bar_atm, nseg & 1, abort_flag, c.status);
      if (!ok) break;
      skipped = !mine;
      const int ntl = sg.t1 - sg.t0;
      // accumulators go round by three; the groups take turns, or the first has them all
      auto advance = [&](int n) {
        b += n;
        if (b >= kAccs) { b -= kAccs; bph ^= 1; }
      };
      if (!mine) {                                 // a unit of one A tile: nothing for the second group
        it += ntl;
        const int on = b + ntl;
        bph ^= (on / kAccs) & 1;
        b = on % kAccs;
        continue;
      }
      const int row0 = sg.u * 256 + grp * 128 + rq;
      const float* rn_new = c.rnorm_new + static_cast<int64_t>(h) * c.max_tokens;
      float best[4];
      int bj[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        best[q] = -INFINITY;
        bj[q] = -1;
      }
      // What a score must reach for its slot to matter (it lacks the row's own factor): the row's maximum starts there, so that a score that
      // finds no match, which most do, is a maximum in a register and nothing else.  Rows past the end have nothing to look for.
      float rn_row[4];                             // (fetched again when the segment is through)
      auto needed = [&](int q) {
        rn_row[q] = SCORE == SCORE_COS && row0 + 8 * q < n ? rn_new[row0 + 8 * q] : 1.f;
        const float need = SCORE == SCORE_COS && rn_row[q] > 0.f ? c.search_floor / rn_row[q] : -INFINITY;
        return row0 + 8 * q >= n ? INFINITY : need > 0.f ? need : -INFINITY;
      };
      if ((lane & 3) == 0)
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float need = needed(q);
          if (need > 0.f) atomicMax(best_s + q, __float_as_int(need));
        }
      __syncwarp();
      for (int t = sg.t0; t < sg.t1; ++t, ++it) {
        Frag f;
        ok = mbar_wait_warp(bar_tfull + 8 * b, bph, abort_flag, c.status);
        if (!ok) break;                            // warp-uniform: TMEM loads are warp-collective
        tc_fence_after();
        // The scores and the rows' maxima are asked for together (one after the other they took half of a tile's time: 8 heads, d = 64,
        // 4 096 new against 16 384 keys 100.1 -> 92.6 us, 12 x 4680, d = 128, 328 -> 320).
        tmem_ld_frag(tmem + lane_addr + b * 128 + cg * 64, f.x[0]);
        tmem_ld_frag(tmem + lane_addr + (16u << 16) + b * 128 + cg * 64, f.x[1]);
        float2 rn[8];
        if (SCORE == SCORE_COS) {
          const float2* rn2 = reinterpret_cast<const float2*>(smem_raw + SM::rn_off + (it % R) * 512 + cg * 256 + (lane & 3) * 8);
#pragma unroll
          for (int i = 0; i < 8; ++i) rn[i] = rn2[4 * i];
        }
        int seen_w[4];
        asm volatile("ld.volatile.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(seen_w[0]), "=r"(seen_w[1]), "=r"(seen_w[2]), "=r"(seen_w[3]) : "r"(smem_u32(best_s)));
        tmem_wait_ld();
        tc_fence_before();
        mbar_arrive_warp(bar_tempty + 8 * b);      // the scores are in registers: release the accumulator
        advance(sg.two ? 2 : 1);
        if (SCORE == SCORE_COS) {
#pragma unroll
          for (int i = 0; i < 8; ++i) {
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
              scale2(f.x[hf][4 * i], f.x[hf][4 * i + 1], rn[i]);
              scale2(f.x[hf][4 * i + 2], f.x[hf][4 * i + 3], rn[i]);
            }
          }
        }
        const int jb = t * 128 + cg * 64 + 2 * (lane & 3), valid = sg.len - jb;
        if (sg.len - t * 128 < 128) {              // only the last tile of a cache has columns to mask
#pragma unroll
          for (int i = 0; i < 16; ++i)
            if (8 * (i >> 1) + (i & 1) >= valid)
#pragma unroll
              for (int hf = 0; hf < 2; ++hf)
                f.x[hf][4 * (i >> 1) + (i & 1)] = f.x[hf][4 * (i >> 1) + 2 + (i & 1)] = __float_as_uint(-INFINITY);
        }
        const float m0 = row_max<0, 0>(f), m1 = row_max<0, 1>(f), m2 = row_max<1, 0>(f), m3 = row_max<1, 1>(f);
        const float s0 = __int_as_float(seen_w[0]), s1 = __int_as_float(seen_w[1]), s2 = __int_as_float(seen_w[2]), s3 = __int_as_float(seen_w[3]);
        if (m0 >= s0 || m1 >= s1 || m2 >= s2 || m3 >= s3) {
          take_max<0, 0>(f, m0, jb, best_s + 0, s0, best[0], bj[0]);
          take_max<0, 1>(f, m1, jb, best_s + 1, s1, best[1], bj[1]);
          take_max<1, 0>(f, m2, jb, best_s + 2, s2, best[2], bj[2]);
          take_max<1, 1>(f, m3, jb, best_s + 3, s3, best[3], bj[3]);
        }
        best[0] = fmaxf(best[0], m0);
        best[1] = fmaxf(best[1], m1);
        best[2] = fmaxf(best[2], m2);
        best[3] = fmaxf(best[3], m3);
      }
      if (!ok) break;
      // A row that has found nothing has its maximum reported by one thread of a quad, with the segment's first slot in its slot's place.
      unsigned long long* out = c.best + static_cast<int64_t>(h) * c.max_tokens;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int row = row0 + 8 * q;
        const float need = needed(q), row_top = __int_as_float(*static_cast<volatile int*>(best_s + q));
        float top = fmaxf(best[q], __shfl_xor_sync(0xffffffffu, best[q], 1));
        top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, 2));
        const bool found = bj[q] >= 0 && best[q] >= row_top, none = need > 0.f && row_top == need && (lane & 3) == 0 && top > -INFINITY && top < need;
        if (row >= n || !(found || none)) continue;
        const float score = found ? best[q] : top, sim = SCORE == SCORE_COS ? score * rn_row[q] : score;
        atomicMax(out + row, (static_cast<unsigned long long>(float_to_ordered(sim)) << 32) |
                                 static_cast<unsigned long long>(0xFFFFFFFFu - static_cast<uint32_t>(found ? bj[q] : sg.t0 * 128)));
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == kMma) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

template <int D, int SCORE>
static int launch_search_t(const CacheView& c, const CUtensorMap& tm_a, const CUtensorMap& tm_b, int n, cudaStream_t st) {
  using SM = Cfg<D, SCORE>;
  auto kern = search_kernel<D, SCORE>;
  const int cfg = ensure_dynamic_smem(reinterpret_cast<const void*>(kern), SM::total);
  if (cfg != FASTAR_OK) return cfg;
  int dev = 0, sm_count = 148, launched = 0;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sm_count, cudaDevAttrMultiProcessorCount, dev);
  for (int h0 = 0; h0 < c.H; h0 += kMaxHeads) {
    const int heads = min(kMaxHeads, c.H - h0);
    // one CTA per SM; fewer only when the whole search has fewer (row unit, key tile) pairs than that
    const int64_t pairs = static_cast<int64_t>(heads) * ((n + 255) / 256) * (c.CAP / 128);
    launch_chained(kern, static_cast<int>(pairs < sm_count ? pairs : sm_count), kThreads, SM::total, st, tm_a, tm_b, c, n, h0, heads);
    if (cudaGetLastError() != cudaSuccess) return FASTAR_ERR_CUDA;
    ++launched;
  }
  return launched;
}

// T1 on the bf16 keys: cosine, or plain dot products (c.raw_dot: rows of A are the probe rows).
int launch_t1_search(const CacheView& c, const CUtensorMap& tm_a, const CUtensorMap& tm_pool_k, int n, cudaStream_t st) {
  if (c.D == 128)
    return c.raw_dot ? launch_search_t<128, SCORE_DOT>(c, tm_a, tm_pool_k, n, st) : launch_search_t<128, SCORE_COS>(c, tm_a, tm_pool_k, n, st);
  return c.raw_dot ? launch_search_t<64, SCORE_DOT>(c, tm_a, tm_pool_k, n, st) : launch_search_t<64, SCORE_COS>(c, tm_a, tm_pool_k, n, st);
}

}  // namespace fastar
