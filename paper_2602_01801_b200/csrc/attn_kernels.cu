// Candidate-set attention on tcgen05 / TMEM (paper Section 5.1: attention over N(q); Lemma 1:
// logits shifted by log m, values are group means):
//   paged  : AnnSA's selected-block attention and the dense Eq. 1 baseline.  A query block attends
//            to the key blocks listed in `sel`; one key block = one cache page = one TMA box, looked
//            up through the page table.
//   gather : AnnCA's attention over the kept prompt tokens of the query's frame; rows of K_p / V_p
//            are gathered by index with 16-byte copies into the same swizzled tile layout.
//
// One CTA per SM takes (head, query block) items in turn, 128 query rows each (TMEM lanes).  The key tiles are cut into sub-tiles of 64
// keys, which are dealt in turn to four soft-max groups of four warps (index t, group t % 4): while one is in its exponentials the
// others load, shift and wait.
//   S    = Q K_j^T                  tcgen05.mma, SMEM x SMEM -> TMEM, a whole key tile
//   P_t  = exp2(S*scale + log2 m - m)       registers -> bf16 -> TMEM
//   O   += P_t V_t                  tcgen05.mma, TMEM x SMEM: V is the MN-major operand straight from its [key][d] page
// What bounds it: 128 x 128 exponentials are 1 024 cycles of an SM's special-function units, the two MMAs of the tile another
// 1 060 of the tensor core, and all of them want the shared-memory read path, which the operand reads of an MMA take first (a
// barrier or a load answers after some 300 cycles meanwhile).  So little goes through shared memory, and nothing waits in line:
//   - P goes through tensor memory (with P in shared memory the MMAs of a tile saturate the read path), beside S and not over
//     it, so that Q K^T of a group's next sub-tile runs while this one is in its exponentials;
//   - that leaves room for one O, so all groups use one running maximum per row.  The four warps that own the same rows hand it
//     on from sub-tile to sub-tile by named barriers.  It is raised lazily, only when a logit exceeds it by more than 24 binary orders
//     (who raises it rescales O: P V of all earlier sub-tiles done, that of this one waiting for its P).  A raise stops all groups
//     for some 4 000 cycles.  Kernel time with a limit of 8 / 12 / 16 / 24 / 64: 12 heads x 4 680 queries on 32 of 220 blocks 124 /
//     144 / 142 / 110 / 110 us, the denoising step 234 / 248 / 240 / 217 / 218, 8 heads on all 16 384 keys 254 / 257 / 253 / 240 /
//     240: keys of a query's own cluster stand some 13 (d = 128) above the first sub-tile's;
//   - the row sums add up the probabilities as rounded to bf16, so that they cancel in a row that one key dominates;
//   - the soft-max warps hold a sub-tile in the 16 x 256-bit fragment shape, four rows x 16 columns a thread: a thread reads 16
//     biases, not 64, and a warp still has its rows to itself;
//   - Q K^T and P V are issued by two warps, so that a barrier that one of them waits for does not hold back the other, with running
//     stage numbers and descriptors: what they do between two barriers is on the way of every sub-tile;
//   - a sub-tile's logits, its biases and the running maximum are asked for together, because each of them takes hundreds of cycles while
//     Q K^T reads both operands from shared memory (eight 64-bit loads by a warp: 203 cycles, 850-2 600 beside such MMAs).  With the two
//     points: denoising step of 12 heads 313 -> 298 us, 8 heads, d = 64, 64 of 1 024 blocks 146 -> 142;
//   - items that do not fill the last round of the SMs are cut by key tiles (see launch_attn), and the soft-max loop is as large as
//     an SM's instruction caches bear (stalls for instructions: a twentieth of a warp's time, and a sixth with a little more code in the
//     kernel), so the cut is a variant of its own;
//   - items whose logits a bound keeps near the first sub-tile's need no maximum at all (see kFlatMin): the loop for them is what the
//     arithmetic needs, some 270 instructions, and the tensor core and the exponentials' units are at 0.76 and 0.67 of the time at d = 128, 0.40
//     and 0.71 at 64;
//   - the CTA stays for its items, and the copies and Q K^T run ahead into the next one, whose first logits are there when the
//     output of the last has left.
// TMEM columns: S 4 x 64, P 4 x 32, O D; with key tiles of 64: S 3 x 64, P, O and Q D / 2 (AttnSmem::QT).  K and V tiles have a TMA ring
// each.
// Measured (B200, kernel time; two groups with whole tiles, a CTA per item, a limit of 8 -> this): 12 heads, d = 128, 4 680 queries on
// 32 of 224 blocks 120.5 -> 105.4 us (0.68 of the measured bf16 peak); the same with the chunk's 4 680 keys beside 241 -> 218 us; 8
// heads, 4 096 queries on all 16 384 keys 275 -> 246 us (108 of 148 CTAs have two items); d = 64, 64 of 1 024 blocks 142 -> 125 us,
// 16 of 160 blocks 49 -> 39.5 us.  With flat items: the first three 99 -> 89, 194 -> 174 and 226 -> 199 us, the last two 118 -> 95 and
// 37.8 -> 32.1.  Row sums by a warp-level product with ones instead of adds: 311 us for 242 (it takes the tensor
// core); sums of the unrounded probabilities: 4 % faster, not as exact.
// Warp roles: warps 0-15 soft-max groups 0-3, 16 copies Q and K (TMA or gather), 17 Q K^T, 18 P V, 19 copies V.
#include "bound.cuh"
#include "common.h"
#include "ptx.cuh"

#include <type_traits>

namespace fastar {

constexpr int kQChunk = 128 * 128;   // bytes of one 128-row x 64-column bf16 chunk
constexpr int kAttnThreads = 640;
constexpr int kGroups = 4;           // soft-max groups of four warps
constexpr int kSoftWarps = 4 * kGroups, kKeyWarp = 16, kQkWarp = 17, kPvWarp = 18, kValueWarp = 19;
// Registers a thread: 640 x 96 at launch, dealt anew by role (16 x 32 x 112 + 4 x 32 x 32 = 640 x 96)
constexpr int kSoftRegs = 112, kIssueRegs = 32;

// shared memory by 32-bit address
__device__ __forceinline__ float2 lds2(uint32_t addr) {
  float2 v;
  asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr));
  return v;
}
__device__ __forceinline__ float4 lds4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr));
  return v;
}

// Probabilities are taken relative to kHead binary orders above the running maximum and the maximum is raised when one would exceed
// 2^kTop, that is when a logit exceeds it by more than kHead + kTop = 24.  So none is above 2^8, and the sums of P V stay in range
// for values up to 2^119 / keys.  What the code calls the maximum, and the warps hand on, is that reference.
constexpr float kHead = 16.f, kTop = 8.f;

// What a cut costs, in times of a tile of BKT keys (0.60 us with 128, 0.32 with 64): a part's way through memory, which is longer by `part`
// for every part there is, adding one up, another stop of a CTA; and the share of the whole that has to be saved (see launch_attn).
template <int BKT>
struct CutCost {
  static constexpr float store = BKT == 64 ? 6.2f : 3.2f, part = BKT == 64 ? 0.066f : 0.029f, add = BKT == 64 ? 1.45f : 0.8f, stop = BKT == 64 ? 14.f : 8.3f;
  static constexpr float gain = 0.05f;
};

__device__ __forceinline__ void sts4(uint32_t addr, const float (&v)[4]) {
  asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]) : "memory");
}
__device__ __forceinline__ float lds1(uint32_t addr) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr));
  return v;
}
// 2^u of two logits on the FMA units, u < 2^22; 0 from -127 down, as the special-function units give it for a logit of -inf.  Adding 1.5 x 2^23
// rounds u to the nearest integer, which goes to the exponent; 2^f of the rest, on [-1/2, 1/2], by a polynomial of degree 5 fitted to the least
// relative error with 2^0 = 1.  Error 1.1e-7 at most, 1.7e-7 as worked out in fp32 (ex2.approx 1.2e-7); rounding to bf16 is 2e-3.
__device__ __forceinline__ float2 poly_exp2(float2 u) {
  auto both = [](float v) { return make_float2(v, v); };
  constexpr float kRound = 12582912.f;                     // 1.5 x 2^23: the sum's last bits are the nearest integer
  u.x = fmaxf(u.x, -127.f);
  u.y = fmaxf(u.y, -127.f);
  const float2 r = fadd2(u, both(kRound)), f = ffma2(fadd2(r, both(-kRound)), both(-1.f), u);
  float2 y = both(0x1.5bba14p-10f);
  y = ffma2(y, f, both(0x1.3cea88p-7f));
  y = ffma2(y, f, both(0x1.c6b752p-5f));
  y = ffma2(y, f, both(0x1.ebf9bcp-3f));
  y = ffma2(y, f, both(0x1.62e42ap-1f));
  y = ffma2(y, f, both(1.f));
  return make_float2(__uint_as_float(__float_as_uint(y.x) + (__float_as_uint(r.x) << 23)), __uint_as_float(__float_as_uint(y.y) + (__float_as_uint(r.y) << 23)));
}
// Both halves of a bf16 pair to a sum each, as they are.
__device__ __forceinline__ void add_bf16x2(float2& s, uint32_t b) {
  asm("{.reg .b16 l, h; mov.b32 {l, h}, %2; add.f32.bf16 %0, l, %0; add.f32.bf16 %1, h, %1;}" : "+f"(s.x), "+f"(s.y) : "r"(b));
}
// Flat items.  What a logit can be at most follows from |q| and from the bounds that the cache keeps for the blocks of an item (BlockBound) and
// that come with a segment.  If that, for the rows of a warp, is not more than kTop above the reference that an item's first sub-tile gives,
// nothing after it can ask for another reference: the sub-tiles that follow need no maximum, no look at the others' and no hand-over, which are
// some 170 of the loop's 440 instructions, and every probability is taken relative to the same number as in the loop that looks.  (One reference
// for the four rows of a thread, within the biases, would spare 24 more and is 1 to 3 % faster, but then the largest probabilities no longer
// lie just below a power of two, where bf16 is finest: error against 64 bits 0.00230 -> 0.00233.  Nor may the bound be further above: with 96, as
// far as fp32 sums bear, items stay flat in which the other loop would have raised, and behind a raise the row's largest probability is a power
// of two.  Keys in the order of their clusters, logits of 1.5 to 4 times the usual size: 0.00209-0.00230 where the maximum is looked for,
// 0.00224-0.00233 so.)  Items of fewer sub-tiles than kFlatMin don't ask; with as many it pays (64 and 444 items of eight, d = 128: 10.6 and 26.6 us,
// looking 11.5 and 28.8; d = 64: 9.4 and 22.4, 10.9 and 25.3).  The bounds are of the item's own blocks: where tokens have merged into its slots
// thousands of times (12 heads, 8-bit search, m up to 2^10) 0.89 of the items are flat, by the bounds of a head 0.60, and if |k| and m are
// bounded apart 0.01.
constexpr int kFlatMin = 8;
// Pairs of every sixteen whose exponentials the FMA units work out: the special-function units take 512 cycles for a sub-tile's, the tensor
// core 270 at d = 64 and 540 at 128.  Kernel time with 0 / 2 / 4 of sixteen: d = 64, 256 items of 128 sub-tiles 97.9 / 94.1 / 95.0 us; at d = 128 it
// makes no difference (256 of 256 201 / 200 / 202), and has the same two.
constexpr int kPolyPairs = 2;

template <int D, int BKT>
struct AttnSmem {
  static constexpr int q_bytes = (D / 64) * kQChunk;
  static constexpr int kv_bytes = (D / 64) * BKT * 128;          // one K or V tile
  // Stages of the two rings.  K and V tiles have one each: a barrier's parity tells two phases apart, so the warp that waits for a
  // stage has to be the one that waited for its tile before (in one ring, a copy that is overtaken by the next five would let Q K^T
  // pass for a tile whose stage is still being filled).
  static constexpr int RS = 160 * 1024 / kv_bytes > 12 ? 12 : 160 * 1024 / kv_bytes;
  static constexpr int RK = (RS + 1) / 2, RV = RS / 2;
  static constexpr int SUB = BKT / 64;                           // sub-tiles of a key tile
  // Q as the MMAs' operand in tensor memory (QT) or in shared memory.  A 128 x 64 x 16 MMA with both operands in shared memory waits for
  // them (48 cycles, 32 with Q in tensor memory), so tiles of 64 keys take the former, which leaves columns for the logits of three
  // sub-tiles instead of four; with 128 keys the latter is as fast, and a fourth sub-tile ahead is worth more (denoising step 311 / 298 us
  // a pass, 161 items of 596 tiles of 64 keys 588 / 633).
  static constexpr bool QT = BKT == 64;
  static constexpr int NSB = QT ? 3 : kGroups / SUB;             // sub-tiles (QT) or key tiles whose logits are in tensor memory
  // Bias rows: one is overwritten when NB (16 or 32) tiles later the key tile is fetched, at most six key tiles behind one that is
  // consumed, whose logits went where those of a tile at least two rounds of the groups after this one had been.
  static constexpr int NB = 2048 / BKT;
  static constexpr int q_off = 0;
  static constexpr int ring_off = q_off + q_bytes;
  static constexpr int bias_off = ring_off + RS * kv_bytes;
  static constexpr int xchg_off = bias_off + NB * BKT * 4;       // [2][kGroups][128] (maximum, sum) of the groups' rows, by item
  static constexpr int max_off = xchg_off + 2 * kGroups * 1024;  // [4][8][4] running maxima: warp of the group, lane / 4, row / 8
  static constexpr int flat_off = max_off + 512;                 // [4] by warp of the group: the item is flat (see kFlatMin)
  static constexpr int stat_off = flat_off + 16;                 // the bounds of an item's keys: |k|, log2 m, both, |k| of the segment
  static constexpr int bar_off = flat_off + 64;
  static constexpr int total = bar_off + 512;
  static constexpr int p_col = (QT ? 3 : kGroups) * 64, o_col = p_col + kGroups * 32, q_col = o_col + D;      // TMEM columns (S at 0)
  static constexpr int tmem_cols = 512;
};

// A query block of a head, and the key tiles it attends to.
struct AttnItem {
  int h, q0, valid_rows;
  int nt;                               // key tiles
  int ntc;                              // paged mode: tiles taken from the cache; tiles [ntc, nt) are segment tiles
  int keep_n;                           // gather mode: kept prompt tokens
  const int32_t* list;                  // paged mode: kept blocks (null: all); gather mode: kept tokens
};

// SPLIT: the items of the last, partly filled round lie on a line, each as `units` units, and CTA b of `pieces` takes the units
// [n b / pieces, n (b + 1) / pieces).  An item's tiles are dealt to its units in proportion, so that every role knows its way without
// the others' tile counts; units is the most tiles that an item can have, and what it has wherever the lists are full.
struct AttnPart {
  int item;                             // of the last round's items
  int lo, hi;                           // its units
};
struct AttnPiece {                      // a CTA's piece: stops 0 .. n - 1 are the items first, first + 1, ...
  int first, n, lo, hi;                 // lo: first unit of the first, hi: end of the last
};
__device__ __forceinline__ AttnPiece piece_of_cta(const AttnArgs& a) {      // (the launch keeps these products below 2^31)
  const unsigned n = a.last_items * a.units, b = blockIdx.x, units = a.units, pieces = a.pieces;
  const unsigned x0 = n * b / pieces, x1 = n * (b + 1) / pieces;
  AttnPiece p{};
  if (b >= pieces || x1 == x0) return p;
  p.first = x0 / units;
  p.n = (x1 - 1) / units - p.first + 1;
  p.lo = x0 - p.first * units;
  p.hi = x1 - (p.first + p.n - 1) * units;
  return p;
}
__device__ __forceinline__ int piece_at(const AttnArgs& a, int x) {         // the piece that unit x belongs to
  return (static_cast<unsigned>(x + 1) * a.pieces - 1) / static_cast<unsigned>(a.last_items * a.units);
}
__device__ __forceinline__ int tile_at(const AttnArgs& a, int nt, int unit) {       // the tile that a unit of an item of nt tiles begins with
  return static_cast<unsigned>(nt * unit) / static_cast<unsigned>(a.units);
}
// Where a CTA's part of a cut item goes: a piece has two cut items at most, the one that it begins in and the one that it ends in.
__device__ __forceinline__ int slot_of(int piece, bool begins) { return 2 * piece + (begins ? 1 : 0); }

// A warp's 32 rows x 32 columns of a part (v, relative to the reference m, with the rows' sums) go to memory.
template <int D>
__device__ __forceinline__ float4* part_rows(const CacheView& c, int slot, int g, int r) {
  return reinterpret_cast<float4*>(c.part_o) + (static_cast<int64_t>(slot) * (D / 4) + g * 8) * 128 + r;
}
__device__ __forceinline__ float2* part_stat(const CacheView& c, int slot, int g, int r) {
  return c.part_ml + (static_cast<int64_t>(slot) * kGroups + g) * 128 + r;
}
template <int D>
__device__ __forceinline__ void store_part(const CacheView& c, int slot, int g, int r, const uint32_t (&v)[32], float m, float sum) {
  float4* dst = part_rows<D>(c, slot, g, r);
#pragma unroll
  for (int q = 0; q < 8; ++q)
    __stcg(dst + q * 128, make_float4(__uint_as_float(v[4 * q]), __uint_as_float(v[4 * q + 1]), __uint_as_float(v[4 * q + 2]), __uint_as_float(v[4 * q + 3])));
  __stcg(part_stat(c, slot, g, r), make_float2(m, sum));
}
// Adds up a warp's share of the `parts` parts of an item, in the order of the pieces; returns the rows' sums.  A part without a live key
// has a reference of -inf, a sum of 0 and no rows; one whose logits are NaN has the same reference and a sum of NaN, which has to reach the row.
template <int D>
__device__ __forceinline__ float merge_parts(const CacheView& c, int first_piece, int parts, int g, int r, uint32_t (&v)[32]) {
  float m = -INFINITY, sum = 0.f;
#pragma unroll 4
  for (int p = 0; p < parts; ++p) m = fmaxf(m, __ldcg(part_stat(c, slot_of(first_piece + p, p == 0), g, r)).x);
#pragma unroll
  for (int q = 0; q < 32; ++q) v[q] = 0u;
#pragma unroll 1
  for (int p = 0; p < parts; ++p) {
    const int slot = slot_of(first_piece + p, p == 0);
    const float2 ml = __ldcg(part_stat(c, slot, g, r));
    const float4* src = part_rows<D>(c, slot, g, r);
    float4 x[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) x[q] = __ldcg(src + q * 128);
    if (ml.x == -INFINITY && ml.y == 0.f) continue;
    const float f = fast_exp2(ml.x - m);
    sum = fmaf(ml.y, f, sum);
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const float2 a = ffma2(make_float2(x[q].x, x[q].y), make_float2(f, f), make_float2(__uint_as_float(v[4 * q]), __uint_as_float(v[4 * q + 1])));
      const float2 b = ffma2(make_float2(x[q].z, x[q].w), make_float2(f, f), make_float2(__uint_as_float(v[4 * q + 2]), __uint_as_float(v[4 * q + 3])));
      v[4 * q] = __float_as_uint(a.x);
      v[4 * q + 1] = __float_as_uint(a.y);
      v[4 * q + 2] = __float_as_uint(b.x);
      v[4 * q + 3] = __float_as_uint(b.y);
    }
  }
  return sum;
}
// 32 columns of a row, divided by the row's sum.
__device__ __forceinline__ void write_row(const AttnArgs& a, int64_t off, const uint32_t (&v)[32], float sum) {
  const float inv = sum > 0.f ? 1.f / sum : 0.f;
  if (a.out_fp32) {
    float4* dst = reinterpret_cast<float4*>(static_cast<float*>(a.out) + off);
#pragma unroll
    for (int q = 0; q < 8; ++q)
      dst[q] = make_float4(__uint_as_float(v[4 * q]) * inv, __uint_as_float(v[4 * q + 1]) * inv, __uint_as_float(v[4 * q + 2]) * inv,
                           __uint_as_float(v[4 * q + 3]) * inv);
  } else {
    uint4* dst = reinterpret_cast<uint4*>(static_cast<__nv_bfloat16*>(a.out) + off);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      uint32_t o[4];
#pragma unroll
      for (int e = 0; e < 4; ++e)
        o[e] = pack_bf16x2(__uint_as_float(v[8 * q + 2 * e]) * inv, __uint_as_float(v[8 * q + 2 * e + 1]) * inv);
      dst[q] = make_uint4(o[0], o[1], o[2], o[3]);
    }
  }
}

// SEG (paged mode only): tiles of an un-cached K/V segment follow the cache tiles.  CUT (paged mode only): the last round's items are
// cut by key tiles if the longest of all items has `whole_below` tiles at least.  The launch knows how many tiles there can be, the device how
// many there are; the kernel has both ways through it, and a CTA runs one of them.
template <int D, int BKT, bool GATHER, bool SEG, bool CUT>
__global__ void __launch_bounds__(kAttnThreads, 1)
attn_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
            const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_sk,
            const __grid_constant__ CUtensorMap tm_sv, const CacheView c, const AttnArgs a) {
  using SM = AttnSmem<D, BKT>;
  constexpr bool FLAT = !GATHER;                     // prompt tokens have no bounds, and few tiles
  // An item's first sub-tile as code of its own: in the loop, what only it does takes a twentieth of the loop's time, but items that are flat
  // then run through more code.  In the loop -> apart: 12 heads x 4680 queries on 32 of 220 blocks, all of whose items look 110 -> 105 us, flat 95.8 ->
  // 95.9; 8 x 4096 on 16 384 keys 240 -> 225 and 200.9 -> 201.6.  At d = 64, 64 of 1 024 blocks 124 -> 117, but flat 89.4 -> 91.4, 16 of 160 41.3 -> 39.9 and
  // 31.7 -> 32.1; where items are cut (12 x 1560, 16 of 110 blocks, flat) 36.6 -> 38.3.
  constexpr bool kApart = FLAT && D == 128 && !CUT;
  constexpr int kFirst = 1, kOther = 0, kAny = 2;
  constexpr int RS = SM::RS, RK = SM::RK, RV = SM::RV, NB = SM::NB, SUB = SM::SUB;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const uint32_t sbase = smem_u32(smem_raw);
  if (sbase & 1023u) {                  // swizzled tiles need 1024-byte alignment; uniform for the CTA
    if (threadIdx.x == 0) record_status(c.status, FASTAR_ERR_CUDA);
    return;
  }
  const uint32_t q_s = sbase + SM::q_off;
  const uint32_t ring_s = sbase + SM::ring_off;
  const uint32_t bias_s = sbase + SM::bias_off;
  const uint32_t bar = sbase + SM::bar_off;
  const uint32_t bar_q_full = bar;
  const uint32_t bar_q_empty = bar + 8;              // the MMAs (or copies) that read Q, and the warps that look at it (FLAT)
  const uint32_t bar_r_full = bar + 16;              // [RS] the K stages, then the V stages
  const uint32_t bar_r_empty = bar_r_full + 8 * RS;  // [RS]
  const uint32_t bar_s_full = bar_r_empty + 8 * RS;  // [4] by key tile, QT by group: the MMAs' commit, and the issuing warp once the biases are there
  const uint32_t bar_pv_done = bar_s_full + 32;      // [4] by sub-tile
  const uint32_t bar_s_empty = bar_pv_done + 32;     // [4] by key tile: the warps of its groups
  const uint32_t bar_p_full = bar_s_empty + 32;      // [4] by sub-tile: the warps of its group
  const uint32_t bar_xchg = bar_p_full + 32;         // [1] the groups meet here before an item's epilogue
  const uint32_t bar_o_free = bar_xchg + 8;          // [1] the soft-max warps: O of the item has been read
  const uint32_t bar_done = bar_xchg + 16;           // [1] the soft-max warps are through
  const uint32_t bar_parts = bar_xchg + 24;          // [1] SPLIT: the warps that store parts are through
  const uint32_t bar_last = bar_xchg + 32;           // [1] SPLIT: last_s is there
  const uint32_t bar_qk_done = bar_xchg + 40;        // [1] Q K^T of an item is complete
  const uint32_t bar_stat = bar_xchg + 48;           // [1] FLAT: the bounds of an item's keys are there
  // and [4] FLAT, by warp of a group: the first sub-tile's maxima and what follows from them are there
  constexpr int kNumBars = 2 + 2 * RS + 27;
  static_assert(kNumBars * 8 + 12 <= 512, "barrier area");
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem_raw + SM::bar_off + kNumBars * 8);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem_raw + SM::bar_off + kNumBars * 8 + 4);
  volatile int* done_flag = abort_flag + 1;          // stays 0: the waits that go on after an abort, for what every soft-max warp gets to

  const int warp = warp_index(), lane = threadIdx.x & 31;
  const int row_blocks = GATHER ? (a.rows_per_frame + 127) / 128 : (a.nq + a.block_q - 1) / a.block_q;
  const int items = row_blocks * c.H * (GATHER ? a.n_frames : 1);
  // Rows of item `it` (valid_rows <= 0: none, gather mode only).  Consecutive items are neighbouring query blocks of a head, which
  // share most of their key tiles.
  auto rows_of = [&](int it) {
    AttnItem w{};
    const int x = it % row_blocks, y = it / row_blocks;
    w.h = y % c.H;
    w.q0 = GATHER ? (y / c.H) * a.rows_per_frame + x * 128 : x * a.block_q;
    w.valid_rows = GATHER ? min(128, min(a.rows_per_frame - x * 128, a.nq - w.q0)) : min(a.block_q, a.nq - w.q0);
    return w;
  };
  if (GATHER && rows_of(blockIdx.x).valid_rows <= 0) return;   // uniform for the CTA (it has one item); nothing allocated yet

  // one thread per barrier
  if (threadIdx.x < kNumBars) {
    const int i = static_cast<int>(threadIdx.x) - (kNumBars - 27);        // s_full, pv_done, s_empty, p_full, xchg, o_free, done, parts, last, qk_done, stat, looked
    mbar_init(bar + 8 * threadIdx.x, FLAT && threadIdx.x == 1 ? 5 : i >= 20 ? 1 : i == 19 ? 4 * (D / 32) : i >= 16 ? kSoftWarps : i >= 12 || (i >= 8 && SM::QT) ? 4 : i >= 8 ? 4 * SUB : i >= 4 || i < 0 ? 1 : 2);
    fence_mbar_init();
  }
  if (threadIdx.x == 0) *abort_flag = *done_flag = 0;
  AttnPiece* piece_s = reinterpret_cast<AttnPiece*>(smem_raw + SM::bar_off + 480);
  volatile uint32_t* last_s = reinterpret_cast<volatile uint32_t*>(smem_raw + SM::bar_off + 496);      // cut items that this CTA has the last part of
  static_assert(kNumBars * 8 + 12 <= 480, "this CTA's piece");
  if (CUT && threadIdx.x == 64) *piece_s = piece_of_cta(a);
  if (warp == kKeyWarp && lane == 0) {
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

  auto run = [&](auto way) {
    constexpr bool SPLIT = decltype(way)::value;
    // The item with its key tiles (warp-uniform)
    auto item_of = [&](int it) {
      AttnItem w = rows_of(it);
      if (!GATHER) {
        if (a.sel == nullptr) {
          w.ntc = (__shfl_sync(0xffffffffu, c.len[w.h], 0) + BKT - 1) / BKT;
        } else {
          w.ntc = __shfl_sync(0xffffffffu, a.nsel[w.h], 0);
          w.list = a.sel + static_cast<int64_t>(w.h) * a.sel_head_stride + static_cast<int64_t>(it % row_blocks) * a.sel_stride;
        }
        w.nt = w.ntc + (SEG ? a.seg_tiles : 0);
      } else {
        const int f = it / (row_blocks * c.H);
        w.keep_n = a.keep;
        if (a.keep_frames) w.keep_n = __shfl_sync(0xffffffffu, a.keep_frames[static_cast<int64_t>(w.h) * a.keep_frames_stride + f], 0);
        w.nt = (w.keep_n + BKT - 1) / BKT;
        w.list = a.sel + static_cast<int64_t>(w.h) * a.sel_head_stride + static_cast<int64_t>(f) * a.sel_stride;
      }
      return w;
    };

    // The stops of a CTA: the items it, it + gridDim.x, ...; SPLIT: `rounds` of those, as it = 0, 1, ..., then its piece of the last round.
    const int it_first = SPLIT ? 0 : blockIdx.x, it_step = SPLIT ? 1 : gridDim.x;
    auto part_of = [&](int k) {
      return AttnPart{piece_s->first + k, k == 0 ? piece_s->lo : 0, k + 1 == piece_s->n ? piece_s->hi : a.units};
    };
    auto more = [&](int it) { return SPLIT ? __shfl_sync(0xffffffffu, it < a.rounds + piece_s->n ? 1 : 0, 0) != 0 : it < items; };
    auto item_at = [&](int it) {
      if (!SPLIT) return it;
      return __shfl_sync(0xffffffffu, static_cast<int>(it < a.rounds ? blockIdx.x + it * gridDim.x : a.rounds * gridDim.x + piece_s->first + it - a.rounds), 0);
    };
    auto tiles_of = [&](int it) {
      if (GATHER) return item_of(it).nt;
      const int h = item_at(it) / row_blocks % c.H;
      const int nt = (a.sel ? __shfl_sync(0xffffffffu, a.nsel[h], 0) : (__shfl_sync(0xffffffffu, c.len[h], 0) + BKT - 1) / BKT) + (SEG ? a.seg_tiles : 0);
      if (!SPLIT || it < a.rounds) return nt;
      const AttnPart p = part_of(it - a.rounds);
      return __shfl_sync(0xffffffffu, tile_at(a, nt, p.hi) - tile_at(a, nt, p.lo), 0);
    };

    // Everything is counted through the items of a CTA: tile0 key tiles, tile0 * SUB sub-tiles before.  Key tile n is in K stage n % RK
    // and V stage RK + n % RV.

    if (warp >= kSoftWarps) {
      setmaxnreg_dec<kIssueRegs>();
      if (warp == kKeyWarp || warp == kValueWarp) {
        // ================================================================ copies: Q, K and the biases, or V
        const bool is_k = warp == kKeyWarp;
        const uint32_t first = is_k ? 0 : RK, end = is_k ? RK : RS;
        uint32_t st = first, empty_phase = 1, copied = 0, n_q = 0, n_stat = 0;
        bool ok = true;
        for (int it = it_first; more(it) && ok; it += it_step) {
          AttnItem w = item_of(item_at(it));
          if (SPLIT && it >= a.rounds) {          // tiles [j0, j0 + nt): the list from there, or for all blocks in order the first block itself
            const AttnPart p = part_of(it - a.rounds);
            const int j0 = __shfl_sync(0xffffffffu, tile_at(a, w.nt, p.lo), 0);
            w.list = a.sel ? w.list + j0 : reinterpret_cast<const int32_t*>(static_cast<intptr_t>(j0));
            w.ntc -= j0;
            w.nt = __shfl_sync(0xffffffffu, tile_at(a, w.nt, p.hi), 0) - j0;
          }
          const int nt = w.nt;
          if (nt == 0) continue;
          // The bounds of the item's keys, by the warp that has the most time: the first tile of V is waited for later than Q and K.  They
          // follow those of the item before once these have been read: a barrier's parity tells two phases apart, and V's ring may have room for
          // all of an item.
          if (FLAT && !is_k) {
            if (n_stat > 0) ok = mbar_wait_warp<kIssueWaitHintNs>(bar_q_empty, (n_stat - 1) & 1, abort_flag, c.status);
            if (!ok) break;
            if (nt * SUB >= kFlatMin) {
              float4 keys = make_float4(0.f, 0.f, 0.f, 0.f);      // |k|, log2 m, both, |k| of the segment
              uint32_t seg = 0;
              if (SEG)
#pragma unroll
                for (int i = 0; i < kSegParts / 32; ++i) seg = max(seg, a.seg_bound[w.h * kSegParts + 32 * i + lane]);
#pragma unroll 2
              for (int jj = lane; jj < min(w.ntc, nt); jj += 32) {
                const int b = FASTAR_IDX(a.sel ? w.list[jj] : SPLIT ? static_cast<int>(reinterpret_cast<intptr_t>(w.list)) + jj : jj, c.CAPB, c.status);
                const float4 x = *reinterpret_cast<const float4*>(c.bound + static_cast<int64_t>(w.h) * c.CAPB + b);
                keys.x = fmaxf(keys.x, x.x);
                keys.y = fmaxf(keys.y, x.y);
                keys.z = fmaxf(keys.z, x.z);
              }
              auto most = [](float x) { return __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(x))); };      // (none is negative)
              const float v[4] = {most(keys.x), most(keys.y), most(keys.z), sqrtf(most(__uint_as_float(seg)))};
              if (lane == 0) sts4(sbase + SM::stat_off, v);
            }
            if (lane == 0) mbar_arrive(bar_stat);
            ++n_stat;
          }
          if (is_k) {
            if (n_q > 0) ok = mbar_wait_warp<kIssueWaitHintNs>(bar_q_empty, (n_q - 1) & 1, abort_flag, c.status);
            if (!ok) break;
            if (lane == 0) {
              mbar_arrive_expect_tx(bar_q_full, SM::q_bytes);
              for (int kc = 0; kc < D / 64; ++kc) tma_load_3d(q_s + kc * kQChunk, &tm_q, bar_q_full, kc * 64, w.q0, w.h);
            }
            ++n_q;
          }
          // paged mode: block ids and page ids of 32 tiles at a time, one coalesced load each and one window ahead; lane 0 copies
          int blk = 0, page = 0, blk_n = 0, page_n = 0;
          auto fetch = [&](int j0) {
            const int jj = j0 + lane;
            if (GATHER) return;
            if (SPLIT && jj >= nt) return;
            if (jj < w.ntc) {
              blk_n = FASTAR_IDX(a.sel ? w.list[jj] : SPLIT ? static_cast<int>(reinterpret_cast<intptr_t>(w.list)) + jj : jj, c.CAPB, c.status);
              page_n = FASTAR_IDX(c.page_table[static_cast<int64_t>(w.h) * c.CAPB + blk_n], c.pool_pages, c.status);
            } else if (SEG && jj < nt) {        // tile of the un-cached segment: its index, no page
              blk_n = jj - w.ntc;
              page_n = -1;
            }
          };
          auto announce = [&](uint32_t stage) {     // gather mode: this warp's copies into the stage have landed
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_r_full + 8 * stage);
          };
          auto token = [&](int i) { return GATHER && i < w.keep_n ? FASTAR_IDX(w.list[i], a.np, c.status) : 0; };
          int next = token(lane);                  // gather mode: 32 kept tokens, one per lane
          fetch(0);
          for (int j = 0; j < nt; ++j) {
            if ((j & 31) == 0) {
              blk = blk_n; page = page_n;
              fetch(j + 32);
            }
            const int b = GATHER ? 0 : __shfl_sync(0xffffffffu, blk, j & 31), p = GATHER ? 0 : __shfl_sync(0xffffffffu, page, j & 31);
            ok = mbar_wait_warp<kIssueWaitHintNs>(bar_r_empty + 8 * st, empty_phase, abort_flag, c.status);
            if (!ok) break;
            const uint32_t dst = ring_s + st * SM::kv_bytes;
            if (!GATHER) {
              if (lane == 0) {
                const bool seg = SEG && p < 0;   // rows past the segment's end arrive as zeros and carry a -inf bias
                const CUtensorMap* tm = seg ? (is_k ? &tm_sk : &tm_sv) : (is_k ? &tm_k : &tm_v);
                mbar_arrive_expect_tx(bar_r_full + 8 * st, SM::kv_bytes + (is_k ? BKT * 4 : 0));
                for (int kc = 0; kc < D / 64; ++kc)
                  tma_load_3d(dst + kc * BKT * 128, tm, bar_r_full + 8 * st, kc * 64, seg ? b * BKT : 0, seg ? w.h : p);
                if (is_k) {
                  const float* bias_src = seg ? a.seg_bias + static_cast<int64_t>(b) * BKT : c.log2m + static_cast<int64_t>(w.h) * c.CAP + b * BKT;
                  bulk_load_1d(bias_s + (copied % NB) * BKT * 4, bias_src, BKT * 4, bar_r_full + 8 * st);
                }
              }
            } else {
              // Rows of K_p / V_p by index, as asynchronous 16-byte copies to their swizzled position.  A tile is announced when the
              // copies of the next one are under way (it needs a stage that the tile before the announced one has left).
              constexpr int CPR = D / 8, RPI = 32 / CPR;       // 16-byte chunks per row, rows per instruction
              const int ch = lane % CPR;
              const __nv_bfloat16* src = (is_k ? a.kp : a.vp) + static_cast<int64_t>(w.h) * a.p_head_stride + ch * 8;
#pragma unroll 1
              for (int i0 = 0; i0 < BKT; i0 += 32) {
                const int idx = next;
                next = token(j * BKT + i0 + 32 + lane);
#pragma unroll 4
                for (int r = 0; r < 32; r += RPI) {
                  const int i = i0 + r + lane / CPR;
                  const int tok = __shfl_sync(0xffffffffu, idx, i & 31);
                  cp_async16(dst + (ch >> 3) * (BKT * 128) + i * 128 + (((ch & 7) ^ (i & 7)) << 4),
                             src + static_cast<int64_t>(tok) * a.p_token_stride, j * BKT + i < w.keep_n);
                }
              }
              if (is_k)
                for (int i = lane; i < BKT; i += 32)
                  asm volatile("st.shared.f32 [%0], %1;" ::"r"(bias_s + ((j % NB) * BKT + i) * 4), "f"((j * BKT + i < w.keep_n) ? 0.f : -INFINITY)
                               : "memory");
              asm volatile("cp.async.commit_group;" ::: "memory");
              if (j > 0) asm volatile("cp.async.wait_group 1;" ::: "memory");
              if (j > 0) announce(st == first ? end - 1 : st - 1);
              if (j + 1 == nt) {
                asm volatile("cp.async.wait_all;" ::: "memory");
                announce(st);
              }
            }
            ++copied;
            if (++st == end) { st = first; empty_phase ^= 1; }
          }
          if (GATHER) break;                       // one item
        }
        // what is still in flight must land before the CTA may exit (normally the MMAs have consumed all of it)
        if (GATHER) asm volatile("cp.async.wait_all;" ::: "memory");
        if (lane == 0) {
          if (n_q > 0) mbar_wait(bar_q_full, (n_q - 1) & 1, abort_flag, c.status);
          if (!GATHER)
            for (uint32_t s = first; s < end; ++s) {           // the last tile of stage s, if it has had one
              const uint32_t r = end - first, had = (copied + r - 1 - (s - first)) / r;
              if (had > 0) mbar_wait(bar_r_full + 8 * s, (had - 1) & 1, abort_flag, c.status);
            }
        }
      } else if (warp == kQkWarp) {
        // ================================================================ S = Q K_j^T
        const uint32_t lead = elect_lane();
        constexpr bool QT = SM::QT;
        constexpr uint32_t idesc = make_idesc_bf16(128, QT ? 64 : BKT, 0);
        const uint64_t qd = make_smem_desc(q_s, 16, 1024), kd0 = make_smem_desc(ring_s, 16, 1024);
        bool ok = true;
        uint32_t nq_used = 0, st = 0, r_phase = 0, b = 0, s_phase = 1, full_b = 0;       // stage, logits' columns and their barriers
        for (int it = it_first; more(it) && ok; it += it_step) {
          const int nt = tiles_of(it);
          if (nt == 0) continue;
          ok = mbar_wait_warp<kIssueWaitHintNs>(bar_q_full, nq_used & 1, abort_flag, c.status);
          if (QT && ok && nq_used > 0) ok = mbar_wait_warp(bar_qk_done, (nq_used - 1) & 1, abort_flag, c.status);
          if (!ok) break;
          ++nq_used;
          if (QT) {      // Q to tensor memory; the copies and the MMAs that read them are issued by one thread and execute in order
            tc_fence_after();
#pragma unroll
            for (int kk = 0; kk < D / 16; ++kk) tmem_copy_128x256b(tmem + SM::q_col + kk * 8, qd + (((kk >> 2) * kQChunk + (kk & 3) * 32) >> 4), lead);
            umma_commit(bar_q_empty, lead);
          }
          for (int j = 0; j < nt && ok; ++j) {
            // the columns are free once the groups hold the logits before in registers
            ok = mbar_wait<kIssueWaitHintNs>(bar_r_full + 8 * st, r_phase, abort_flag, c.status) && mbar_wait(bar_s_empty + 8 * b, s_phase, abort_flag, c.status);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            tc_fence_after();
            const uint64_t kd = kd0 + st * (SM::kv_bytes >> 4);
            const uint32_t s_col = tmem + b * (QT ? 64 : BKT);
#pragma unroll
            for (int kk = 0; kk < D / 16; ++kk) {
              const uint64_t bd = kd + (((kk >> 2) * (BKT * 128) + (kk & 3) * 32) >> 4);
              if (QT) umma_ts(s_col, tmem + SM::q_col + kk * 8, bd, idesc, kk != 0, lead);
              else umma_ss(s_col, qd + (((kk >> 2) * kQChunk + (kk & 3) * 32) >> 4), bd, idesc, kk != 0, lead);
            }
            const uint32_t full = bar_s_full + 8 * (QT ? full_b : b);
            umma_commit(full, lead);
            umma_commit(bar_r_empty + 8 * st, lead);
            if (j + 1 == nt) umma_commit(QT ? bar_qk_done : bar_q_empty, lead);
            if (lead) mbar_arrive(full);                   // what this warp has seen land (the biases) is there for the waiting warps
            full_b = (full_b + 1) % kGroups;
            if (++st == RK) { st = 0; r_phase ^= 1; }
            if (++b == SM::NSB) { b = 0; s_phase ^= 1; }
          }
        }
      } else if (warp == kPvWarp) {
        // ================================================================ O += P V_j
        const uint32_t lead = elect_lane();
        constexpr uint32_t idesc = make_idesc_bf16(128, D, 1);
        const uint64_t vd0 = make_smem_desc(ring_s + RK * SM::kv_bytes, BKT * 128, 1024);
        bool ok = true;
        uint32_t n_done = 0, st = 0, r_phase = 0, b = 0, p_phase = 0;
        for (int it = it_first; more(it) && ok; it += it_step) {
          const int nt = tiles_of(it);
          if (nt == 0) continue;
          if (n_done > 0) ok = mbar_wait_warp(bar_o_free, (n_done - 1) & 1, abort_flag, c.status);
          ++n_done;
          for (int j = 0; j < nt && ok; ++j) {
            ok = mbar_wait_warp(bar_r_full + 8 * (RK + st), r_phase, abort_flag, c.status);
            const uint64_t vd = vd0 + st * (SM::kv_bytes >> 4);
#pragma unroll
            for (int sub = 0; sub < SUB; ++sub) {
              ok = ok && mbar_wait_warp(bar_p_full + 8 * b, p_phase, abort_flag, c.status);
              if (!ok) break;
              tc_fence_after();
#pragma unroll
              for (int ks = 0; ks < 4; ++ks)
                umma_ts(tmem + SM::o_col, tmem + SM::p_col + b * 32 + ks * 8, vd + (((sub * 4 + ks) * 2048) >> 4), idesc, (j | sub | ks) != 0, lead);
              umma_commit(bar_pv_done + 8 * b, lead);
              if (++b == kGroups) { b = 0; p_phase ^= 1; }
            }
            if (!ok) break;
            umma_commit(bar_r_empty + 8 * (RK + st), lead);
            if (++st == RV) { st = 0; r_phase ^= 1; }
          }
        }
        // tensor memory goes back when the soft-max warps are through (all of them get there, none waits for long)
        mbar_wait_warp(bar_done, 0, done_flag, c.status);
        tc_fence_after();
        tmem_dealloc(tmem, SM::tmem_cols);
      }
    } else {
      // ================================================================== soft-max groups + epilogue (512 threads)
      setmaxnreg_inc<kSoftRegs>();
      constexpr uint32_t kHalf = 16u << 16;               // the second sixteen lanes
      // After a time-out a warp goes on to its last sub-tile without waiting, so that no other is ever left at a named barrier.
      // (It reads and writes its columns of tensor memory all the same: with the loads behind `if (ok)` the logits would have to
      // outlive their loop, which the registers do not allow.)
      bool ok = true, s_ready = false;
      int sub0 = 0, n_done = 0;                           // sub-tiles and items before
      for (int it = it_first; more(it); it += it_step) {
        const int ns = tiles_of(it) * SUB;
        // what follows from these four is worked out again for every item: kept over the items it would not fit the registers
        uint32_t sb_ = sbase, tm_ = tmem;
        int wp_ = warp, ln_ = lane;
        asm volatile("" : "+r"(sb_), "+r"(tm_), "+r"(wp_), "+r"(ln_));
        const uint32_t sbase = sb_, tmem = tm_;
        const int warp = wp_, lane = ln_;
        const uint32_t bar_s_full = sbase + SM::bar_off + 16 + 16 * RS, bar_pv_done = bar_s_full + 32, bar_s_empty = bar_pv_done + 32;
        const uint32_t bar_p_full = bar_s_empty + 32, bar_xchg = bar_p_full + 32, bar_o_free = bar_xchg + 8;
        const int g = warp >> 2;                          // soft-max group: sub-tiles with index % kGroups == g
        const uint32_t lane_t = tmem + (static_cast<uint32_t>((warp & 3) * 32) << 16);
        const float scale = rsqrtf(static_cast<float>(D)) * 1.4426950408889634f;
        const uint32_t p_t = lane_t + SM::p_col + g * 32, o_t = lane_t + SM::o_col;
        const uint32_t max_s = sbase + SM::max_off + ((warp & 3) * 8 + (lane >> 2)) * 16;
        const uint32_t bias_t = sbase + SM::bias_off + 8 * (lane & 3), flat_s = sbase + SM::flat_off + 4 * (warp & 3);
        // the barriers of the hand-over (all sixteen: nothing else uses one after the roles part): this warp waits for the look at the
        // sub-tile before, and tells of its own
        const uint32_t heard = 4 * g + (warp & 3), told = 4 * ((g + 1) % kGroups) + (warp & 3);
        float m[4];
        float2 l[4];                                      // running maxima of rows 8 q + lane / 4; sums over the even and the odd columns
#pragma unroll
        for (int q = 0; q < 4; ++q) { m[q] = -INFINITY; l[q] = make_float2(0.f, 0.f); }
        // the logits' barriers: QT has one per group for their arrival (a barrier's parity tells two phases apart) and one per place for their leaving
        const uint32_t full = bar_s_full + 8 * (SM::QT ? g : g / SUB), empty = bar_s_empty + 8 * (SM::QT ? 0 : g / SUB);
        int t = (g - sub0) & (kGroups - 1);
        if (FLAT && t == 0 && ns > 0) {
          ok = ok && mbar_wait_warp(bar_s_full + 176, n_done & 1, abort_flag, c.status);      // the bounds of the item's keys
          if (ns >= kFlatMin) {
            ok = ok && mbar_wait_warp(sbase + SM::bar_off, n_done & 1, abort_flag, c.status);
            const uint32_t row = sbase + SM::q_off + ((warp & 3) * 32 + lane) * 128;
            float sq = 0.f;
#pragma unroll
            for (int ch = 0; ch < D / 8; ++ch) {
              uint4 v;
              asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(row + (ch >> 3) * kQChunk + (((ch & 7) ^ (lane & 7)) << 4)));
              sq = square_sum8(v, sq);
            }
            // (1.001: the roundings of the norms, of the products' sums and of what follows; 1e-20: components whose squares are below the
            // smallest float.  Where q or a key is not finite, `apart` is not either, or no number, and so is the lesser of the two.)
            const float4 keys = lds4(sbase + SM::stat_off);
            const float y = (sqrtf(sq) + 1e-20f) * (scale * 1.001f), norm = keys.x + 1e-20f;
            const float together = keys.z + fmaxf(y - kJoint, 0.f) * norm, apart = y * norm + keys.y;
            float most = together < apart ? together : apart;
            if (SEG) most = most >= y * (keys.w + 1e-20f) ? most : y * (keys.w + 1e-20f);
            // what the rows' logits may be, less kTop, to where the maxima will be: nobody looks there yet, and it would not fit the registers
            float need[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) need[q] = __shfl_sync(0xffffffffu, most, (lane >> 2) + 8 * q) - kTop;
            if ((lane & 3) == 0) sts4(max_s, need);
          }
          mbar_arrive_warp(sbase + SM::bar_off + 8);
        }
        const uint32_t looked = bar_s_full + 184 + 8 * (warp & 3);
        bool flat = false;
        if (FLAT && ns >= kFlatMin && t > 0) {            // the first sub-tile's warp says whether the item is flat
          // (not given up with the other waits: all warps of the rows have to go the same way, and the one that says which gets there)
          ok = mbar_wait_warp(looked, n_done & 1, done_flag, c.status, 2 * kWaitLimitNs) && ok;
          flat = lds1(flat_s) != 0.f;
          if (flat) {
            const float4 ref = lds4(max_s);
            m[0] = ref.x; m[1] = ref.y; m[2] = ref.z; m[3] = ref.w;
          }
        }
        // A sub-tile whose maximum is looked for: an item's first one (kFirst), another one (kOther), or whichever it is.
        auto look = [&](auto way) {
          constexpr int WAY = decltype(way)::value;
          const bool first = WAY == kAny ? t == 0 : WAY == kFirst;
          const int tg = sub0 + t, jg = tg / SUB;
          const uint32_t sb = SM::QT ? tg % SM::NSB : 0;
          if (!s_ready) ok = ok && mbar_wait_warp(full, (tg / kGroups) & 1, abort_flag, c.status);
          tc_fence_after();
          // the logits of this warp's rows: x[hf][4 k + 2 e + c] is row 16 hf + 8 e + lane / 4, column 8 k + 2 (lane & 3) + c
          uint32_t x[2][32];
#pragma unroll
          for (int hf = 0; hf < 2; ++hf)
            tmem_ld_frag(lane_t + (SM::QT ? sb : g) * 64 + hf * kHalf, x[hf]);
          const uint32_t bp = bias_t + ((jg % NB) * BKT + (tg % SUB) * 64) * 4;
          float2 bias[8];
#pragma unroll
          for (int k = 0; k < 8; ++k) bias[k] = lds2(bp + 32 * k);
          if (!first) named_barrier_sync(heard, 64);
          const float4 seen = first ? make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY) : lds4(max_s);
          bool p_free = tg < kGroups || mbar_test_wait(bar_pv_done + 8 * g, (tg / kGroups - 1) & 1);
          tmem_wait_ld();
          tc_fence_before();
          mbar_arrive_warp(empty + 8 * sb);                // the logits are in registers
          float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
          for (int k = 0; k < 8; ++k) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              uint32_t* v = &x[q >> 1][4 * k + 2 * (q & 1)];
              const float2 y = ffma2(make_float2(__uint_as_float(v[0]), __uint_as_float(v[1])), make_float2(scale, scale), bias[k]);
              v[0] = __float_as_uint(y.x);
              v[1] = __float_as_uint(y.y);
              mx[q] = fmax3(mx[q], y.x, y.y);
            }
          }
          // A logit makes this warp raise the maximum if it exceeds the last one by as much.  If none does, and nobody has raised it since
          // this warp looked, the hand-over goes on at once: the maximum cannot change before this sub-tile is through, because whoever
          // raises it waits for P V of all sub-tiles before.
          // The first sub-tile's warp always goes the long way: it puts the maxima where the others read them, also those of a sub-tile
          // without a live key (-inf; what lies there is an earlier item's).
          bool may = first;
          if (WAY != kFirst) {
#pragma unroll
            for (int q = 0; q < 4; ++q) may |= mx[q] > m[q] + kTop;
            may = __any_sync(0xffffffffu, may);
          }
          if (!may && t + 1 < ns) named_barrier_arrive(told, 64);
          const float cur[4] = {seen.x, seen.y, seen.z, seen.w};
          bool change = first, becomes_flat = false;
#pragma unroll
          for (int q = 0; q < 4; ++q) change |= mx[q] > cur[q] + kTop || cur[q] != m[q];
          if (__any_sync(0xffffffffu, change)) {
            float alpha[4];
            bool raised = first;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              // the same for the four threads of a row
              mx[q] = fmaxf(mx[q], __shfl_xor_sync(0xffffffffu, mx[q], 1));
              mx[q] = fmaxf(mx[q], __shfl_xor_sync(0xffffffffu, mx[q], 2));
              float top = cur[q];
              alpha[q] = 1.f;
              if (mx[q] > cur[q] + kTop) {
                top = mx[q] + kHead;
                alpha[q] = cur[q] == -INFINITY ? 0.f : fast_exp2(cur[q] - top);
                raised = true;
              }
              // this thread's sum follows both the others' raises and its own
              if (m[q] != top) {
                const float f = m[q] == -INFINITY ? 0.f : fast_exp2(m[q] - top);
                l[q].x *= f;
                l[q].y *= f;
              }
              m[q] = top;
            }
            if (FLAT && first) {
              if (ns >= kFlatMin) {
                const float4 need = lds4(max_s);
                becomes_flat = need.x <= m[0] && need.y <= m[1] && need.z <= m[2] && need.w <= m[3] && fminf(fminf(m[0], m[1]), fminf(m[2], m[3])) > -INFINITY;
                becomes_flat = __all_sync(0xffffffffu, becomes_flat);
              }
              if (lane == 0) asm volatile("st.shared.f32 [%0], %1;" ::"r"(flat_s), "f"(becomes_flat ? 1.f : 0.f) : "memory");
            }
            if (__any_sync(0xffffffffu, raised)) {
              if (!first) {
                // O is relative to the old maxima: P V of the sub-tile before must be in it, that of this one follows its P.
                // (A parity tells only two phases apart, so the phase before has to be over: P V of sub-tile t - 4, which this group
                // has to see done in any case, comes after that of t - 5.)
                if (!__all_sync(0xffffffffu, p_free)) ok = ok && mbar_wait_warp(bar_pv_done + 8 * g, (tg / kGroups - 1) & 1, abort_flag, c.status);
                p_free = true;
                ok = ok && mbar_wait_warp(bar_pv_done + 8 * ((tg - 1) % kGroups), ((tg - 1) / kGroups) & 1, abort_flag, c.status);
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
                    for (int q = 0; q < 16; ++q) v[q] = __float_as_uint(__uint_as_float(v[q]) * ((q & 2) ? a1 : a0));
                    tmem_st_frag16(o_c, v);
                  }
              }
              if ((lane & 3) == 0) sts4(max_s, m);
              __syncwarp();
              if (FLAT && first) mbar_arrive_warp(looked);
            }
            if (becomes_flat) may = false;                 // nobody hands on in a flat item
          }
          if (may && t + 1 < ns) named_barrier_arrive(told, 64);
          // P is free once P V of the group's last sub-tile has read it
          if (!__all_sync(0xffffffffu, p_free)) ok = ok && mbar_wait_warp(bar_pv_done + 8 * g, (tg / kGroups - 1) & 1, abort_flag, c.status);
          tc_fence_after();
          // exponentials -> bf16 P
#pragma unroll
          for (int hf = 0; hf < 2; ++hf) {
            float2 neg[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) neg[e].x = neg[e].y = m[2 * hf + e] == -INFINITY ? 0.f : -m[2 * hf + e];
            uint32_t p[16];
#pragma unroll
            for (int k = 0; k < 8; ++k)
#pragma unroll
              for (int e = 0; e < 2; ++e) {
                const uint32_t* v = &x[hf][4 * k + 2 * e];
                const float2 u = fadd2(make_float2(__uint_as_float(v[0]), __uint_as_float(v[1])), neg[e]);
                const float2 pr = make_float2(fast_exp2(u.x), fast_exp2(u.y));
                const uint32_t b = pack_bf16x2(pr.x, pr.y);
                p[2 * k + e] = b;
                l[2 * hf + e] = fadd2(l[2 * hf + e], make_float2(__uint_as_float(b << 16), __uint_as_float(b & 0xFFFF0000u)));
              }
            tmem_st_half_frag(p_t + hf * kHalf, p);
          }
          s_ready = mbar_test_wait(full, (tg / kGroups + 1) & 1);      // (asked here, needed later: a barrier answers slowly while MMAs run)
          tmem_wait_st();
          tc_fence_before();
          mbar_arrive_warp(bar_p_full + 8 * g);
          s_ready = __all_sync(0xffffffffu, s_ready);
          if (WAY == kFirst) flat = becomes_flat;
        };
        if (kApart) {
          if (t == 0 && ns > 0) {
            look(std::integral_constant<int, kFirst>{});
            t += kGroups;
          }
          if (!flat)                                      // (a condition of its own: in the loop's it costs a twentieth)
            for (; t < ns; t += kGroups) look(std::integral_constant<int, kOther>{});
        } else if (!flat) {
          for (; t < ns; t += kGroups) {
            look(std::integral_constant<int, kAny>{});
            if (FLAT && t == 0 && lds1(flat_s) != 0.f) {
              t += kGroups;
              break;
            }
          }
        }
        if (FLAT) {
          const float2 scale2 = make_float2(scale, scale);
          for (; t < ns; t += kGroups) {
            const int tg = sub0 + t, jg = tg / SUB;
            const uint32_t phase = (tg / kGroups) & 1, sb = SM::QT ? tg % SM::NSB : 0;
            if (!s_ready) ok = ok && mbar_wait_warp(full, phase, abort_flag, c.status);
            tc_fence_after();
            uint32_t x[2][32];
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) tmem_ld_frag(lane_t + (SM::QT ? sb : g) * 64 + hf * kHalf, x[hf]);
            const uint32_t bp = bias_t + ((jg % NB) * BKT + (tg % SUB) * 64) * 4;
            float2 bias[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) bias[k] = lds2(bp + 32 * k);
            const bool p_free = mbar_test_wait(bar_pv_done + 8 * g, phase ^ 1);
            tmem_wait_ld();
            tc_fence_before();
            mbar_arrive_warp(empty + 8 * sb);
            uint32_t p[2][16];
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
#pragma unroll
              for (int k = 0; k < 8; ++k)
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                  const uint32_t* v = &x[hf][4 * k + 2 * e];
                  const float ref = -m[2 * hf + e];
                  const float2 u = fadd2(ffma2(make_float2(__uint_as_float(v[0]), __uint_as_float(v[1])), scale2, bias[k]), make_float2(ref, ref));
                  float2 pr;
                  if (2 * k + e < kPolyPairs) pr = poly_exp2(u);
                  else pr = make_float2(fast_exp2(u.x), fast_exp2(u.y));
                  const uint32_t b = pack_bf16x2(pr.x, pr.y);
                  p[hf][2 * k + e] = b;
                  add_bf16x2(l[2 * hf + e], b);
                }
            }
            // P is free once P V of the group's last sub-tile has read it; waited for here, behind the exponentials
            if (!__all_sync(0xffffffffu, p_free)) ok = ok && mbar_wait_warp(bar_pv_done + 8 * g, phase ^ 1, abort_flag, c.status);
            tc_fence_after();
            tmem_st_half_frag(p_t, p[0]);
            tmem_st_half_frag(p_t + kHalf, p[1]);
            s_ready = mbar_test_wait(full, phase ^ 1);
            tmem_wait_st();
            tc_fence_before();
            mbar_arrive_warp(bar_p_full + 8 * g);
            s_ready = __all_sync(0xffffffffu, s_ready);
          }
        }
        // ---- the groups meet: (m, l) of every row through shared memory ----
        const uint32_t xchg = sbase + SM::xchg_off + (n_done & 1) * kGroups * 1024;
        if (ns > 0) {
          // the group of the last sub-tile waits for the last P V, the others for that group
          const int last = sub0 + ns - 1;
          if (g == last % kGroups) ok = ok && mbar_wait_warp(bar_pv_done + 8 * g, (last / kGroups) & 1, abort_flag, c.status);
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            float sum = l[q].x + l[q].y;
            sum += __shfl_xor_sync(0xffffffffu, sum, 1);
            sum += __shfl_xor_sync(0xffffffffu, sum, 2);
            if ((lane & 3) == 0)
              asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(xchg + (g * 128 + (warp & 3) * 32 + (lane >> 2) + 8 * q) * 8), "f"(m[q]), "f"(sum)
                           : "memory");
          }
          mbar_arrive_warp(bar_xchg);
          // (nor is this given up with the others: after a time-out too the warps go from item to item together)
          ok = mbar_wait_warp(bar_xchg, n_done & 1, done_flag, c.status, 2 * kWaitLimitNs) && ok;
          tc_fence_after();
        }
        const int r = (warp & 3) * 32 + lane;         // from here on a thread owns one row, 32 of its columns
        if (ok && g < D / 32) {
          // O is relative to the last maximum, which the group of the last sub-tile knows; the others may be some raises behind
          uint32_t v[32];
          float m_all = -INFINITY, denom = 0.f;
          if (ns > 0) {
            float2 part[kGroups];
#pragma unroll
            for (int q = 0; q < kGroups; ++q) {
              part[q] = lds2(xchg + (q * 128 + r) * 8);
              m_all = fmaxf(m_all, part[q].x);
            }
#pragma unroll
            for (int q = 0; q < kGroups; ++q) denom += part[q].y * ((part[q].x == -INFINITY) ? 0.f : fast_exp2(part[q].x - m_all));
            tmem_ld32(o_t + g * 32, v);
            tmem_wait_ld();
          } else {
#pragma unroll
            for (int q = 0; q < 32; ++q) v[q] = 0u;
          }
          tc_fence_before();
          if (ns > 0) mbar_arrive_warp(bar_o_free);
          AttnPart cut{};
          if (SPLIT && it >= a.rounds) cut = part_of(it - a.rounds);
          if (SPLIT && it >= a.rounds && cut.hi - cut.lo < a.units) {
            store_part<D>(c, slot_of(blockIdx.x, cut.lo == 0), g, r, v, m_all, denom);
          } else {
            const AttnItem w = rows_of(item_at(it));
            if (r < w.valid_rows)               // loads are warp-collective, only the stores are per row
              write_row(a, static_cast<int64_t>(w.h) * a.out_head_stride + static_cast<int64_t>(w.q0 + r) * a.out_token_stride + g * 32, v, denom);
          }
        } else if (ns > 0) {
          mbar_arrive_warp(bar_o_free);
        }
        if (ns > 0) ++n_done;
        sub0 += ns;
      }
      const AttnPiece piece = SPLIT ? *piece_s : AttnPiece{};
      if (SPLIT && (warp >> 2) < D / 32 && piece.n > 0) {
        // The parts of cut items: the CTA that finds that the other parts of an item have come adds them up.  Asked at the end, so that no
        // answer is waited for between two items; by one warp, because a fence by each of sixteen takes as long as ten tiles; for both cut
        // items at once, by two lanes.  After a time-out the warps come here too, so that the counters go back to zero.
        const int g = warp >> 2, r = (warp & 3) * 32 + lane;
        auto cut_at = [&](int e) { return part_of(e == 0 ? 0 : piece.n - 1); };
        auto parts_of = [&](int item, int& first) {
          first = piece_at(a, item * a.units);
          return piece_at(a, item * a.units + a.units - 1) - first + 1;
        };
        mbar_arrive_warp(bar_parts);
        if (warp == 0) {
          ok = mbar_wait_warp(bar_parts, 0, abort_flag, c.status) && ok;
          const AttnPart cut = cut_at(lane & 1);
          int last = 0, first;
          if (lane < min(piece.n, 2) && cut.hi - cut.lo < a.units) {
            last = atomic_add_acq_rel(c.part_count + cut.item, 1) == parts_of(cut.item, first) - 1 ? 1 : 0;
            if (last) c.part_count[cut.item] = 0;
          }
          const uint32_t both = __ballot_sync(0xffffffffu, last);
          if (lane == 0) *last_s = both;
          mbar_arrive_warp(bar_last);
        }
        ok = mbar_wait_warp(bar_last, 0, abort_flag, c.status) && ok;
#pragma unroll 1
        for (int e = 0; e < 2; ++e)
          if (ok && ((*last_s >> e) & 1)) {
            uint32_t v[32];
            int first;
            const int item = cut_at(e).item, parts = parts_of(item, first);
            const float sum = merge_parts<D>(c, first, parts, g, r, v);
            const AttnItem w = rows_of(a.rounds * gridDim.x + item);
            if (r < w.valid_rows)
              write_row(a, static_cast<int64_t>(w.h) * a.out_head_stride + static_cast<int64_t>(w.q0 + r) * a.out_token_stride + g * 32, v, sum);
          }
      }
      tc_fence_before();
      mbar_arrive_warp(bar_done);
    }  };
  if constexpr (CUT) {
    const int32_t* live = a.sel ? a.nsel : c.len;            // tiles, or keys
    int longest = live[min(lane, c.H - 1)];
#pragma unroll 1
    for (int h = lane + 32; h < c.H; h += 32) longest = max(longest, live[h]);
    longest = __reduce_max_sync(0xffffffffu, longest);
    if ((a.sel ? longest : (longest + BKT - 1) / BKT) + (SEG ? a.seg_tiles : 0) >= a.whole_below) run(std::true_type{});
    else run(std::false_type{});
  } else {
    run(std::false_type{});
  }
}

template <int D, int BKT, bool GATHER, bool SEG, bool CUT = false>
static int launch_attn_t(const CUtensorMap& tq, const CUtensorMap& tk, const CUtensorMap& tv, const CUtensorMap& tsk,
                         const CUtensorMap& tsv, const CacheView& c, const AttnArgs& a, int grid, cudaStream_t st) {
  using SM = AttnSmem<D, BKT>;
  auto kern = attn_kernel<D, BKT, GATHER, SEG, CUT>;
  const int cfg = ensure_dynamic_smem(reinterpret_cast<const void*>(kern), SM::total);
  if (cfg != FASTAR_OK) return cfg;
  launch_chained(kern, grid, kAttnThreads, SM::total, st, tq, tk, tv, tsk, tsv, c, a);
  return cudaGetLastError() == cudaSuccess ? 1 : FASTAR_ERR_CUDA;
}

template <int D, int BKT, bool GATHER, bool SEG>
static int launch_attn(const CUtensorMap& tq, const CUtensorMap& tk, const CUtensorMap& tv, const CUtensorMap& tsk,
                       const CUtensorMap& tsv, const CacheView& c, const AttnArgs& a, int items, cudaStream_t st) {
  // One CTA per SM takes the items in turn; gather mode (more than 64 kept prompt tokens, or up to that many by the bucket rule) has
  // one item per CTA.  Its rows come in by asynchronous copies, a tile ahead: 12 heads x 4680 queries, 512 kept 385 -> 94 us for the
  // whole call (loads and stores through registers: 385; with 64 registers a thread 286), 40 x 10800 2420 -> 479, 128 kept 71 -> 64.
  int dev = 0, sm_count = 148;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sm_count, cudaDevAttrMultiProcessorCount, dev);
  if constexpr (!GATHER) {
    // Items that do not fill the last round of the SMs are cut by key tiles where that pays by CutCost: either every item into k equal
    // pieces, which leaves a CTA one stop, or all are dealt to all CTAs.  What is decided here for the most tiles that an item can have, the
    // kernel does if there is an item of so many (whole_below) that it pays: a cache that is a tenth full is attended as if it had no more room.
    // Dense calls of 288 shapes (4 to 440 items of 4 to 256 tiles, both dimensions, both tiles) were measured uncut, in as many equal pieces as
    // fit, and dealt; this picks a time 1.01 times the best of the three in the geometric mean.  Kernel time uncut and cut: 18 items of 128
    // 128-key tiles 85 -> 27 us, 72 of 32 28 -> 23, 156 of 64 93 -> 71; 160 of 128 64-key tiles 91 -> 63, 18 of 64 26 -> 18; 108 of 256 64-key
    // tiles, dealt, 87 -> 77; 256 of 128 128-key tiles, d = 64, dealt, 156 -> 149.  Where it would not pay: 72 of 16 128-key tiles 18.0 and
    // 18.1, 108 of 64, dealt, 43 and 45, 4 of 8 12.5 and 13.8.
    // With room for more keys than there are: 4 x 1 024 queries on 512 keys in a cache of 32 768, 64-key tiles 10.8 us, cut by the room 21.6, now
    // 11.3 (the look at the lengths is 0.4 of it); 8 x 1 560 on 2 048, 128-key tiles 21.9, 30.5, 21.8.
    using Cost = CutCost<BKT>;
    const int grid = min(min(sm_count, kAttnMaxGrid), c.max_pieces), full = min(sm_count, kAttnMaxGrid), rounds = items / full, left = items % full;
    const int tiles = (a.sel ? a.keep : c.CAPB) + a.seg_tiles;           // at most
    const float share = 1.f - Cost::gain * (rounds + 1);                 // of its tiles' time that a cut item may take
    AttnArgs cut = a;
    cut.rounds = rounds;
    cut.last_items = left;
    cut.units = tiles;
    float best = tiles * share;
    for (int k = 2; left > 0 && k * left <= grid && k * kAttnMinPiece <= tiles; ++k) {
      const float dealt = 1.f / k, cost = Cost::store + Cost::part * k * left + Cost::add * k, t = tiles * dealt + cost;
      if (t < best) { best = t; cut.pieces = k * left; cut.whole_below = static_cast<int>(cost / (share - dealt)) + 1; }
    }
    if (left > 0 && grid > left) {
      const float dealt = static_cast<float>(left) / grid, cost = Cost::stop + Cost::store + Cost::part * (grid + left) + Cost::add * (static_cast<float>(grid) / left + 1.f);
      if (tiles * dealt + cost < best && static_cast<int64_t>(left) * tiles >= static_cast<int64_t>(grid) * kAttnMinPiece) {
        cut.pieces = grid;
        cut.whole_below = static_cast<int>(cost / (share - dealt)) + 1;
      }
    }
    const int64_t largest = static_cast<int64_t>(tiles) * max(left * (cut.pieces + 1), tiles);      // of the kernel's products
    if (cut.pieces > 0 && !a.no_cut && largest < (1ll << 31)) return launch_attn_t<D, BKT, GATHER, SEG, true>(tq, tk, tv, tsk, tsv, c, cut, full, st);
  }
  return launch_attn_t<D, BKT, GATHER, SEG>(tq, tk, tv, tsk, tsv, c, a, GATHER ? items : min(items, sm_count), st);
}

// tm_seg_k / tm_seg_v: maps of the un-cached segment (box {64, page_tokens, 1}); nullptr when a.seg_tiles == 0.
int launch_attention_paged(const CacheView& c, const CUtensorMap& tm_q, const CUtensorMap& tm_pool_k,
                           const CUtensorMap& tm_pool_v, const CUtensorMap* tm_seg_k, const CUtensorMap* tm_seg_v,
                           const AttnArgs& a, cudaStream_t st) {
  if (a.seg_tiles > 0 && (!tm_seg_k || !tm_seg_v || !a.seg_bias)) return FASTAR_ERR_INVALID_ARG;
  const CUtensorMap& sk = a.seg_tiles > 0 ? *tm_seg_k : tm_q;      // never read without segment tiles
  const CUtensorMap& sv = a.seg_tiles > 0 ? *tm_seg_v : tm_q;
  const int items = (a.nq + a.block_q - 1) / a.block_q * c.H;
  if (c.D == 128 && c.PT == 128) return a.seg_tiles > 0 ? launch_attn<128, 128, false, true>(tm_q, tm_pool_k, tm_pool_v, sk, sv, c, a, items, st)
                                                          : launch_attn<128, 128, false, false>(tm_q, tm_pool_k, tm_pool_v, sk, sv, c, a, items, st);
  if (c.D == 128 && c.PT == 64) return a.seg_tiles > 0 ? launch_attn<128, 64, false, true>(tm_q, tm_pool_k, tm_pool_v, sk, sv, c, a, items, st)
                                                          : launch_attn<128, 64, false, false>(tm_q, tm_pool_k, tm_pool_v, sk, sv, c, a, items, st);
  if (c.D == 64 && c.PT == 128) return a.seg_tiles > 0 ? launch_attn<64, 128, false, true>(tm_q, tm_pool_k, tm_pool_v, sk, sv, c, a, items, st)
                                                          : launch_attn<64, 128, false, false>(tm_q, tm_pool_k, tm_pool_v, sk, sv, c, a, items, st);
  if (c.D == 64 && c.PT == 64) return a.seg_tiles > 0 ? launch_attn<64, 64, false, true>(tm_q, tm_pool_k, tm_pool_v, sk, sv, c, a, items, st)
                                                          : launch_attn<64, 64, false, false>(tm_q, tm_pool_k, tm_pool_v, sk, sv, c, a, items, st);
  return FASTAR_ERR_UNSUPPORTED_SHAPE;
}

int launch_attention_gather(const CacheView& c, const CUtensorMap& tm_q, const AttnArgs& a, cudaStream_t st) {
  // one key tile of 64: a kernel of its own, which keeps the tile and streams the queries (12 x 4680 queries, 64 kept: 34.2 -> 11.5 us)
  if (a.keep <= 64) return launch_attention_prompt64(c, tm_q, a, st);
  const int items = (a.rows_per_frame + 127) / 128 * c.H * a.n_frames;
  if (c.D == 128) return launch_attn<128, 128, true, false>(tm_q, tm_q, tm_q, tm_q, tm_q, c, a, items, st);
  return launch_attn<64, 128, true, false>(tm_q, tm_q, tm_q, tm_q, tm_q, c, a, items, st);
}

}  // namespace fastar
