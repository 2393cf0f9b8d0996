// Attention over the paged store for f32, head_dim 64 (Sec. 3.3, Eq. 5) on the tensor cores, at the precision of fp32 arithmetic.
// Every operand is split into three bf16 numbers, x = h + m + l (8 significant bits each, so nothing of x is lost, see kLift), and a product
// is the six products of pieces that are larger than 2^-24 of it, the small ones summed first:
//   S = Ql Kh + Qh Kl + Qm Km + Qm Kh + Qh Km + Qh Kh,  and P V alike.
// A CTA of 256 threads, two per SM, owns 128 query rows of one slice and streams its keys in tiles of 64:
//   warps 4-7 : operands.  They load K and V rows (the pages' or, for a map that has not been copied there, the caller's), split
//               them and leave the pieces in 128B-swizzled shared memory; the next tile's rows wait in registers meanwhile.
//               Warp 4 issues S of a tile as soon as its keys lie there, into the other of two buffers, under the softmax of
//               the tile before.
//   warps 0-3 : softmax, a thread per query row (TMEM lane).  The products of a tile of V land in TMEM and are added to the row's
//               64 columns in registers: the tensor core cuts its sums off where fp32 arithmetic rounds them, which over the tiles of a
//               long cache would show.  P goes back to TMEM in three pieces, over the scores it comes from.  Warp 0 issues P V when all
//               four warps have met; its result is added behind the softmax of the next tile.
// With two CTAs an SM's tensor pipe works for the one while the other is in its softmax.
// Scores that are not numbers (an infinite key: its products with the pieces of a query may differ in sign) are taken again, by signs or fp32 FMA
// (repair_scores).  Rows whose sum or columns are none all the same, an infinite value's, are done again at the end by fp32 FMA (redo_rows).
// The observation window's logits are taken by CTAs of their own behind those of all slices, in plain fp32 (see the launch).
// gridDim.z CTAs of a cluster share a slice's keys and combine: O = sum_e 2^(c (m_e - M)) O_e / sum_e 2^(c (m_e - M)) l_e, through distributed
// shared memory.
// What bounds it: the issue of MMAs, six products standing for one (48 a tile and CTA; one of N = 64 holds the path for 65 cycles, as long as one of
// N = 128, though its work is half of that: the pipe counts 37 % at 1 600 queries), and the instructions of the softmax and of the splitting (issue slots
// 48 %); a step of two CTAs that share an SM takes about 8 000 cycles.  (Working copies that skip work, us per layer, 16 slices x 1 600 queries: whole 130; one
// product of six 102; P not split 115; K and V not split 112.)  S of the next tile under the softmax of this one, from two buffers, and
// fewer instructions: 139 -> 123.  The loop of exponentials and splitting over a tile's 16-column pieces is not unrolled (that of the maximum is), and the
// operands' part of a step stands once: 123 -> 113 (fewer spills, less code to fetch in short launches).  us per layer and step, 16 slices behind 92 to 772 entries with their compresses,
// by packed fp32 FMA (66 % of that pipe), a copy of the map and three launches per compress -> here: 16 queries 15.4 -> 8.7, 64: 25.7 -> 16, 256: 35.8 -> 20,
// 400: 65 -> 31, 576: 91 -> 40, 1 024: 179 -> 63, 1 600: 331 -> 113.
// Error against 64 bits, full caches of 29 to 4 436 entries, queries and keys normal, queries times 0.25 / 1 / 3: outputs 0.9 to 1.6 / 1.0 to
// 2.1 / 1.5 to 4.0 e-7 (by FMA 1.1 to 11.9 / 2.2 to 12.3 / 3.3 to 15.2), lse 1.1 to 3.2 / 1.1 to 3.4 / 2.9 to 3.7 e-7 rms (1.1 to 3.2 / 1.4 to 3.3 /
// 5.2 to 8.2).
#pragma once
#include <cfloat>
#include <type_traits>

#include "attend_tc.cuh"
#include "kernels_simt.cuh"
#include "key_split.h"

namespace scalekv {
namespace f32 {

using tc::tc_fence_after;
using tc::tc_fence_before;

constexpr int kRows = 128, kKeys = 64, kThreads = 256;
constexpr uint32_t kPieceQ = kRows * 128, kPieceK = kKeys * 128;                  // bytes of one bf16 piece of an operand tile
constexpr uint32_t kOffQ = 0, kOffK = kOffQ + 3 * kPieceQ, kOffV = kOffK + 3 * kPieceK, kOffBar = kOffV + 3 * kPieceK;
constexpr uint32_t kSmemBytes = kOffBar + 64;
constexpr uint32_t kOffStat = kOffQ + kRows * 256;          // references and sums of the rows, behind their columns (where Q was)
static_assert(kOffStat + kRows * 8 <= kOffK, "the parts of a row have to fit where Q was");
static_assert(2 * (kSmemBytes + 1024) <= 233472, "two CTAs have to fit an SM");
// What a score loses, of its size and on average, because the tensor core cuts its sums off: about half a unit in the last place (2^-24)
// in each of the four steps over the large pieces, less in those where the sum is still growing.  It is given back (without: lse of queries
// times 3 low by 6.6e-7 on average, 7.4e-7 rms; so by 0.1 to 0.5e-7, 3.2 to 3.4e-7 rms): to the differences between a row's products and their
// reference, and to the reference where it enters a log-sum-exp.  (Given to the products alone, it would leave the largest weight at 2^(7e-8 m),
// m its exponent: of scores near -1e9 the weights would lie where their pieces run out of range.)
constexpr float kCutOff = 1.2f / 16777216.f;
// Queries and values are lifted by 2^24 before they are split, and products and outputs taken down again, so that the pieces of small ones
// are not bf16's subnormal numbers (of values near 1e-36 the output would be off by 1e-5 of it): every query and value of normal size is held
// whole.  Keys are not: theirs below 2^-110 lose up to 2^-134, which the largest query that can be split, 2^103, does not make 2^-30 of a score.  What
// the lift takes beyond the range - queries and values from 2^103, products from 2^104 - is an infinity and done by fp32 FMA, as those are.
constexpr float kLift = 16777216.f;
// TMEM: two buffers of 96 columns for scores and P, 64 columns for products with V.  The 16 keys of step kk have their scores in columns
// 16 kk .. of a buffer, and their P there (h in the first eight, m in the next) and in columns 64 + 8 kk .. (l).
constexpr uint32_t kTmemCols = 256, kBufCols = 96, kColPm = 8, kColPl = 64, kColO = 192;
enum { bV = 0, bPv = 1, bS = 2 };                           // barriers: V is there; P V has landed; S has, by buffer

struct Params {
  LayerView lv;
  TensorView Q, O, K, V;       // K, V: a current map outside the pages (fused)
  float *lse;
  int n_k, room;               // room: entries that a slice's pages hold
  int fused, copy_in, n_prev;  // copy_in: the map's rows go to the pages on the way
  float scale;
  float weight_scale;          // what a difference of two rows' products is multiplied with to make a weight's exponent: |scale| log2(e), and kCutOff
  int win_tiles;               // key tiles of a slice whose logits with the window's w rows the CTAs behind the slices' (blockIdx.y) take
  float *win_logits;           // base-2 logits by slot, [slice][rank][ld_l]
  int ld_l, w;
  int win_pos[kMaxWindow];
};

// Four steps (of 16) of one product of pieces, issued by the elected lane of a converged warp.
__device__ __forceinline__ void mma4_ss(uint32_t d, uint32_t a_lo, uint32_t b_lo, uint32_t hi, uint32_t idesc, uint32_t accumulate_first) {
  asm volatile(
      "{\n\t.reg .pred e, pf, pt;\n\t.reg .b64 da, db;\n\t.reg .b32 al, bl;\n\t"
      "elect.sync _|e, 0xffffffff;\n\tsetp.ne.b32 pf, %5, 0;\n\tsetp.eq.b32 pt, 0, 0;\n\t"
      "mov.b64 da, {%1, %3};\n\tmov.b64 db, {%2, %3};\n\t@e tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, pf;\n\t"
      "add.u32 al, %1, 2;\n\tadd.u32 bl, %2, 2;\n\tmov.b64 da, {al, %3};\n\tmov.b64 db, {bl, %3};\n\t@e tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, pt;\n\t"
      "add.u32 al, %1, 4;\n\tadd.u32 bl, %2, 4;\n\tmov.b64 da, {al, %3};\n\tmov.b64 db, {bl, %3};\n\t@e tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, pt;\n\t"
      "add.u32 al, %1, 6;\n\tadd.u32 bl, %2, 6;\n\tmov.b64 da, {al, %3};\n\tmov.b64 db, {bl, %3};\n\t@e tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, pt;\n\t"
      "}" ::"r"(d),
      "r"(a_lo), "r"(b_lo), "r"(hi), "r"(idesc), "r"(accumulate_first)
      : "memory");
}
template <int STEP>              // columns of P from one step to the next
__device__ __forceinline__ void mma4_ts(uint32_t d, uint32_t a, uint32_t b_lo, uint32_t hi, uint32_t idesc, uint32_t accumulate_first) {
  asm volatile(
      "{\n\t.reg .pred e, pf, pt;\n\t.reg .b64 db;\n\t.reg .b32 at, bl;\n\t"
      "elect.sync _|e, 0xffffffff;\n\tsetp.ne.b32 pf, %5, 0;\n\tsetp.eq.b32 pt, 0, 0;\n\t"
      "mov.b64 db, {%2, %3};\n\t@e tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], db, %4, pf;\n\t"
      "add.u32 at, %1, %6;\n\tadd.u32 bl, %2, 128;\n\tmov.b64 db, {bl, %3};\n\t@e tcgen05.mma.cta_group::1.kind::f16 [%0], [at], db, %4, pt;\n\t"
      "add.u32 at, %1, %7;\n\tadd.u32 bl, %2, 256;\n\tmov.b64 db, {bl, %3};\n\t@e tcgen05.mma.cta_group::1.kind::f16 [%0], [at], db, %4, pt;\n\t"
      "add.u32 at, %1, %8;\n\tadd.u32 bl, %2, 384;\n\tmov.b64 db, {bl, %3};\n\t@e tcgen05.mma.cta_group::1.kind::f16 [%0], [at], db, %4, pt;\n\t"
      "}" ::"r"(d),
      "r"(a), "r"(b_lo), "r"(hi), "r"(idesc), "r"(accumulate_first), "n"(STEP), "n"(2 * STEP), "n"(3 * STEP)
      : "memory");
}
__device__ __forceinline__ void tc_st8(uint32_t taddr, const uint32_t *v) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]),
               "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
               : "memory");
}

// the largest, or no number where one of them is none
__device__ __forceinline__ float max3_nan(float a, float b, float c) {
  float r;
  asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

// A pair of numbers in three pairs of bf16 numbers that sum to them.  (What h and m leave of 24 bits fits the eight of l, so l is the
// upper half of what is left.)
__device__ __forceinline__ void split2(float x, float y, uint32_t &h, uint32_t &m, uint32_t &l) {
  const uint64_t minus = tc::pack2(-1.f, -1.f);
  h = tc::pack_bf16(x, y);
  tc::unpack2(tc::fma2(tc::pack2(__uint_as_float(h << 16), __uint_as_float(h & 0xffff0000u)), minus, tc::pack2(x, y)), x, y);
  m = tc::pack_bf16(x, y);
  tc::unpack2(tc::fma2(tc::pack2(__uint_as_float(m << 16), __uint_as_float(m & 0xffff0000u)), minus, tc::pack2(x, y)), x, y);
  l = __byte_perm(__float_as_uint(x), __float_as_uint(y), 0x7632);
}
__device__ __forceinline__ void store16(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ float4 times(const float4 &x, float f) {
  const uint64_t ff = tc::pack2(f, f);
  float4 y;
  tc::unpack2(tc::mul2(tc::pack2(x.x, x.y), ff), y.x, y.y);
  tc::unpack2(tc::mul2(tc::pack2(x.z, x.w), ff), y.z, y.w);
  return y;
}
// eight columns (chunk c) of row r of an operand tile: the pieces' 16 bytes, 128B-swizzled
__device__ __forceinline__ void put_split(uint32_t tile, uint32_t piece_bytes, int r, int c, const float4 &a, const float4 &b) {
  uint32_t h[4], m[4], l[4];
  split2(a.x, a.y, h[0], m[0], l[0]);
  split2(a.z, a.w, h[1], m[1], l[1]);
  split2(b.x, b.y, h[2], m[2], l[2]);
  split2(b.z, b.w, h[3], m[3], l[3]);
  const uint32_t at = tile + (uint32_t)(r * 128 + ((c ^ (r & 7)) << 4));
  store16(at, h[0], h[1], h[2], h[3]);
  store16(at + piece_bytes, m[0], m[1], m[2], m[3]);
  store16(at + 2 * piece_bytes, l[0], l[1], l[2], l[3]);
}
// row `slot` of a slice's keys or values
__device__ __forceinline__ const float *entry(const Params &prm, bool values, int slice, int b, int h, int hist, int slot) {
  if (prm.fused && slot >= hist) return row_ptr<float>(values ? prm.V : prm.K, b, h, slot - hist);
  return reinterpret_cast<const float *>((values ? prm.lv.v_pool : prm.lv.k_pool) + slot_row(prm.lv, slice, slot) * 256);
}

// The log-sum-exp of a row from its reference, the largest of its products, and its sum: the logarithm is taken to base e (to base 2 both are
// of larger numbers), and what the sum of the two is rounded by is put right together with kCutOff's part, which by itself would be lost in it.
__device__ __forceinline__ float row_lse_f32(float m, float l, float scale) {
  const float lg = logf(l), sum = fmaf(m, scale, lg);
  if (!(fabsf(sum) < INFINITY)) return sum;
  const float rest = fabsf(m * scale) > fabsf(lg) ? fmaf(m, scale, -sum) + lg : fmaf(m, scale, lg - sum);      // (exact: the larger first)
  return sum + fmaf(m, scale * kCutOff, rest);
}

// Scores that are not numbers, for they are the sums of products with a query's pieces that differ in sign: an infinite key's, or those of numbers near
// the range's end.  A warp takes them again, a thread its row's, 32 keys at a time.  A score with an infinite column is decided by signs: a lane reads
// one key's and hands its masks round.  The others are taken by fp32 FMA, four keys at a time: two columns of each in a lane, handed round likewise,
// and the query put together from its pieces eight columns at a time.  (Few registers, so that the softmax around it spills hardly more than without: with
// the query in 64 of them every launch took 4 % longer.  us per launch of 16 slices x 1 600 queries behind 772
// entries, of keys masked by -inf in a column: none 142, one 164, 32 in a row 179, 32 apart 316, 300 in a row 403; with fp32 FMA for each 142, 171,
// 248, 334, 1 038; fp32 FMA throughout 398.)
struct Repaired { float max; int hopeless; };      // hopeless: the row has a score that is +inf or no number all the same, and so no output that is one
__device__ __noinline__ Repaired repair_scores(const Params &prm, const uint8_t *q_tile, uint32_t buf, int row, int slice, int b, int h, int hist,
                                               int key0, int valid) {
  const int lane = threadIdx.x & 31;
  auto query = [&](int c, float (&q)[8]) {         // columns 8 c .., lifted
    const uint8_t *at = q_tile + row * 128 + ((c ^ (row & 7)) << 4);
    const uint4 h4 = *reinterpret_cast<const uint4 *>(at), m4 = *reinterpret_cast<const uint4 *>(at + kPieceQ), l4 = *reinterpret_cast<const uint4 *>(at + 2 * kPieceQ);
    const uint32_t hw[4] = {h4.x, h4.y, h4.z, h4.w}, mw[4] = {m4.x, m4.y, m4.z, m4.w}, lw[4] = {l4.x, l4.y, l4.z, l4.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      q[2 * i] = (__uint_as_float(hw[i] << 16) + __uint_as_float(mw[i] << 16)) + __uint_as_float(lw[i] << 16);
      q[2 * i + 1] = (__uint_as_float(hw[i] & 0xffff0000u) + __uint_as_float(mw[i] & 0xffff0000u)) + __uint_as_float(lw[i] & 0xffff0000u);
    }
  };
  float over = 0.f;
  uint64_t q_pos = 0, q_neg = 0;         // by column
#pragma unroll 1
  for (int c = 0; c < 8; ++c) {
    float q[8];
    uint32_t pos = 0, neg = 0;
    query(c, q);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      over += q[i] - q[i];
      if (q[i] > 0.f) pos |= 1u << i;
      if (q[i] < 0.f) neg |= 1u << i;
    }
    q_pos |= (uint64_t)pos << (8 * c);
    q_neg |= (uint64_t)neg << (8 * c);
  }
  const bool row_ok = over == 0.f;       // (a query that cannot be split spoils all its scores: its row is done again in the end)
  Repaired r{-INFINITY, 0};
#pragma unroll 1
  for (int j0 = 0; j0 < valid; j0 += 32) {
    uint32_t bad = 0;
#pragma unroll 1
    for (int j = 0; j < 32; j += 8) {
      uint32_t x[8];
      asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];" : "=r"(x[0]), "=r"(x[1]), "=r"(x[2]), "=r"(x[3]),
                   "=r"(x[4]), "=r"(x[5]), "=r"(x[6]), "=r"(x[7]) : "r"(buf + j0 + j));
      tc::tc_wait_ld();
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const float y = __uint_as_float(x[e]);
        if (j0 + j + e >= valid) continue;
        if (__any_sync(0xffffffffu, y != y && row_ok)) bad |= 1u << (j + e);
        r.max = fmaxf(r.max, y);
      }
    }
    if (bad == 0) continue;
    const uint64_t key = (uint64_t)entry(prm, false, slice, b, h, hist, key0 + min(j0 + lane, valid - 1));
    uint64_t k_pos = 0, k_neg = 0;       // the lane's key: its infinite columns
    bool nan = false;
    if ((bad >> lane) & 1u) {
#pragma unroll 1
      for (int c = 0; c < 16; c += 4) {
        float4 z[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) z[i] = reinterpret_cast<const float4 *>(key)[c + i];
        uint32_t pos = 0, neg = 0;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const float y = i % 4 == 0 ? z[i / 4].x : i % 4 == 1 ? z[i / 4].y : i % 4 == 2 ? z[i / 4].z : z[i / 4].w;
          if (y == INFINITY) pos |= 1u << i;
          if (y == -INFINITY) neg |= 1u << i;
          nan = nan || y != y;
        }
        k_pos |= (uint64_t)pos << (4 * c);
        k_neg |= (uint64_t)neg << (4 * c);
      }
    }
    const uint32_t signs = __ballot_sync(0xffffffffu, nan || (k_pos | k_neg) != 0), nans = __ballot_sync(0xffffffffu, nan);
    // a score, not lifted, to its column in TMEM
    auto put = [&](int j, float y) {
      uint32_t x;
      asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(x) : "r"(buf + j0 + j));
      tc::tc_wait_ld();
      if (row_ok && __uint_as_float(x) != __uint_as_float(x)) {
        if (!(y < INFINITY)) r.hopeless = 1;
        x = __float_as_uint(y * kLift);
        r.max = fmaxf(r.max, y * kLift);
      }
      __syncwarp();
      asm volatile("tcgen05.st.sync.aligned.32x32b.x1.b32 [%0], {%1};" ::"r"(buf + j0 + j), "r"(x) : "memory");
    };
#pragma unroll 1
    for (uint32_t left = signs; left != 0; left &= left - 1) {
      const int j = __ffs(left) - 1;
      const uint64_t pos = __shfl_sync(0xffffffffu, k_pos, j), neg = __shfl_sync(0xffffffffu, k_neg, j);
      const bool up = ((pos & q_pos) | (neg & q_neg)) != 0, down = ((pos & q_neg) | (neg & q_pos)) != 0;
      const bool none = ((nans >> j) & 1u) || (up && down) || ((pos | neg) & ~(q_pos | q_neg)) != 0;
      put(j, none ? NAN : up ? INFINITY : -INFINITY);
    }
    bad &= ~signs;
#pragma unroll 1
    while (bad != 0) {
      uint32_t rest = bad;
      float2 k[4];
      float s[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int j = rest != 0 ? __ffs(rest) - 1 : 0;
        rest &= rest - 1;
        k[e] = reinterpret_cast<const float2 *>(__shfl_sync(0xffffffffu, key, j))[lane];
        s[e] = 0.f;
      }
#pragma unroll 1
      for (int c = 0; c < 8; ++c) {
        float q[8];
        query(c, q);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float x = q[i] * (1.f / kLift);
#pragma unroll
          for (int e = 0; e < 4; ++e) s[e] = fmaf(x, __shfl_sync(0xffffffffu, i & 1 ? k[e].y : k[e].x, 4 * c + (i >> 1)), s[e]);
        }
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        if (bad == 0) break;
        put(__ffs(bad) - 1, s[e] * (1.f - kCutOff));       // (as the tensor core would leave it)
        bad &= bad - 1;
      }
    }
  }
  tc::tc_wait_st();
  return r;
}

// Rows whose sums or columns by pieces are no numbers all the same (an infinite value's all, an infinite query's own), by fp32 FMA over the entries
// [from, to): two threads per row, which share its columns by 16-byte pieces, keys and values in tiles of 64 where their pieces lay.  For rows that few
// will ever need, so without pipelining: 16 slices x 1 600 queries behind 772 entries, all rows, 683 us.
__device__ __noinline__ void redo_rows(const Params &prm, uint8_t *smem, const uint32_t *marks) {
  const int tid = threadIdx.x, row = tid >> 1, half = tid & 1;
  // (worked out once more: passed, they would have to outlive the softmax)
  const int slice = blockIdx.y, b = slice / prm.lv.n_heads, h = slice - b * prm.lv.n_heads, q0 = blockIdx.x * kRows;
  const int hist = prm.lv.hist_len[slice], L = min(hist + prm.n_k, prm.room), tiles = (L + kKeys - 1) / kKeys;
  const int from = tiles * (int)blockIdx.z / (int)gridDim.z * kKeys, to = min(tiles * ((int)blockIdx.z + 1) / (int)gridDim.z * kKeys, L);
  float *Ks = reinterpret_cast<float *>(smem + kOffK), *Vs = reinterpret_cast<float *>(smem + kOffV);
  const float cut = copysignf(1.f - kCutOff, prm.scale), c = prm.weight_scale;       // (products as the tensor core would leave them)
  float4 q[8], o[8];
  const float4 *qp = reinterpret_cast<const float4 *>(row_ptr<float>(prm.Q, b, h, min(q0 + row, prm.n_k - 1)));
#pragma unroll
  for (int i = 0; i < 8; ++i) { q[i] = qp[2 * i + half]; o[i] = make_float4(0.f, 0.f, 0.f, 0.f); }
  float m = kNoMax, l = 0.f;
#pragma unroll 1
  for (int t0 = from; t0 < to; t0 += kKeys) {
    __syncthreads();                     // the tile before has been read
    {
      const int r = tid >> 2;
      const bool there = t0 + r < to;
      const float4 *k = reinterpret_cast<const float4 *>(entry(prm, false, slice, b, h, hist, there ? t0 + r : from));
      const float4 *v = reinterpret_cast<const float4 *>(entry(prm, true, slice, b, h, hist, there ? t0 + r : from));
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int piece = (tid & 3) + 4 * u;
        const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f), x = there ? k[piece] : zero, y = there ? v[piece] : zero;
        reinterpret_cast<float4 *>(Ks)[r * 16 + piece] = x;
        reinterpret_cast<float4 *>(Vs)[r * 16 + piece] = y;
      }
    }
    __syncthreads();
    const int n = min(kKeys, to - t0);
#pragma unroll 1
    for (int j = 0; j < n; j += 8) {
      float s[8], mx = m;
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        float a = 0.f, a2 = 0.f;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float4 z = reinterpret_cast<const float4 *>(Ks)[(j + e) * 16 + 2 * i + half];
          a = fmaf(q[i].x, z.x, a);
          a2 = fmaf(q[i].y, z.y, a2);
          a = fmaf(q[i].z, z.z, a);
          a2 = fmaf(q[i].w, z.w, a2);
        }
        a += a2;
        a += __shfl_xor_sync(0xffffffffu, a, 1);
        s[e] = j + e < n ? a * cut : -INFINITY;
        mx = fmaxf(mx, s[e]);
      }
      const float f = exp2f((m - mx) * c);
      float sum = 0.f;
#pragma unroll
      for (int i = 0; i < 8; ++i) o[i] = make_float4(o[i].x * f, o[i].y * f, o[i].z * f, o[i].w * f);
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const float p = exp2f((s[e] - mx) * c);
        sum += p;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float4 z = reinterpret_cast<const float4 *>(Vs)[(j + e) * 16 + 2 * i + half];
          o[i] = make_float4(fmaf(p, z.x, o[i].x), fmaf(p, z.y, o[i].y), fmaf(p, z.z, o[i].z), fmaf(p, z.w, o[i].w));
        }
      }
      l = fmaf(l, f, sum);
      m = mx;
    }
  }
  if ((marks[row >> 5] >> (row & 31)) & 1u) {
#pragma unroll
    for (int i = 0; i < 8; ++i) *reinterpret_cast<float4 *>(smem + kOffQ + row * 256 + (((2 * i + half) ^ (row & 7)) << 4)) = o[i];
    if (half == 0) {
      reinterpret_cast<float2 *>(smem + kOffStat)[row] = make_float2(m, l);
      if (gridDim.z == 1 && prm.lse != nullptr) prm.lse[(size_t)slice * prm.n_k + q0 + row] = row_lse_f32(m, l, fabsf(prm.scale));
    }
  }
}

// The window's logits against the 64 entries of a tile, as score_logits_kernel takes them from the pages.
__device__ __noinline__ void window_logits(const Params &prm, float *sm, int slice, int b, int h, int hist, int L, int tile) {
  constexpr int LD = 68;
  float *Qs = sm, *Ks = sm + 64 * LD;
  const int c = threadIdx.x & 15, j0 = tile * kKeys;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int r = (threadIdx.x >> 4) + 16 * u;
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    const float4 q = r < prm.w ? reinterpret_cast<const float4 *>(row_ptr<float>(prm.Q, b, h, prm.win_pos[r]))[c] : zero;
    const float4 k = j0 + r < L ? reinterpret_cast<const float4 *>(entry(prm, false, slice, b, h, hist, j0 + r))[c] : zero;
    *reinterpret_cast<float4 *>(Qs + r * LD + 4 * c) = q;
    *reinterpret_cast<float4 *>(Ks + r * LD + 4 * c) = k;
  }
  __syncthreads();
  tile_logits<64>(Qs, Ks, prm.w, j0, L, prm.win_logits + (size_t)slice * prm.w * prm.ld_l, prm.ld_l, prm.scale);
}

// grid (ceil(n_k / 128), n_slices and, where the window is recorded, as many as its key tiles take, split); dynamic shared memory kSmemBytes.
__global__ void __launch_bounds__(kThreads, 2) attend_f32_tc_kernel(const __grid_constant__ Params prm) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t base = tc::smem_u32(smem_raw);
  auto bar = [&](int i) { return base + kOffBar + 8u * (uint32_t)i; };
  volatile uint32_t *tmem_slot = reinterpret_cast<volatile uint32_t *>(smem_raw + kOffBar + 32);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(smem_raw + kOffBar + 36);
  volatile int *leave_slot = reinterpret_cast<volatile int *>(smem_raw + kOffBar + 40);
  uint32_t *marks = reinterpret_cast<uint32_t *>(smem_raw + kOffBar + 44);      // rows that are to be done again, by warp
  const LayerView &lv = prm.lv;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int slice = blockIdx.y, b = slice / lv.n_heads, h = slice - b * lv.n_heads;
  const int q0 = blockIdx.x * kRows, n_k = prm.n_k, n_split = gridDim.z;
  int *status = lv.status;
  if (slice >= lv.n_slices) {
    const int e = ((slice - lv.n_slices) * (int)gridDim.x + (int)blockIdx.x) * n_split + (int)blockIdx.z;
    const int sl = e / prm.win_tiles, tile = e - sl * prm.win_tiles;
    if (sl >= lv.n_slices) return;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int hist = lv.hist_len[sl], L = min(hist + n_k, prm.room);
    if (tile * kKeys < L) window_logits(prm, reinterpret_cast<float *>(smem_raw), sl, sl / lv.n_heads, sl % lv.n_heads, hist, L, tile);
    return;
  }
  if (tid == 0) {
    tc::mbar_init(bar(bV), 4);           // (one lane of each operand warp)
    for (int i = bPv; i <= bS + 1; ++i) tc::mbar_init(bar(i), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  } else if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(base + kOffBar + 32), "r"(kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  // (what is above runs while the kernel before this one ends; see attend_tc_kernel)
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int hist = lv.hist_len[slice];
  // A slice that outgrows its pages is cut off, so that no slot behind the page table is looked up.
  const int L = min(hist + n_k, prm.room);
  const int tiles = (L + kKeys - 1) / kKeys;
  const int lo = tiles * (int)blockIdx.z / n_split;
  if (tid == 0) {
    *abort_flag = 0;
    // (an earlier CTA's wait has run out: do not pile on.  One thread decides for the CTA.)
    int leave = *reinterpret_cast<volatile int *>(status) == kDevTimeout;
    if (base & 1023u) { atomicExch(status, kDevCheck); leave = 1; }
    if (hist + n_k > prm.room) atomicExch(status, kDevCheck);
    *leave_slot = leave;
    if (!leave && blockIdx.x == 0 && blockIdx.z == 0) lv.next_len[slice] = L;      // unless a compress of this scale evicts
  }
  const int c = tid & 7, r0 = (tid & 127) >> 3;
  // The operand warps' part of a tile: chunk c of rows r0, r0 + 16, ..
  long long at[4];                     // where the rows of the tile whose keys were loaded last lie in the pages, in bytes
  auto load = [&](bool values, int tile, float4 (&x)[4][2]) {      // (the keys of a tile before its values)
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int slot = tile * kKeys + r0 + 16 * u;
      const bool outside = prm.fused && slot >= hist;
      x[u][0] = x[u][1] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (slot < L) {
        if (!values && !outside) at[u] = (long long)slot_row(lv, slice, slot) * 256;
        const char *row = outside ? reinterpret_cast<const char *>(row_ptr<float>(values ? prm.V : prm.K, b, h, slot - hist))
                                  : (values ? lv.v_pool : lv.k_pool) + at[u];
        x[u][0] = reinterpret_cast<const float4 *>(row)[2 * c];
        x[u][1] = reinterpret_cast<const float4 *>(row)[2 * c + 1];
      }
    }
  };
  float4 kx[4][2], vx[4][2];
  if (warp >= 4 && lo < tiles * ((int)blockIdx.z + 1) / n_split) {       // (on their way while Q is split)
    load(false, lo, kx);
    load(true, lo, vx);
  }
  // Q: a thread takes one chunk of eight columns of four rows.  (Of a negative scale Q takes the sign, so that the largest product is
  // the largest score.)
  const float lift = copysignf(kLift, prm.scale);
  {
    float4 x[4][2];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int r = (tid >> 3) + 32 * u, c = tid & 7;
      x[u][0] = x[u][1] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (q0 + r < n_k) {
        const float4 *src = reinterpret_cast<const float4 *>(row_ptr<float>(prm.Q, b, h, q0 + r)) + 2 * c;
        x[u][0] = times(__ldg(src), lift);
        x[u][1] = times(__ldg(src + 1), lift);
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) put_split(base + kOffQ, kPieceQ, (tid >> 3) + 32 * u, tid & 7, x[u][0], x[u][1]);
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const bool leave = *leave_slot != 0;
  const int nt = leave ? 0 : tiles * ((int)blockIdx.z + 1) / n_split - lo;
  const uint32_t tmem = *tmem_slot;
  float *rows_out = reinterpret_cast<float *>(smem_raw + kOffQ);               // [row][64], 16-byte pieces permuted by the row
  float2 *stat_out = reinterpret_cast<float2 *>(smem_raw + kOffStat);
  constexpr uint32_t dhi = tc::desc_hi(1024);
  constexpr uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((64u >> 3) << 17) | ((128u >> 4) << 24);    // bf16, N = 64, M = 128
  constexpr uint32_t idesc_pv = idesc | (1u << 16);                                                            // B is MN-major
  // S of tile i and P V of tile i have landed (waits)
  auto s_landed = [&](int i) { return tc::mbar_wait_warp(bar(bS + (i & 1)), (i >> 1) & 1, abort_flag, status); };
  auto pv_landed = [&](int i) { return tc::mbar_wait_warp(bar(bPv), i & 1, abort_flag, status); };

  if (warp >= 4) {
    // ---------------------------------------------------------------- operands
    auto put = [&](bool values, int tile, const float4 (&x)[4][2]) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (values) put_split(base + kOffV, kPieceK, r0 + 16 * u, c, times(x[u][0], kLift), times(x[u][1], kLift));
        else put_split(base + kOffK, kPieceK, r0 + 16 * u, c, x[u][0], x[u][1]);
      }
      if (prm.copy_in && tile * kKeys + kKeys > hist && tile % (int)gridDim.x == (int)blockIdx.x) {      // (the CTAs of a slice take turns)
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int slot = tile * kKeys + r0 + 16 * u;
          if (slot < hist || slot >= L) continue;
          const size_t row = slot_row(lv, slice, slot);
          float4 *dst = reinterpret_cast<float4 *>((values ? lv.v_pool : lv.k_pool) + row * 256) + 2 * c;
          dst[0] = x[u][0];
          dst[1] = x[u][1];
          if (!values && c == 0) lv.pos_pool[row] = prm.n_prev + slot - hist;
        }
      }
    };
    const uint32_t q_lo = tc::desc_lo(base + kOffQ, 16), k_lo = tc::desc_lo(base + kOffK, 16);
    int issued = 0;                      // products S issued by warp 4
    auto mma_s = [&](int i) {            // products of pieces, the smallest first
      constexpr int A[6] = {2, 0, 1, 1, 0, 0}, B[6] = {0, 2, 1, 0, 1, 0};
      tc_fence_after();
#pragma unroll
      for (int e = 0; e < 6; ++e) mma4_ss(tmem + kBufCols * (i & 1), q_lo + A[e] * (kPieceQ >> 4), k_lo + B[e] * (kPieceK >> 4), dhi, idesc, e > 0);
      if (tc::elect_one()) tc::tc_commit(bar(bS + (i & 1)));
      __syncwarp();
      issued = i + 1;
    };
    auto keys_there = [&] {              // all four warps have left their part
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      asm volatile("bar.sync 3, 128;" ::: "memory");
    };
    auto announce_v = [&] {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(bar(bV));
    };
    bool ok = true;
    // (a warp whose wait gives up goes on to meet the others at the named barrier, which knows no limit)
#pragma unroll 1
    for (int i = -1; i < nt; ++i) {
      const bool more = i + 1 < nt;
      ok = ok && (i < 0 || s_landed(i));                      // K_i has been read
      if (more) {
        if (ok) put(false, lo + i + 1, kx);
        if (i < 0 && nt > 1) load(false, lo + 1, kx);
        keys_there();
      }
      ok = ok && (i <= 0 || pv_landed(i - 1));                // V_{i-1} has been read, and P_{i-1}
      if (warp == 4 && more && ok) mma_s(i + 1);
      if (ok && i != 0 && nt > 0) {                           // (V_0 before the softmax of tile 0)
        put(true, lo + max(i, 0), vx);
        announce_v();
      }
      if (ok && i >= 0) {
        if (more) load(true, lo + i + 1, vx);
        if (i + 2 < nt) load(false, lo + i + 2, kx);
      }
    }
    // (given up: what has been issued must be through before TMEM and shared memory are anybody else's)
    if (!ok && issued > 0) tc::mbar_drain(bar(bS + ((issued - 1) & 1)), ((issued - 1) >> 1) & 1);
  } else {
    // ---------------------------------------------------------------- softmax
    const uint32_t v_lo = tc::desc_lo(base + kOffV, 16);
    auto mma_pv = [&](int i) {
      const uint32_t p = tmem + kBufCols * (i & 1);
      constexpr uint32_t step_v = kPieceK >> 4;
      tc_fence_after();
      mma4_ts<8>(tmem + kColO, p + kColPl, v_lo, dhi, idesc_pv, 0);
      mma4_ts<16>(tmem + kColO, p, v_lo + 2 * step_v, dhi, idesc_pv, 1);
      mma4_ts<16>(tmem + kColO, p + kColPm, v_lo + step_v, dhi, idesc_pv, 1);
      mma4_ts<16>(tmem + kColO, p + kColPm, v_lo, dhi, idesc_pv, 1);
      mma4_ts<16>(tmem + kColO, p, v_lo + step_v, dhi, idesc_pv, 1);
      mma4_ts<16>(tmem + kColO, p, v_lo, dhi, idesc_pv, 1);
      if (tc::elect_one()) tc::tc_commit(bar(bPv));
      __syncwarp();
    };
    const int row = warp * 32 + lane;
    const uint32_t lane_addr = tmem + ((uint32_t)(warp * 32) << 16);
    const float c = prm.weight_scale * (1.f / kLift);
    uint64_t o[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) o[i] = 0ull;
    float m = kNoMax, l = 0.f, l_rest = 0.f;       // l_rest: what the additions to l have rounded off
    int hopeless = 0;                              // the row has a score that makes its output no number
    // (o + P V of the tile before) f
    auto add_products = [&](float f, bool scale) {
      const uint64_t ff = tc::pack2(f, f);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        uint32_t x[16];
        tc::tc_ld16(lane_addr + kColO + 16 * e, x);
        tc::tc_wait_ld();
#pragma unroll
        for (int i = 0; i < 8; ++i) o[8 * e + i] = tc::add2(o[8 * e + i], tc::pack2(__uint_as_float(x[2 * i]), __uint_as_float(x[2 * i + 1])));
      }
      if (scale) {
#pragma unroll
        for (int i = 0; i < 32; ++i) o[i] = tc::mul2(o[i], ff);
      }
    };
    // The softmax of tile i (masked: a ragged one).  f: what the sums so far are to be scaled by; returns whether any is not 1.
    auto sweep = [&](int i, float &f, auto masked) {
      const int valid = L - (lo + i) * kKeys;
      const uint32_t buf = lane_addr + kBufCols * (i & 1);
      auto real = [&](int key) { return !decltype(masked)::value || key < valid; };
      float mx = -INFINITY;
#pragma unroll 4                       // (all of it; a plain unroll is scheduled otherwise, with 20 bytes more of spills)
      for (int e = 0; e < 4; ++e) {
        uint32_t x[16];
        tc::tc_ld16(buf + 16 * e, x);
        tc::tc_wait_ld();
#pragma unroll
        for (int q = 0; q < 16; q += 2)
          mx = max3_nan(mx, real(16 * e + q) ? __uint_as_float(x[q]) : -INFINITY, real(16 * e + q + 1) ? __uint_as_float(x[q + 1]) : -INFINITY);
      }
      if (__any_sync(0xffffffffu, mx != mx)) {
        const Repaired r = repair_scores(prm, smem_raw + kOffQ, buf, row, slice, b, h, hist, (lo + i) * kKeys, min(valid, kKeys));
        mx = r.max;
        hopeless |= r.hopeless;
      }
      mx = fmaxf(m, mx);
      const bool scale = __any_sync(0xffffffffu, mx > m);
      if (scale) {
        f = tc::ex2((m - mx) * c);
        l *= f;
        l_rest *= f;
        m = mx;
      }
      const uint64_t c2 = tc::pack2(c, c), negm2 = tc::pack2(-m, -m);
      uint64_t sum2[2] = {0ull, 0ull};
#pragma unroll 1
      for (int e = 0; e < 4; ++e) {
        uint32_t x[16], ph[8], pm[8], pl[8];
        tc::tc_ld16(buf + 16 * e, x);
        tc::tc_wait_ld();
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          float a0, a1;
          const uint64_t s2 = tc::pack2(__uint_as_float(x[2 * q]), __uint_as_float(x[2 * q + 1]));
          tc::unpack2(tc::mul2(tc::add2(s2, negm2), c2), a0, a1);
          a0 = real(16 * e + 2 * q) ? tc::ex2(a0) : 0.f;
          a1 = real(16 * e + 2 * q + 1) ? tc::ex2(a1) : 0.f;
          sum2[q & 1] = tc::add2(sum2[q & 1], tc::pack2(a0, a1));
          split2(a0, a1, ph[q], pm[q], pl[q]);
        }
        tc_st8(buf + 16 * e, ph);
        tc_st8(buf + 16 * e + kColPm, pm);
        tc_st8(buf + 8 * e + kColPl, pl);
      }
      float s0, s1, s2, s3;
      tc::unpack2(sum2[0], s0, s1);
      tc::unpack2(sum2[1], s2, s3);
      const float add = (s0 + s1) + (s2 + s3), sum = l + add, part = sum - l;
      l_rest += (l - (sum - part)) + (add - part);
      l = sum;
      return scale;
    };
    bool ok = true;
    int issued = 0;                      // products P V issued by warp 0
    for (int i = 0; i < nt; ++i) {
      // (a warp whose wait gives up goes on to meet the others at the named barrier, which knows no limit)
      ok = ok && s_landed(i);
      if (ok) {
        tc_fence_after();
        float f = 1.f;
        const bool scale = L - (lo + i) * kKeys < kKeys ? sweep(i, f, std::true_type{}) : sweep(i, f, std::false_type{});
        if (i > 0) {
          ok = pv_landed(i - 1);
          tc_fence_after();
          if (ok) add_products(f, scale);
        }
        tc::tc_wait_st();
        tc_fence_before();
      }
      asm volatile("bar.sync 2, 128;" ::: "memory");
      if (warp == 0) {
        ok = ok && tc::mbar_wait_warp(bar(bV), i & 1, abort_flag, status);
        if (ok) {
          mma_pv(i);
          ++issued;
        }
      }
    }
    if (warp == 0) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (nt > 0) ok = ok && pv_landed(nt - 1);
    tc_fence_after();
    if (ok && nt > 0) add_products(1.f, false);
    // (given up: as above)
    if (!ok && issued > 0) tc::mbar_drain(bar(bPv), (issued - 1) & 1);
    l += l_rest;
    if (m != kNoMax) m *= 1.f / kLift;
    float *mine = rows_out + row * 64;
    float amax = 0.f;
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      float x0, x1, x2, x3;
      tc::unpack2(o[2 * q], x0, x1);
      tc::unpack2(o[2 * q + 1], x2, x3);
      amax += (x0 - x0) + (x1 - x1) + (x2 - x2) + (x3 - x3);      // zero, unless one of them is not a number
      *reinterpret_cast<float4 *>(mine + ((q ^ (row & 7)) << 2)) = times(make_float4(x0, x1, x2, x3), 1.f / kLift);
    }
    const unsigned spoiled = __ballot_sync(0xffffffffu, nt > 0 && ok && q0 + row < n_k && !hopeless && !(amax == 0.f && l > 0.f && l < INFINITY));
    if (lane == 0) marks[warp] = spoiled;
    stat_out[row] = make_float2(m, ok && !leave ? l : -1.f);             // (no sum is negative: a part that has been given up)
    if (n_split == 1 && ok && nt > 0 && q0 + row < n_k) {
      if (prm.lse != nullptr) prm.lse[(size_t)slice * n_k + q0 + row] = row_lse_f32(m, l, fabsf(prm.scale));
    }
    tc_fence_before();
  }
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
  }
  if ((marks[0] | marks[1] | marks[2] | marks[3]) != 0u) {
    redo_rows(prm, smem_raw, marks);
    __syncthreads();
  }
  const int ty = tid >> 4, tx = tid & 15, rows = min(kRows, n_k - q0);
  if (n_split == 1) {
    if (leave) return;
    for (int r = ty; r < rows; r += 16) {
      const float sum = stat_out[r].y;
      if (sum < 0.f) continue;
      const float inv = 1.f / sum;
      const float4 x = *reinterpret_cast<const float4 *>(rows_out + r * 64 + ((tx ^ (r & 7)) << 2));
      *reinterpret_cast<float4 *>(const_cast<float *>(row_ptr<float>(prm.O, b, h, q0 + r)) + tx * 4) = make_float4(x.x * inv, x.y * inv, x.z * inv, x.w * inv);
    }
    return;
  }
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
  auto peer = [&](const void *p, int cta) { return tc::remote((uint32_t)__cvta_generic_to_shared(p), cta); };
  const int r_lo = rows * (int)blockIdx.z / n_split, r_hi = leave ? r_lo : rows * ((int)blockIdx.z + 1) / n_split;
  for (int r = r_lo + ty; r < r_hi; r += 16) {
    float4 x[kMaxSplit];
    float me[kMaxSplit], le[kMaxSplit], M = kNoMax;
    bool whole = true;
#pragma unroll
    for (int e = 0; e < kMaxSplit; ++e) {
      x[e] = make_float4(0.f, 0.f, 0.f, 0.f);
      me[e] = kNoMax; le[e] = 0.f;
      if (e < n_split) {
        asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(me[e]), "=f"(le[e]) : "r"(peer(stat_out + r, e)));
        asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(x[e].x), "=f"(x[e].y), "=f"(x[e].z), "=f"(x[e].w)
                     : "r"(peer(rows_out + r * 64 + ((tx ^ (r & 7)) << 2), e)));
      }
    }
#pragma unroll
    for (int e = 0; e < kMaxSplit; ++e) {
      M = fmaxf(M, me[e]);
      whole = whole && !(le[e] < 0.f);
    }
    if (!whole) continue;
    float sum = 0.f, a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
#pragma unroll
    for (int e = 0; e < kMaxSplit; ++e) {
      const float f = exp2f((me[e] - M) * prm.weight_scale);
      sum = fmaf(f, le[e], sum);
      a0 = fmaf(f, x[e].x, a0); a1 = fmaf(f, x[e].y, a1); a2 = fmaf(f, x[e].z, a2); a3 = fmaf(f, x[e].w, a3);
    }
    const float inv = 1.f / sum;
    *reinterpret_cast<float4 *>(const_cast<float *>(row_ptr<float>(prm.O, b, h, q0 + r)) + tx * 4) = make_float4(a0 * inv, a1 * inv, a2 * inv, a3 * inv);
    if (tx == 0 && prm.lse != nullptr) prm.lse[(size_t)slice * n_k + q0 + r] = row_lse_f32(M, sum, fabsf(prm.scale));
  }
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");     // nobody leaves while a peer still reads here
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

}  // namespace f32
}  // namespace scalekv
