// Tiles of the staged FP64 kernel: its two shapes and the choice of a tile's inner and tail
// splits, shared by the forward schedule (numeric_fp64.cu) and the adjoint's (adjoint.cu).
#pragma once
#include "bst_internal.h"

namespace bst {
namespace {

// Two shapes of the kernel (MR accumulators per lane, tiles up to 32 MR elements):
// * MR = 10, slots of at most 896 doubles: four 4-warp CTAs per SM (at most 128
//   registers, 4 x (2 x 4 x 896 x 8 B + 1 KB) <= 228 KB).  The FP64 pipe takes 16 SM
//   cycles per warp FMA and idles when no resident warp has one ready: with 17
//   accumulators and 1184-double slots 12 warps fitted and the pipe was 94 % busy on the
//   banded product (20.8 ms); 16 warps keep it 96 % busy (18.9 ms with the tail split).  A
//   23 x 23 block is then cut into tiles of 13 and 10 rows.
// * MR = 17, slots of 1184 doubles, three CTAs per SM ("wide"): for plans with rows of C
//   of 321 to 544 elements, and for contractions read in place as slabs (which need whole
//   C blocks) with blocks of 321 to 544 elements.
constexpr int kNarrowR = 10, kWideR = 17;
constexpr int kNarrowSlot = 896, kWideSlot = 1184;
constexpr int kStageWarps = 4;    // warps per CTA
constexpr int kF64Desc = kF64DescWords;

__device__ __forceinline__ int f64_split_word(int s, int tail, int fresh = 0) {
  return s | (tail << 8) | (fresh << 16);
}

// Whether a tile sums every panel by itself and adds it to the output once (split instances
// only): long sums without a whole-tile split, over panels wide enough that the extra add
// costs at most 1/16.  One chain over 300 inner elements rounds twice as far as the partial
// sums of the whole-tile split that the tail split replaces (relative error of the rank-3
// contraction with gradients 2.1e-15, so 0.8e-15, for 1 % of its time).
__device__ __forceinline__ int f64_fresh(long long w1, int ne, int split, int tail) {
  return split == 1 && tail > 1 && w1 >= 128 && w1 >= 16ll * ne;
}

// Inner split of every tile (descriptor word 7): the s <= smax of the tile's class that
// needs the fewest FP64 warp instructions -- ceil(s mt n / 32) for each of the
// ceil(w / s) steps of a panel of width w, plus (s - 1) ceil(mt n / 32) adds for the
// final sums -- when it saves anything on a tile with at least kSplitLongInner inner
// elements in all, at least 1/8 of the unsplit count on one with kSplitMinInner or more,
// else 1 (on short tiles the final sums cost more than the idle lanes).  The plan-wide
// sums of the unsplit counts and of the savings decide whether the plan splits at all
// (refresh_f64_split).
constexpr int kMaxSplit = 16;
constexpr int kSplitMinInner = 48;
constexpr int kSplitLongInner = 128;

// FP64 instructions of a tile split s ways whose steps number W, and whether the best of
// them (cb) is worth it against c1 unsplit ones on w1 inner elements
__device__ __forceinline__ long long split_cost(int s, int mn, long long W) {
  return (long long)((s * mn + 31) / 32) * W + (s - 1) * ((mn + 31) / 32);
}
__device__ __forceinline__ bool split_pays(long long cb, long long c1, long long w1) {
  return w1 >= kSplitMinInner && (w1 >= kSplitLongInner ? cb < c1 : 8 * cb <= 7 * c1);
}

__device__ inline int f64_split_of(int32_t *__restrict__ d, const int4 *__restrict__ ents,
                                   int smax, int tile, int slot_elems, long long c1,
                                   long long &saved) {
  const int mn = (d[3] & 0xfff) * ((d[3] >> 12) & 0xfff), ne = d[2];
  // s m n partial sums fit the accumulators and, for the final sums, one slot
  smax = min(min(smax, kMaxSplit), min(tile, slot_elems) / max(mn, 1));
  int best = 1;
  saved = 0;
  // short tiles (most of a plan of small products) never split: one pass over the widths
  long long w1 = 0;
  for (int e = 0; e < ne; ++e) w1 += ents[(int64_t)d[1] + e].z;
  if (w1 < kSplitMinInner || smax < 2) return 1;
  long long W[kMaxSplit + 1];
  for (int s = 1; s <= max(smax, 1); ++s) W[s] = 0;
  for (int e = 0; e < ne; ++e) {
    const int w = ents[(int64_t)d[1] + e].z;
    for (int s = 1; s <= max(smax, 1); ++s) W[s] += (w + s - 1) / s;
  }
  long long cb = c1;
  for (int s = 2; s <= smax; ++s) {
    const long long c = split_cost(s, mn, W[s]);
    if (c < cb) {
      cb = c;
      best = s;
    }
  }
  if (!split_pays(cb, c1, W[1])) best = 1;
  if (best > 1) saved = c1 - cb;
  return best;
}

// Tail split of a tile (descriptor word 7, bits 8 and up): the t <= 32 / rem lane groups
// over which its last partial round of rem outputs spreads the inner dimension, by FP64
// warp instructions: sum of ceil(w / t) over the entries plus ceil(log2 t) adds, against
// the unsplit sum of w.  The most groups that fit and half of them are compared (13 x 13,
// one product of 13: 6 against 13; 5 x 13: 1 + 4 against 13), bounded like the tile's
// inner split.
struct TailCost {
  int t[2];
  unsigned inv[2];  // ceil(2^16 / t): n / t = n inv >> 16 for n < 4096 and t <= 16
  long long c[2], w1;
};

__device__ __forceinline__ TailCost tail_cost(int mn, int smax) {
  TailCost C;
  const int rem = mn & 31;
  C.t[0] = rem ? min(32 / rem, min(smax, kMaxSplit)) : 1;
  C.t[1] = (C.t[0] + 1) >> 1;
  C.w1 = 0;
  for (int i = 0; i < 2; ++i) {
    C.c[i] = 32 - __clz(C.t[i] - 1);  // ceil(log2 t)
    C.inv[i] = (65535 + C.t[i]) / C.t[i];
  }
  return C;
}

__device__ __forceinline__ void tail_add(TailCost &C, int w) {
  C.w1 += w;
  // panels are at most a slot wide, w <= kWideSlot
  C.c[0] += ((unsigned)(w + C.t[0] - 1) * C.inv[0]) >> 16;
  C.c[1] += ((unsigned)(w + C.t[1] - 1) * C.inv[1]) >> 16;
}

// FP64 instructions of the unsplit tile
__device__ __forceinline__ long long tail_total(const TailCost &C, int mn) {
  return (mn >> 5) * C.w1 + ((mn & 31) ? min(C.w1, min(C.c[0], C.c[1])) : 0);
}

__device__ __forceinline__ int tail_of(const TailCost &C) {
  const int i = C.c[1] < C.c[0] ? 1 : 0;
  return C.t[i] > 1 && C.c[i] < C.w1 ? C.t[i] : 1;
}

}  // namespace
}  // namespace bst
