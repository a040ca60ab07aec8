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
//   accumulators and 1184-double slots 12 warps fitted and the pipe was 91 % busy on the
//   2000 x 2000 banded product; 16 warps keep it 94 % busy (4000 x 4000: 20.8 and, with the
//   tail split, 18.6 ms).  A 23 x 23 block is then cut into tiles of 13 and 10 rows.
// * MR = 17, slots of 1184 doubles, three CTAs per SM ("wide"): for plans with rows of C
//   of 321 to 544 elements, for contractions read in place as slabs (which need whole
//   C blocks) with blocks of 321 to 544 elements, and where its splits and panels save
//   instructions (wide_saves).
constexpr int kNarrowR = 10, kWideR = 17;
constexpr int kNarrowSlot = 896, kWideSlot = 1184;
constexpr int kStageWarps = 4;    // warps per CTA
constexpr int kF64Desc = kF64DescWords;

// descriptor word 7: whole-tile split, tail split, and whether every panel is summed by itself
// and then added (full rounds, tail)
__host__ __device__ __forceinline__ int f64_split_word(int s, int tail, int fresh = 0,
                                                       int tail_fresh = 0) {
  return s | (tail << 8) | (fresh << 16) | (tail_fresh << 17);
}

// Inner split of a tile (descriptor word 7): the s <= smax of the tile's class that needs the
// fewest FP64 warp instructions -- ceil(s mt n / 32) for each of the ceil(w / s) steps of a
// panel of width w, plus (s - 1) ceil(mt n / 32) adds for the final sums -- when it saves
// anything on a tile with at least kSplitLongInner inner elements in all, at least 1/8 of the
// other count on one with kSplitMinInner or more, else 1 (on short tiles the final sums cost
// more than the idle lanes).  choose_tile weighs it against the tail split.
constexpr int kMaxSplit = 16;
constexpr int kSplitMinInner = 48;
constexpr int kSplitLongInner = 128;

// FP64 instructions of a tile split s ways whose steps number W, and whether the best of
// them (cb) is worth it against c1 unsplit ones on w1 inner elements
__host__ __device__ __forceinline__ long long split_cost(int s, int mn, long long W) {
  return (long long)((s * mn + 31) / 32) * W + (s - 1) * ((mn + 31) / 32);
}
__host__ __device__ __forceinline__ bool split_pays(long long cb, long long c1, long long w1) {
  return w1 >= kSplitMinInner && (w1 >= kSplitLongInner ? cb < c1 : 8 * cb <= 7 * c1);
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

__host__ __device__ __forceinline__ TailCost tail_cost(int mn, int smax) {
  TailCost C;
  const int rem = mn & 31;
  C.t[0] = 1;
  if (rem) {
    const int most = smax < kMaxSplit ? smax : kMaxSplit;
    C.t[0] = 32 / rem < most ? 32 / rem : most;
  }
  C.t[1] = (C.t[0] + 1) >> 1;
  C.w1 = 0;
  for (int i = 0; i < 2; ++i) {
    C.c[i] = (C.t[i] > 1) + (C.t[i] > 2) + (C.t[i] > 4) + (C.t[i] > 8);  // ceil(log2 t)
    C.inv[i] = (65535 + C.t[i]) / C.t[i];
  }
  return C;
}

__host__ __device__ __forceinline__ void tail_add(TailCost &C, int w) {
  C.w1 += w;
  // panels are at most a slot wide, w <= kWideSlot
  C.c[0] += ((unsigned)(w + C.t[0] - 1) * C.inv[0]) >> 16;
  C.c[1] += ((unsigned)(w + C.t[1] - 1) * C.inv[1]) >> 16;
}

// FP64 instructions of the tile without a whole-tile split
__host__ __device__ __forceinline__ long long tail_total(const TailCost &C, int mn) {
  const long long t = C.c[0] < C.c[1] ? C.c[0] : C.c[1];
  return (mn >> 5) * C.w1 + ((mn & 31) ? (t < C.w1 ? t : C.w1) : 0);
}

__host__ __device__ __forceinline__ int tail_of(const TailCost &C) {
  const int i = C.c[1] < C.c[0] ? 1 : 0;
  return C.t[i] > 1 && C.c[i] < C.w1 ? C.t[i] : 1;
}

// What a whole-tile split's cost is formed from: steps[s] = sum of ceil(w / s) over the panels
// (32 bits hold a tile's: its inner elements are elements of A, which 31 bits index)
template <class T>
struct SplitSteps {
  T steps[kMaxSplit + 1] = {};
  __host__ __device__ __forceinline__ void add(int w, T times = 1) {
#pragma unroll
    for (int s = 2; s <= kMaxSplit; ++s) steps[s] += times * (T)((unsigned)(w + s - 1) / s);
  }
};

// an add of a fresh panel waits for the panel's chain, with no other FMA of the warp behind it:
// 4.7 % of the time of 10 x 10 and 5 x 13 blocks over panels of 35, 12 % over panels of 13,
// where the added instructions are 2.7 % and 7.3 %
constexpr int kFreshAdd = 2;

struct TileChoice {
  int split = 1, tail = 1, fresh = 0, tail_fresh = 0;
  long long plain = 0;      // instructions with the tail split alone
  long long cost = 0;       // of what was chosen
  long long saved = 0;      // plain minus cost where a whole-tile split was chosen
  long long unsplit = 0;    // without any split
  long long reference = 0;  // what the reference split saves of that
};

// the largest whole-tile split whose partial sums fit `elems` accumulators and a slot
__host__ __device__ __forceinline__ int split_bound(int smax, int mn, int elems, int slot) {
  const int room = (elems < slot ? elems : slot) / (mn > 1 ? mn : 1);
  const int most = smax < kMaxSplit ? smax : kMaxSplit;
  return room < most ? room : most;
}

// Whether choose_tile may split a tile and reads `steps`.  A split saves at most the idle lanes,
// so short tiles (which split for 1/8 of the instructions) need 1/8 of them idle: the 1.3 M tiles
// of the 4000 x 4000 banded plan are mostly short, and going through their splits took 0.25 ms.
__host__ __device__ __forceinline__ bool tile_may_split(long long w1, int smax, int mn, int tile,
                                                        int slot, bool whole) {
  const int lanes = (mn + 31) & ~31, idle = lanes - mn;
  return w1 >= kSplitMinInner && idle > 0 && (w1 >= kSplitLongInner || 8 * idle >= lanes) &&
         split_bound(smax, mn, whole ? 32 * kWideR : tile, slot) >= 2;
}

// the choice for a tile that tile_may_split turns down (see below)
__host__ __device__ __forceinline__ TileChoice choose_tile(const TailCost &C, int mn, long long ne) {
  TileChoice R;
  R.tail = tail_of(C);
  R.plain = R.cost = tail_total(C, mn);
  R.unsplit = ((mn + 31) >> 5) * C.w1;
  R.fresh = R.tail > 1 && mn >= 32 && C.w1 >= kSplitLongInner && C.w1 >= 16 * ne;
  R.cost += R.fresh ? kFreshAdd * (mn >> 5) * ne : 0;
  return R;
}

// How a tile of mn outputs, ne panels and C.w1 inner elements in all sums them (tile: elements
// of the largest tile of the plan's shape; slot: doubles of its slots; whole: the tile is a whole
// block).
//
// An output of one chain over w1 elements rounds as sqrt(w1); the s partial sums of a whole-tile
// split as sqrt(w1 / s + s), panels summed by themselves ("fresh") as sqrt(w1 / ne + ne), at one
// add per output and panel.  The tail split is often cheaper than a whole-tile split but leaves the
// full rounds one chain: the relative error of 13 x 13 blocks with 60 products of 35 was 1.2e-15
// that way, 4.4e-16 with the sums split in three.  So where a whole-tile split would pay (at
// least 1/25 of the unsplit instructions, by the accumulators of the wide shape), it is the
// reference: the tile takes the cheapest form whose chains are no longer than that split's.  Parts
// of blocks have none (in the wide shape they would be larger), nor have panels that the slot cuts
// to four elements, whose adds cost a third of the time (200 x 200 blocks 64 -> 84 ms).
// Long sums over wide panels beside a tail split are fresh in any case (an add per 16 elements at
// most; the rank-3 contraction with gradients 2.1e-15, so 0.8e-15, for 1 % of its time): a
// whole-tile split with longer chains takes their place only where the narrow shape's is cheaper
// than the tail split alone.  Elsewhere one chain stays.
template <class T>
__host__ __device__ inline TileChoice choose_tile(const TailCost &C, const SplitSteps<T> &S, int mn,
                                                  long long ne, int smax, int tile, int slot,
                                                  bool whole) {
  TileChoice R = choose_tile(C, mn, ne);
  const long long w1 = C.w1;
  if (!tile_may_split(w1, smax, mn, tile, slot, whole)) return R;
  const unsigned inner = w1 < (1ll << 31) ? (unsigned)w1 : 1u << 31;  // for the chains' lengths
  const int full = R.tail > 1 ? mn >> 5 : (mn + 31) >> 5;
  int s0 = 1;
  long long c0 = R.unsplit, cn = R.unsplit;
  const int narrow = split_bound(smax, mn, 32 * kNarrowR, slot);
  const int now = split_bound(smax, mn, tile, slot);
  const int most = whole && w1 > 4 * ne ? split_bound(smax, mn, 32 * kWideR, slot) : 1;
#pragma unroll
  for (int s = 2; s <= kMaxSplit; ++s) {
    const long long c = split_cost(s, mn, S.steps[s]);
    if (s <= most && c < c0) {
      c0 = c;
      s0 = s;
    }
    if (s <= narrow && c < cn) cn = c;
  }
  const bool narrow_pays = split_pays(cn, R.plain, w1);
  if (!split_pays(c0, R.unsplit, w1) || 25 * (R.unsplit - c0) < R.unsplit) s0 = 1;
  R.reference = s0 > 1 ? R.unsplit - c0 : 0;
  const long long width = (inner + (unsigned)ne - 1) / (unsigned)ne;  // of a panel, on average
  long long limit = s0 > 1 ? inner / (unsigned)s0 + s0 : w1 + ne;
  if (R.fresh && !narrow_pays && width + ne < limit) limit = width + ne;
  long long chain = 0;  // the longest without a whole-tile split
  if (full > 0) {
    if (s0 > 1 && !R.fresh) {
      R.fresh = 1;
      R.cost += kFreshAdd * full * ne;
    }
    chain = R.fresh ? width + ne : w1;
  }
  if (R.tail > 1) {
    const long long one = inner / (unsigned)R.tail + R.tail;
    R.tail_fresh = one > limit;
    R.cost += R.tail_fresh ? kFreshAdd * ne : 0;
    const long long t = R.tail_fresh ? (width + R.tail - 1) / R.tail + ne : one;
    chain = chain > t ? chain : t;
  }
  int best = 1, shortest = 1;
  long long cb = 0, least = chain;
#pragma unroll
  for (int s = 2; s <= kMaxSplit; ++s) {
    const long long c = split_cost(s, mn, S.steps[s]), ch = inner / (unsigned)s + s;
    if (s > now) continue;
    if (ch < least) {
      shortest = s;
      least = ch;
    }
    if (ch <= limit && (best == 1 || c < cb)) {
      best = s;
      cb = c;
    }
  }
  if (chain > limit) {
    if (best == 1) best = shortest;
  } else if (best > 1 && !split_pays(cb, R.cost, w1)) {
    best = 1;
  }
  if (best > 1) {
    R.split = best;
    R.cost = 0;
#pragma unroll
    for (int s = 2; s <= kMaxSplit; ++s)
      if (s == best) R.cost = split_cost(s, mn, S.steps[s]);
    R.saved = R.plain > R.cost ? R.plain - R.cost : 0;
  }
  return R;
}

// Plan-wide sums that decide whether a plan's tiles split at all (apply_split_gate)
struct SplitSums {
  unsigned long long plain, saved, unsplit, reference, marked;
};

__host__ __device__ __forceinline__ int choice_word(const TileChoice &R) {
  return f64_split_word(R.split, R.tail, R.fresh, R.tail_fresh);
}

}  // namespace
}  // namespace bst
