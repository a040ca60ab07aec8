// Passes of the stable counting sort (prims.cu) for n items of nkeys keys.  Host arithmetic only.
#pragma once
#include <cstdint>

namespace bst {

// A pass counts its keys per segment of items (a warp walks a segment): keys x segments cells of
// the histogram and of its scan, 4 bytes each, at most kPartCells of them.
constexpr int64_t kPartCells = int64_t(1) << 24;
// Segment length from which two passes are faster than one: grouping the 3.2 M products of the
// 2000 x 2000 banded plan by 80 000 blocks took 0.95 ms in one pass of segments of 16 384
// (two passes: 0.3 ms), the ragged product by 64 000 size buckets 0.37 ms.
constexpr int64_t kTwoPassSegment = 1024;
// and above which three passes take the place of two: a warp then walks 2048 batches of 32 items
// one after another
constexpr int64_t kThreePassSegment = 1 << 16;

struct PartitionPlan {
  int passes = 1;
  int bits = 31;             // of a pass's digit, lowest first
  int64_t segment[3] = {};   // items per segment of every pass
  int64_t keys[3] = {};      // digit values of every pass
};

// shortest segment of at least `from` items whose cells fit
inline int64_t partition_segment(int64_t n, int64_t keys, int64_t from) {
  int64_t L = from;
  while (L < n && keys * ((n + L - 1) / L) > kPartCells) L *= 2;
  return L;
}

inline PartitionPlan partition_plan(int64_t n, int64_t nkeys) {
  PartitionPlan P;
  P.keys[0] = nkeys;
  P.segment[0] = partition_segment(n, nkeys, 256);
  if (P.segment[0] < kTwoPassSegment && nkeys <= kPartCells) return P;
  int total = 1;  // bits of the largest key
  while ((int64_t(1) << total) < nkeys) ++total;
  for (P.passes = 2;; ++P.passes) {
    P.bits = (total + P.passes - 1) / P.passes;
    int64_t longest = 0;
    for (int i = 0; i < P.passes; ++i) {
      const int64_t rest = ((nkeys - 1) >> (i * P.bits)) + 1, most = int64_t(1) << P.bits;
      P.keys[i] = rest < most ? rest : most;
      P.segment[i] = partition_segment(n, P.keys[i], kTwoPassSegment);
      longest = P.segment[i] > longest ? P.segment[i] : longest;
    }
    if (P.passes == 3 || longest <= kThreePassSegment) return P;
  }
}

}  // namespace bst
