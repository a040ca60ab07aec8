// Adjoint of the block-sparse multiply (sampled block-sparse products), native FP64.
//
// For C_out = alpha op(A) op(B) + beta C_in with the filter decisions held fixed (a
// kept product stays kept; its derivative through the filter threshold is zero):
//     dop(A)_ik = alpha sum_{j: (i,k,j) kept} dC_ij op(B)_kj^T   on pattern(A)
//     dop(B)_kj = alpha sum_{i: (i,k,j) kept} op(A)_ik^T dC_ij   on pattern(B)
//     dC_in     = beta dC                                        on pattern(C_in)
// The paper defines only the forward product; this is its exact adjoint.
//
// The plan's stack entries are grouped by stored A block and by stored B block once (stable
// counting sort), and every output block sums over its group; no two warps write the same
// element.  Two routes:
// * staged: a stored gradient block is itself a sum of block products X Y whose factors are
//   dC and the other operand, each as stored or transposed, so the forward's staged kernel
//   computes it from a schedule of its own (tiles of gradient blocks, "schedule" below):
//   operands through shared memory, the inner dimension of a tile's last partial round
//   split over idle lanes, tiles dealt by decreasing cost;
// * direct (k_adj_a, k_adj_b): lanes own output elements in passes of 32 RA = 128, one warp
//   per pass, and read dC and the other operand from L1/L2.  It needs no schedule: it runs
//   small plans, plans of large blocks and blocks with a dimension of 2^15 or more.
#include <algorithm>
#include <atomic>
#include <cmath>

#include "bst_internal.h"
#include "fp64_tiles.h"

namespace bst {

// Gradients of one operand: the groups of the direct kernels, or the staged schedule
struct AdjSide {
  int32_t *grp = nullptr, *ptr = nullptr;  // entries grouped by stored block of the operand
  bool staged = false;
  TileLaunch t;
};

// work counters of the first launches of a plan that are captured into graphs (other launches
// allocate theirs)
constexpr int kAdjCounters = 64;

struct AdjState {
  Arena ar;
  AdjSide a, b;
  unsigned long long *counters = nullptr;
  std::atomic<int> next_counter{0};
};

namespace {

inline unsigned nblk(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

constexpr int RA = 4;  // outputs per lane per pass (8 and 2 measured: 4 the best balance)

struct AdjArgs {
  const double *A, *B, *dC;
  double *dA, *dB;
  double alpha;
  int ta, tb;
  const int32_t *grp, *ptr;        // entries of each output block
  const int32_t *s_a, *s_b, *s_c, *s_cb;
  const int32_t *c_row, *c_col, *c_rsz, *c_csz;  // C block index and sizes
  // stored blocks of the output side; each is cut into nch chunks of `span` outputs
  // (consecutive passes), one warp per (block, chunk), so that large blocks spread over
  // several warps
  int64_t nblocks;
  int32_t nch, span;
  const int32_t *row, *col, *rsz, *csz;
  const int64_t *off;
};

// dop(A) for stored A block b: lanes own (p, l) of the m x k op block, numbered column
// by column (o = l m + p), so that a pass of 32 RA outputs covers every row p of a few
// columns l and reads each op(B) row it needs once per product.  (Numbered row by row,
// a pass covered one or two rows p and every op(B) row came in again for each of the m
// rows: on the rank-3 adjoint the kernel read 14.6 GB from DRAM for about 2 GB of
// operands.)  The sums run over the entries, then q, in the same order either way.
__global__ void k_adj_a(AdjArgs P) {
  const int lane = threadIdx.x & 31;
  const int64_t w = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int64_t b = w / P.nch;
  if (b >= P.nblocks) return;
  const int R = P.rsz[P.row[b]], Cc = P.csz[P.col[b]];
  const int m = P.ta ? Cc : R, k = P.ta ? R : Cc;
  const int64_t ob = (w - b * P.nch) * (int64_t)P.span;
  if (ob >= m * k) return;
  const int o1 = (int)min((int64_t)m * k, ob + P.span);
  const int e0 = P.ptr[b], e1 = P.ptr[b + 1];
  double *out = P.dA + P.off[b];
  for (int o0 = (int)ob; o0 < o1; o0 += 32 * RA) {
    double acc[RA];
    int pr[RA], lr[RA];
#pragma unroll
    for (int r = 0; r < RA; ++r) {
      const int o = o0 + lane + 32 * r;
      lr[r] = o / m;
      pr[r] = o - lr[r] * m;
      acc[r] = 0.0;
    }
    for (int q0 = e0; q0 < e1; ++q0) {
      const int e = P.grp[q0];
      const int c = P.s_cb[e];
      const int n = P.c_csz[P.c_col[c]];
      const double *g = P.dC + P.s_c[e];   // m x n
      const double *bb = P.B + P.s_b[e];   // op(B): k x n
      const int b_sl = P.tb ? 1 : n, b_sq = P.tb ? k : 1;
#pragma unroll
      for (int r = 0; r < RA; ++r) {
        if (o0 + lane + 32 * r < m * k) {
          const double *gr = g + pr[r] * n, *br = bb + lr[r] * b_sl;
          double s = acc[r];
          for (int q = 0; q < n; ++q) s = fma(__ldg(gr + q), __ldg(br + q * b_sq), s);
          acc[r] = s;
        }
      }
    }
#pragma unroll
    for (int r = 0; r < RA; ++r) {
      if (o0 + lane + 32 * r < m * k)
        out[P.ta ? lr[r] * m + pr[r] : pr[r] * k + lr[r]] = P.alpha * acc[r];
    }
  }
}

// dop(B) for stored B block b: lanes own (l, q) of the k x n op block
__global__ void k_adj_b(AdjArgs P) {
  const int lane = threadIdx.x & 31;
  const int64_t w = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int64_t b = w / P.nch;
  if (b >= P.nblocks) return;
  const int R = P.rsz[P.row[b]], Cc = P.csz[P.col[b]];
  const int k = P.tb ? Cc : R, n = P.tb ? R : Cc;
  const int64_t ob = (w - b * P.nch) * (int64_t)P.span;
  if (ob >= k * n) return;
  const int o1 = (int)min((int64_t)k * n, ob + P.span);
  const int e0 = P.ptr[b], e1 = P.ptr[b + 1];
  double *out = P.dB + P.off[b];
  for (int o0 = (int)ob; o0 < o1; o0 += 32 * RA) {
    double acc[RA];
#pragma unroll
    for (int r = 0; r < RA; ++r) acc[r] = 0.0;
    for (int q0 = e0; q0 < e1; ++q0) {
      const int e = P.grp[q0];
      const int c = P.s_cb[e];
      const int m = P.c_rsz[P.c_row[c]];
      const double *g = P.dC + P.s_c[e];  // m x n
      const double *aa = P.A + P.s_a[e];  // op(A): m x k
      const int a_sp = P.ta ? 1 : k, a_sl = P.ta ? m : 1;
#pragma unroll
      for (int r = 0; r < RA; ++r) {
        const int o = o0 + lane + 32 * r;
        if (o < k * n) {
          const int l = o / n, q = o % n;
          const double *ar = aa + l * a_sl, *gq = g + q;
          double s = acc[r];
          if (m >= 32) {
            // long inner sums (e.g. the 169-row folds of a rank-4 contraction): eight p at
            // a time, their 16 loads issued before the dependent FMAs (rank-4 adjoint
            // 21.0 -> 20.2 ms; unrolled for short sums too, the rank-3 adjoint lost 5 %)
#pragma unroll 8
            for (int p = 0; p < m; ++p) s = fma(__ldg(ar + p * a_sp), __ldg(gq + p * n), s);
          } else {
            for (int p = 0; p < m; ++p) s = fma(__ldg(ar + p * a_sp), __ldg(gq + p * n), s);
          }
          acc[r] = s;
        }
      }
    }
#pragma unroll
    for (int r = 0; r < RA; ++r) {
      const int o = o0 + lane + 32 * r;
      if (o < k * n) {
        const int l = o / n, q = o % n;
        out[P.tb ? q * k + l : l * n + q] = P.alpha * acc[r];
      }
    }
  }
}

// dC_in = beta dC on the C_in blocks (one warp per C block that carries a C_in block)
__global__ void k_adj_cin(int64_t nc, const int32_t *c_cin, const int64_t *c_off,
                          const int64_t *cin_off, const int32_t *c_row, const int32_t *c_col,
                          const int32_t *rsz, const int32_t *csz, const double *dC, double *dCin,
                          double beta) {
  const int lane = threadIdx.x & 31;
  const int64_t c = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (c >= nc) return;
  const int ci = c_cin[c];
  if (ci < 0) return;
  const int len = rsz[c_row[c]] * csz[c_col[c]];
  for (int e = lane; e < len; e += 32) dCin[cin_off[ci] + e] = beta * dC[c_off[c] + e];
}

// Chunks of kAdjChunkPasses passes (of 32 RA outputs) per warp, as many per block as
// the largest stored block of the output side needs; a warp whose chunk lies past its
// block's end returns at once.  Without host block sizes: one chunk per block.  One
// pass per chunk: more warps and shorter tails than 4 (the rank-4 adjoint's dU grid
// was 3.4 waves of resident CTAs): rank-4 adjoint 20.2 -> 16.8 ms, rank-3 86 -> 80.5 ms
// with passes of 256 outputs; passes of 128 (RA = 4): 16.5 and 79.8 ms.
constexpr int kAdjChunkPasses = 1;

void chunking(AdjArgs &P, const bst_matrix &M) {
  int32_t r = 0, c = 0;
  for (int32_t v : M.h_rsz) r = std::max(r, v);
  for (int32_t v : M.h_csz) c = std::max(c, v);
  const int64_t span = (int64_t)kAdjChunkPasses * 32 * RA;
  const int64_t most = (int64_t)r * c;
  if (M.h_rsz.empty() || M.h_csz.empty() || most <= span) {
    P.nch = 1;
    P.span = 1 << 30;
  } else {
    P.nch = (int32_t)((most + span - 1) / span);
    P.span = (int32_t)span;
  }
}

// ---- schedule of the staged route -----------------------------------------------------
//
// Per stored block of the operand (R x Cc, stored layout) the gradient is sum over its
// group's entries of X Y, X with R rows and Y with Cc columns, over an inner dimension I:
//   dA, op = N:  X = dC (m x n),           Y = op(B)^T   (I = n)
//   dA, op = T:  X = op(B) (k x n),        Y = dC^T      (I = n)
//   dB, op = N:  X = op(A)^T (k x m),      Y = dC        (I = m)
//   dB, op = T:  X = dC^T (n x m),         Y = op(A)     (I = m)
// A block of more than 320 elements is cut into rectangular tiles of about equal size, an
// inner dimension that does not fit a slot into panels; the entries (first X element, first
// Y element, panel width, row strides) are those of the whole block, and each of its tiles
// adds its own first row and column.  Wide blocks need rectangles: a 13 x 390 block in tiles
// of 13 x 23 stages 4 doubles per 32 outputs and inner step, in rows of 320 it would be 32.

struct AdjTile {
  int tr, tc, wmax;  // tile rows and columns, largest panel width
};

struct AdjSched {
  int64_t nblocks, T;
  int32_t D2;             // column classes of op(operand)
  int32_t trans, tx, ty;  // the operand's op; X, Y stored transposed
  int32_t x_c;            // X is dC and Y the other operand, else the other way round
  const int32_t *row, *col, *rsz, *csz;  // stored blocks of the operand
  const int32_t *cls1, *cls2;            // size class of every row / column of op(operand)
  const int64_t *off;
  const int32_t *grp, *ptr;
  const int32_t *s_o, *s_c, *s_ob, *s_cb;  // other operand's and C's offsets; own and C block
  const int32_t *c_dim, *c_sz;             // C block row (or column) index, and its sizes
  const AdjTile *tile;                     // per (class, class)
  const int32_t *epos;                     // first entry of every product (null: itself)
  int4 *ents;
  int32_t *desc, *key;
  const int64_t *tbeg;  // first tile of every block (null: the block itself)
  int32_t slot;
};

__device__ __forceinline__ AdjTile adj_tile_of(const AdjSched &S, int64_t b) {
  const int r = S.row[b], c = S.col[b];
  return S.tile[S.cls1[S.trans ? c : r] * S.D2 + S.cls2[S.trans ? r : c]];
}

__global__ void k_adj_panels(AdjSched S, int32_t *__restrict__ cnt) {
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= S.T) return;
  const int e = S.grp[q];
  const int I = S.c_sz[S.c_dim[S.s_cb[e]]], wmax = adj_tile_of(S, S.s_ob[e]).wmax;
  cnt[q] = (I + wmax - 1) / wmax;
}

__global__ void k_adj_ents(AdjSched S) {
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= S.T) return;
  const int e = S.grp[q];
  const int64_t b = S.s_ob[e];
  const int I = S.c_sz[S.c_dim[S.s_cb[e]]], wmax = adj_tile_of(S, b).wmax;
  const int R = S.rsz[S.row[b]], Cc = S.csz[S.col[b]];
  const int sx = S.tx ? R : I, sy = S.ty ? I : Cc;  // stored row lengths of X and Y
  const int c = S.s_c[e], o = S.s_o[e];
  const int x = S.x_c ? c : o, y = S.x_c ? o : c;
  const int np = (I + wmax - 1) / wmax, w = (I + np - 1) / np;
  int4 *out = S.ents + (S.epos ? S.epos[q] : (int32_t)q);
  for (int i = 0; i < np; ++i) {
    const int l0 = i * w;
    out[i] = make_int4(x + (S.tx ? l0 * sx : l0), y + (S.ty ? l0 : l0 * sy), min(w, I - l0),
                       sx | (sy << 16));
  }
}

__global__ void k_adj_tile_count(AdjSched S, int32_t *__restrict__ cnt) {
  const int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= S.nblocks) return;
  const AdjTile t = adj_tile_of(S, b);
  cnt[b] = ((S.rsz[S.row[b]] + t.tr - 1) / t.tr) * ((S.csz[S.col[b]] + t.tc - 1) / t.tc);
}

__device__ __forceinline__ long long warp_sum(long long v) {
#pragma unroll
  for (int d = 16; d >= 1; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
  return v;
}

// Descriptors and cost keys, a warp per block.  A block's tiles come in at most four shapes
// (the last row and the last column of tiles may be smaller); the lanes sum the costs of a
// shape over the block's entries together, then write a descriptor each.  (A lane per tile,
// each reading all entries, took 0.69 ms a side on the 2000 x 2000 banded product.)
__global__ void k_adj_desc(AdjSched S) {
  const int lane = threadIdx.x & 31;
  const int64_t b = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (b >= S.nblocks) return;
  const AdjTile t = adj_tile_of(S, b);
  const int R = S.rsz[S.row[b]], Cc = S.csz[S.col[b]];
  const int nr = (R + t.tr - 1) / t.tr, nc = (Cc + t.tc - 1) / t.tc;
  const int q0 = S.ptr[b], q1 = S.ptr[b + 1];
  const int e0 = S.epos ? S.epos[q0] : q0, e1 = S.epos ? S.epos[q1] : q1;
  const int64_t tile0 = S.tbeg ? S.tbeg[b] : b;
  for (int sh = 0; sh < 4; ++sh) {
    // tiles [i0, i1) x [j0, j1): all but the last row / column of tiles, or that one
    const int i0 = (sh & 1) ? nr - 1 : 0, i1 = (sh & 1) ? nr : nr - 1;
    const int j0 = (sh & 2) ? nc - 1 : 0, j1 = (sh & 2) ? nc : nc - 1;
    if (i0 >= i1 || j0 >= j1) continue;
    const int m = min(t.tr, R - i0 * t.tr), n = min(t.tc, Cc - j0 * t.tc), mn = m * n;
    TailCost tc = tail_cost(mn, kMaxSplit), part = tc;
    part.c[0] = part.c[1] = 0;
    for (int e = e0 + lane; e < e1; e += 32) tail_add(part, S.ents[e].z);
    tc.w1 = warp_sum(part.w1);
    tc.c[0] += warp_sum(part.c[0]);
    tc.c[1] += warp_sum(part.c[1]);
    const long long c1 = tail_total(tc, mn);
    const int smax = min(kMaxSplit, min(32 * kNarrowR, S.slot) / mn);
    int split = 1;
    if (tc.w1 >= kSplitMinInner && smax >= 2) {
      long long cb = c1;
      for (int s = 2; s <= smax; ++s) {
        long long W = 0;
        for (int e = e0 + lane; e < e1; e += 32) W += (S.ents[e].z + s - 1) / s;
        const long long c = split_cost(s, mn, warp_sum(W));
        if (c < cb) {
          cb = c;
          split = s;
        }
      }
      if (!split_pays(cb, c1, tc.w1)) split = 1;
    }
    const int word = f64_split_word(split, tail_of(tc));
    const int key = __clzll((unsigned long long)tc.w1 * mn + 1ull);
    const int nj = j1 - j0, cnt = (i1 - i0) * nj;
    for (int x = lane; x < cnt; x += 32) {
      const int i = i0 + x / nj, j = j0 + x % nj, r0 = i * t.tr, c0 = j * t.tc;
      const int64_t tile = tile0 + (int64_t)i * nc + j;
      int4 *d = reinterpret_cast<int4 *>(S.desc + tile * kF64Desc);
      d[0] = make_int4((int32_t)(S.off[b] + (int64_t)r0 * Cc + c0), e0, e1 - e0, m | (n << 12));
      d[1] = make_int4(r0 | (c0 << 16), Cc, (int32_t)b, word);
      S.key[tile] = key;
    }
  }
}

// Tile of an R x Cc block: whole up to 320 elements, else the candidate that needs the least
// time per inner step by the FP64 instructions (16 cycles each, a quarter of one lost per
// tile to its tail) and the staged doubles (about a cycle each).
AdjTile adj_tile(int R, int Cc) {
  constexpr int most = 32 * kNarrowR;
  AdjTile best{R, Cc, 1};
  if ((int64_t)R * Cc > most) {
    double low = 0.0;
    for (int want : {most / std::min(Cc, most), 8, 12, 16, 20, 24, 32, R}) {
      int tr = std::min({std::max(want, 1), R, most});
      int tc = std::min(Cc, most / tr);
      tr = (R + (R + tr - 1) / tr - 1) / ((R + tr - 1) / tr);  // about equal tiles
      tc = (Cc + (Cc + tc - 1) / tc - 1) / ((Cc + tc - 1) / tc);
      const double nt = double((R + tr - 1) / tr) * ((Cc + tc - 1) / tc);
      const double cost = nt * (16.0 * (tr * tc / 32.0 + 0.25) + tr + tc);
      if (low == 0.0 || cost < low) {
        low = cost;
        best = AdjTile{tr, tc, 1};
      }
    }
  }
  best.wmax = std::max(1, kNarrowSlot / (best.tr + best.tc));
  return best;
}

// The staged route is taken where it saves time.  It needs a schedule (about 25 launches a
// side the first time a plan's adjoint runs), which a plan used once gets back from about
// 5e8 flops a side on (a 200 x 200-block banded product, 0.6 GF: 2.72 -> 2.67 ms for forward
// and backward).  And what it saves are the idle lanes of last partial rounds: with blocks of
// 5, 13 and 23 the direct kernels issue 1.1 times the FP64 instructions of full rounds and
// take 20.8 ms against 18.0 (2000 x 2000 banded, 21 GF); with a rank-3 contraction's blocks
// of 750 to 5070 elements 1.01 times, and both routes take 19.4 ms.
constexpr double kAdjStagedFlops = 5e8, kAdjLaneWaste = 1.05;

// One side's groups and, where the staged route takes it, what the schedule needs before
// its tiles are counted.  is_a: the gradient of A, else of B.
struct SideBuild {
  bool is_a;
  AdjSide *side;
  const bst_matrix *M;
  AdjSched S{};
  int64_t nents = 0, ntiles = 0;
  bool panels = false, tiled = false;
};

void side_begin(bst_plan *p, SideBuild &B, AdjState &st, Arena &scratch, cudaStream_t s) {
  const bst_matrix &M = *B.M;
  AdjSide &D = *B.side;
  const bool trans = B.is_a ? p->ta : p->tb;
  const std::vector<int32_t> &v1 = B.is_a ? p->m_vals : p->k_vals,
                             &v2 = B.is_a ? p->k_vals : p->n_vals,
                             &vi = B.is_a ? p->n_vals : p->m_vals;
  // tiles and panels of every size class of the operand's blocks
  int64_t most = 0, tiles_max = 1;
  for (const auto *v : {&v1, &v2, &vi})
    for (int32_t x : *v) most = std::max<int64_t>(most, x);
  D.staged = p->T > 0 && M.nblocks > 0 && most < (1 << 15) && p->stats.flops >= kAdjStagedFlops;
  if (D.staged) {  // FP64 instructions of the direct kernels against full rounds
    double issued = 0.0, full = 0.0;
    for (int32_t q = 0; q < p->nb_all; ++q) {
      const double n = (double)(p->h_bucket_ptr[q + 1] - p->h_bucket_ptr[q]);
      if (n == 0.0) continue;
      const int32_t kc = q % p->Dk, nc = (q / p->Dk) % p->Dn, mc = q / (p->Dk * p->Dn);
      const double out = (double)p->k_vals[kc] * (B.is_a ? p->m_vals[mc] : p->n_vals[nc]);
      const double inner = n * (B.is_a ? p->n_vals[nc] : p->m_vals[mc]);
      issued += inner * std::ceil(out / 32.0);
      full += inner * out / 32.0;
    }
    D.staged = issued >= kAdjLaneWaste * full;
  }
  std::vector<AdjTile> tab;
  int64_t slot = 1;
  if (D.staged) {
    tab.resize(v1.size() * v2.size());
    for (size_t i = 0; i < v1.size(); ++i)
      for (size_t j = 0; j < v2.size(); ++j) {
        const int R = trans ? v2[j] : v1[i], Cc = trans ? v1[i] : v2[j];
        const AdjTile t = tab[i * v2.size() + j] = adj_tile(R, Cc);
        tiles_max = std::max<int64_t>(tiles_max, (int64_t)((R + t.tr - 1) / t.tr) * ((Cc + t.tc - 1) / t.tc));
      }
    for (int32_t q = 0; q < p->nb_all; ++q) {
      const int64_t n = p->h_bucket_ptr[q + 1] - p->h_bucket_ptr[q];
      if (n == 0) continue;
      const int32_t kc = q % p->Dk, nc = (q / p->Dk) % p->Dn, mc = q / (p->Dk * p->Dn);
      const AdjTile t = B.is_a ? tab[(size_t)mc * v2.size() + kc] : tab[(size_t)kc * v2.size() + nc];
      const int64_t I = B.is_a ? p->n_vals[nc] : p->m_vals[mc];
      const int64_t np = (I + t.wmax - 1) / t.wmax;
      B.panels = B.panels || np > 1;
      B.nents += n * np;
      slot = std::max(slot, (I + np - 1) / np * (t.tr + t.tc));
    }
    B.tiled = tiles_max > 1;
    D.staged = B.nents < INT32_MAX && M.nblocks * tiles_max < INT32_MAX;
  }
  // the direct kernels read the groups on every call, a schedule only while it is built
  Arena &ga = D.staged ? scratch : st.ar;
  D.grp = ga.alloc_n<int32_t>((size_t)p->T);
  const int32_t nkeys = (int32_t)std::max<int64_t>(M.nblocks, 1);  // an operand without blocks too
  D.ptr = ga.alloc_n<int32_t>((size_t)nkeys + 1);
  stable_partition(B.is_a ? p->s_ab : p->s_bb, p->T, nkeys, D.grp, D.ptr, scratch, s);
  if (!D.staged) return;
  AdjSched &S = B.S;
  S.nblocks = M.nblocks;
  S.T = p->T;
  S.D2 = (int32_t)v2.size();
  S.trans = trans;
  if (B.is_a) {
    S.tx = p->ta ? p->tb : 0;
    S.ty = p->ta ? 1 : !p->tb;
    S.x_c = !p->ta;
    S.cls1 = p->m_cls;
    S.cls2 = p->k_cls;
    S.s_o = p->s_b;
    S.s_ob = p->s_ab;
    S.c_dim = p->C->col;
    S.c_sz = p->C->csz;
  } else {
    S.tx = p->tb ? 1 : !p->ta;
    S.ty = p->tb ? p->ta : 0;
    S.x_c = p->tb;
    S.cls1 = p->k_cls;
    S.cls2 = p->n_cls;
    S.s_o = p->s_a;
    S.s_ob = p->s_bb;
    S.c_dim = p->C->row;
    S.c_sz = p->C->rsz;
  }
  S.s_c = p->s_c;
  S.s_cb = p->s_cb;
  S.row = M.row;
  S.col = M.col;
  S.rsz = M.rsz;
  S.csz = M.csz;
  S.off = M.off;
  S.grp = D.grp;
  S.ptr = D.ptr;
  S.slot = (int32_t)slot;
  AdjTile *d_tab = scratch.alloc_n<AdjTile>(tab.size());
  {
    Upload up(p->ctx, s);
    up.add(d_tab, tab.data(), sizeof(AdjTile) * tab.size());
    up.done_async();  // read by this stream's kernels; adjoint_fp64 synchronises below
  }
  S.tile = d_tab;
  if (B.panels) {
    int32_t *cnt = scratch.alloc_n<int32_t>((size_t)p->T);
    int32_t *epos = scratch.alloc_n<int32_t>((size_t)p->T + 1);
    k_adj_panels<<<nblk(p->T, 256), 256, 0, s>>>(S, cnt);
    BST_CHECK_LAUNCH();
    exscan_i32(cnt, epos, p->T, scratch, s);
    S.epos = epos;
  }
  B.ntiles = M.nblocks;
  if (B.tiled) {
    int32_t *cnt = scratch.alloc_n<int32_t>((size_t)M.nblocks);
    int64_t *tbeg = scratch.alloc_n<int64_t>((size_t)M.nblocks + 1);
    k_adj_tile_count<<<nblk(M.nblocks, 256), 256, 0, s>>>(S, cnt);
    BST_CHECK_LAUNCH();
    exscan_i32_i64(cnt, tbeg, M.nblocks, scratch, s);
    S.tbeg = tbeg;
  }
}

void side_finish(SideBuild &B, AdjState &st, Arena &scratch, cudaStream_t s) {
  AdjSched &S = B.S;
  TileLaunch &t = B.side->t;
  S.ents = st.ar.alloc_n<int4>((size_t)B.nents);
  S.desc = st.ar.alloc_n<int32_t>((size_t)B.ntiles * kF64Desc);
  S.key = scratch.alloc_n<int32_t>((size_t)B.ntiles);
  k_adj_ents<<<nblk(S.T, 256), 256, 0, s>>>(S);
  BST_CHECK_LAUNCH();
  k_adj_desc<<<nblk(S.nblocks, 8), 256, 0, s>>>(S);
  BST_CHECK_LAUNCH();
  int64_t *it0 = scratch.alloc_n<int64_t>((size_t)B.ntiles);
  int64_t *items = st.ar.alloc_n<int64_t>((size_t)B.ntiles);
  plan_items(B.ntiles, it0, s);
  sort_items(it0, S.key, B.ntiles, items, scratch, s);
  t.items = items;
  t.nitems = B.ntiles;
  t.desc = S.desc;
  t.ents = S.ents;
  t.slot = S.slot;
  t.tx = S.tx;
  t.ty = S.ty;
  t.tiled = B.tiled || B.panels;
}

}  // namespace

void adj_state_free(bst_plan *p) {
  delete p->adj;
  p->adj = nullptr;
}

void adjoint_info(const bst_plan *p, int32_t *info) {
  for (int i = 0; i < 2; ++i) {
    const AdjSide *D = p->adj ? (i ? &p->adj->b : &p->adj->a) : nullptr;
    info[2 * i] = D && D->staged;
    info[2 * i + 1] = D && D->staged && D->t.tiled;
  }
}

static void adj_build(bst_plan *p, AdjState &S, cudaStream_t s) {
  S.ar.ctx = static_cast<Ctx *>(p->ctx);
  S.ar.stream = s;
  Arena scratch;
  scratch.ctx = S.ar.ctx;
  scratch.stream = s;
  scratch.chunk = kScratchChunk;
  S.counters = S.ar.alloc_n<unsigned long long>(kAdjCounters);
  SideBuild sides[2] = {{true, &S.a, p->A}, {false, &S.b, p->B}};
  for (SideBuild &B : sides) side_begin(p, B, S, scratch, s);
  {
    ReadBack rb(p->ctx, s);
    for (SideBuild &B : sides)
      if (B.S.tbeg) rb.add(&B.ntiles, B.S.tbeg + B.S.nblocks, 8);
    if (rb.used) rb.done();
  }
  for (SideBuild &B : sides)
    if (B.side->staged) side_finish(B, S, scratch, s);
  BST_CUDA(cudaStreamSynchronize(s));  // the state serves later calls on any stream
}

// one side's gradient: out = alpha X Y by the staged schedule
static void side_staged(bst_plan *p, const AdjSide &D, const double *X, const double *Y, double *out,
                        double alpha, cudaStream_t s) {
  // Adjoints of one plan may overlap on several streams, so each launch has its own work
  // counter: from the stream's pool, or (a captured launch must not allocate) one of the plan's.
  // Graphs keep theirs, and replays of different graphs may overlap too, so none is handed out
  // twice; once they are used up, a captured launch deals its tiles out in turn (banded_backward
  // 29.5 -> 30.6 ms).
  AdjState &S = *p->adj;
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  BST_CUDA(cudaStreamIsCapturing(s, &cap));
  Arena scratch;
  scratch.ctx = static_cast<Ctx *>(p->ctx);
  scratch.stream = s;
  unsigned long long *counter = nullptr;
  if (cap == cudaStreamCaptureStatusNone) {
    counter = scratch.alloc_n<unsigned long long>(1);
  } else if (S.next_counter.load() < kAdjCounters) {
    const int i = S.next_counter.fetch_add(1);
    if (i < kAdjCounters) counter = S.counters + i;
  }
  launch_fp64_tiles(D.t, X, Y, out, alpha, p->ctx->num_sms, counter, s);
  scratch.release_all();
}

void adjoint_fp64(bst_plan *p, const double *A, const double *B, const double *dC, double *dA,
                  double *dB, double alpha, cudaStream_t s) {
  const bst_matrix *Am = p->A, *Bm = p->B;
  if (!p->adj) {
    auto *st = new AdjState();
    try {
      adj_build(p, *st, s);
    } catch (...) {
      delete st;
      throw;
    }
    p->adj = st;
  }
  AdjState &S = *p->adj;
  AdjArgs P{};
  P.A = A;
  P.B = B;
  P.dC = dC;
  P.dA = dA;
  P.dB = dB;
  P.alpha = alpha;
  P.ta = p->ta;
  P.tb = p->tb;
  P.s_a = p->s_a;
  P.s_b = p->s_b;
  P.s_c = p->s_c;
  P.s_cb = p->s_cb;
  P.c_row = p->C->row;
  P.c_col = p->C->col;
  P.c_rsz = p->C->rsz;
  P.c_csz = p->C->csz;
  const int wpb = 8;
  if (Am->nblocks > 0 && dA && S.a.staged) {
    side_staged(p, S.a, p->ta ? B : dC, p->ta ? dC : B, dA, alpha, s);
  } else if (Am->nblocks > 0 && dA) {
    P.grp = S.a.grp;
    P.ptr = S.a.ptr;
    P.nblocks = Am->nblocks;
    P.row = Am->row;
    P.col = Am->col;
    P.rsz = Am->rsz;
    P.csz = Am->csz;
    P.off = Am->off;
    chunking(P, *Am);
    k_adj_a<<<nblk(Am->nblocks * P.nch, wpb), 32 * wpb, 0, s>>>(P);
    BST_CHECK_LAUNCH();
  }
  if (Bm->nblocks > 0 && dB && S.b.staged) {
    side_staged(p, S.b, p->tb ? dC : A, p->tb ? A : dC, dB, alpha, s);
  } else if (Bm->nblocks > 0 && dB) {
    P.grp = S.b.grp;
    P.ptr = S.b.ptr;
    P.nblocks = Bm->nblocks;
    P.row = Bm->row;
    P.col = Bm->col;
    P.rsz = Bm->rsz;
    P.csz = Bm->csz;
    P.off = Bm->off;
    chunking(P, *Bm);
    k_adj_b<<<nblk(Bm->nblocks * P.nch, wpb), 32 * wpb, 0, s>>>(P);
    BST_CHECK_LAUNCH();
  }
}

void scale_cin_grad(bst_plan *p, const double *dC, double *dCin, double beta, cudaStream_t s) {
  const int64_t nc = p->C->nblocks;
  if (!p->Cin || !dCin || nc == 0) return;
  const int wpb = 8;
  k_adj_cin<<<nblk(nc, wpb), 32 * wpb, 0, s>>>(nc, p->c_cin, p->C->off, p->Cin->off, p->C->row,
                                               p->C->col, p->C->rsz, p->C->csz, dC, dCin, beta);
  BST_CHECK_LAUNCH();
}

}  // namespace bst
