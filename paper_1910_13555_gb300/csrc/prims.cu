// Device primitives of the symbolic phase: exclusive scans, a stable counting sort
// (partition by a small integer key) and an LSD radix sort built on it.
//
// All of them are deterministic: the counting sort is stable because every warp
// owns one contiguous segment of the input and emits it in order, with the ranks of
// equal keys inside a 32-element batch taken from __match_any_sync.
#include <algorithm>
#include <cstring>

#include "bst_internal.h"
#include "partition.h"

namespace bst {

namespace {

constexpr int kScanThreads = 256;
constexpr int kScanItems = 8;
constexpr int kScanTile = kScanThreads * kScanItems;

template <class T>
__device__ __forceinline__ T warp_incl_scan(T v) {
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    T o = __shfl_up_sync(0xffffffffu, v, d);
    if ((threadIdx.x & 31) >= d) v += o;
  }
  return v;
}

// block-wide exclusive scan of one value per thread; returns the exclusive prefix,
// *total gets the block sum.
template <class T>
__device__ __forceinline__ T block_excl_scan(T v, T *total) {
  constexpr int NW = kScanThreads / 32;
  __shared__ T warp_sums[NW];
  __shared__ T tot;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  T inc = warp_incl_scan(v);
  if (lane == 31) warp_sums[wid] = inc;
  __syncthreads();
  if (wid == 0) {
    T w = lane < NW ? warp_sums[lane] : T(0);
    T wi = warp_incl_scan(w);
    if (lane < NW) warp_sums[lane] = wi - w;
    if (lane == NW - 1) tot = wi;
  }
  __syncthreads();
  T excl = inc - v + warp_sums[wid];
  *total = tot;
  __syncthreads();  // the shared slots are reused by the next call
  return excl;
}

template <class TI, class TO>
__global__ void k_tile_sums(const TI *__restrict__ in, int64_t n, TO *__restrict__ sums) {
  int64_t base = (int64_t)blockIdx.x * kScanTile;
  TO acc = 0;
#pragma unroll
  for (int r = 0; r < kScanItems; ++r) {
    int64_t i = base + (int64_t)r * kScanThreads + threadIdx.x;
    if (i < n) acc += (TO)in[i];
  }
  TO total;
  block_excl_scan<TO>(acc, &total);
  if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

// single-CTA exclusive scan of the tile sums (in place), carry across chunks
template <class TO>
__global__ void k_scan_sums(TO *sums, int64_t nt) {
  TO carry = 0;
  for (int64_t c0 = 0; c0 < nt; c0 += kScanThreads) {
    int64_t i = c0 + threadIdx.x;
    TO v = i < nt ? sums[i] : TO(0);
    TO total;
    TO ex = block_excl_scan<TO>(v, &total);
    if (i < nt) sums[i] = ex + carry;
    carry += total;
  }
}

template <class TI, class TO>
__global__ void k_tile_scan(const TI *__restrict__ in, int64_t n, const TO *__restrict__ sums,
                            TO *__restrict__ out) {
  // each thread takes kScanItems consecutive elements
  int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
  TO v[kScanItems];
  TO acc = 0;
#pragma unroll
  for (int r = 0; r < kScanItems; ++r) {
    int64_t i = base + r;
    v[r] = i < n ? (TO)in[i] : TO(0);
    acc += v[r];
  }
  TO total;
  TO ex = block_excl_scan<TO>(acc, &total) + sums[blockIdx.x];
#pragma unroll
  for (int r = 0; r < kScanItems; ++r) {
    int64_t i = base + r;
    if (i < n) out[i] = ex;
    ex += v[r];
  }
  // the grand total goes to out[n]
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == kScanThreads - 1) out[n] = ex;
}

// the whole scan by one CTA: three launches on a few thousand elements are mostly latency
constexpr int kOneThreads = 1024, kOneTile = kOneThreads * kScanItems;

// (one CTA per array: up to three of the same length at once)
template <class TI, class TO>
__global__ void __launch_bounds__(kOneThreads)
    k_scan_one(const TI *__restrict__ in0, const TI *__restrict__ in1, const TI *__restrict__ in2,
               int64_t n, TO *__restrict__ out0, TO *__restrict__ out1, TO *__restrict__ out2) {
  const TI *in = blockIdx.x == 0 ? in0 : blockIdx.x == 1 ? in1 : in2;
  TO *out = blockIdx.x == 0 ? out0 : blockIdx.x == 1 ? out1 : out2;
  __shared__ TO sums[32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t base = (int64_t)threadIdx.x * kScanItems;
  TO v[kScanItems];
  TO acc = 0;
#pragma unroll
  for (int r = 0; r < kScanItems; ++r) {
    v[r] = base + r < n ? (TO)in[base + r] : TO(0);
    acc += v[r];
  }
  const TO inc = warp_incl_scan(acc);
  if (lane == 31) sums[wid] = inc;
  __syncthreads();
  if (wid == 0) {
    const TO w = sums[lane];
    sums[lane] = warp_incl_scan(w) - w;
  }
  __syncthreads();
  TO ex = inc - acc + sums[wid];
#pragma unroll
  for (int r = 0; r < kScanItems; ++r) {
    if (base + r < n) out[base + r] = ex;
    ex += v[r];
  }
  if (threadIdx.x == kOneThreads - 1) out[n] = ex;
}

template <class TI, class TO>
void exscan_impl(const TI *in, TO *out, int64_t n, Arena &ar, cudaStream_t s) {
  if (n == 0) {
    BST_CUDA(cudaMemsetAsync(out, 0, sizeof(TO), s));
    return;
  }
  if (n <= kOneTile) {
    k_scan_one<TI, TO><<<1, kOneThreads, 0, s>>>(in, in, in, n, out, out, out);
    BST_CHECK_LAUNCH();
    return;
  }
  int64_t nt = (n + kScanTile - 1) / kScanTile;
  TO *sums = ar.alloc_n<TO>((size_t)nt);
  k_tile_sums<TI, TO><<<(unsigned)nt, kScanThreads, 0, s>>>(in, n, sums);
  BST_CHECK_LAUNCH();
  k_scan_sums<TO><<<1, kScanThreads, 0, s>>>(sums, nt);
  BST_CHECK_LAUNCH();
  k_tile_scan<TI, TO><<<(unsigned)nt, kScanThreads, 0, s>>>(in, n, sums, out);
  BST_CHECK_LAUNCH();
}

// ---- stable counting sort ------------------------------------------------------

__global__ void k_part_hist(const int32_t *__restrict__ keys, int64_t n, int64_t L, int64_t G,
                            int32_t *__restrict__ hist) {
  const int lane = threadIdx.x & 31;
  int64_t g = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (g >= G) return;
  int64_t p0 = g * L, p1 = min(n, p0 + L);
  for (int64_t b = p0; b < p1; b += 32) {
    int64_t p = b + lane;
    unsigned act = __ballot_sync(0xffffffffu, p < p1);
    if (p < p1) {
      int32_t key = keys[p];
      unsigned peers = __match_any_sync(act, key);
      if ((int)(__ffs(peers) - 1) == lane) atomicAdd(&hist[(int64_t)key * G + g], __popc(peers));
    }
  }
}

__global__ void k_part_keyptr(const int32_t *__restrict__ base, int32_t nkeys, int64_t G,
                              int32_t *__restrict__ key_ptr) {
  int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k <= nkeys) key_ptr[k] = base[k * G];
}

__global__ void k_part_scatter(const int32_t *__restrict__ keys, int64_t n, int64_t L, int64_t G,
                               int32_t *__restrict__ base, int32_t *__restrict__ perm) {
  const int lane = threadIdx.x & 31;
  int64_t g = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (g >= G) return;
  int64_t p0 = g * L, p1 = min(n, p0 + L);
  for (int64_t b = p0; b < p1; b += 32) {
    int64_t p = b + lane;
    unsigned act = __ballot_sync(0xffffffffu, p < p1);
    int32_t key = 0;
    unsigned peers = 0;
    int32_t pos = 0;
    if (p < p1) {
      key = keys[p];
      peers = __match_any_sync(act, key);
      unsigned lt = peers & ((1u << lane) - 1u);
      pos = base[(int64_t)key * G + g] + __popc(lt);
      perm[pos] = (int32_t)p;
    }
    __syncwarp();
    if (p < p1 && (int)(__ffs(peers) - 1) == lane) base[(int64_t)key * G + g] += __popc(peers);
    __syncwarp();
  }
}

// The whole partition by one CTA, for short inputs: five launches otherwise.  Each of the 32
// warps owns a segment; its key counts, scanned in (key, segment) order, become its write
// cursors.
constexpr int kOnePartKeys = 256, kOnePartItems = 8192;

__global__ void __launch_bounds__(1024)
    k_part_one(const int32_t *__restrict__ keys, int n, int nkeys, int32_t *__restrict__ perm,
               int32_t *__restrict__ key_ptr) {
  __shared__ int32_t cur[kOnePartKeys * 32];
  __shared__ int32_t sums[32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int cells = nkeys * 32;
  for (int i = threadIdx.x; i < cells; i += 1024) cur[i] = 0;
  __syncthreads();
  const int L = (n + 31) / 32, p0 = min(w * L, n), p1 = min(p0 + L, n);
  for (int p = p0 + lane; p < p1; p += 32) atomicAdd(&cur[keys[p] * 32 + w], 1);
  __syncthreads();
  // exclusive scan of the cells, cells / 1024 (at most 8) consecutive ones per thread
  const int per = (cells + 1023) / 1024, c0 = threadIdx.x * per;
  int acc = 0;
  for (int i = c0; i < min(c0 + per, cells); ++i) acc += cur[i];
  const int inc = warp_incl_scan(acc);
  if (lane == 31) sums[w] = inc;
  __syncthreads();
  if (w == 0) {
    const int v = sums[lane];
    sums[lane] = warp_incl_scan(v) - v;
  }
  __syncthreads();
  int ex = inc - acc + sums[w];
  for (int i = c0; i < min(c0 + per, cells); ++i) {
    const int v = cur[i];
    cur[i] = ex;
    if ((i & 31) == 0) key_ptr[i >> 5] = ex;
    ex += v;
  }
  if (threadIdx.x == 0) key_ptr[nkeys] = n;
  __syncthreads();
  for (int b = p0; b < p1; b += 32) {
    const int p = b + lane;
    const unsigned act = __ballot_sync(0xffffffffu, p < p1);
    int cell = 0;
    unsigned peers = 0;
    if (p < p1) {
      cell = keys[p] * 32 + w;
      peers = __match_any_sync(act, cell);
      perm[cur[cell] + __popc(peers & ((1u << lane) - 1u))] = p;
    }
    __syncwarp();
    if (p < p1 && (int)(__ffs(peers) - 1) == lane) cur[cell] += __popc(peers);
    __syncwarp();
  }
}

// digit of key[perm[i]] (perm null: key[i]): the bits of mask from `shift` on
__global__ void k_key_digit(const int32_t *__restrict__ keys, const int32_t *__restrict__ perm,
                            int64_t n, int shift, int32_t mask, int32_t *__restrict__ dig) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  dig[i] = (keys[perm ? perm[i] : i] >> shift) & mask;
}

// perm[i] = p1[p2[i]], and the key there
__global__ void k_compose_sorted(const int32_t *__restrict__ keys, const int32_t *__restrict__ p1,
                                 const int32_t *__restrict__ p2, int64_t n,
                                 int32_t *__restrict__ perm, int32_t *__restrict__ sorted) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int32_t p = p1[p2[i]];
  perm[i] = p;
  sorted[i] = keys[p];
}

// where every key starts among the sorted ones: a search per key (an item filling the gap before
// its key left one thread with all the keys of a sparse range)
__global__ void k_key_starts(const int32_t *__restrict__ sorted, int64_t n, int32_t nkeys,
                             int32_t *__restrict__ key_ptr) {
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q > nkeys) return;
  int64_t lo = 0, hi = n;
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if (sorted[mid] < q)
      lo = mid + 1;
    else
      hi = mid;
  }
  key_ptr[q] = (int32_t)lo;
}

__global__ void k_iota(int32_t *p, int64_t n) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) p[i] = (int32_t)i;
}

__global__ void k_fill(int32_t *p, int32_t v, int64_t n) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) p[i] = v;
}

__global__ void k_gather(const int32_t *__restrict__ src, const int32_t *__restrict__ idx,
                         int32_t *__restrict__ dst, int64_t n) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) dst[i] = src[idx[i]];
}

__global__ void k_digits(const uint64_t *__restrict__ keys, const int32_t *__restrict__ perm,
                         int64_t n, int shift, int32_t *__restrict__ dig) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) dig[i] = (int32_t)((keys[perm[i]] >> shift) & 0xffu);
}

inline unsigned nblk(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

void exscan_i32_i64(const int32_t *in, int64_t *out, int64_t n, Arena &ar, cudaStream_t s) {
  exscan_impl<int32_t, int64_t>(in, out, n, ar, s);
}
void exscan3_i32_i64(const int32_t *const (&in)[3], int64_t *const (&out)[3], int64_t n, Arena &ar,
                     cudaStream_t s) {
  if (n == 0 || n > kOneTile) {
    for (int i = 0; i < 3; ++i) exscan_i32_i64(in[i], out[i], n, ar, s);
    return;
  }
  k_scan_one<int32_t, int64_t><<<3, kOneThreads, 0, s>>>(in[0], in[1], in[2], n, out[0], out[1],
                                                         out[2]);
  BST_CHECK_LAUNCH();
}
void exscan_i64(const int64_t *in, int64_t *out, int64_t n, Arena &ar, cudaStream_t s) {
  exscan_impl<int64_t, int64_t>(in, out, n, ar, s);
}
void exscan_i32(const int32_t *in, int32_t *out, int64_t n, Arena &ar, cudaStream_t s) {
  exscan_impl<int32_t, int32_t>(in, out, n, ar, s);
}

void iota_i32(int32_t *p, int64_t n, cudaStream_t s) {
  if (n <= 0) return;
  k_iota<<<nblk(n, 256), 256, 0, s>>>(p, n);
  BST_CHECK_LAUNCH();
}
// The copies of a ReadBack or an Upload, up to kCopyItems per launch (one row of CTAs each;
// a launch per item was a fifth of the launches of a small plan): 16-byte words where both
// ends are 16-byte aligned, the rest byte by byte.
constexpr int kCopyItems = 16;
struct CopyItems {
  unsigned char *dst[kCopyItems];
  const unsigned char *src[kCopyItems];
  int64_t n[kCopyItems];
};

__global__ void k_copy_items(CopyItems C) {
  unsigned char *dst = C.dst[blockIdx.y];
  const unsigned char *src = C.src[blockIdx.y];
  const int64_t n = C.n[blockIdx.y], stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool aligned = ((reinterpret_cast<uintptr_t>(dst) | reinterpret_cast<uintptr_t>(src)) & 15) == 0;
  const int64_t nw = aligned ? n >> 4 : 0;
  for (int64_t i = i0; i < nw; i += stride)
    reinterpret_cast<uint4 *>(dst)[i] = reinterpret_cast<const uint4 *>(src)[i];
  for (int64_t i = (nw << 4) + i0; i < n; i += stride) dst[i] = src[i];
}

static void copy_items(const CopyItems &C, int count, cudaStream_t s) {
  if (count == 0) return;
  int64_t most = 0;
  for (int i = 0; i < count; ++i) most = std::max(most, C.n[i]);
  const int blocks = (int)std::min<int64_t>(512, (most + 4095) / 4096);
  k_copy_items<<<dim3((unsigned)std::max(blocks, 1), (unsigned)count), 256, 0, s>>>(C);
  BST_CHECK_LAUNCH();
}

ReadBack::ReadBack(bst_ctx *c, cudaStream_t st) : ctx(c), s(st) {
  ctx->rb_mutex.lock();
  locked = true;
}

ReadBack::~ReadBack() {
  if (locked) {
    // an exception left copies in flight: let them land before the buffer is reused
    if (!items.empty()) (void)cudaStreamSynchronize(s);
    ctx->rb_mutex.unlock();
  }
}

void ReadBack::done() {
  finish();
  if (locked) {
    locked = false;
    ctx->rb_mutex.unlock();
  }
}

void ReadBack::add(void *host_dst, const void *dev_src, size_t bytes) {
  if (bytes == 0) return;
  const size_t off = (used + 15) & ~(size_t)15;
  if (off + bytes > ctx->rb_cap) {
    // grow (geometrically, never shrinking: freeing pinned memory synchronises the whole
    // device): earlier items of this ReadBack are still pending, so finish them first
    if (!items.empty()) finish();
    const size_t cap = std::max<size_t>({(size_t)1 << 20, 2 * ctx->rb_cap, 2 * (off + bytes)});
    BST_CUDA(cudaStreamSynchronize(s));
    if (ctx->rb_host) BST_CUDA(cudaFreeHost(ctx->rb_host));
    ctx->rb_host = nullptr;
    ctx->rb_cap = 0;
    BST_CUDA(cudaHostAlloc(&ctx->rb_host, cap, cudaHostAllocMapped));
    ctx->rb_cap = cap;
    return add(host_dst, dev_src, bytes);
  }
  items.push_back({host_dst, dev_src, off, bytes});
  used = off + bytes;
}

void ReadBack::finish() {
  void *dev_view = nullptr;
  if (!items.empty()) BST_CUDA(cudaHostGetDevicePointer(&dev_view, ctx->rb_host, 0));
  CopyItems C;
  int count = 0;
  for (const Item &it : items) {
    C.dst[count] = static_cast<unsigned char *>(dev_view) + it.off;
    C.src[count] = static_cast<const unsigned char *>(it.src);
    C.n[count] = (int64_t)it.bytes;
    if (++count == kCopyItems) {
      copy_items(C, count, s);
      count = 0;
    }
  }
  copy_items(C, count, s);
  BST_CUDA(cudaStreamSynchronize(s));
  for (const Item &it : items)
    std::memcpy(it.dst, static_cast<const char *>(ctx->rb_host) + it.off, it.bytes);
  items.clear();
  used = 0;
}

Upload::Upload(bst_ctx *c, cudaStream_t st) : ctx(c), s(st) {
  ctx->up_mutex.lock();
  locked = true;
  if (ctx->up_pending) {
    if (ctx->up_stream == s)
      used = ctx->up_tail;  // behind the copies in flight
    else
      wait_pending();  // no throw here: the lock is held
  }
}

void Upload::wait_pending() {
  if (!ctx->up_pending) return;
  ctx->up_pending = false;
  (void)cudaEventSynchronize(ctx->up_event);
}

Upload::~Upload() {
  if (locked) {
    // an exception left copies in flight: let them land before the buffer is reused
    if (!items.empty() || used) {
      (void)cudaStreamSynchronize(s);
      ctx->up_pending = false;
    }
    ctx->up_mutex.unlock();
  }
}

void Upload::done() {
  flush();
  if (locked) {
    locked = false;
    ctx->up_mutex.unlock();
  }
}

void Upload::done_async() {
  if (!items.empty()) {
    launch();
    if (!ctx->up_event) BST_CUDA(cudaEventCreateWithFlags(&ctx->up_event, cudaEventDisableTiming));
    // the event covers the earlier copies too, whatever became of their stream
    if (ctx->up_pending) BST_CUDA(cudaStreamWaitEvent(s, ctx->up_event, 0));
    BST_CUDA(cudaEventRecord(ctx->up_event, s));
    ctx->up_pending = true;
    ctx->up_stream = s;
    ctx->up_tail = used;
    items.clear();
    used = 0;
  }
  if (locked) {
    locked = false;
    ctx->up_mutex.unlock();
  }
}

void Upload::add(void *dev_dst, const void *host_src, size_t bytes) {
  if (bytes == 0) return;
  const size_t off = (used + 15) & ~(size_t)15;
  if (off + bytes > ctx->up_cap) {
    // full: once the copies in flight and the items staged so far are out, start over, or
    // grow (geometrically, never shrinking: freeing pinned memory synchronises the whole
    // device)
    wait_pending();
    flush();
    used = 0;
    if (4 * bytes <= ctx->up_cap) return add(dev_dst, host_src, bytes);
    const size_t cap = std::max<size_t>({(size_t)1 << 20, 2 * ctx->up_cap, 8 * bytes});
    if (ctx->up_host) BST_CUDA(cudaFreeHost(ctx->up_host));
    ctx->up_host = nullptr;
    ctx->up_cap = 0;
    BST_CUDA(cudaHostAlloc(&ctx->up_host, cap, cudaHostAllocMapped));
    ctx->up_cap = cap;
    return add(dev_dst, host_src, bytes);
  }
  std::memcpy(static_cast<char *>(ctx->up_host) + off, host_src, bytes);
  items.push_back({dev_dst, off, bytes});
  used = off + bytes;
}

void Upload::flush() {
  if (items.empty()) return;
  launch();
  BST_CUDA(cudaStreamSynchronize(s));
  items.clear();
  ctx->up_pending = false;  // on this stream, so it is over too
  used = 0;
}

void Upload::launch() {
  void *dev_view = nullptr;
  BST_CUDA(cudaHostGetDevicePointer(&dev_view, ctx->up_host, 0));
  CopyItems C;
  int count = 0;
  for (const Item &it : items) {
    C.dst[count] = static_cast<unsigned char *>(it.dst);
    C.src[count] = static_cast<const unsigned char *>(dev_view) + it.off;
    C.n[count] = (int64_t)it.bytes;
    if (++count == kCopyItems) {
      copy_items(C, count, s);
      count = 0;
    }
  }
  copy_items(C, count, s);
}

void fill_i32(int32_t *p, int32_t v, int64_t n, cudaStream_t s) {
  if (n <= 0) return;
  k_fill<<<nblk(n, 256), 256, 0, s>>>(p, v, n);
  BST_CHECK_LAUNCH();
}
void gather_i32(const int32_t *src, const int32_t *idx, int32_t *dst, int64_t n, cudaStream_t s) {
  if (n <= 0) return;
  k_gather<<<nblk(n, 256), 256, 0, s>>>(src, idx, dst, n);
  BST_CHECK_LAUNCH();
}

// one counting-sort pass with segments of L items, one warp each
static void partition_pass(const int32_t *keys, int64_t n, int32_t nkeys, int64_t L, int32_t *perm,
                           int32_t *key_ptr, Arena &ar, cudaStream_t s);

void stable_partition(const int32_t *keys, int64_t n, int32_t nkeys, int32_t *perm,
                      int32_t *key_ptr, Arena &ar, cudaStream_t s) {
  BST_REQUIRE(nkeys >= 1, BST_ERR_INVALID_ARG, "stable_partition: nkeys < 1");
  if (n == 0) {
    BST_CUDA(cudaMemsetAsync(key_ptr, 0, sizeof(int32_t) * ((size_t)nkeys + 1), s));
    return;
  }
  if (n <= kOnePartItems && nkeys <= kOnePartKeys) {
    k_part_one<<<1, 1024, 0, s>>>(keys, (int)n, nkeys, perm, key_ptr);
    BST_CHECK_LAUNCH();
    return;
  }
  const PartitionPlan P = partition_plan(n, nkeys);
  if (P.passes == 1) {
    partition_pass(keys, n, nkeys, P.segment[0], perm, key_ptr, ar, s);
    return;
  }
  // so many keys that a warp would walk thousands of items one batch after another: stable passes
  // over the digits of the key instead
  int32_t *dig = ar.alloc_n<int32_t>((size_t)n), *order = ar.alloc_n<int32_t>((size_t)n),
          *p2 = ar.alloc_n<int32_t>((size_t)n);
  const int64_t most = std::max({P.keys[0], P.keys[1], P.keys[2]});
  int32_t *kp = ar.alloc_n<int32_t>((size_t)most + 1);
  const int32_t mask = (int32_t)((int64_t(1) << P.bits) - 1);
  for (int i = 0; i < P.passes; ++i) {
    k_key_digit<<<nblk(n, 256), 256, 0, s>>>(keys, i ? order : nullptr, n, i * P.bits, mask, dig);
    BST_CHECK_LAUNCH();
    partition_pass(dig, n, (int32_t)P.keys[i], P.segment[i], i ? p2 : order, kp, ar, s);
    if (i == 0) continue;
    int32_t *out = i + 1 == P.passes ? perm : ar.alloc_n<int32_t>((size_t)n);
    k_compose_sorted<<<nblk(n, 256), 256, 0, s>>>(keys, order, p2, n, out, dig);
    BST_CHECK_LAUNCH();
    order = out;
  }
  k_key_starts<<<nblk((int64_t)nkeys + 1, 256), 256, 0, s>>>(dig, n, nkeys, key_ptr);
  BST_CHECK_LAUNCH();
}

static void partition_pass(const int32_t *keys, int64_t n, int32_t nkeys, int64_t L, int32_t *perm,
                           int32_t *key_ptr, Arena &ar, cudaStream_t s) {
  int64_t G = (n + L - 1) / L;
  int64_t cells = (int64_t)nkeys * G;
  int32_t *hist = ar.alloc_n<int32_t>((size_t)cells);
  int32_t *base = ar.alloc_n<int32_t>((size_t)cells + 1);
  BST_CUDA(cudaMemsetAsync(hist, 0, sizeof(int32_t) * (size_t)cells, s));
  const int wpb = 8;
  k_part_hist<<<nblk(G, wpb), 32 * wpb, 0, s>>>(keys, n, L, G, hist);
  BST_CHECK_LAUNCH();
  exscan_i32(hist, base, cells, ar, s);
  // key_ptr[k] = base[k * G]; the entry for k = nkeys reads base[cells] = n
  k_part_keyptr<<<nblk((int64_t)nkeys + 1, 256), 256, 0, s>>>(base, nkeys, G, key_ptr);
  BST_CHECK_LAUNCH();
  k_part_scatter<<<nblk(G, wpb), 32 * wpb, 0, s>>>(keys, n, L, G, base, perm);
  BST_CHECK_LAUNCH();
}

void radix_sort_perm(const uint64_t *keys, int64_t n, int bits, int32_t *perm, Arena &ar,
                     cudaStream_t s) {
  iota_i32(perm, n, s);
  if (n <= 1 || bits <= 0) return;
  int32_t *dig = ar.alloc_n<int32_t>((size_t)n);
  int32_t *p2 = ar.alloc_n<int32_t>((size_t)n);
  int32_t *cur = ar.alloc_n<int32_t>((size_t)n);
  int32_t *kp = ar.alloc_n<int32_t>(257);
  for (int shift = 0; shift < bits; shift += 8) {
    k_digits<<<nblk(n, 256), 256, 0, s>>>(keys, perm, n, shift, dig);
    BST_CHECK_LAUNCH();
    stable_partition(dig, n, 256, p2, kp, ar, s);
    // new perm[i] = perm[p2[i]]
    gather_i32(perm, p2, cur, n, s);
    BST_CUDA(cudaMemcpyAsync(perm, cur, sizeof(int32_t) * (size_t)n, cudaMemcpyDeviceToDevice, s));
  }
}

}  // namespace bst
