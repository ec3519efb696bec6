// a10: the set union of Algorithm 2 (§3.2).
//
// 1. every candidate row gets a 64-bit hash (16-byte vector loads);
// 2. rows are inserted into an open-addressing table of row indices with
//    linear probing.  Rows are fully written before the insert kernel runs,
//    so an insert only ever compares against complete rows: a lock-free CAS
//    on an empty slot makes a row the representative of its value, and a
//    match (hash, then bytes) marks it a duplicate.  The table holds at least
//    twice as many slots as rows, so every probe sequence meets an empty slot
//    and the loop is bounded by the table size;
// 3. representatives are compacted (order not fixed by the hardware) and
//    then sorted lexicographically, which fixes the output order
//    independently of the atomics.  The key of a row is the first 64 bits of
//    its bytes in an order-preserving prefix code (2 bits for a 0, 3 for a
//    +-1, up to 16): about 30 coordinates of a sparse row, 14 of a dense one,
//    where the raw bytes gave 8, which most rows of a set share.  A merge sort
//    of (key, row index) pairs, 2048 to a block in shared memory, then merge
//    passes over pairs of runs; equal keys are decided by the rows themselves,
//    16 bytes at a time.  (The bitonic network on raw 8-byte keys with a
//    second sort of the runs of equal keys took 3.2 ms for the 90 000 distinct
//    of 120 000 rows of 200 bytes and 7.3 ms for 225 000 of 300 000 rows of
//    2000, the whole stage; with this sort it takes 0.50 and 1.26 ms.)
#include "common.cuh"

#include <algorithm>
#include <mutex>
#include <vector>

namespace {

constexpr uint32_t kEmpty = 0xffffffffu;

__device__ __forceinline__ uint64_t mix64(uint64_t x) {
  x ^= x >> 31;
  x *= 0x7fb5d329728ea185ull;
  x ^= x >> 27;
  x *= 0x81dadef4bc2dd44dull;
  x ^= x >> 33;
  return x;
}

__device__ __forceinline__ void hash_row(const int8_t* __restrict__ rows, int64_t r, int ldc,
                                         uint64_t* __restrict__ h) {
  const uint4* p = reinterpret_cast<const uint4*>(rows + r * ldc);
  uint64_t acc = 0x243f6a8885a308d3ull ^ (uint64_t)ldc;
  for (int c = 0; c < ldc / 16; ++c) {
    uint4 v = p[c];
    acc = mix64(acc ^ (((uint64_t)v.y << 32) | v.x));
    acc = mix64(acc + (((uint64_t)v.w << 32) | v.z));
  }
  h[r] = acc;
}

__global__ void hash_rows_kernel(const int8_t* __restrict__ rows, int64_t count, int ldc,
                                 uint64_t* __restrict__ h) {
  int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (r >= count) return;
  hash_row(rows, r, ldc, h);
}

__device__ __forceinline__ bool rows_equal(const int8_t* a, const int8_t* b, int ldc) {
  const uint4* pa = reinterpret_cast<const uint4*>(a);
  const uint4* pb = reinterpret_cast<const uint4*>(b);
  for (int c = 0; c < ldc / 16; ++c) {
    uint4 x = pa[c], y = pb[c];
    if (x.x != y.x || x.y != y.y || x.z != y.z || x.w != y.w) return false;
  }
  return true;
}

__device__ __forceinline__ void insert_row(const int8_t* __restrict__ rows, const uint64_t* __restrict__ h,
                                           int64_t r, int ldc, uint32_t* __restrict__ table, uint64_t mask,
                                           uint8_t* __restrict__ is_rep) {
  uint64_t hr = h[r];
  uint64_t slot = hr & mask;
  uint8_t rep = 0;
  for (uint64_t probe = 0; probe <= mask; ++probe) {
    uint32_t cur = table[slot];
    if (cur == kEmpty) {
      uint32_t old = atomicCAS(&table[slot], kEmpty, (uint32_t)r);
      if (old == kEmpty) { rep = 1; break; }
      cur = old;
    }
    if (h[cur] == hr && rows_equal(rows + (int64_t)cur * ldc, rows + r * ldc, ldc)) break;
    slot = (slot + 1) & mask;
  }
  is_rep[r] = rep;
}

__global__ void insert_kernel(const int8_t* __restrict__ rows, const uint64_t* __restrict__ h, int64_t count,
                              int ldc, uint32_t* __restrict__ table, uint64_t mask,
                              uint8_t* __restrict__ is_rep) {
  int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (r >= count) return;
  insert_row(rows, h, r, ldc, table, mask, is_rep);
}

__device__ __forceinline__ void compact_row(const uint8_t* __restrict__ is_rep, int64_t r,
                                            uint32_t* __restrict__ idx, unsigned long long* __restrict__ K) {
  if (!is_rep[r]) return;
  unsigned long long at = atomicAdd(K, 1ull);
  idx[at] = (uint32_t)r;
}

__global__ void compact_reps_kernel(const uint8_t* __restrict__ is_rep, int64_t count,
                                    uint32_t* __restrict__ idx, unsigned long long* __restrict__ K) {
  int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (r >= count) return;
  compact_row(is_rep, r, idx, K);
}

// ---- the sort -------------------------------------------------------------------

// Prefix code of a signed byte, order-preserving: codes compare as bit strings
// (first bit most significant) as the bytes do.  Zero is 10; a positive m is
// 11 and the code of its magnitude, a negative one 0 and that code inverted.
// Magnitudes: 0 (1), 10 (2), 110 (3), then k + 1 ones, a zero and k bits for
// [2^k, 2^(k+1)), k = 2 .. 5, and seven ones and 7 bits from 64 on.  Length in the
// upper half, bits (right-aligned) in the lower.
__device__ __forceinline__ uint32_t byte_code(int v) {
  if (v == 0) return (2u << 16) | 2u;
  const uint32_t m = (uint32_t)(v < 0 ? -v : v);
  uint32_t len, bits;
  if (m <= 3) {
    len = m;
    bits = (1u << m) - 2u;
  } else if (m < 64) {
    const uint32_t k = 31u - (uint32_t)__clz((int)m);  // 2 .. 5
    len = 2u * k + 2u;
    bits = ((((1u << (k + 1u)) - 1u) << 1) << k) | (m - (1u << k));
  } else {
    len = 14;
    bits = (127u << 7) | (m - 64u);
  }
  if (v > 0) return ((len + 2u) << 16) | (3u << len) | bits;
  return ((len + 1u) << 16) | (~bits & ((1u << len) - 1u));
}

// the first 64 bits of the row's code (tab: byte_code of every byte)
__device__ __forceinline__ uint64_t row_key(const int8_t* __restrict__ row, int ldc, const uint32_t* tab) {
  uint64_t acc = 0;
  int left = 64;
  for (int c = 0; c < ldc / 16 && left > 0; ++c) {
    const uint4 q = reinterpret_cast<const uint4*>(row)[c];
    const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int b = 0; b < 16; ++b) {
      if (left > 0) {
        const uint32_t e = tab[(w[b >> 2] >> (8 * (b & 3))) & 0xffu];
        const int len = (int)(e >> 16);
        const uint64_t bits = e & 0xffffu;
        left -= len;
        acc |= left >= 0 ? bits << left : bits >> -left;
      }
    }
  }
  return acc;
}

// Lexicographic order of the signed bytes of two rows: a before b
__device__ __forceinline__ bool row_less(const int8_t* __restrict__ rows, int ldc, uint32_t a, uint32_t b) {
  const uint4* pa = reinterpret_cast<const uint4*>(rows + (int64_t)a * ldc);
  const uint4* pb = reinterpret_cast<const uint4*>(rows + (int64_t)b * ldc);
  for (int c = 0; c < ldc / 16; ++c) {
    const uint4 x = pa[c], y = pb[c];
    const uint32_t xs[4] = {x.x, x.y, x.z, x.w}, ys[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (xs[k] != ys[k])
        return (__byte_perm(xs[k], 0, 0x0123) ^ 0x80808080u) < (__byte_perm(ys[k], 0, 0x0123) ^ 0x80808080u);
  }
  return false;
}

// One set's arrays: (key, row) pairs in two buffers, K of them.
struct SortView {
  const int8_t* rows;
  int64_t K;
  int ldc;
  uint64_t* key[2];
  uint32_t* idx[2];
};

__device__ __forceinline__ bool pair_less(const SortView& d, uint64_t ka, uint32_t a, uint64_t kb, uint32_t b) {
  return ka != kb ? ka < kb : (a != b && row_less(d.rows, d.ldc, a, b));
}

constexpr int kSortThreads = 256;
constexpr int kSortItems = 8;  // consecutive pairs of a thread
constexpr int kSortTile = kSortThreads * kSortItems;

// Merge path (Green, Odeh and Birk): where the merge of A (na sorted pairs) and B (nb) has given `diag` pairs:
// how many of them come from A (from A first among equals).  ka/ia/kb/ib read
// a pair.
template <typename KA, typename IA, typename KB, typename IB>
__device__ __forceinline__ int merge_split(const SortView& d, KA ka, IA ia, int na, KB kb, IB ib, int nb, int diag) {
  int lo = diag > nb ? diag - nb : 0, hi = diag < na ? diag : na;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    // is A[mid] among the first diag?  yes unless B[diag - 1 - mid] is before it
    if (pair_less(d, kb(diag - 1 - mid), ib(diag - 1 - mid), ka(mid), ia(mid))) hi = mid;
    else lo = mid + 1;
  }
  return lo;
}

// kSortItems pairs of the merge of the shared runs [a, a1) and [b, b1)
__device__ __forceinline__ void merge_items(const SortView& d, const uint64_t* sk, const uint32_t* si, int a, int a1,
                                            int b, int b1, uint64_t (&k)[kSortItems], uint32_t (&i)[kSortItems]) {
#pragma unroll
  for (int u = 0; u < kSortItems; ++u) {
    const bool has_a = a < a1, has_b = b < b1;
    bool take_a = has_a;
    if (has_a && has_b) take_a = !pair_less(d, sk[b], si[b], sk[a], si[a]);
    const int p = take_a ? a : (has_b ? b : 0);
    k[u] = sk[p];
    i[u] = si[p];
    if (take_a) ++a; else ++b;
  }
}

// Sorts tile t of a set: each thread its kSortItems pairs (insertion by a
// network of neighbours), then runs doubling in shared memory.
__device__ __forceinline__ void sort_tile(const SortView& d, int64_t t) {
  __shared__ uint64_t sk[kSortTile];
  __shared__ uint32_t si[kSortTile];
  __shared__ uint32_t tab[256];
  tab[threadIdx.x] = byte_code((int)(int8_t)threadIdx.x);
  __syncthreads();
  const int64_t base = t * kSortTile;
  const int n = (int)(d.K - base < kSortTile ? d.K - base : kSortTile);
  for (int p = threadIdx.x; p < kSortTile; p += kSortThreads) {
    const uint32_t r = p < n ? d.idx[0][base + p] : 0u;
    si[p] = r;
    if (p < n) sk[p] = row_key(d.rows + (int64_t)r * d.ldc, d.ldc, tab);
  }
  __syncthreads();
  const int p0 = threadIdx.x * kSortItems;
  uint64_t k[kSortItems];
  uint32_t i[kSortItems];
#pragma unroll
  for (int u = 0; u < kSortItems; ++u) {
    k[u] = sk[p0 + u];
    i[u] = si[p0 + u];
  }
#pragma unroll
  for (int s = 0; s < kSortItems; ++s)  // odd-even transposition; pairs past the end stay there
#pragma unroll
    for (int u = s & 1; u + 1 < kSortItems; u += 2)
      if (p0 + u + 1 < n && pair_less(d, k[u + 1], i[u + 1], k[u], i[u])) {
        const uint64_t tk = k[u];
        const uint32_t ti = i[u];
        k[u] = k[u + 1];
        i[u] = i[u + 1];
        k[u + 1] = tk;
        i[u + 1] = ti;
      }
  for (int w = kSortItems; w < n; w <<= 1) {  // w: sorted runs; the threads of 2 w pairs merge them
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kSortItems; ++u) {
      sk[p0 + u] = k[u];
      si[p0 + u] = i[u];
    }
    __syncthreads();
    const int a0 = p0 / (2 * w) * (2 * w);
    const int a1 = min(a0 + w, n), b1 = min(a0 + 2 * w, n);
    if (p0 < n) {
      const int diag = p0 - a0;
      const int na = max(0, a1 - a0), nb = max(0, b1 - a1);
      const uint64_t *ka = sk + a0, *kb = sk + a1;
      const uint32_t *ia = si + a0, *ib = si + a1;
      const int x = merge_split(d, [&](int q) { return ka[q]; }, [&](int q) { return ia[q]; }, na,
                                [&](int q) { return kb[q]; }, [&](int q) { return ib[q]; }, nb, diag);
      merge_items(d, sk, si, a0 + x, a1, a1 + diag - x, b1, k, i);
    }
  }
#pragma unroll
  for (int u = 0; u < kSortItems; ++u)
    if (p0 + u < n) {
      d.key[0][base + p0 + u] = k[u];
      d.idx[0][base + p0 + u] = i[u];
    }
}

// Outputs [t, t + 1) kSortTile of the pass that merges runs of w pairs (from
// buffer `from` into the other).  Two warps find the ends of the block's
// stretch in the two runs, 32 probes at a time.
__device__ __forceinline__ void merge_tile(const SortView& d, int64_t w, int from, int64_t t) {
  __shared__ uint64_t sk[kSortTile];
  __shared__ uint32_t si[kSortTile];
  __shared__ int64_t s_split[2];
  const int64_t base = t * kSortTile;
  const int64_t a0 = base / (2 * w) * (2 * w);
  const int64_t a1 = a0 + w < d.K ? a0 + w : d.K, b1 = a0 + 2 * w < d.K ? a0 + 2 * w : d.K;
  const int64_t na = a1 - a0, nb = b1 - a1;
  const uint64_t *ka = (from ? d.key[1] : d.key[0]) + a0, *kb = ka + na;
  const uint32_t *ia = (from ? d.idx[1] : d.idx[0]) + a0, *ib = ia + na;
  uint64_t* const kout = from ? d.key[0] : d.key[1];
  uint32_t* const iout = from ? d.idx[0] : d.idx[1];
  const int64_t end = base + kSortTile < b1 ? base + kSortTile : b1;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp < 2) {
    const int64_t diag = (warp == 0 ? base : end) - a0;
    int64_t lo = diag > nb ? diag - nb : 0, hi = diag < na ? diag : na;
    while (lo < hi) {
      const int64_t step = (hi - lo + 31) / 32;
      const int64_t mid = lo + lane * step;
      // true: A[mid] is among the first diag
      bool in = false;
      if (mid < hi) in = !pair_less(d, kb[diag - 1 - mid], ib[diag - 1 - mid], ka[mid], ia[mid]);
      const int c = __popc(__ballot_sync(0xffffffffu, in));  // the probes that are form a prefix
      if (c == 0) {
        hi = lo;
      } else {
        const int64_t nlo = lo + (c - 1) * step + 1, nhi = lo + c * step;
        lo = nlo;
        hi = nhi < hi ? nhi : hi;
      }
    }
    if (lane == 0) s_split[warp] = lo;
  }
  __syncthreads();
  const int64_t x0 = s_split[0], x1 = s_split[1];
  const int ca = (int)(x1 - x0), n = (int)(end - base);
  const int64_t y0 = base - a0 - x0;
  for (int p = threadIdx.x; p < n; p += kSortThreads) {
    const bool fa = p < ca;
    const int64_t q = fa ? x0 + p : y0 + (p - ca);
    sk[p] = fa ? ka[q] : kb[q];
    si[p] = fa ? ia[q] : ib[q];
  }
  __syncthreads();
  const int p0 = threadIdx.x * kSortItems;
  if (p0 >= n) return;
  const uint64_t* skb = sk + ca;
  const uint32_t* sib = si + ca;
  const int x = merge_split(d, [&](int q) { return sk[q]; }, [&](int q) { return si[q]; }, ca,
                            [&](int q) { return skb[q]; }, [&](int q) { return sib[q]; }, n - ca, p0);
  uint64_t k[kSortItems];
  uint32_t i[kSortItems];
  merge_items(d, sk, si, x, ca, ca + p0 - x, n, k, i);
#pragma unroll
  for (int u = 0; u < kSortItems; ++u)
    if (p0 + u < n) {
      kout[base + p0 + u] = k[u];
      iout[base + p0 + u] = i[u];
    }
}

__global__ void __launch_bounds__(kSortThreads) sort_tiles_kernel(SortView d) { sort_tile(d, blockIdx.x); }
__global__ void __launch_bounds__(kSortThreads) merge_tiles_kernel(SortView d, int64_t w, int from) {
  merge_tile(d, w, from, blockIdx.x);
}

__global__ void gather_rows_kernel(const int8_t* __restrict__ rows, int ldc, const uint32_t* __restrict__ idx,
                                   int64_t K, int8_t* __restrict__ out) {
  int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  int chunks = ldc / 16;
  int64_t r = t / chunks;
  int c = (int)(t % chunks);
  if (r >= K) return;
  reinterpret_cast<uint4*>(out + r * ldc)[c] = reinterpret_cast<const uint4*>(rows + (int64_t)idx[r] * ldc)[c];
}

uint64_t next_pow2(uint64_t x) {
  uint64_t p = 1;
  while (p < x) p <<= 1;
  return p;
}

}  // namespace

namespace mape_detail {

// Sorts the K pairs of the view; the buffer that holds the result.
int sort_pairs(const SortView& d, cudaStream_t st) {
  if (d.K < 2) return 0;  // every row the same: 5 us of 90 for 3000 rows
  const unsigned tiles = (unsigned)ceil_div(d.K, kSortTile);
  launch(sort_tiles_kernel, tiles, kSortThreads, 0, st, d);
  int from = 0;
  for (int64_t w = kSortTile; w < d.K; w <<= 1, from ^= 1) launch(merge_tiles_kernel, tiles, kSortThreads, 0, st, d, w, from);
  return from;
}

uint64_t dedup_table_slots(int64_t count) { return next_pow2((uint64_t)(count > 0 ? count : 1) * 2); }

}  // namespace mape_detail

extern "C" size_t mape_dedup_workspace_bytes(int64_t count, int32_t ldc) {
  (void)ldc;
  if (count < 0) return 0;
  mape_detail::Sizer s;
  s.take<uint64_t>((size_t)count);                               // hashes, then sort keys
  s.take<uint32_t>((size_t)mape_detail::dedup_table_slots(count)); // table, then sorted indices
  s.take<uint8_t>((size_t)count);                                 // representative flags
  s.take<uint32_t>((size_t)(count > 0 ? count : 1));              // sorted indices
  s.take<uint64_t>((size_t)(count > 0 ? count : 1));              // their sort keys
  s.take<unsigned long long>(1);                                  // counter
  return s.bytes();
}

extern "C" int mape_dedup(const int8_t* cand, int64_t count, int32_t n, int32_t ldc, int8_t* uniq,
                          int64_t uniq_cap, int64_t* K_out, void* workspace, size_t workspace_bytes,
                          void* stream) {
  using namespace mape_detail;
  if (!K_out || count < 0 || n <= 0 || ldc < n || ldc % 16 != 0 || uniq_cap < 0) return MAPE_ERR_INVALID_ARG;
  if (count > 0 && !cand) return MAPE_ERR_INVALID_ARG;
  if (count >= (int64_t)kEmpty) return MAPE_ERR_SHAPE;
  *K_out = 0;
  if (count == 0) return MAPE_OK;
  Carver cv(workspace, workspace_bytes);
  uint64_t* h = cv.take<uint64_t>((size_t)count);
  uint64_t slots = dedup_table_slots(count);
  uint32_t* table = cv.take<uint32_t>((size_t)slots);
  uint8_t* is_rep = cv.take<uint8_t>((size_t)count);
  uint32_t* idx = cv.take<uint32_t>((size_t)count);
  uint64_t* keys = cv.take<uint64_t>((size_t)count);
  unsigned long long* dK = cv.take<unsigned long long>(1);
  if (!cv.ok) return MAPE_ERR_CAPACITY;
  cudaStream_t st = as_stream(stream);
  unsigned g = (unsigned)ceil_div(count, 256);
  MAPE_CUDA_TRY(cudaMemsetAsync(table, 0xff, slots * sizeof(uint32_t), st));
  MAPE_CUDA_TRY(cudaMemsetAsync(dK, 0, sizeof(unsigned long long), st));
  mape_detail::launch(hash_rows_kernel, g, 256, 0, st, cand, count, ldc, h);
  mape_detail::launch(insert_kernel, g, 256, 0, st, cand, h, count, ldc, table, slots - 1, is_rep);
  mape_detail::launch(compact_reps_kernel, g, 256, 0, st, is_rep, count, idx, dK);
  MAPE_LAUNCH_CHECK();
  unsigned long long K = 0;
  MAPE_CUDA_TRY(cudaMemcpyAsync(&K, dK, sizeof(K), cudaMemcpyDeviceToHost, st));
  MAPE_CUDA_TRY(cudaStreamSynchronize(st));
  *K_out = (int64_t)K;
  if ((int64_t)K > uniq_cap) return MAPE_ERR_CAPACITY;
  if (!uniq) return MAPE_ERR_INVALID_ARG;
  // the hashes and the table have served: they are the sort's second buffer
  const SortView sv{cand, (int64_t)K, ldc, {keys, h}, {idx, table}};
  const int at = sort_pairs(sv, st);
  int64_t chunks = (int64_t)K * (ldc / 16);
  mape_detail::launch(gather_rows_kernel, (unsigned)ceil_div(chunks, 256), 256, 0, st, cand, ldc, sv.idx[at], (int64_t)K, uniq);
  MAPE_LAUNCH_CHECK();
  MAPE_CUDA_TRY(cudaStreamSynchronize(st));
  return MAPE_OK;
}

// ---- the same stage without any device allocation ----------------------------
//
// For callers that cannot allocate device memory at the point where they
// dedup: hosts that reserve all device memory up front and forbid allocations
// later (fixed-memory long-running loops), or plugins whose host owns the
// device allocator.  The call stays synchronous (it reads the distinct count
// back and synchronises the stream), so it cannot run inside a stream capture.
// The scratch lives in a file-scope device array that every GPU loading this
// library holds until the process exits.  Host code cannot pass that array's
// name to a kernel (in host code it is only a host-side stand-in), so its
// device address is looked up once per device, with that device current, by
// cudaGetSymbolAddress, and cached; a CUDA error forgets the cached address
// (a cudaDeviceReset invalidates it), so the next call looks it up again.

namespace {

constexpr int64_t kStaticDedupRows = (int64_t)1 << 18;       // candidate rows per call
constexpr size_t kStaticDedupBytes = (size_t)10 << 20;        // >= mape_dedup_workspace_bytes(2^18, any ldc)
static __device__ __align__(256) unsigned char g_dedup_scratch[kStaticDedupBytes];

constexpr int kMaxDevices = 64;
std::mutex g_scratch_mu;
void* g_scratch_ptr[kMaxDevices] = {};

// Device address of g_dedup_scratch on the current device (looked up once).
int static_dedup_scratch(void** out) {
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) {
    mape_detail::record_cuda_error(e, "cudaGetDevice", __FILE__, __LINE__);
    return MAPE_ERR_CUDA;
  }
  if (dev < 0 || dev >= kMaxDevices) {
    mape_detail::record_message("mape_dedup_static: device index beyond the 64 devices it supports");
    return MAPE_ERR_INVALID_ARG;
  }
  std::lock_guard<std::mutex> lk(g_scratch_mu);
  if (g_scratch_ptr[dev] == nullptr) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_dedup_scratch);
    if (e != cudaSuccess || p == nullptr) {
      mape_detail::record_cuda_error(e, "cudaGetSymbolAddress(g_dedup_scratch)", __FILE__, __LINE__);
      return MAPE_ERR_CUDA;
    }
    g_scratch_ptr[dev] = p;
  }
  *out = g_scratch_ptr[dev];
  return MAPE_OK;
}

// Drops the cached address of the current device (after a CUDA error, which
// may come from a reset context): the next call looks it up again.
void forget_static_dedup_scratch() {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return;
  std::lock_guard<std::mutex> lk(g_scratch_mu);
  g_scratch_ptr[dev] = nullptr;
}

}  // namespace

extern "C" int64_t mape_dedup_static_max_rows(void) { return kStaticDedupRows; }

extern "C" int mape_dedup_static(const int8_t* cand, int64_t count, int32_t n, int32_t ldc, int8_t* uniq,
                                 int64_t uniq_cap, int64_t* K_out, void* stream) {
  if (!K_out || count < 0 || n <= 0 || ldc < n || ldc % 16 != 0 || uniq_cap < 0) return MAPE_ERR_INVALID_ARG;
  *K_out = 0;
  if (count > kStaticDedupRows) return MAPE_ERR_CAPACITY;  // more rows than the static scratch holds
  if (mape_dedup_workspace_bytes(count, ldc) > kStaticDedupBytes) return MAPE_ERR_CAPACITY;
  if (count == 0) return MAPE_OK;
  void* scratch = nullptr;
  int rc = static_dedup_scratch(&scratch);
  if (rc != MAPE_OK) return rc;
  // the table and the counter are cleared by the stage itself on every call
  rc = mape_dedup(cand, count, n, ldc, uniq, uniq_cap, K_out, scratch, kStaticDedupBytes, stream);
  if (rc == MAPE_ERR_CUDA) forget_static_dedup_scratch();
  return rc;
}

// ---- many candidate sets at once -------------------------------------------
//
// mape_dedup for `count` independent sets in one sequence of launches: every
// kernel of the stage runs once over the rows (or sort positions, runs,
// output pieces) of all sets, each thread, warp or block finding its set by
// binary search over the launch's prefix table.  Each set keeps its own hash
// table, sort arrays and output, carved from its own workspace exactly as
// mape_dedup carves it, so its output is the same.  The merge passes run for
// the largest set; a set already sorted is copied along.

namespace {

struct DedupView {
  const int8_t* rows;
  int64_t count;
  int ldc;
  uint64_t* h;
  uint32_t* table;
  uint64_t mask;
  uint8_t* is_rep;
  uint32_t* idx;
  uint64_t* key;
  int8_t* uniq;
  int64_t K;  // distinct rows
};

__device__ __forceinline__ SortView sort_view(const DedupView& d) {
  return SortView{d.rows, d.K, d.ldc, {d.key, d.h}, {d.idx, d.table}};
}

__device__ __forceinline__ int find_set(const int64_t* __restrict__ prefix, int count, int64_t x) {
  int lo = 0, hi = count - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (prefix[mid] <= x) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// prefix: rows (count + 1 entries)
__global__ void hash_insert_batch_kernel(const DedupView* __restrict__ v, const int64_t* __restrict__ prefix, int count,
                                         int phase, unsigned long long* __restrict__ K) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= prefix[count]) return;
  const int i = find_set(prefix, count, t);
  const DedupView& d = v[i];
  const int64_t r = t - prefix[i];
  if (phase == 0) hash_row(d.rows, r, d.ldc, d.h);
  else if (phase == 1) insert_row(d.rows, d.h, r, d.ldc, d.table, d.mask, d.is_rep);
  else compact_row(d.is_rep, r, d.idx, K + i);
}

// prefix: sort tiles
__global__ void __launch_bounds__(kSortThreads) sort_batch_kernel(const DedupView* __restrict__ v,
                                                                 const int64_t* __restrict__ prefix, int count) {
  const int i = find_set(prefix, count, blockIdx.x);
  sort_tile(sort_view(v[i]), blockIdx.x - prefix[i]);
}
__global__ void __launch_bounds__(kSortThreads) merge_batch_kernel(const DedupView* __restrict__ v,
                                                                  const int64_t* __restrict__ prefix, int count,
                                                                  int64_t w, int from) {
  const int i = find_set(prefix, count, blockIdx.x);
  merge_tile(sort_view(v[i]), w, from, blockIdx.x - prefix[i]);
}

// prefix: 16-byte pieces of the distinct rows
__global__ void gather_batch_kernel(const DedupView* __restrict__ v, const int64_t* __restrict__ prefix, int count,
                                    int at) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= prefix[count]) return;
  const int i = find_set(prefix, count, t);
  const DedupView& d = v[i];
  const int64_t e = t - prefix[i];
  const int chunks = d.ldc / 16;
  const int64_t r = e / chunks;
  const int c = (int)(e % chunks);
  reinterpret_cast<uint4*>(d.uniq + r * d.ldc)[c] = reinterpret_cast<const uint4*>(d.rows + (int64_t)(at ? d.table : d.idx)[r] * d.ldc)[c];
}

}  // namespace

// prefix tables of the batch launches, `count` + 1 entries each
enum { kPxRows, kPxTiles, kPxPieces, kPxTables };

extern "C" size_t mape_dedup_batch_workspace_bytes(int32_t count) {
  if (count <= 0) return 0;
  mape_detail::Sizer s;
  s.take<DedupView>((size_t)count);
  s.take<int64_t>((size_t)kPxTables * (count + 1));  // prefix tables
  s.take<unsigned long long>((size_t)count);         // distinct-row counters
  return s.bytes();
}

extern "C" int mape_dedup_batch(mape_dedup_item* items, int32_t count, void* workspace, size_t workspace_bytes,
                                void* stream) {
  using namespace mape_detail;
  if (!items || count <= 0) return MAPE_ERR_INVALID_ARG;
  for (int i = 0; i < count; ++i) {
    const mape_dedup_item& it = items[i];
    if (it.count < 0 || it.n <= 0 || it.ldc < it.n || it.ldc % 16 != 0 || it.uniq_cap < 0) return MAPE_ERR_INVALID_ARG;
    if (it.count > 0 && !it.cand) return MAPE_ERR_INVALID_ARG;
    if (it.count >= (int64_t)kEmpty) return MAPE_ERR_SHAPE;
  }
  Carver bc(workspace, workspace_bytes);
  DedupView* d_views = bc.take<DedupView>((size_t)count);
  int64_t* d_px = bc.take<int64_t>((size_t)kPxTables * (count + 1));
  unsigned long long* d_K = bc.take<unsigned long long>((size_t)count);
  if (!bc.ok) return MAPE_ERR_CAPACITY;
  cudaStream_t st = as_stream(stream);
  const int n1 = count + 1;
  std::vector<int64_t> px((size_t)kPxTables * n1, 0);
  // prefix table `t` over units(i), returning its total
  auto prefix = [&](int t, auto units) -> int64_t {
    int64_t* p = px.data() + (size_t)t * n1;
    p[0] = 0;
    for (int i = 0; i < count; ++i) p[i + 1] = p[i] + units(i);
    return p[count];
  };
  auto dpx = [&](int t) -> const int64_t* { return d_px + (size_t)t * n1; };
  std::vector<DedupView> v((size_t)count);
  for (int i = 0; i < count; ++i) {
    mape_dedup_item& it = items[i];
    it.K = 0;
    it.status = MAPE_OK;
    DedupView& d = v[(size_t)i];
    d = DedupView{};
    d.rows = it.cand;
    d.count = it.count;
    d.ldc = it.ldc;
    d.uniq = it.uniq;
    if (it.count == 0) continue;
    // the same carve as mape_dedup
    Carver cv(it.workspace, it.workspace_bytes);
    d.h = cv.take<uint64_t>((size_t)it.count);
    const uint64_t slots = dedup_table_slots(it.count);
    d.table = cv.take<uint32_t>((size_t)slots);
    d.mask = slots - 1;
    d.is_rep = cv.take<uint8_t>((size_t)it.count);
    d.idx = cv.take<uint32_t>((size_t)it.count);
    d.key = cv.take<uint64_t>((size_t)it.count);
    cv.take<unsigned long long>(1);
    if (!cv.ok) {
      it.status = MAPE_ERR_CAPACITY;
      return MAPE_ERR_CAPACITY;
    }
    MAPE_CUDA_TRY(cudaMemsetAsync(d.table, 0xff, slots * sizeof(uint32_t), st));
  }
  // 1. hash, insert, compact over the rows of every set
  const int64_t rows = prefix(kPxRows, [&](int i) { return v[(size_t)i].count; });
  MAPE_CUDA_TRY(cudaMemcpyAsync(d_views, v.data(), sizeof(DedupView) * count, cudaMemcpyHostToDevice, st));
  MAPE_CUDA_TRY(cudaMemcpyAsync(d_px, px.data(), sizeof(int64_t) * n1, cudaMemcpyHostToDevice, st));
  MAPE_CUDA_TRY(cudaMemsetAsync(d_K, 0, sizeof(unsigned long long) * count, st));
  if (rows > 0) {
    const unsigned g = (unsigned)ceil_div(rows, 256);
    for (int phase = 0; phase < 3; ++phase)
      launch(hash_insert_batch_kernel, g, 256, 0, st, (const DedupView*)d_views, dpx(kPxRows), (int)count, phase, d_K);
    MAPE_LAUNCH_CHECK();
  }
  std::vector<unsigned long long> hK((size_t)count, 0);
  MAPE_CUDA_TRY(cudaMemcpyAsync(hK.data(), d_K, sizeof(unsigned long long) * count, cudaMemcpyDeviceToHost, st));
  MAPE_CUDA_TRY(cudaStreamSynchronize(st));
  int first_err = MAPE_OK;
  int64_t max_K = 0;
  for (int i = 0; i < count; ++i) {
    mape_dedup_item& it = items[i];
    DedupView& d = v[(size_t)i];
    it.K = (int64_t)hK[(size_t)i];
    d.K = it.K;
    if (it.K > it.uniq_cap || (it.K > 0 && !it.uniq)) {  // as mape_dedup: the count only
      it.status = it.K > it.uniq_cap ? MAPE_ERR_CAPACITY : MAPE_ERR_INVALID_ARG;
      if (first_err == MAPE_OK) first_err = it.status;
      d.K = 0;
    }
    max_K = std::max(max_K, d.K);
  }
  // 2. the sort, with the merge passes of the largest set
  const int64_t tiles = prefix(kPxTiles, [&](int i) { return ceil_div(v[(size_t)i].K, kSortTile); });
  const int64_t pieces = prefix(kPxPieces, [&](int i) { return v[(size_t)i].K * (v[(size_t)i].ldc / 16); });
  MAPE_CUDA_TRY(cudaMemcpyAsync(d_views, v.data(), sizeof(DedupView) * count, cudaMemcpyHostToDevice, st));
  MAPE_CUDA_TRY(cudaMemcpyAsync(d_px, px.data(), sizeof(int64_t) * kPxTables * n1, cudaMemcpyHostToDevice, st));
  int at = 0;
  if (tiles > 0) {
    launch(sort_batch_kernel, (unsigned)tiles, kSortThreads, 0, st, (const DedupView*)d_views, dpx(kPxTiles), (int)count);
    for (int64_t w = kSortTile; w < max_K; w <<= 1, at ^= 1)
      launch(merge_batch_kernel, (unsigned)tiles, kSortThreads, 0, st, (const DedupView*)d_views, dpx(kPxTiles),
             (int)count, w, at);
    MAPE_LAUNCH_CHECK();
  }
  // 3. the distinct rows in order
  if (pieces > 0)
    launch(gather_batch_kernel, (unsigned)ceil_div(pieces, 256), 256, 0, st, (const DedupView*)d_views,
           dpx(kPxPieces), (int)count, at);
  MAPE_LAUNCH_CHECK();
  MAPE_CUDA_TRY(cudaStreamSynchronize(st));
  return first_err;
}
