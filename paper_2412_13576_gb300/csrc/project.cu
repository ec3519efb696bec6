// a2: starting points z0 = (B^T B)^{-1} B^T g (§3.2, Algorithm 2).
//
// Per instance: H = B^T B (exact in int64, rounded to FP32), its Cholesky
// factor L (blocked, right-looking, panels of 64 columns, d <= 4096) and
// W = B H^{-1} (n x d) by a forward and a backward triangular solve per row
// of B.  Per start: z0 = W^T g, i.e. Z0 = G0 W for all starts at once with a
// tiled FP32 GEMM (64 x 64 output tiles, 4 x 4 per thread).
#include "common.cuh"
#include "tc_ptx.cuh"

#include <algorithm>

namespace {

// One block per column k: its nonzeros (a kernel basis has few) are listed in
// shared memory, a piece of the rows at a time, and every thread adds them up
// for its rows j >= k of H.  Exact in int64, so the order does not matter.  (One
// thread per entry over all n rows took 172 us for n = 1000, d = 800.)
constexpr int kGramThreads = 256, kGramList = 1024, kGramPer = 16;

__global__ void __launch_bounds__(kGramThreads) gram_kernel(const int32_t* __restrict__ B, int n, int d,
                                                            float* __restrict__ H) {
  __shared__ int s_row[kGramList];
  __shared__ int s_val[kGramList];
  __shared__ int s_n;
  const int k = blockIdx.x;
  for (int jb = k; jb < d; jb += kGramThreads * kGramPer) {
    long long acc[kGramPer];
#pragma unroll
    for (int q = 0; q < kGramPer; ++q) acc[q] = 0;
    for (int i0 = 0; i0 < n; i0 += kGramList) {
      if (threadIdx.x == 0) s_n = 0;
      __syncthreads();
      for (int i = i0 + threadIdx.x; i < n && i < i0 + kGramList; i += kGramThreads) {
        const int v = B[(int64_t)i * d + k];
        if (v != 0) {
          const int at = atomicAdd(&s_n, 1);
          s_row[at] = i;
          s_val[at] = v;
        }
      }
      __syncthreads();
      const int cnt = s_n;
      for (int e = 0; e < cnt; ++e) {
        const long long v = s_val[e];
        const int32_t* row = B + (int64_t)s_row[e] * d;
#pragma unroll
        for (int q = 0; q < kGramPer; ++q) {
          const int j = jb + q * kGramThreads + threadIdx.x;
          if (j < d) acc[q] += v * row[j];
        }
      }
      __syncthreads();
    }
#pragma unroll
    for (int q = 0; q < kGramPer; ++q) {
      const int j = jb + q * kGramThreads + threadIdx.x;
      if (j < d) {
        H[(int64_t)j * d + k] = (float)acc[q];
        H[(int64_t)k * d + j] = (float)acc[q];
      }
    }
  }
}

// The same for small n, a thread per entry over all rows, eight loads at once:
// the list's barriers outweigh its gain (n = 20: 3.7 us against 5.4)
constexpr int kGramSmall = 128;
__global__ void gram_small_kernel(const int32_t* __restrict__ B, int n, int d, float* __restrict__ H) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x, k = blockIdx.y;
  if (j >= d || j < k) return;  // lower triangle: row j >= column k
  long long acc = 0;
#pragma unroll 8
  for (int i = 0; i < n; ++i) acc += (long long)B[(int64_t)i * d + j] * B[(int64_t)i * d + k];
  H[(int64_t)j * d + k] = (float)acc;
  H[(int64_t)k * d + j] = (float)acc;
}

// Blocked right-looking Cholesky of the lower triangle of H (row-major,
// d x d), panel width kNB: per panel, (1) the diagonal block is factored in
// shared memory by one CTA, (2) the rows below it are solved against it
// (L21 = A21 L11^{-T}, one thread per row), (3) the trailing matrix takes the
// rank-kNB update A22 -= L21 L21^T on 64 x 64 tiles of its lower triangle.
// Only the lower triangle is read and written; the upper one is left as is.
constexpr int kNB = 64;

// In both kernels four threads share a row, thread c of them its columns
// 4 q + c in registers; step t finishes column t and takes its product from the
// columns behind it, so that every entry sees its terms in the order t = 0, 1,
// ..., one fused multiply-add each.  Four steps on, the finished column group
// leaves and the registers move down one, so that the loop's code is four
// steps long (64 unrolled steps were bound by fetching them: 38 and 22 us).  A
// panel is a chain of 64 steps of one division and a few multiply-adds; with
// the rows in shared memory and integer divisions for the addresses (diagonal
// block), or as a chain of 2048 dependent products (panel), it took 58 + 66 us
// per panel, 24 + 21 us now.
constexpr int kRowThreads = 4, kRowCols = kNB / kRowThreads;

__global__ void __launch_bounds__(kNB * kRowThreads) chol_diag_kernel(float* __restrict__ H, int d, int k0,
                                                                      int32_t* __restrict__ status) {
  __shared__ float col[2][kNB];
  const int nb = min(kNB, d - k0);
  const int i = threadIdx.x / kRowThreads, c = threadIdx.x % kRowThreads;
  float x[kRowCols];
#pragma unroll
  for (int q = 0; q < kRowCols; ++q) {
    const int j = kRowThreads * q + c;
    x[q] = i < nb && j <= i ? H[(int64_t)(k0 + i) * d + k0 + j] : 0.f;
  }
#pragma unroll 1
  for (int t0 = 0; t0 < nb; t0 += kRowThreads) {
#pragma unroll
    for (int s = 0; s < kRowThreads; ++s) {
      const int t = t0 + s;
      if (t < nb) {  // block-uniform
        float* cb = col[s & 1];
        float v = __shfl_sync(0xffffffffu, x[0], (threadIdx.x & 28) | s);
        if (i == t) {
          if (!(v > 0.f)) {
            if (c == 0) *status = 1;
            v = 1.f;
          }
          v = sqrtf(v);
          if (c == 0) cb[t] = v;
        }
        __syncthreads();
        if (i > t) v /= cb[t];
        if (i >= t && c == s) x[0] = v;
        if (i > t && c == 0) cb[i] = v;
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kRowCols; ++q) {
          const int j = t0 + kRowThreads * q + c;
          if (j > t && j <= i) x[q] -= v * cb[j];
        }
      }
    }
    const int j = t0 + c;
    if (i < nb && j <= i) H[(int64_t)(k0 + i) * d + k0 + j] = x[0];
#pragma unroll
    for (int q = 0; q + 1 < kRowCols; ++q) x[q] = x[q + 1];
  }
}

constexpr int kPanelRows = 64;

__global__ void __launch_bounds__(kPanelRows * kRowThreads) chol_panel_kernel(float* __restrict__ H, int d, int k0) {
  // a full panel: rows below it exist only then; zeros past the last column
  __shared__ float L11[2 * kNB][kNB + 1];
  for (int e = threadIdx.x; e < 2 * kNB * kNB; e += kPanelRows * kRowThreads) {
    const int i = e / kNB, j = e % kNB;
    L11[i][j] = i < kNB && j <= i ? H[(int64_t)(k0 + i) * d + k0 + j] : 0.f;
  }
  const int i = k0 + kNB + blockIdx.x * kPanelRows + threadIdx.x / kRowThreads, c = threadIdx.x % kRowThreads;
  float x[kRowCols];
#pragma unroll
  for (int q = 0; q < kRowCols; ++q) x[q] = i < d ? H[(int64_t)i * d + k0 + kRowThreads * q + c] : 0.f;
  __syncthreads();
#pragma unroll 1
  for (int t0 = 0; t0 < kNB; t0 += kRowThreads) {
#pragma unroll
    for (int s = 0; s < kRowThreads; ++s) {
      const int t = t0 + s;
      const float v = __shfl_sync(0xffffffffu, x[0], (threadIdx.x & 28) | s) / L11[t][t];
      if (c == s) x[0] = v;
#pragma unroll
      for (int q = 0; q < kRowCols; ++q) {
        const int j = t0 + kRowThreads * q + c;
        if (j > t) x[q] -= v * L11[j][t];
      }
    }
    if (i < d) H[(int64_t)i * d + k0 + t0 + c] = x[0];
#pragma unroll
    for (int q = 0; q + 1 < kRowCols; ++q) x[q] = x[q + 1];
  }
}

__global__ void __launch_bounds__(256) chol_update_kernel(float* __restrict__ H, int d, int k0) {
  const int nb = min(kNB, d - k0), base = k0 + nb;
  const int ti = blockIdx.y, tj = blockIdx.x;
  if (tj > ti) return;  // lower-triangular tiles only
  const int r0 = base + ti * 64, c0 = base + tj * 64;
  __shared__ float sa[kNB][64 + 4];
  __shared__ float sb[kNB][64 + 4];
  for (int e = threadIdx.x; e < 64 * nb; e += 256) {
    const int r = e / nb, t = e % nb;
    sa[t][r] = r0 + r < d ? H[(int64_t)(r0 + r) * d + k0 + t] : 0.f;
    sb[t][r] = c0 + r < d ? H[(int64_t)(c0 + r) * d + k0 + t] : 0.f;
  }
  __syncthreads();
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  float acc[4][4] = {};
  for (int t = 0; t < nb; ++t) {
    float av[4], bv[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) { av[q] = sa[t][ty * 4 + q]; bv[q] = sb[t][tx * 4 + q]; }
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[p][q] = fmaf(av[p], bv[q], acc[p][q]);
  }
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    const int i = r0 + ty * 4 + p;
    if (i >= d) continue;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int j = c0 + tx * 4 + q;
      if (j < d && j <= i) H[(int64_t)i * d + j] -= acc[p][q];
    }
  }
}

// Lt = L^T (upper triangle; the strict lower part of Lt is zero)
__global__ void transpose_lower_kernel(const float* __restrict__ L, int d, float* __restrict__ Lt) {
  __shared__ float tile[32][33];
  const int bx = blockIdx.x * 32, by = blockIdx.y * 32;
  for (int y = threadIdx.y; y < 32; y += blockDim.y) {
    const int i = by + y, j = bx + threadIdx.x;
    tile[y][threadIdx.x] = (i < d && j < d && j <= i) ? L[(int64_t)i * d + j] : 0.f;
  }
  __syncthreads();
  for (int y = threadIdx.y; y < 32; y += blockDim.y) {
    const int i = bx + y, j = by + threadIdx.x;  // Lt[i][j] = L[j][i]
    if (i < d && j < d) Lt[(int64_t)i * d + j] = tile[threadIdx.x][y];
  }
}

// Row r of W = B H^{-1} = H^{-1} B_r^T (H symmetric): forward solve L u = B_r^T,
// backward solve L^T w = u.  A warp solves one row with its vector in shared
// memory (lane l sums the terms k = l, l + 32, ... of a step, the 32 sums are
// added by a butterfly); the eight warps of a block take the rows of L (then
// L^T) from a ring filled several steps ahead by asynchronous copies.  A step
// waits for the one before, so what counts is its latency: with every warp
// loading its row of L itself, one right-hand side at a time, a step waited for
// L2 (2.59 ms for n = 1000, d = 800; 0.95 ms now).
constexpr int kSolveWarps = 8;
constexpr int kSolveRows = 1;   // per warp
constexpr int kSolveBatch = 16;  // terms of a lane loaded at once
constexpr int kSolveRing = 8;  // rows of L ahead, at most

__host__ __device__ inline size_t solve_row_bytes(int d) { return ((size_t)d * 4 + 15) / 16 * 16; }

// kTail: terms of a lane that the last batch of a step may have, 2 while d <= 64
// (16 predicated ones a step were most of the instructions at d = 15)
template <int kTail>
__global__ void __launch_bounds__(32 * kSolveWarps) w_solve_kernel(const int32_t* __restrict__ B, const float* __restrict__ L,
                                                          const float* __restrict__ Lt, int n, int d, int ring,
                                                          float* __restrict__ W) {
  extern __shared__ __align__(16) float s_vec[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rp = (int)(solve_row_bytes(d) / 4);  // pitch of a staged row
  float* const srow = s_vec;                     // [ring][rp]
  const int r0 = (blockIdx.x * kSolveWarps + warp) * kSolveRows;
  float* u[kSolveRows];
#pragma unroll
  for (int q = 0; q < kSolveRows; ++q) {
    u[q] = s_vec + (size_t)ring * rp + (size_t)(warp * kSolveRows + q) * rp;
    for (int i = lane; i < d; i += 32) u[q][i] = r0 + q < n ? (float)B[(int64_t)(r0 + q) * d + i] : 0.f;
  }
  // step s of a sweep uses row i(s) = s forward, d - 1 - s backward, of `src`;
  // only its entries up to (from) the diagonal are copied, in 16-byte pieces
  // where a row starts on one
  const bool vec = (d & 3) == 0;
  auto fetch = [&](const float* src, int s, int slot, bool back) {  // slot: s % ring
    if (s < d) {
      const int i = back ? d - 1 - s : s;
      const float* g = src + (int64_t)i * d;
      float* t = srow + (size_t)slot * rp;
      const int k0 = back ? i : 0, k1 = back ? d : i + 1;
      if (vec) {
        for (int k = (k0 & ~3) + 4 * (int)threadIdx.x; k < k1; k += 4 * 32 * kSolveWarps)
          mape_tc::cp_async16(mape_tc::smem_u32(t + k), g + k);
      } else {
        for (int k = k0 + (int)threadIdx.x; k < k1; k += 32 * kSolveWarps)
          asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(mape_tc::smem_u32(t + k)), "l"(g + k) : "memory");
      }
    }
    mape_tc::cp_async_commit();
  };
  auto sweep = [&](const float* src, bool back) {
    for (int s = 0; s < ring - 1; ++s) fetch(src, s, s, back);
    int slot = 0, prev = ring - 1;  // of steps s and s - 1
#pragma unroll 1
    for (int s = 0; s < d; ++s) {
      // rows s .. s + ring - 2 are on their way; row s has to be here
      if (ring == 8) mape_tc::cp_async_wait<6>();
      else if (ring == 4) mape_tc::cp_async_wait<2>();
      else mape_tc::cp_async_wait<0>();
      __syncthreads();  // ... for every thread's copies, and row s - 1 is no longer read
      const int i = back ? d - 1 - s : s;
      const float* row = srow + (size_t)slot * rp;
      float part[kSolveRows];
#pragma unroll
      for (int q = 0; q < kSolveRows; ++q) part[q] = 0.f;
      const float diag = row[i];
      float ui[kSolveRows];
#pragma unroll
      for (int q = 0; q < kSolveRows; ++q) ui[q] = u[q][i];
      int k = back ? i + 1 + lane : lane;
      const int ke = back ? d : i;
#pragma unroll 1
      for (; k + (kSolveBatch - 1) * 32 < ke; k += kSolveBatch * 32) {
        float l[kSolveBatch], v[kSolveRows][kSolveBatch];
#pragma unroll
        for (int e = 0; e < kSolveBatch; ++e) {
          l[e] = row[k + 32 * e];
#pragma unroll
          for (int q = 0; q < kSolveRows; ++q) v[q][e] = u[q][k + 32 * e];
        }
#pragma unroll
        for (int e = 0; e < kSolveBatch; ++e)
#pragma unroll
          for (int q = 0; q < kSolveRows; ++q) part[q] = fmaf(l[e], v[q][e], part[q]);
      }
      {
        float l[kTail], v[kSolveRows][kTail];
#pragma unroll
        for (int e = 0; e < kTail; ++e) {  // the rest; an absent term is skipped, not added as 0
          const bool in = k + 32 * e < ke;
          l[e] = in ? row[k + 32 * e] : 0.f;
#pragma unroll
          for (int q = 0; q < kSolveRows; ++q) v[q][e] = in ? u[q][k + 32 * e] : 0.f;
        }
#pragma unroll
        for (int e = 0; e < kTail; ++e)
#pragma unroll
          for (int q = 0; q < kSolveRows; ++q)
            if (k + 32 * e < ke) part[q] = fmaf(l[e], v[q][e], part[q]);
      }
      fetch(src, s + ring - 1, prev, back);
      prev = slot;
      slot = slot + 1 == ring ? 0 : slot + 1;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int q = 0; q < kSolveRows; ++q) part[q] += __shfl_xor_sync(0xffffffffu, part[q], o);
#pragma unroll
      for (int q = 0; q < kSolveRows; ++q) {
        ui[q] = (ui[q] - part[q]) / diag;
        if (lane == 0) u[q][i] = ui[q];
      }
      __syncwarp();
    }
    __syncthreads();  // the ring is free for the next sweep
  };
  __syncwarp();
  sweep(L, false);
  sweep(Lt, true);
#pragma unroll
  for (int q = 0; q < kSolveRows; ++q)
    if (r0 + q < n)
      for (int i = lane; i < d; i += 32) W[(int64_t)(r0 + q) * d + i] = u[q][i];
}

// Z0 [P x d] = G0 [P x n] . W [n x d]: 128 x 64 output tiles, 8 x 4 per thread,
// K in steps of 16 through two shared buffers, the next step's loads in
// registers meanwhile; every entry is one chain of multiply-adds in the order
// k = 0, 1, ....  (64 x 64 tiles of 4 x 4 with one buffer took 440 us for P =
// 4096, n = 1000, d = 800; 189 us now.)
constexpr int kTM = 128, kTN = 64, kTK = 16;

__global__ void __launch_bounds__(256) gemm_kernel(const float* __restrict__ G0, const float* __restrict__ W, int P,
                                                    int n, int d, float* __restrict__ Z) {
  __shared__ __align__(16) float sA[2][kTK][kTM + 4];
  __shared__ __align__(16) float sB[2][kTK][kTN];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int row0 = blockIdx.y * kTM, col0 = blockIdx.x * kTN;
  float acc[8][4] = {};
  float ra[8], rb[4];
  // thread e of the A tile: column e % 16, rows e / 16 + 16 q; of B: row e / 64
  // + 4 q, column e % 64
  const int ak = threadIdx.x & 15, ar = threadIdx.x >> 4, bc = threadIdx.x & 63, bk = threadIdx.x >> 6;
  auto load = [&](int k0) {
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int gr = row0 + ar + 16 * q, gk = k0 + ak;
      ra[q] = (gr < P && gk < n) ? G0[(int64_t)gr * n + gk] : 0.f;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int gk = k0 + bk + 4 * q, gc = col0 + bc;
      rb[q] = (gk < n && gc < d) ? W[(int64_t)gk * d + gc] : 0.f;
    }
  };
  auto put = [&](int b) {
#pragma unroll
    for (int q = 0; q < 8; ++q) sA[b][ak][ar + 16 * q] = ra[q];
#pragma unroll
    for (int q = 0; q < 4; ++q) sB[b][bk + 4 * q][bc] = rb[q];
  };
  load(0);
  put(0);
  __syncthreads();
  int b = 0;
  for (int k0 = 0; k0 < n; k0 += kTK, b ^= 1) {
    if (k0 + kTK < n) load(k0 + kTK);
#pragma unroll
    for (int k = 0; k < kTK; ++k) {
      const float4 a0 = *reinterpret_cast<const float4*>(&sA[b][k][ty * 8]),
                   a1 = *reinterpret_cast<const float4*>(&sA[b][k][ty * 8 + 4]),
                   b0 = *reinterpret_cast<const float4*>(&sB[b][k][tx * 4]);
      const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w}, bb[4] = {b0.x, b0.y, b0.z, b0.w};
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], bb[j], acc[i][j]);
    }
    if (k0 + kTK < n) put(b ^ 1);
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int r = row0 + ty * 8 + i;
    if (r >= P) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int c = col0 + tx * 4 + j;
      if (c < d) Z[(int64_t)r * d + c] = acc[i][j];
    }
  }
}

}  // namespace

extern "C" size_t mape_project_prepare_workspace_bytes(int32_t n, int32_t d) {
  (void)n;
  if (d <= 0) return 0;
  mape_detail::Sizer s;
  s.take<float>((size_t)d * d);   // H, then its Cholesky factor L
  s.take<float>((size_t)d * d);   // L^T
  s.take<float>((size_t)d * d);   // (reserved)
  s.take<int32_t>(1);
  return s.bytes();
}

extern "C" int mape_project_prepare(const int32_t* B, int32_t n, int32_t d, float* W, void* workspace,
                                    size_t workspace_bytes, void* stream) {
  using namespace mape_detail;
  if (!B || !W || n <= 0 || d <= 0 || d > n) return MAPE_ERR_INVALID_ARG;
  if (d > 4096) return MAPE_ERR_SHAPE;
  Carver cv(workspace, workspace_bytes);
  float* H = cv.take<float>((size_t)d * d);
  float* Lt = cv.take<float>((size_t)d * d);
  cv.take<float>((size_t)d * d);
  int32_t* status = cv.take<int32_t>(1);
  if (!cv.ok) return MAPE_ERR_CAPACITY;
  cudaStream_t st = as_stream(stream);
  MAPE_CUDA_TRY(cudaMemsetAsync(status, 0, sizeof(int32_t), st));
  if (n <= kGramSmall)
    mape_detail::launch(gram_small_kernel, dim3((unsigned)ceil_div(d, 128), (unsigned)d), 128, 0, st, B, n, d, H);
  else
    mape_detail::launch(gram_kernel, (unsigned)d, kGramThreads, 0, st, B, n, d, H);
  for (int k0 = 0; k0 < d; k0 += kNB) {
    mape_detail::launch(chol_diag_kernel, 1, kNB * kRowThreads, 0, st, H, d, k0, status);
    const int rest = d - k0 - kNB;
    if (rest > 0) {
      mape_detail::launch(chol_panel_kernel, (unsigned)ceil_div(rest, kPanelRows), kPanelRows * kRowThreads, 0, st, H, d,
                          k0);
      const unsigned T = (unsigned)ceil_div(rest, 64);
      mape_detail::launch(chol_update_kernel, dim3(T, T), 256, 0, st, H, d, k0);
    }
  }
  const unsigned g32 = (unsigned)ceil_div(d, 32);
  mape_detail::launch(transpose_lower_kernel, dim3(g32, g32), dim3(32, 8), 0, st, H, d, Lt);
  size_t lim = 0;
  const auto solve = d <= 64 ? w_solve_kernel<2> : w_solve_kernel<kSolveBatch>;
  const int rc = allow_max_dynamic_smem((const void*)solve, &lim);
  if (rc != MAPE_OK) return rc;
  // the vectors of the block's rows, and as many rows of L ahead as fit
  const size_t rb = solve_row_bytes(d), vecs = (size_t)kSolveWarps * kSolveRows * rb;
  const int ring = vecs + kSolveRing * rb <= lim ? kSolveRing : vecs + 4 * rb <= lim ? 4 : 2;
  const size_t smem = vecs + (size_t)ring * rb;
  if (smem > lim) return MAPE_ERR_SHAPE;
  mape_detail::launch(solve, (unsigned)ceil_div(n, kSolveWarps * kSolveRows), 32 * kSolveWarps, smem, st, B, H, Lt,
                      n, d, ring, W);
  MAPE_LAUNCH_CHECK();
  int32_t h_status = 0;
  MAPE_CUDA_TRY(cudaMemcpyAsync(&h_status, status, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
  MAPE_CUDA_TRY(cudaStreamSynchronize(st));
  return h_status ? MAPE_ERR_NUMERIC : MAPE_OK;
}

extern "C" int mape_project_apply(const float* W, int32_t n, int32_t d, const float* G0, int32_t P, float* Z0,
                                  void* stream) {
  using namespace mape_detail;
  if (!W || n <= 0 || d <= 0 || d > n || P < 0 || (P > 0 && (!G0 || !Z0))) return MAPE_ERR_INVALID_ARG;
  if (P == 0) return MAPE_OK;
  mape_detail::launch(gemm_kernel, dim3((unsigned)ceil_div(d, kTN), (unsigned)ceil_div(P, kTM)), 256, 0,
                      as_stream(stream), G0, W, P, n, d, Z0);
  MAPE_LAUNCH_CHECK();
  return MAPE_OK;
}

extern "C" size_t mape_project_workspace_bytes(int32_t n, int32_t d) {
  if (d <= 0 || n <= 0) return 0;
  mape_detail::Sizer s;
  s.take<float>((size_t)n * d);                                   // W
  s.take<char>(mape_project_prepare_workspace_bytes(n, d));
  return s.bytes();
}

extern "C" int mape_project_starts(const int32_t* B, int32_t n, int32_t d, const float* G0, int32_t P,
                                   float* Z0, void* workspace, size_t workspace_bytes, void* stream) {
  using namespace mape_detail;
  if (!B || n <= 0 || d <= 0 || d > n || P < 0 || (P > 0 && (!G0 || !Z0))) return MAPE_ERR_INVALID_ARG;
  if (d > 4096) return MAPE_ERR_SHAPE;
  Carver cv(workspace, workspace_bytes);
  float* W = cv.take<float>((size_t)n * d);
  size_t pb = mape_project_prepare_workspace_bytes(n, d);
  char* pw = cv.take<char>(pb);
  if (!cv.ok) return MAPE_ERR_CAPACITY;
  int rc = mape_project_prepare(B, n, d, W, pw, pb, stream);
  if (rc != MAPE_OK) return rc;
  return mape_project_apply(W, n, d, G0, P, Z0, stream);
}
