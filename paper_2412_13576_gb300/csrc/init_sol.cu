// Initial feasible solutions of model (1), Eq. (4) (§3.3): projected Adam on
// ||A x - b||_2^2 + lambda3 sum_i (x_i - floor x_i)(ceil x_i - x_i) over the
// box [l, u] from many starts at once; after every `period`-th step the
// rounded iterate (ties to even) is tested exactly (A round(x) = b in int64;
// the box holds by the projection) and, if it changed since the start's
// previous collection in this call, appended as a row of bytes round(x) - l.
//
// One block (dense A: one warp) per start, persistent over the T steps: it keeps
// x in shared memory (the broadcast operand of both products), its threads take
// the rows of A for r = A x - b and the coordinates for 2 A^T r, the gradient
// term of the integrality penalty, Adam and the projection.  FP32 SIMT, the
// precision of the paper's PyTorch version.
//
// The products run over the nonzeros of A, kept by rows and by columns in
// groups of 32 (entry e of the group's 32 rows or columns side by side, each
// list padded with zeros to the group's longest), and for n <= 512 a thread keeps
// Adam's moments of its coordinates in registers.  Skipping a zero changes no
// bit: x and r are finite, and a term 0 x leaves an FP32 sum as it is.  A step
// is bound by the latency of these short lists (17 entries a row on the medium
// workload, where the dense loops ran over 200: 6.0 ms for 1024 starts and 200
// steps, 0.97 ms now).  An A with a row or column more than half full takes
// the dense loops, with A as FP32 in both orientations (in shared memory when
// it fits, else through L2); which of the two kernels works is decided by the
// device, so that the call stays asynchronous.
#include "common.cuh"

#include <cmath>
#include <vector>

namespace {

constexpr int kWarps = 4;
constexpr uint32_t kSmemLimit = 200 * 1024;

struct InitParams {
  int n, m, P, t0, T, period;
  const float* Af;    // [m x n]
  const float* At;    // [n x m]
  const int64_t* b;
  const int32_t* l;
  const int32_t* u;
  float* X;
  float* M;
  float* V;
  const float2* bias;  // (lr / (1 - beta1^t), 1 / sqrt(1 - beta2^t)) per step
  float lambda3, eps, beta1, beta2, omb1, omb2;
  uint8_t* sol;
  int lds;
  int64_t cap;
  unsigned long long* count;
  int32_t* flags;
  float* dbg_f;
  float* dbg_grad;
  int a_smem;  // 1: A and A^T are copied into shared memory
  // the nonzeros: (value, index) lists by rows and by columns
  float2* rows;      // group g of 32 rows at g * 32 * cap_r: entry e of row i at e * 32 + i % 32
  float2* cols;      // the same for columns, cap_c entries
  int32_t* width;    // longest list per group of rows, then per group of columns
  int cap_r, cap_c;
};

// by every lane of a warp: some list of A is longer than its capacity
__device__ __forceinline__ bool lists_overflow(const InitParams& p) {
  const int gr = (p.m + 31) / 32, groups = gr + (p.n + 31) / 32;
  bool over = false;
  for (int i = threadIdx.x & 31; i < groups; i += 32) over |= p.width[i] > (i < gr ? p.cap_r : p.cap_c);
  return __any_sync(0xffffffffu, over) != 0;
}

__device__ __forceinline__ float warp_sum_f(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ void dense_steps(const InitParams& p, float* sm) {
  const int n = p.n, m = p.m;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* sAf = sm;
  float* sAt = sm + (p.a_smem ? (size_t)m * n : 0);
  float* base = sm + (p.a_smem ? 2 * (size_t)m * n : 0);
  float* xs = base + (size_t)warp * (n + m);
  float* rs = xs + n;
  if (p.a_smem) {
    for (int e = threadIdx.x; e < m * n; e += blockDim.x) {
      sAf[e] = p.Af[e];
      sAt[e] = p.At[e];
    }
  }
  __syncthreads();
  const float* Af = p.a_smem ? sAf : p.Af;
  const float* At = p.a_smem ? sAt : p.At;
  const int64_t pg = (int64_t)blockIdx.x * kWarps + warp;
  if (pg >= p.P) return;  // warp-uniform; no block barrier follows
  float* X = p.X + pg * n;
  float* Mv = p.M + pg * n;
  float* Vv = p.V + pg * n;
  for (int j = lane; j < n; j += 32) xs[j] = fminf(fmaxf(X[j], (float)p.l[j]), (float)p.u[j]);
  __syncwarp();
  bool changed = true;  // the first collection of a call always counts
  for (int s = 0; s < p.T; ++s) {
    const int t = p.t0 + s + 1;
    // r = A x - b, one row per lane
    for (int i = lane; i < m; i += 32) {
      float acc = -(float)p.b[i];
      for (int j = 0; j < n; ++j) acc = fmaf(At[(size_t)j * m + i], xs[j], acc);
      rs[i] = acc;
    }
    __syncwarp();
    const bool dbg = s == 0 && (p.dbg_f || p.dbg_grad);
    float fr = 0.f;
    if (dbg && p.dbg_f)
      for (int i = lane; i < m; i += 32) fr += rs[i] * rs[i];
    const float2 ad = p.bias[s];
    bool moved = false;
    for (int j = lane; j < n; j += 32) {
      float g = 0.f;
      for (int i = 0; i < m; ++i) g = fmaf(Af[(size_t)i * n + j], rs[i], g);
      const float x = xs[j];
      const float fl = floorf(x);
      // ceil x + floor x = 2 floor x + [x not an integer]
      const float grad = 2.f * g + p.lambda3 * (2.f * fl + (x != fl ? 1.f : 0.f) - 2.f * x);
      if (dbg) {
        if (p.dbg_f) fr += p.lambda3 * (x - fl) * (ceilf(x) - x);
        if (p.dbg_grad) p.dbg_grad[pg * n + j] = grad;
      }
      const float mm = p.beta1 * Mv[j] + p.omb1 * grad;
      const float vv = p.beta2 * Vv[j] + p.omb2 * grad * grad;
      const float den = (vv > 0.f ? vv * rsqrtf(vv) : 0.f) * ad.y + p.eps;
      float xn = x - ad.x * __fdividef(mm, den);
      xn = fminf(fmaxf(xn, (float)p.l[j]), (float)p.u[j]);
      Mv[j] = mm;
      Vv[j] = vv;
      moved |= rintf(xn) != rintf(x);
      xs[j] = xn;
    }
    if (dbg && p.dbg_f) {
      fr = warp_sum_f(fr);
      if (lane == 0) p.dbg_f[pg] = fr;
    }
    changed |= __any_sync(0xffffffffu, moved);
    __syncwarp();
    if (t % p.period == 0) {
      if (changed) {
        // exact test of A round(x) = b in int64
        bool ok = true;
        for (int i = lane; i < m; i += 32) {
          long long acc = 0;
          for (int j = 0; j < n; ++j) acc += (long long)Af[(size_t)i * n + j] * (long long)rintf(xs[j]);
          ok &= acc == p.b[i];
        }
        ok = __all_sync(0xffffffffu, ok);
        long long slot = -1;
        if (ok && lane == 0) {
          const unsigned long long at = atomicAdd(p.count, 1ull);
          if ((int64_t)at < p.cap) slot = (long long)at;
          else atomicOr(p.flags, 1);
        }
        slot = __shfl_sync(0xffffffffu, slot, 0);
        if (slot >= 0) {
          uint8_t* row = p.sol + slot * p.lds;
          for (int j = lane; j < p.lds; j += 32) row[j] = j < n ? (uint8_t)((int)rintf(xs[j]) - p.l[j]) : 0;
        }
      }
      changed = false;
    }
  }
  for (int j = lane; j < n; j += 32) X[j] = xs[j];
}

// What the steps read of A, in one launch (small calls are bound by their
// launches: a kernel each and a cleared flag cost 256 starts of a 20 x 5 matrix
// 6% of 175 us).  The first blocks: the nonzeros of 32 rows, a warp per row, in
// column order.  The next: those of 32 x 32 columns, a warp per 32 columns, in
// row order.  The rest: A as FP32 in both orientations.
constexpr int kSetupThreads = 1024;

__global__ void __launch_bounds__(kSetupThreads) init_setup_kernel(const int32_t* __restrict__ A, InitParams p,
                                                                   float* __restrict__ Af, float* __restrict__ At) {
  const int n = p.n, m = p.m, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int gr = (m + 31) / 32, gc = (n + 31) / 32;
  int b = blockIdx.x;
  if (b < gr) {
    __shared__ int s_most[kSetupThreads / 32];
    const int w = b * 32 + warp;
    int at = 0;
    if (w < m) {
      float2* out = p.rows + (size_t)b * 32 * p.cap_r + warp;
      for (int j0 = 0; j0 < n; j0 += 32) {
        const int j = j0 + lane;
        const int v = j < n ? A[(int64_t)w * n + j] : 0;
        const unsigned bal = __ballot_sync(0xffffffffu, v != 0);
        const int e = at + __popc(bal & ((1u << lane) - 1));
        if (v != 0 && e < p.cap_r) out[(size_t)e * 32] = make_float2((float)v, __int_as_float(j));
        at += __popc(bal);
      }
      for (int e = at + lane; e < p.cap_r; e += 32) out[(size_t)e * 32] = make_float2(0.f, __int_as_float(0));
    }
    if (lane == 0) s_most[warp] = at;
    __syncthreads();
    if (warp == 0) {
      const int most = (int)__reduce_max_sync(0xffffffffu, (unsigned)s_most[lane]);
      if (lane == 0) p.width[b] = most;
    }
    return;
  }
  b -= gr;
  if (b < (gc + 31) / 32) {
    const int g = b * 32 + warp;  // group of columns
    if (g >= gc) return;
    const int j = g * 32 + lane;
    float2* out = p.cols + (size_t)g * 32 * p.cap_c + lane;
    int at = 0;
#pragma unroll 4
    for (int i = 0; i < m; ++i) {
      const int v = j < n ? A[(int64_t)i * n + j] : 0;
      if (v != 0) {
        if (at < p.cap_c) out[(size_t)at * 32] = make_float2((float)v, __int_as_float(i));
        ++at;
      }
    }
    const int most = (int)__reduce_max_sync(0xffffffffu, (unsigned)at);
    if (lane == 0) p.width[gr + g] = most;
    for (int e = at; e < most && e < p.cap_c; ++e) out[(size_t)e * 32] = make_float2(0.f, __int_as_float(0));
    return;
  }
  b -= (gc + 31) / 32;
  const int64_t e = b * (int64_t)kSetupThreads + threadIdx.x;
  if (e >= (int64_t)m * n) return;
  const int i = (int)(e / n), j = (int)(e % n);
  const float v = (float)A[e];
  Af[e] = v;
  At[(int64_t)j * m + i] = v;
}

// sum of value x vec[index] over a list of `width` entries, from acc, in order
__device__ __forceinline__ float list_dot(const float2* __restrict__ l, int width, const float* vec, float acc) {
  int e = 0;
  for (; e + 4 <= width; e += 4) {
    float2 q[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) q[u] = l[(e + u) * 32];
#pragma unroll
    for (int u = 0; u < 4; ++u) acc = fmaf(q[u].x, vec[__float_as_int(q[u].y)], acc);
  }
  for (; e < width; ++e) {
    const float2 q = l[e * 32];
    acc = fmaf(q.x, vec[__float_as_int(q.y)], acc);
  }
  return acc;
}

constexpr int kListThreads = 128;  // per start

// One block per start: with a warp per start the lists of seven groups of
// columns and their Adam updates followed one another (1.8 ms on the medium
// workload); four warps share them at two block barriers a step.
// kNT > 0: n <= 128 kNT, the moments and bounds of a thread's coordinates in
// registers for the whole call; 0: any n, in global memory.
template <int kNT>
__device__ __forceinline__ void list_steps(const InitParams& p, float* sm) {
  const int n = p.n, m = p.m;
  const int tid = threadIdx.x, lane = tid & 31;
  float* xs = sm;
  float* rs = sm + n;
  const int64_t pg = blockIdx.x;
  float* X = p.X + pg * n;
  float* Mv = p.M + pg * n;
  float* Vv = p.V + pg * n;
  const int ngr = (m + 31) / 32;
  constexpr int kR = kNT > 0 ? kNT : 1;
  float rM[kR], rV[kR], rl[kR], ru[kR];
  int rw[kR];
  if (kNT > 0) {
#pragma unroll
    for (int t = 0; t < kR; ++t) {
      const int j = t * kListThreads + tid;
      const bool in = j < n;
      rM[t] = in ? Mv[j] : 0.f;
      rV[t] = in ? Vv[j] : 0.f;
      rl[t] = in ? (float)p.l[j] : 0.f;
      ru[t] = in ? (float)p.u[j] : 0.f;
      rw[t] = in ? p.width[ngr + (j >> 5)] : 0;
    }
  }
  const int w0 = tid < m ? p.width[tid >> 5] : 0;  // of the thread's first row
  const float nb0 = tid < m ? -(float)p.b[tid] : 0.f;
  for (int j = tid; j < n; j += kListThreads) xs[j] = fminf(fmaxf(X[j], (float)p.l[j]), (float)p.u[j]);
  __syncthreads();
  bool changed = true;  // the first collection of a call always counts
  for (int s = 0; s < p.T; ++s) {
    const int t1 = p.t0 + s + 1;
    for (int i = tid; i < m; i += kListThreads) {  // r = A x - b, a row per thread
      const float2* l = p.rows + (size_t)(i >> 5) * 32 * p.cap_r + lane;
      rs[i] = list_dot(l, i == tid ? w0 : p.width[i >> 5], xs, i == tid ? nb0 : -(float)p.b[i]);
    }
    __syncthreads();
    const bool dbg = s == 0 && (p.dbg_f || p.dbg_grad);
    float fr = 0.f;
    if (dbg && p.dbg_f)
      for (int i = tid; i < m; i += kListThreads) fr += rs[i] * rs[i];
    const float2 ad = p.bias[s];
    bool moved = false;
    auto coordinate = [&](int j, int width, float& mo, float& vo, float lo, float hi) {
      const float gsum = list_dot(p.cols + (size_t)(j >> 5) * 32 * p.cap_c + lane, width, rs, 0.f);
      const float x = xs[j];
      const float fl = floorf(x);
      // ceil x + floor x = 2 floor x + [x not an integer]
      const float grad = fmaf(p.lambda3, 2.f * fl + (x != fl ? 1.f : 0.f) - 2.f * x, 2.f * gsum);
      if (dbg) {
        if (p.dbg_f) fr += p.lambda3 * (x - fl) * (ceilf(x) - x);
        if (p.dbg_grad) p.dbg_grad[pg * n + j] = grad;
      }
      const float mm = p.beta1 * mo + p.omb1 * grad;
      const float vv = p.beta2 * vo + p.omb2 * grad * grad;
      const float den = (vv > 0.f ? vv * rsqrtf(vv) : 0.f) * ad.y + p.eps;
      float xn = x - ad.x * __fdividef(mm, den);
      xn = fminf(fmaxf(xn, lo), hi);
      mo = mm;
      vo = vv;
      moved |= rintf(xn) != rintf(x);
      xs[j] = xn;
    };
    if (kNT > 0) {
#pragma unroll
      for (int t = 0; t < kR; ++t) {
        const int j = t * kListThreads + tid;
        if (j < n) coordinate(j, rw[t], rM[t], rV[t], rl[t], ru[t]);
      }
    } else {
      for (int j = tid; j < n; j += kListThreads) {
        float mo = Mv[j], vo = Vv[j];
        coordinate(j, p.width[ngr + (j >> 5)], mo, vo, (float)p.l[j], (float)p.u[j]);
        Mv[j] = mo;
        Vv[j] = vo;
      }
    }
    if (dbg && p.dbg_f) {
      __shared__ float s_f[kListThreads / 32];
      fr = warp_sum_f(fr);
      if (lane == 0) s_f[tid >> 5] = fr;
      __syncthreads();
      if (tid == 0) {
        float f = 0.f;
        for (int w = 0; w < kListThreads / 32; ++w) f += s_f[w];
        p.dbg_f[pg] = f;
      }
    }
    changed |= __syncthreads_or(moved) != 0;
    if (t1 % p.period == 0) {
      if (changed) {
        // exact test of A round(x) = b in int64
        bool ok = true;
        for (int i = tid; i < m; i += kListThreads) {
          const float2* l = p.rows + (size_t)(i >> 5) * 32 * p.cap_r + lane;
          long long acc = 0;
          const int wd = p.width[i >> 5];
          for (int e = 0; e < wd; ++e) {
            const float2 q = l[e * 32];
            acc += (long long)q.x * (long long)rintf(xs[__float_as_int(q.y)]);
          }
          ok &= acc == p.b[i];
        }
        if (__syncthreads_and(ok)) {
          __shared__ long long s_slot;
          if (tid == 0) {
            long long slot = -1;
            const unsigned long long at = atomicAdd(p.count, 1ull);
            if ((int64_t)at < p.cap) slot = (long long)at;
            else atomicOr(p.flags, 1);
            s_slot = slot;
          }
          __syncthreads();
          const long long slot = s_slot;
          if (slot >= 0) {
            uint8_t* row = p.sol + slot * p.lds;
            for (int j = tid; j < p.lds; j += kListThreads)
              row[j] = j < n ? (uint8_t)((int)rintf(xs[j]) - p.l[j]) : 0;
          }
          __syncthreads();  // xs and the slot are read before the next step writes them
        }
      }
      changed = false;
    }
  }
  if (kNT > 0) {
#pragma unroll
    for (int t = 0; t < kR; ++t) {
      const int j = t * kListThreads + tid;
      if (j < n) {
        Mv[j] = rM[t];
        Vv[j] = rV[t];
      }
    }
  }
  for (int j = tid; j < n; j += kListThreads) X[j] = xs[j];
}

__global__ void __launch_bounds__(32 * kWarps) init_sol_kernel(InitParams p) {
  extern __shared__ __align__(16) float sm[];
  if (lists_overflow(p)) dense_steps(p, sm);
}
// the registers that the moments leave: 12, 10, 8 and 9 blocks an SM
template <int kNT>
__global__ void __launch_bounds__(kListThreads, kNT == 1 ? 12 : kNT == 2 ? 10 : kNT == 4 ? 8 : 9)
init_sol_lists_kernel(InitParams p) {
  extern __shared__ __align__(16) float sm[];
  if (!lists_overflow(p)) list_steps<kNT>(p, sm);
}
// the two in one launch, of a block per start: for the smallest A (a launch for
// nothing is 3 us; with the 9.5 KB of 64 x 16 entries the dense steps take 475 us
// here, 440 in their own kernel)
static_assert(kListThreads == 32 * kWarps);
constexpr size_t kBothSmem = 4 * 1024;
__global__ void __launch_bounds__(kListThreads) init_sol_both_kernel(InitParams p) {
  extern __shared__ __align__(16) float sm[];
  if (!lists_overflow(p)) list_steps<1>(p, sm);
  else if (blockIdx.x < (unsigned)((p.P + kWarps - 1) / kWarps)) dense_steps(p, sm);
}

int list_cap(int x) { return x / 2 + 1; }
size_t list_entries(int lists, int cap) { return (size_t)((lists + 31) / 32) * 32 * cap; }

}  // namespace

extern "C" size_t mape_initial_solutions_workspace_bytes(int32_t n, int32_t m, int32_t T) {
  if (n <= 0 || m <= 0 || T < 0) return 0;
  mape_detail::Sizer s;
  s.take<float>((size_t)m * n);
  s.take<float>((size_t)m * n);
  s.take<float2>((size_t)(T > 0 ? T : 1));
  s.take<float2>(list_entries(m, list_cap(n)));
  s.take<float2>(list_entries(n, list_cap(m)));
  s.take<int32_t>((size_t)(m + 31) / 32 + (n + 31) / 32);
  return s.bytes();
}

extern "C" int mape_initial_solutions(const mape_init_args* a, void* stream) {
  using namespace mape_detail;
  if (!a) return MAPE_ERR_INVALID_ARG;
  const int n = a->n, m = a->m, P = a->P;
  if (n <= 0 || m <= 0 || P < 0 || a->T < 0 || a->t0 < 0 || a->period <= 0) return MAPE_ERR_INVALID_ARG;
  if (!a->A || !a->b || !a->l || !a->u || !a->sol_count || !a->flags) return MAPE_ERR_INVALID_ARG;
  if (P > 0 && (!a->X || !a->M || !a->V)) return MAPE_ERR_INVALID_ARG;
  if (a->lds < n || a->sol_cap < 0 || (a->sol_cap > 0 && !a->sol)) return MAPE_ERR_INVALID_ARG;
  if (n > 48 * 1024) return MAPE_ERR_SHAPE;
  if (P == 0 || a->T == 0) return MAPE_OK;
  if (a->workspace_bytes < mape_initial_solutions_workspace_bytes(n, m, a->T)) return MAPE_ERR_CAPACITY;
  cudaStream_t st = as_stream(stream);
  Carver cv(a->workspace, a->workspace_bytes);
  float* Af = cv.take<float>((size_t)m * n);
  float* At = cv.take<float>((size_t)m * n);
  float2* bias = cv.take<float2>((size_t)a->T);
  float2* rows = cv.take<float2>(list_entries(m, list_cap(n)));
  float2* cols = cv.take<float2>(list_entries(n, list_cap(m)));
  const int gr = (m + 31) / 32, gc = (n + 31) / 32;
  int32_t* width = cv.take<int32_t>((size_t)gr + gc);
  if (!cv.ok) return MAPE_ERR_CAPACITY;
  std::vector<float2> bc((size_t)a->T);
  for (int s = 0; s < a->T; ++s) {
    const double t = (double)a->t0 + s + 1;
    const double bc1 = 1.0 - std::pow(a->beta1, t), bc2 = 1.0 - std::pow(a->beta2, t);
    bc[s] = make_float2((float)((double)a->lr / bc1), (float)(1.0 / std::sqrt(bc2)));
  }
  MAPE_CUDA_TRY(cudaMemcpyAsync(bias, bc.data(), sizeof(float2) * bc.size(), cudaMemcpyHostToDevice, st));
  InitParams p{};
  p.n = n; p.m = m; p.P = P; p.t0 = a->t0; p.T = a->T; p.period = a->period;
  p.Af = Af; p.At = At; p.b = a->b; p.l = a->l; p.u = a->u; p.X = a->X; p.M = a->M; p.V = a->V; p.bias = bias;
  p.lambda3 = a->lambda3; p.eps = a->eps;
  p.beta1 = (float)a->beta1; p.beta2 = (float)a->beta2;
  p.omb1 = (float)(1.0 - a->beta1); p.omb2 = (float)(1.0 - a->beta2);
  p.sol = a->sol; p.lds = a->lds; p.cap = a->sol_cap; p.count = a->sol_count; p.flags = a->flags;
  p.dbg_f = a->dbg_f; p.dbg_grad = a->dbg_grad;
  p.rows = rows; p.cols = cols; p.width = width;
  p.cap_r = list_cap(n); p.cap_c = list_cap(m);
  launch(init_setup_kernel, (unsigned)(gr + ceil_div(gc, 32) + ceil_div((int64_t)m * n, kSetupThreads)), kSetupThreads, 0,
         st, a->A, p, Af, At);
  const size_t per_warp = (size_t)kWarps * (n + m) * sizeof(float);
  const size_t with_a = 2 * (size_t)m * n * sizeof(float) + per_warp;
  p.a_smem = with_a <= kSmemLimit ? 1 : 0;
  const size_t smem = p.a_smem ? with_a : per_warp;
  if (smem > kSmemLimit) return MAPE_ERR_SHAPE;
  {
    size_t lim = 0;
    const int rc = allow_max_dynamic_smem((const void*)init_sol_kernel, &lim);
    if (rc != MAPE_OK) return rc;
    if ((size_t)smem > lim) return MAPE_ERR_SHAPE;
  }
  const size_t lsm = (size_t)(n + m) * sizeof(float);
  if (n <= 128 && smem <= kBothSmem) {  // holds the lists' lsm, too
    launch(init_sol_both_kernel, (unsigned)P, kListThreads, smem, st, p);
    MAPE_LAUNCH_CHECK();
    return MAPE_OK;
  }
  launch(init_sol_kernel, (unsigned)ceil_div(P, kWarps), 32 * kWarps, smem, st, p);
  auto lists = n <= 128 ? init_sol_lists_kernel<1> : n <= 256 ? init_sol_lists_kernel<2>
             : n <= 512 ? init_sol_lists_kernel<4> : init_sol_lists_kernel<0>;
  if (lsm > kSmemUnasked) {
    size_t lim = 0;
    const int rc = allow_max_dynamic_smem((const void*)lists, &lim);
    if (rc != MAPE_OK) return rc;
  }
  launch(lists, (unsigned)P, kListThreads, lsm, st, p);
  MAPE_LAUNCH_CHECK();
  return MAPE_OK;
}
