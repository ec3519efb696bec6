// Algorithm 2 (§3.2) on the tensor cores for identity-topped bases whose tile
// does not fit the resident kernel: one launch runs all T steps.  A cluster of
// C thread blocks (C = 1, 2, 4 or 8) owns a tile of 128 starts for the whole
// call; block c of it owns a slice of the coordinates (whose z, m, v only it
// reads and writes) and a slice of the rows of Bm, the rows of B below the
// identity.  Per step:
//   forward   every block multiplies its rows of Bm with the tile's z operands
//             (all coordinates): D1 = hi(Z) Bm^T + lo(Z) Bm^T, M = 128 starts,
//             N = its rows, K = d in chunks of 32; S = sign(D1) goes to global
//             memory as the gradient's A operand.  On collecting steps the same
//             chunks give D2 = round(Z) Bm^T, tested against C4 and staged.
//   barrier   of the cluster: S of every block is visible to all of them.
//   gradient  G = S Bm[:, slice] (M = 128, N = coordinates of the slice, K = rows
//             of Bm), then Adam on the FP32 state of the slice; the epilogue
//             writes the next step's BF16 (or e4m3) operands of z.
//   barrier   of the cluster: the operands of every block are visible.
// The blocks exchange operands and signs through global memory (L2: 0.3 to 1.3
// MB a tile at n = 2000), so the only thing a step waits for is the cluster's own hardware
// barrier: no launch, no host, and no other tile.  What that replaces: three
// launches per step over all tiles of the call, each with a grid of at most a
// few blocks per SM and one pipeline fill.
// Bound: HBM for many tiles.  n = 2000, P = 65536, e4m3: a step 0.48 ms, 2.78 GB of
// DRAM traffic (the state once each way is 2.52; the rest are operands and signs
// that L2 evicts), 0.86 of the measured copy rate; step by step 0.60 ms.  For few
// tiles the chain of a step, 20 us at n = 487 and P = 1024.
//
// Eight warps convert accumulators (two per TMEM lane quarter).  Before they
// do, warp 0 issues the phase's MMAs and warp 1 its bulk copies, over a ring
// whose stages are cut to the phase's chunks, so that about 100 KB are in flight.
// Both run their loops with all lanes and elect one for the instructions: with
// a single thread doing both, its instruction latency (descriptors moved to
// uniform registers one by one, 1 650 cycles per 32 coordinates) was two thirds
// of a step.  (A ninth warp for the issue would leave 96 registers a thread.)
// Shared memory (112 KB) and registers allow two blocks per SM, each with 256
// TMEM columns, so one tile's forward pass overlaps another tile's epilogue on
// the same SM; the resident kernel (116 KB, 512 columns) never shares an SM with
// them.
//
// The tensor-memory loads and their waits are for a converged warp, which the
// code between them does not leave (lane 0 arrives on a barrier, lanes write
// their debug outputs): without a __syncwarp before each, halves of a warp
// took a chunk's gradient before it was there.  The four cost 1% of a step.
//
// Accumulation order: K ascends in steps of 16, hi before lo, into one FP32
// accumulator per (start, row), the order of the step-by-step kernels of
// extract_stream.cu; the gradient's sums are integers.  Both give the same
// bits.
#include "common.cuh"
#include "extract_internal.cuh"
#include "refill_stage.cuh"
#include "tc_ptx.cuh"

#include <algorithm>
#include <cmath>
#include <memory>
#include <type_traits>
#include <vector>

namespace {
using namespace mape_tc;

constexpr int kTM = 128;                  // starts per tile
constexpr int kThreads = 256;             // 8 warps: two per TMEM lane quarter
constexpr int kKC = 32;                   // K per chunk
constexpr int kMaxStages = 10;            // of the copy ring; how many a phase uses depends on its bytes per chunk
constexpr int kStageMost = 32768;         // chunks are copied in groups of up to this size
constexpr int kChunk16 = kTM * kKC * 2;   // a 128 x 32 BF16 operand chunk (8 KB)
constexpr int kChunk8 = kTM * kKC;        // the same in e4m3 (4 KB)
constexpr int kRowBlk = 128;              // rows of Bm per forward accumulator
constexpr int kColBlk = 256;              // coordinates per gradient accumulator
constexpr int kTmemCols = 256;            // D1 at 0, D2 at 128; the gradient from 0
constexpr int kColD2 = 128;
constexpr int kEStages = 4;               // ring of the epilogue's state: 8 coordinates of z, m, v a stage
constexpr int kEArr = kTM * 8 * 4, kEBytes = 3 * kEArr;
constexpr int kDynSmem = 112 * 1024;      // the spans of the slice, the operand ring (its end: the state ring)
constexpr int kDynSmemOne = 220 * 1024;   // where one block per SM is all there is
constexpr int kMaxC = 8;
constexpr int kSms = 152;
constexpr int kNoNz = 0x7fffffff;
constexpr uint32_t kChanged = 1, kUnexact = 2;
// byte offsets within a K = 32 chunk (8-row groups of 4 or 2 core matrices)
__host__ __device__ __forceinline__ uint32_t off16(int r, int k) {
  return (uint32_t)((((r >> 3) * 4 + (k >> 3)) << 7) + ((r & 7) << 4) + ((k & 7) << 1));
}
__host__ __device__ __forceinline__ uint32_t off8(int r, int k) {
  return (uint32_t)((((r >> 3) * 2 + (k >> 4)) << 7) + ((r & 7) << 4) + (k & 15));
}
constexpr uint32_t kSbo16 = 512, kSbo8 = 256;

struct ClParams {
  int n, d, P, R;       // R: rows of Bm = n - d
  int d32, R32;         // padded to 32
  int tiles, C, dyn;    // blocks per cluster; dynamic shared memory of a block
  int ldc, ldi;         // candidate pitch; pitch of the staged identity rows
  const uint8_t* Bf;    // forward operand: per block and 128-row block, [d32/32][rows x 32] chunks
  const uint8_t* Bf8;   // the same in e4m3
  const uint8_t* Bg;    // gradient operand: per block and 256-coordinate block, [R32/32][coordinates x 32]
  const int32_t* span;
  float* Zt;
  float* Mt;
  float* Vt;            // blocked [tiles][d32/4][128][4]
  // z operands (z_tile): tiles below z1 at Zh[0], the next up to z2 at Zh[1],
  // the rest at Zh[2]
  uint8_t* Zh[3];
  int z1, z2;
  int z_out;            // 1: they lie in the caller's M, V and Z
  uint8_t* S;           // [tiles][R32/32] chunks
  // staged candidate rows: the identity rows [2][tiles*128][ldi] by step parity
  // (those of a step are written while the last step's are read), the Bm rows
  // [tiles*128][R32] (written before a step's gradient, read during it)
  int8_t *stage, *stage_map;
  unsigned long long* zkey;  // [2][tiles*128]: (|z|_inf bits << 32) | (~first argmax)
  uint32_t* acc;        // [2][..] rounding changed / unexact since the last collection
  uint32_t* oob;        // Bm rows of the staged candidate out of the box
  uint32_t* idw;        // [2][..] identity rows out of the box
  int32_t* first;       // [2][..] first nonzero identity row
  const float2* bias;   // (lr / (1 - beta1^t), 1 / sqrt(1 - beta2^t)) per step
  float lambda1, lambda2, eps, beta1, beta2, omb1, omb2;
  int nterms, f8;
  int t0, T, period;
  int8_t* cand;
  int64_t cap;
  unsigned long long* count;
  int32_t* flags;
  float* dbg_phi;
  float* dbg_grad;
};

// slice of rank c: units of 16 spread evenly, the first (units % C) ranks one more
__host__ __device__ __forceinline__ void slice_of(int padded, int C, int c, int& begin, int& len) {
  const int u = padded / 16, base = u / C, rem = u % C;
  begin = 16 * (c * base + (c < rem ? c : rem));
  len = 16 * (base + (c < rem ? 1 : 0));
}

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void fence_async_all() { asm volatile("fence.proxy.async;" ::: "memory"); }

// Descriptor words of a K-major no-swizzle tile (LBO 128).  Low: the shared
// address (whose bits above 18 name the block within its cluster, and are not
// the descriptor's) in units of 16 bytes, so that an offset is an addition.
__device__ __forceinline__ uint32_t desc_lo(uint32_t saddr) { return (8u << 16) | ((saddr & 0x3FFFFu) >> 4); }
__host__ __device__ constexpr uint32_t desc_hi(uint32_t sbo) { return (sbo >> 4) | (1u << 14); }

__device__ __forceinline__ float scale_of(unsigned long long key) {
  const float zinf = __uint_as_float((uint32_t)(key >> 32));
  if (!(zinf > 0.f)) return 1.f;
  int e;
  frexpf(zinf, &e);
  e = max(-100, min(100, 8 - e));
  return ldexpf(1.f, e);
}

// The epilogue's arithmetic.  One step of a coordinate was about 120
// instructions, and the epilogue is issue-bound; these forms give the same
// values with about 40:
//  * rint by adding and subtracting 1.5 2^23 (round to nearest even, exact for
//    |z| < 2^22; the sum's low byte is the integer's), not the quarter-rate
//    rounding instruction;
//  * a sign as |x| 2^75 2^75 saturated to [0, 1] with the sign of x copied on
//    (two exact scalings, so that a subnormal x also reaches 1; NaN gives 0);
//  * ceil z + floor z - 2 z as sign(e) - 2 e with e = z - rint(z);
//  * the index of the first maximiser of |z| kept only below 1, where the
//    inverse-norm term needs it.
// The plain forms replace them for |z| beyond 2^22, and for an Adam epsilon so
// small that a subnormal second moment shows.  (One copy of the loop: the kernel
// runs phases of long straight code, and its size costs instruction fetches.)
constexpr float kRintMagic = 12582912.f;  // 1.5 2^23
constexpr float kRintMost = 4194304.f;    // 2^22
__device__ __forceinline__ float sgn_sat(float x) {
  const float t = fabsf(x) * 0x1p75f;
  float a;
  asm("mul.sat.f32 %0, %1, %2;" : "=f"(a) : "f"(t), "f"(0x1p75f));
  return copysignf(a, x);
}
__device__ __forceinline__ float rsqrt_ftz(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rcp_ftz(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// A tile's z operands: per 32 coordinates z_bytes of hi and lo (or e4m3) and
// 8 KB of round(z).  A call that collects after every step has them side by
// side, one copy moves both; else round(z) has its own part behind all of z.
__device__ __forceinline__ uint32_t z_bytes(const ClParams& p) {
  return p.f8 ? (uint32_t)kChunk8 : (uint32_t)p.nterms * kChunk16;
}
__device__ __forceinline__ uint32_t z_stride(const ClParams& p) {
  return z_bytes(p) + (p.period == 1 ? (uint32_t)kChunk16 : 0u);
}
__device__ __forceinline__ uint8_t* z_tile(const ClParams& p, int tile) {
  const size_t bytes = (size_t)(p.d32 / kKC) * (z_bytes(p) + kChunk16);
  if (tile < p.z1) return p.Zh[0] + tile * bytes;
  if (tile < p.z2) return p.Zh[1] + (tile - p.z1) * bytes;
  return p.Zh[2] + (tile - p.z2) * bytes;
}

// the BF16 operand words of 8 coordinates: hi, and lo = bf16(z - hi)
__device__ __forceinline__ void split8(const float (&z)[8], uint32_t (&wh)[4], uint32_t (&wl)[4]) {
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    wh[k] = pack_bf16x2(z[2 * k], z[2 * k + 1]);
    const float2 hf = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&wh[k]));
    wl[k] = pack_bf16x2(z[2 * k] - hf.x, z[2 * k + 1] - hf.y);
  }
}

// A candidate row of start pg from its staged row, in canonical sign, by the
// calling warp: 4 bytes per lane where the pieces are aligned
__device__ __forceinline__ void write_row(const ClParams& p, const int8_t* src, const int8_t* map, int8_t* dst, bool neg) {
  const int lane = threadIdx.x & 31;
  const int d = p.d, n = p.n;
  const bool words = (reinterpret_cast<uintptr_t>(dst) & 3) == 0;
#pragma unroll 1
  for (int b = 4 * lane; b < p.ldc; b += 128) {
    uint32_t v = 0;
    if (b + 4 <= d) {
      v = __ldcg(reinterpret_cast<const unsigned int*>(src + b));
    } else if (b >= d && (d & 3) == 0 && b + 4 <= n) {
      v = __ldcg(reinterpret_cast<const unsigned int*>(map + (b - d)));
    } else {
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int i = b + k;
        if (i < n) {
          const int8_t x = (int8_t)__ldcg(reinterpret_cast<const signed char*>(i < d ? src + i : map + (i - d)));
          v |= (uint32_t)(uint8_t)x << (8 * k);
        }
      }
    }
    if (neg) v = __vneg4(v);
    if (words) {
      *reinterpret_cast<uint32_t*>(dst + b) = v;
    } else {
#pragma unroll
      for (int k = 0; k < 4; ++k) dst[b + k] = (int8_t)(v >> (8 * k));
    }
  }
}

__device__ __forceinline__ void cluster_body(const ClParams& p, const int tile, const int rank) {
  extern __shared__ __align__(1024) uint8_t smem[];
  // full, empty, accumulator ready, accumulator free; state ring full, empty
  __shared__ __align__(8) uint64_t bars[2 * kMaxStages + 2 + 2 * kEStages];
  __shared__ uint32_t s_tmem;
  __shared__ int s_abort;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int uwarp = __shfl_sync(0xffffffffu, warp, 0);  // warp-uniform for the compiler, too
  const uint32_t lead = elect_lead();
  const int C = p.C;
  int row0, RS, col0, CS;  // this block's rows of Bm and coordinates
  slice_of(p.R32, C, rank, row0, RS);
  slice_of(p.d32, C, rank, col0, CS);
  const int nkF = p.d32 / kKC, nkG = p.R32 / kKC;
  const int64_t P2 = (int64_t)p.tiles * kTM;
  float* s_span = reinterpret_cast<float*>(smem);  // of the slice (at most 4096 floats)
  // the forward pass's operands take the whole ring; the gradient pass leaves
  // its end to the epilogue's state
  const uint32_t ring0 = (uint32_t)(CS * 4 + 1023) / 1024 * 1024;
  const uint32_t ring_fwd = (uint32_t)p.dyn - ring0, ring_grad = ring_fwd - kEStages * kEBytes;
  const uint32_t ering0 = ring0 + ring_grad;

  if (tid == 0) {
    for (int b = 0; b < 2 * kMaxStages + 1; ++b) mbar_init(smem_u32(&bars[b]), 1);
    mbar_init(smem_u32(&bars[2 * kMaxStages + 1]), kThreads / 32);
    for (int b = 0; b < kEStages; ++b) {
      mbar_init(smem_u32(&bars[2 * kMaxStages + 2 + b]), 1);
      mbar_init(smem_u32(&bars[2 * kMaxStages + 2 + kEStages + b]), 4);  // the four warps that read a chunk
    }
    s_abort = (*(volatile int32_t*)p.flags & 16) ? 1 : 0;
  }
  if (warp == 0) tmem_alloc(smem_u32(&s_tmem), kTmemCols);
#pragma unroll 1
  for (int k = tid; k < CS; k += kThreads) s_span[k] = col0 + k < p.d ? (float)p.span[col0 + k] : 0.f;
  mbar_init_fence();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = s_tmem;
  const uint32_t full0 = smem_u32(&bars[0]), empty0 = smem_u32(&bars[kMaxStages]),
                 accr = smem_u32(&bars[2 * kMaxStages]), accf = smem_u32(&bars[2 * kMaxStages + 1]);
  const uint32_t ring = smem_u32(smem) + ring0, ering = smem_u32(smem) + ering0;
  const uint32_t efull0 = smem_u32(&bars[2 * kMaxStages + 2]), eempty0 = efull0 + 8 * kEStages;

  // epilogue geometry: two warps per TMEM lane quarter, alternate chunks of columns
  const int q = warp & 3, h = warp >> 2;
  const int r = q * 32 + lane;
  const int64_t pg = (int64_t)tile * kTM + r;
  const bool row_live = pg < p.P;
  const uint32_t lane_base = (uint32_t)(q * 32) << 16;
  float4* const zt = reinterpret_cast<float4*>(p.Zt) + (size_t)tile * (p.d32 / 4) * kTM + r;
  float4* const mt = reinterpret_cast<float4*>(p.Mt) + (size_t)tile * (p.d32 / 4) * kTM + r;
  float4* const vt = reinterpret_cast<float4*>(p.Vt) + (size_t)tile * (p.d32 / 4) * kTM + r;
  const uint32_t zstride = z_stride(p), zbytes = z_bytes(p);
  uint8_t* const zh = z_tile(p, tile);
  uint8_t* const zr = zh + (p.period == 1 ? zbytes : nkF * zbytes);
  const uint32_t rstride = p.period == 1 ? zstride : (uint32_t)kChunk16;
  uint8_t* const Sg = p.S + (size_t)tile * nkG * kChunk16;

  uint32_t ph = ~0u;       // warps 0 and 1: bit s = phase parity of the current use of stage s
  uint32_t accph = 0;      // phase of the accumulator-ready barrier
  uint32_t ec = 0;         // chunks of state read before this step (stage ec % 4, phase (ec / 4) & 1)
  uint32_t freeph = 0;     // warp 0: phase of the accumulator-free barrier
  uint32_t accbits = kChanged;  // the first collection of a call always counts
  float sc = 1.f;               // FP8: the start's e4m3 scale
  float zmost = 0.f;            // largest |z| of this thread's coordinates after its last step
  if (p.f8) sc = scale_of(__ldcg(&p.zkey[pg]));

  // One chain of MMAs over nk chunks of `bytes` bytes, copied in groups of
  // neighbouring chunks; every earlier MMA of the block has completed when it
  // starts.  Warp 1: load(n, stage, full) starts the copies of the next n chunks.
  // Warp 0: mma(n, stage descriptor) issues their instructions; the chain ends
  // with the accumulator handed to all warps.  False on time-out.  Each loop is
  // the dependent instruction stream of one warp (about 4 cycles apiece), so
  // addresses advance by additions and the groups are as large as leaves three
  // stages in the ring.
  auto geometry = [&](uint32_t bytes, uint32_t ring_bytes, int& grp, int& nst) {
    grp = max(1, min((int)(kStageMost / bytes), (int)(ring_bytes / (3 * bytes))));
    nst = min((int)(ring_bytes / (grp * bytes)), kMaxStages);
  };
  auto load_chain = [&](int nk, uint32_t bytes, int grp, int nst, auto load) -> bool {
    int st = 0;
    uint32_t dst = ring, bar = 0;
    bool wrapped = false;
#pragma unroll 1
    for (int left = nk; left > 0; left -= grp) {
      if (wrapped) {
        const bool ok = mbar_wait_bounded(empty0 + bar, (ph >> st) & 1u);
        if (!__all_sync(0xffffffffu, ok)) return false;
      }
      ph ^= 1u << st;
      load(min(grp, left), dst, full0 + bar);
      dst += grp * bytes;
      bar += 8;
      if (++st == nst) {
        st = 0;
        bar = 0;
        dst = ring;
        wrapped = true;
      }
    }
    return true;
  };
  auto mma_chain = [&](int nk, uint32_t bytes, int grp, int nst, bool reuse, auto mma) -> bool {
    if (reuse) {  // the accumulator of the block before has been read
      const bool ok = mbar_wait_bounded(accf, freeph);
      if (!__all_sync(0xffffffffu, ok)) return false;
      freeph ^= 1;
      tc_fence_after();
    }
    int st = 0;
    const uint32_t first = desc_lo(ring), units = (grp * bytes) >> 4;
    uint32_t sd = first, bar = 0;
#pragma unroll 1
    for (int left = nk; left > 0; left -= grp) {
      ph ^= 1u << st;
      const bool ok = mbar_wait_bounded(full0 + bar, (ph >> st) & 1u);
      if (!__all_sync(0xffffffffu, ok)) return false;
      tc_fence_after();
      mma(min(grp, left), sd);
      mma_commit_if(lead, empty0 + bar);
      sd += units;
      bar += 8;
      if (++st == nst) {
        st = 0;
        bar = 0;
        sd = first;
      }
    }
    mma_commit_if(lead, accr);
    return true;
  };
  // A time-out: the phase ends for every warp at its next vote (wait_acc) or
  // wait, and the block's remaining steps only take part in the barriers.  A warp
  // leaves its chunks after the one whose wait ran out (what it computed of
  // that one is void, as the flagged call is; refusing it before the stores
  // cost 2 to 3% of every step).
  auto give_up = [&]() {
    *(volatile int*)&s_abort = 1;
    atomicOr(p.flags, 16);
  };
  // Every thread: the accumulator is ready.  Only warp 0 polls; the others
  // sleep at a block barrier (polled by all, they took the issue slots and the
  // shared-memory queue from the two warps that feed the MMAs).  going: false
  // for a warp whose own wait ran out; the answer is the same for every thread.
  auto wait_acc = [&](bool going) -> bool {
    bool ok = going;
    if (uwarp == 0 && ok) ok = mbar_wait_bounded(accr, accph);
    accph ^= 1;
    const bool bad = __syncthreads_or(!ok) != 0;
    tc_fence_after();
    return !bad;
  };
  // a wait of the epilogue: another warp's time-out ends it, too
  auto wait_or_abort = [&](uint32_t bar, uint32_t parity) -> bool {
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    do {
      if (mbar_try_wait(bar, parity)) return true;
    } while (*(volatile int*)&s_abort == 0 && clock64() - t0 < kWaitCycles);
    return false;
  };
  // The state of chunk ch (8 coordinates: 3 x 4 KB, contiguous in the blocked
  // arrays) into its stage, by one lane of the calling warp
  auto load_state = [&](int ch) {
    const uint32_t e = ec + (uint32_t)ch, st = e % kEStages;
    const size_t o = ((size_t)tile * p.d32 + col0 + ch * 8) * kTM;
    const uint32_t dst = ering + st * kEBytes, bar = efull0 + 8 * st;
    mbar_expect_tx_if(lead, bar, kEBytes);
    bulk_g2s_if(lead, dst, p.Zt + o, kEArr, bar);
    bulk_g2s_if(lead, dst + kEArr, p.Mt + o, kEArr, bar);
    bulk_g2s_if(lead, dst + 2 * kEArr, p.Vt + o, kEArr, bar);
  };

  int until = p.period - p.t0 % p.period;  // steps to the next collection
  bool due = false;                         // the candidate of the step before is due
#pragma unroll 1
  for (int s = 0; s <= p.T; ++s) {
    const bool do_fwd = s < p.T;
    const bool coll = due;
    const bool next_coll = do_fwd && --until == 0;  // this step's will be due
    if (next_coll) until = p.period;
    due = next_coll;
    if (!do_fwd && !coll) break;
    bool dead = __syncthreads_or(*(volatile int*)&s_abort) != 0;  // the same for every thread

    // FP8: a start whose ||z||_inf passed a power of two since its operand was
    // written has another scale now: its slice of the operand is written again
    if (p.f8 && s >= 1 && do_fwd) {
      bool redo = false;
      const float ns = scale_of(__ldcg(&p.zkey[(s & 1) * P2 + pg]));
      redo = ns != sc;
      sc = ns;
      if (__syncthreads_or(redo)) {  // the same in every block of the cluster
        if (redo && !dead) {
#pragma unroll 1
          for (int ch = h; ch < CS / 8; ch += 2) {
            const int j0 = col0 + ch * 8;
            const float4 a = zt[(size_t)(j0 / 4) * kTM], b = zt[(size_t)(j0 / 4 + 1) * kTM];
            const float v8[8] = {a.x * sc, a.y * sc, a.z * sc, a.w * sc, b.x * sc, b.y * sc, b.z * sc, b.w * sc};
            *reinterpret_cast<uint2*>(zh + (size_t)(j0 >> 5) * zstride + off8(r, j0 & 31)) = pack_e4m3x8(v8);
          }
        }
        fence_async_all();
        cluster_sync();
      }
    }

    // ---- forward ----
    auto prefetch_state = [&]() {  // warps 0 and 4, which issue these copies
      fence_async_all();
      if (uwarp == 4)
#pragma unroll 1
        for (int ch = 0; ch < kEStages && ch < CS / 8; ++ch) load_state(ch);
      __syncwarp();
    };
    if (do_fwd && RS == 0 && !dead && (uwarp == 0 || uwarp == 4)) prefetch_state();
    if (rank == 0 && h == 0 && do_fwd) p.zkey[((s + 1) & 1) * P2 + pg] = 0ull;  // the next step's maximum
    float l1 = 0.f;
    bool out = false;
    bool acc_ok = true;  // the same for every thread
#pragma unroll 1
    for (int rb = 0; rb < RS && acc_ok; rb += kRowBlk) {
      const int N = RS - rb < kRowBlk ? RS - rb : kRowBlk;
      bool ok = true;
      if (uwarp < 2 && !dead) {
        const bool f16 = do_fwd && !p.f8, f8 = do_fwd && p.f8;
        // a stage holds its chunks' z (hi, lo, round(z)), then Bm, then Bm in e4m3
        const uint32_t zb = do_fwd ? zbytes : 0u, rb16 = coll ? (uint32_t)kChunk16 : 0u;
        const bool both = zb && rb16 && p.period == 1;  // z and round(z) of a chunk side by side
        const uint32_t zS = both ? zstride : zb, rS = both ? zstride : rb16;
        const uint32_t b16 = (f16 || coll) ? (uint32_t)N * kKC * 2 : 0u, b8 = f8 ? (uint32_t)N * kKC : 0u;
        const uint32_t bytes = zb + rb16 + b16 + b8;
        int grp, nst;
        geometry(bytes, ring_fwd, grp, nst);
        if (uwarp == 1) {
          fence_async_all();
          const uint8_t* bf = p.Bf + ((size_t)(row0 + rb) * p.d32) * 2;
          const uint8_t* bf8 = p.Bf8 + (size_t)(row0 + rb) * p.d32;
          const uint8_t *zs = zh, *rs = zr;
          const uint32_t offR = grp * zb, offB = grp * (zb + rb16), offB8 = offB + grp * b16;
          const bool zone = zb && zstride == zb, rone = rb16 && rstride == rb16;
          ok = load_chain(nkF, bytes, grp, nst, [&](int cnt, uint32_t st, uint32_t bar) {
            mbar_expect_tx_if(lead, bar, bytes * cnt);
            if (both) {
              bulk_g2s_if(lead, st, zs, zstride * cnt, bar);
            } else {
              if (zone) bulk_g2s_if(lead, st, zs, zb * cnt, bar);
              if (rone) bulk_g2s_if(lead, st + offR, rs, rb16 * cnt, bar);
              if ((zb && !zone) || (rb16 && !rone)) {
#pragma unroll 1
                for (int u = 0; u < cnt; ++u) {  // one of the two alone where they lie side by side
                  if (zb && !zone) bulk_g2s_if(lead, st + u * zb, zs + (size_t)u * zstride, zb, bar);
                  if (rb16 && !rone) bulk_g2s_if(lead, st + offR + u * rb16, rs + (size_t)u * rstride, rb16, bar);
                }
              }
            }
            if (b16) bulk_g2s_if(lead, st + offB, bf, b16 * cnt, bar);
            if (b8) bulk_g2s_if(lead, st + offB8, bf8, b8 * cnt, bar);
            zs += grp * zstride;
            rs += grp * rstride;
            bf += grp * b16;
            bf8 += grp * b8;
          });
        } else {
          const uint32_t id16 = idesc_bf16(kTM, N), id8 = idesc_e4m3(kTM, N);
          const bool two = p.nterms > 1;
          const uint32_t offR = (both ? zb : grp * zb) >> 4, offB = (grp * (zb + rb16)) >> 4,
                         offB8 = offB + ((grp * b16) >> 4);
          const uint32_t zD = zS >> 4, rD = rS >> 4, bD = b16 >> 4, b8D = b8 >> 4;
          uint32_t a0 = 0;  // the first instruction overwrites the accumulator
          ok = mma_chain(nkF, bytes, grp, nst, rb > 0, [&](int cnt, uint32_t sd) {
            uint32_t zd = sd, rd = sd + offR, bd = sd + offB, b8d = sd + offB8;
            if (f8) {
#pragma unroll 1
              for (int u = 0; u < cnt; ++u) {
                mma_e4m3_if(lead, tmem, zd, b8d, desc_hi(kSbo8), id8, a0 | (uint32_t)u);
                zd += zD;
                b8d += b8D;
              }
            }
            if (b16) {
#pragma unroll 1
              for (int u = 0; u < cnt; ++u) {
                const uint32_t a1 = a0 | (uint32_t)u;
#pragma unroll
                for (int kk = 0; kk < 2; ++kk) {
                  if (f16) mma_bf16_if(lead, tmem, zd + 16 * kk, bd + 16 * kk, desc_hi(kSbo16), id16, a1 | kk);
                  if (f16 && two) mma_bf16_if(lead, tmem, zd + (kChunk16 >> 4) + 16 * kk, bd + 16 * kk, desc_hi(kSbo16), id16, 1u);
                  if (coll) mma_bf16_if(lead, tmem + kColD2, rd + 16 * kk, bd + 16 * kk, desc_hi(kSbo16), id16, a1 | kk);
                }
                zd += zD;
                rd += rD;
                bd += bD;
              }
            }
            a0 = 1;
          });
        }
        if (!ok) give_up();
      }
      __syncwarp();
      if (!dead) {
        acc_ok = wait_acc(ok);
        // the ring is free: the first chunks of the state are on their way
        // before the gradient is
        if (do_fwd && (uwarp == 0 || uwarp == 4) && acc_ok && rb + kRowBlk >= RS) prefetch_state();
        if (acc_ok) {
          const float inv_sc = p.f8 ? 1.f / sc : 1.f;
#pragma unroll 1
          for (int ch = h; ch < N / 16; ch += 2) {
            const int i0 = row0 + rb + ch * 16;
            uint32_t v[16];
            if (do_fwd) {
              __syncwarp();
              tmem_ld16(tmem + lane_base + ch * 16, v);
              tc_wait_ld();
              uint32_t w[8];
#pragma unroll
              for (int k = 0; k < 8; ++k) {
                const float y0 = __uint_as_float(v[2 * k]), y1 = __uint_as_float(v[2 * k + 1]);
                w[k] = pack_bf16x2((float)mape_sign_f(y0), (float)mape_sign_f(y1));
                l1 += (fabsf(y0) + fabsf(y1)) * inv_sc;
              }
              uint8_t* Sp = Sg + (size_t)(i0 >> 5) * kChunk16;
              *reinterpret_cast<uint4*>(Sp + off16(r, i0 & 31)) = make_uint4(w[0], w[1], w[2], w[3]);
              *reinterpret_cast<uint4*>(Sp + off16(r, (i0 & 31) + 8)) = make_uint4(w[4], w[5], w[6], w[7]);
            }
            if (coll) {
              __syncwarp();
              tmem_ld16(tmem + lane_base + kColD2 + ch * 16, v);
              tc_wait_ld();
              uint32_t pk[4] = {0, 0, 0, 0};
#pragma unroll
              for (int k = 0; k < 16; ++k) {
                const int i = i0 + k;
                const int gv = __float2int_rn(__uint_as_float(v[k]));
                if (i < p.R) {
                  const int sp = p.span[p.d + i];
                  if (gv > sp || -gv > sp) out = true;
                }
                pk[k >> 2] |= ((uint32_t)(gv & 0xff)) << (8 * (k & 3));
              }
              if (row_live)
                *reinterpret_cast<uint4*>(p.stage_map + pg * p.R32 + i0) =
                    make_uint4(pk[0], pk[1], pk[2], pk[3]);
            }
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0 && rb + kRowBlk < RS) mbar_arrive(accf);
        } else if (tid == 0) {
          give_up();
        }
      }
    }
    if (row_live) {
      if (out) p.oob[pg] = 1u;  // every writer writes the same word
      if (do_fwd && s == 0 && p.dbg_phi) atomicAdd(&p.dbg_phi[pg], l1);
    }
    tc_fence_before();
    fence_async_all();
    cluster_sync();
    tc_fence_after();
    dead = __syncthreads_or(*(volatile int*)&s_abort) != 0;

    // ---- gradient ----
    auto issue_grad = [&](int cb) -> bool {  // warps 0 and 1
      const int N = CS - cb < kColBlk ? CS - cb : kColBlk;
      const uint32_t nb = (uint32_t)N * kKC * 2;
      int grp, nst;
      geometry(kChunk16 + nb, ring_grad, grp, nst);
      bool ok;
      if (uwarp == 1) {
        const uint8_t *bg = p.Bg + ((size_t)(col0 + cb) * p.R32) * 2, *sg = Sg;
        ok = load_chain(nkG, kChunk16 + nb, grp, nst, [&](int cnt, uint32_t st, uint32_t bar) {
          mbar_expect_tx_if(lead, bar, (kChunk16 + nb) * cnt);
          bulk_g2s_if(lead, st, sg, kChunk16 * cnt, bar);
          bulk_g2s_if(lead, st + grp * kChunk16, bg, nb * cnt, bar);
          sg += grp * kChunk16;
          bg += grp * nb;
        });
      } else {
        const uint32_t idg = idesc_bf16(kTM, N), offB = (grp * kChunk16) >> 4, bD = nb >> 4;
        uint32_t a0 = 0;
        ok = mma_chain(nkG, kChunk16 + nb, grp, nst, cb > 0, [&](int cnt, uint32_t sd) {
          uint32_t ad = sd, bd = sd + offB;
#pragma unroll 1
          for (int u = 0; u < cnt; ++u) {
#pragma unroll
            for (int kk = 0; kk < 2; ++kk)
              mma_bf16_if(lead, tmem, ad + 16 * kk, bd + 16 * kk, desc_hi(kSbo16), idg, a0 | (uint32_t)(u | kk));
            ad += kChunk16 >> 4;
            bd += bD;
          }
          a0 = 1;
        });
      }
      if (!ok) give_up();
      __syncwarp();
      return ok;
    };
    bool ok = true;  // no wait of this warp has run out
    if (do_fwd && uwarp < 2 && !dead && CS > 0) {
      if (uwarp == 1) fence_async_all();
      ok = issue_grad(0);
    }
    __syncwarp();
    // the candidates of step s - 1, the starts spread over the cluster's blocks
    if (coll && !dead && uwarp >= 2) {  // warps 0 and 1 issue meanwhile
      const int per = kTM / C;         // starts of this block
      const int mine = (per + 5) / 6;  // of a warp, one per lane
      const int i = (warp - 2) * mine + lane;
      const int64_t pc = (int64_t)tile * kTM + rank * per + i;
      const int64_t at2 = (s & 1) * P2 + pc;
      long long slot = -1;
      int neg = 0;
      if (lane < mine && i < per && pc < p.P) {
        const uint32_t a = __ldcg(&p.acc[at2]), o = __ldcg(&p.oob[pc]), idout = __ldcg(&p.idw[at2]);
        const int fz = __ldcg(&p.first[at2]);
        if ((a & kChanged) && !o && !idout && fz != kNoNz) {
          if (a & kUnexact) {
            atomicOr(p.flags, 2);
          } else {
            const unsigned long long at = atomicAdd(p.count, 1ull);
            if ((int64_t)at < p.cap) slot = (long long)at;
            else atomicOr(p.flags, 1);
          }
        }
        neg = (fz != kNoNz && (fz & 1)) ? 1 : 0;
        p.acc[at2] = 0u;
        p.idw[at2] = 0u;
        p.first[at2] = kNoNz;
        p.oob[pc] = 0u;
      }
      unsigned todo = __ballot_sync(0xffffffffu, slot >= 0);
      while (todo) {
        const int l = __ffs(todo) - 1;
        todo &= todo - 1;
        const long long sl = __shfl_sync(0xffffffffu, slot, l);
        const int ng = __shfl_sync(0xffffffffu, neg, l);
        const int64_t ps = (int64_t)tile * kTM + rank * per + (warp - 2) * mine + l;
        write_row(p, p.stage + ((s & 1) * P2 + ps) * p.ldi, p.stage_map + ps * p.R32, p.cand + sl * p.ldc, ng != 0);
      }
    }
    if (!do_fwd) break;

    if (!dead) {
      const unsigned long long zk = __ldcg(&p.zkey[(s & 1) * P2 + pg]);
      const float zinf = __uint_as_float((uint32_t)(zk >> 32));
      const int kmax = zk ? (int)(0xffffffffu - (uint32_t)zk) : -1;
      float inv_term = 0.f;
      if (zinf < 1.f && zinf > 0.f) inv_term = -p.lambda2 / (zinf * zinf);  // times sign(z_kmax)
      const float2 ad = p.bias[s];
      const float step = ad.x, rsb2 = ad.y;
      const bool dbg = s == 0 && (p.dbg_phi || p.dbg_grad);
      const bool inv_on = inv_term != 0.f;
      // z of this thread's coordinates as the last step left it (at the first
      // step, of all the start's, where a NaN in coordinate 0 hides the others)
      const bool slow = __any_sync(0xffffffffu, p.eps < 1e-15f || !((s == 0 ? zinf : zmost) < kRintMost / 2));
      float nzinf = 0.f, frac = 0.f, l1_id = 0.f;
      float dsum = 0.f;  // sum of |rint(z_new) - rint(z_old)|: 0 iff no rounding changed
      int nkmax = -1, first_id = kNoNz;  // the first maximiser of |z|; the first nonzero rounding
      bool out_id = false, nan_head = false;
      int8_t* srow = p.stage + (((s + 1) & 1) * P2 + pg) * p.ldi;
#pragma unroll 1
      for (int cb = 0; cb < CS; cb += kColBlk) {
        const int nch = (CS - cb < kColBlk ? CS - cb : kColBlk) / 8;
        if (cb > 0 && uwarp < 2 && ok) ok = issue_grad(cb);
        __syncwarp();
        if (!wait_acc(ok)) {  // every warp leaves here
          ok = false;
          if (tid == 0) give_up();
          break;
        }
        auto chunk = [&](int ch) {
          const int j0 = col0 + cb + ch * 8;
          uint32_t gv[8];
          __syncwarp();
          tmem_ld8(tmem + lane_base + ch * 8, gv);
          const uint32_t e = ec + (uint32_t)(cb / 8 + ch), st = e % kEStages;
          if (!wait_or_abort(efull0 + 8 * st, (e / kEStages) & 1u)) ok = false;
          const float4* es = reinterpret_cast<const float4*>(smem + ering0 + st * kEBytes) + r;
          const float4 cz[2] = {es[0], es[kTM]}, cm[2] = {es[2 * kTM], es[3 * kTM]}, cv[2] = {es[4 * kTM], es[5 * kTM]};
          float zc[8] = {cz[0].x, cz[0].y, cz[0].z, cz[0].w, cz[1].x, cz[1].y, cz[1].z, cz[1].w};
          float mc[8] = {cm[0].x, cm[0].y, cm[0].z, cm[0].w, cm[1].x, cm[1].y, cm[1].z, cm[1].w};
          float vc[8] = {cv[0].x, cv[0].y, cv[0].z, cv[0].w, cv[1].x, cv[1].y, cv[1].z, cv[1].w};
          __syncwarp();
          if (lane == 0) mbar_arrive(eempty0 + 8 * st);
          float g[8], rz[8], rn[8], tn[8];
#pragma unroll
          for (int k = 0; k < 8; ++k) rz[k] = __fadd_rn(__fadd_rn(zc[k], kRintMagic), -kRintMagic);
          if (slow) {
#pragma unroll
            for (int k = 0; k < 8; ++k) rz[k] = rintf(zc[k]);
          }
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            const float e = zc[k] - rz[k];
            g[k] = fmaf(-2.f, e, sgn_sat(e));
          }
          __syncwarp();
          tc_wait_ld();
#pragma unroll
          for (int k = 0; k < 8; ++k) g[k] = fmaf(p.lambda1, g[k], __uint_as_float(gv[k]));
          if (inv_on && (unsigned)(kmax - j0) < 8u) {
#pragma unroll
            for (int k = 0; k < 8; ++k)
              if (j0 + k == kmax) g[k] = fmaf(inv_term, (float)mape_sign_f(zc[k]), g[k]);
          }
#pragma unroll
          for (int k = 0; k < 8; ++k) g[k] += sgn_sat(zc[k]);  // identity row j of B: sign((Bz)_j) = sign(z_j)
          if (dbg && row_live) {
#pragma unroll
            for (int k = 0; k < 8; ++k) {
              if (j0 + k >= p.d) continue;
              const float z = zc[k], fl = floorf(z);
              frac += (z - fl) * (ceilf(z) - z);
              l1_id += fabsf(z);
              if (p.dbg_grad) p.dbg_grad[pg * p.d + j0 + k] = g[k];
            }
          }
          float upd[8];
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            const float grad = g[k];
            mc[k] = p.beta1 * mc[k] + p.omb1 * grad;
            vc[k] = p.beta2 * vc[k] + p.omb2 * grad * grad;
            const float den = vc[k] * rsqrt_ftz(fmaxf(vc[k], 0x1p-126f)) * rsb2 + p.eps;
            upd[k] = mc[k] * rcp_ftz(den);
          }
          if (slow) {
#pragma unroll
            for (int k = 0; k < 8; ++k) {
              const float den = (vc[k] > 0.f ? vc[k] * rsqrtf(vc[k]) : 0.f) * rsb2 + p.eps;
              upd[k] = __fdividef(mc[k], den);
            }
          }
          float cmax = 0.f;
#pragma unroll
          for (int k = 0; k < 8; ++k) {  // padding coordinates stay at 0 and change none of the trackers
            zc[k] = zc[k] - step * upd[k];
            tn[k] = __fadd_rn(zc[k], kRintMagic);
            rn[k] = __fadd_rn(tn[k], -kRintMagic);
            cmax = fmaxf(cmax, fabsf(zc[k]));
          }
          if (slow || cmax >= kRintMost) {  // also a step that leaves the exact range
#pragma unroll
            for (int k = 0; k < 8; ++k) rn[k] = rintf(zc[k]);
          }
#pragma unroll
          for (int k = 0; k < 8; ++k) dsum += fabsf(rn[k] - rz[k]);
          // as in the step-by-step kernels, a NaN counts as the maximum where it
          // heads one of their threads' coordinates (and is passed over elsewhere)
          if ((j0 & 0xF7) == 0) nan_head |= zc[0] != zc[0];
          if (cmax > nzinf) {
            nzinf = cmax;
            if (cmax < 1.f) {
#pragma unroll
              for (int k = 7; k >= 0; --k)
                if (fabsf(zc[k]) == cmax) nkmax = j0 + k;
            } else {
              nkmax = 0;  // not needed
            }
          }
          const size_t o = (size_t)(j0 / 4) * kTM;
          zt[o] = make_float4(zc[0], zc[1], zc[2], zc[3]);
          zt[o + kTM] = make_float4(zc[4], zc[5], zc[6], zc[7]);
          mt[o] = make_float4(mc[0], mc[1], mc[2], mc[3]);
          mt[o + kTM] = make_float4(mc[4], mc[5], mc[6], mc[7]);
          vt[o] = make_float4(vc[0], vc[1], vc[2], vc[3]);
          vt[o + kTM] = make_float4(vc[4], vc[5], vc[6], vc[7]);
          // the next step's operands
          const uint32_t oc = off16(r, j0 & 31);
          uint8_t* const zo = zh + (uint32_t)(j0 >> 5) * zstride;
          if (p.f8) {
            float v8[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) v8[k] = zc[k] * sc;
            *reinterpret_cast<uint2*>(zo + off8(r, j0 & 31)) = pack_e4m3x8(v8);
          } else {
            uint32_t wh[4], wl[4];
            split8(zc, wh, wl);
            *reinterpret_cast<uint4*>(zo + oc) = make_uint4(wh[0], wh[1], wh[2], wh[3]);
            if (p.nterms > 1) *reinterpret_cast<uint4*>(zo + kChunk16 + oc) = make_uint4(wl[0], wl[1], wl[2], wl[3]);
          }
          if (next_coll) {  // round(z): its operand, the identity rows of the candidate and their tests
            uint32_t wr[4], bb[2];
#pragma unroll
            for (int k = 0; k < 4; ++k) wr[k] = pack_bf16x2(rn[2 * k], rn[2 * k + 1]);
            *reinterpret_cast<uint4*>(zr + (uint32_t)(j0 >> 5) * rstride + oc) = make_uint4(wr[0], wr[1], wr[2], wr[3]);
#pragma unroll
            for (int k = 0; k < 2; ++k) {  // low bytes of the roundings (a rounding beyond 8 bits is out of the box)
              const uint32_t lo = __byte_perm(__float_as_uint(tn[4 * k]), __float_as_uint(tn[4 * k + 1]), 0x0040);
              const uint32_t hi = __byte_perm(__float_as_uint(tn[4 * k + 2]), __float_as_uint(tn[4 * k + 3]), 0x0040);
              bb[k] = __byte_perm(lo, hi, 0x5410);
            }
            float asum = 0.f;  // sum of |rounding|: 0 iff all are 0
#pragma unroll
            for (int k = 0; k < 8; ++k) asum += fabsf(rn[k]);
            if (!(asum < kRintMost)) {  // beyond the exact range of the bytes, or a NaN (a 0 in the row)
              bb[0] = bb[1] = 0;
#pragma unroll
              for (int k = 0; k < 8; ++k) bb[k >> 2] |= ((uint32_t)((int)rn[k] & 0xff)) << (8 * (k & 3));
            }
            const float4 s0 = *reinterpret_cast<const float4*>(s_span + cb + ch * 8),
                         s1 = *reinterpret_cast<const float4*>(s_span + cb + ch * 8 + 4);
            const float sp[8] = {s0.x, s0.y, s0.z, s0.w, s1.x, s1.y, s1.z, s1.w};
#pragma unroll
            for (int k = 0; k < 8; ++k) out_id |= fabsf(rn[k]) > sp[k];
            if (first_id == kNoNz && asum != 0.f) {
#pragma unroll
              for (int k = 7; k >= 0; --k)
                if (rn[k] != 0.f) first_id = ((j0 + k) << 1) | (rn[k] < 0.f ? 1 : 0);
            }
            if (row_live && j0 < p.ldi) *reinterpret_cast<uint2*>(srow + j0) = make_uint2(bb[0], bb[1]);
          }
          // the stage's next chunk, once the three other warps have read it
          if (q == 0 && cb / 8 + ch + kEStages < CS / 8) {
            ok = mape_detail::refill_stage(
                ok, [&] { return wait_or_abort(eempty0 + 8 * st, (e / kEStages) & 1u); },
                [](bool b) { return __all_sync(0xffffffffu, b) != 0; }, [&] { load_state(cb / 8 + ch + kEStages); });
            __syncwarp();
          }
        };
#pragma unroll 1
        for (int ch = h; ch < nch; ch += 2) {
          chunk(ch);
          if (!__all_sync(0xffffffffu, ok)) break;
        }
        ok = __all_sync(0xffffffffu, ok);
        if (!ok && lane == 0) give_up();
        tc_fence_before();
        __syncwarp();
        if (lane == 0 && cb + kColBlk < CS) mbar_arrive(accf);
      }
      ec += (uint32_t)(CS / 8);
      zmost = nzinf;
      if (row_live && ok) {
        // |rint z_j| > 256 for some j iff max |z_j| > 256.5 (256.5 rounds to 256)
        accbits |= (dsum != 0.f ? kChanged : 0u) | (nzinf > 256.5f ? kUnexact : 0u);
        const int64_t nb = ((s + 1) & 1) * P2 + pg;
        if (nan_head) {
          atomicMax(&p.zkey[nb], 0x7fffffffull << 32);
        } else if (nkmax >= 0) {
          atomicMax(&p.zkey[nb], ((unsigned long long)__float_as_uint(nzinf) << 32) | (0xffffffffu - (uint32_t)nkmax));
        }
        if (next_coll) {
          if (accbits) atomicOr(&p.acc[nb], accbits);
          accbits = 0u;
          if (out_id) p.idw[nb] = 1u;
          if (first_id != kNoNz) atomicMin(&p.first[nb], first_id);
        }
        if (dbg && p.dbg_phi) {
          float add = p.lambda1 * frac + l1_id;
          if (rank == 0 && h == 0) add += p.lambda2 * (zinf > 0.f ? fmaxf(1.f / zinf - 1.f, 0.f) : INFINITY);
          atomicAdd(&p.dbg_phi[pg], add);
        }
      }
    }
    tc_fence_before();
    fence_async_all();
    cluster_sync();
    tc_fence_after();
  }
  // after a time-out: what was started lands before the memory goes away
  if (*(volatile int*)&s_abort) {
    const long long t0 = clock64();
    while (clock64() - t0 < 2000000) {}  // 1 ms: copies and MMAs in flight are far shorter
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
}

__global__ void __launch_bounds__(kThreads, 2) cluster_kernel(const __grid_constant__ ClParams p) {
  cluster_body(p, blockIdx.x / p.C, blockIdx.x % p.C);
}

// many instances: cluster w runs tile work[w].y of instance work[w].x
__global__ void __launch_bounds__(kThreads, 2) cluster_batch_kernel(const ClParams* __restrict__ table,
                                                                   const int2* __restrict__ work, int C) {
  __shared__ ClParams s_p;
  const int2 w = work[blockIdx.x / C];
  if (threadIdx.x == 0) s_p = table[w.x];
  __syncthreads();
  cluster_body(s_p, w.y, blockIdx.x % C);
}

// ---------------------------------------------------------------- set-up kernels

// Bm in the layouts of the two operands, per block of the cluster; *bad = 1
// (and flags |= 8) if an entry is not exact in BF16 (or e4m3 for FP8)
__global__ void cl_pack_b_kernel(const int32_t* __restrict__ B, int d, int R, int d32, int R32, int C, int f8,
                                 uint8_t* __restrict__ Bf, uint8_t* __restrict__ Bf8, uint8_t* __restrict__ Bg,
                                 int32_t* bad, int32_t* flags) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= (int64_t)R32 * d32) return;
  const int i = (int)(e / d32), j = (int)(e % d32);
  const int v = (i < R && j < d) ? B[(int64_t)(d + i) * d + j] : 0;
  bool inexact = v > 256 || v < -256;
  int begin = 0, len = 0;
  for (int c = 0; c < C; ++c) {
    slice_of(R32, C, c, begin, len);
    if (i < begin + len) break;
  }
  const int rb = (i - begin) / kRowBlk * kRowBlk;
  const int Nf = min(kRowBlk, len - rb), il = i - begin - rb;
  const size_t fo = (size_t)(begin + rb) * d32 + (size_t)(j / kKC) * Nf * kKC;
  if (f8) {
    const __nv_fp8_storage_t qv = __nv_cvt_float_to_fp8((float)v, __NV_SATFINITE, __NV_E4M3);
    const __half_raw hr = __nv_cvt_fp8_to_halfraw(qv, __NV_E4M3);
    if (__half2float(*reinterpret_cast<const __half*>(&hr)) != (float)v) inexact = true;
    Bf8[fo + off8(il, j % kKC)] = (uint8_t)qv;
  }
  if (inexact) {
    atomicOr(bad, 1);
    atomicOr(flags, 8);
  }
  const __nv_bfloat16 hb = __float2bfloat16_rn((float)v);
  const uint16_t hv = *reinterpret_cast<const uint16_t*>(&hb);
  *reinterpret_cast<uint16_t*>(Bf + fo * 2 + off16(il, j % kKC)) = hv;
  for (int c = 0; c < C; ++c) {
    slice_of(d32, C, c, begin, len);
    if (j < begin + len) break;
  }
  const int cb = (j - begin) / kColBlk * kColBlk;
  const int Ng = min(kColBlk, len - cb), jl = j - begin - cb;
  *reinterpret_cast<uint16_t*>(Bg + ((size_t)(begin + cb) * R32 + (size_t)(i / kKC) * Ng * kKC) * 2 +
                               off16(jl, i % kKC)) = hv;
}

// The call's state in the blocked layout, the operands of z0 and the per-start
// words.  One block per 32 starts of a tile: a warp reads 32 coordinates of a
// start at a time (coalesced), shared memory turns them.
constexpr int kInitRows = 32;

// the operands of z0 from the blocked state, 8 coordinates of a start per thread
__device__ __forceinline__ void z_operands(const ClParams& p, int tile, int rq) {
  const int row = rq * kInitRows + (threadIdx.x & 31), part = threadIdx.x >> 5;
  const size_t base = (size_t)tile * (p.d32 / 4) * kTM + row;
  const float sc = p.f8 ? scale_of(__ldcg(&p.zkey[(int64_t)tile * kTM + row])) : 1.f;
  for (int j0 = 8 * part; j0 < p.d32; j0 += 64) {
    const size_t o = base + (size_t)(j0 / 4) * kTM;
    const float4 a = reinterpret_cast<const float4*>(p.Zt)[o], b = reinterpret_cast<const float4*>(p.Zt)[o + kTM];
    uint8_t* const zo = z_tile(p, tile) + (size_t)(j0 >> 5) * z_stride(p);
    if (p.f8) {
      const float v8[8] = {a.x * sc, a.y * sc, a.z * sc, a.w * sc, b.x * sc, b.y * sc, b.z * sc, b.w * sc};
      *reinterpret_cast<uint2*>(zo + off8(row, j0 & 31)) = pack_e4m3x8(v8);
    } else {
      const float z[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
      uint32_t wh[4], wl[4];
      split8(z, wh, wl);
      const uint32_t oc = off16(row, j0 & 31);
      *reinterpret_cast<uint4*>(zo + oc) = make_uint4(wh[0], wh[1], wh[2], wh[3]);
      if (p.nterms > 1) *reinterpret_cast<uint4*>(zo + kChunk16 + oc) = make_uint4(wl[0], wl[1], wl[2], wl[3]);
    }
  }
}

__global__ void __launch_bounds__(256) cl_init_kernel(ClParams p, const float* __restrict__ Z,
                                                      const float* __restrict__ M, const float* __restrict__ V) {
  __shared__ float t[3][kInitRows][33];
  __shared__ float s_best[kInitRows][8];
  __shared__ int s_at[kInitRows][8];
  const int tile = blockIdx.x / (kTM / kInitRows), rq = blockIdx.x % (kTM / kInitRows);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t pg0 = (int64_t)tile * kTM + rq * kInitRows;
  const int64_t P2 = (int64_t)p.tiles * kTM;
  const int rr = tid & 31, part = tid >> 5;  // the turned side: start rr, coordinates 4 part ..
  const size_t base = (size_t)tile * (p.d32 / 4) * kTM + rq * kInitRows + rr;
  float best = 0.f;
  int kb = -1;
  for (int j0 = 0; j0 < p.d32; j0 += 32) {
    for (int a = warp; a < kInitRows; a += 8) {
      const int64_t row = pg0 + a;
      const int j = j0 + lane;
      const bool in = row < p.P && j < p.d;
      t[0][a][lane] = in ? Z[row * p.d + j] : 0.f;
      t[1][a][lane] = in ? M[row * p.d + j] : 0.f;
      t[2][a][lane] = in ? V[row * p.d + j] : 0.f;
    }
    __syncthreads();
    const int c = 4 * part;
    const size_t o = base + (size_t)((j0 + c) / 4) * kTM;
    reinterpret_cast<float4*>(p.Zt)[o] = make_float4(t[0][rr][c], t[0][rr][c + 1], t[0][rr][c + 2], t[0][rr][c + 3]);
    reinterpret_cast<float4*>(p.Mt)[o] = make_float4(t[1][rr][c], t[1][rr][c + 1], t[1][rr][c + 2], t[1][rr][c + 3]);
    reinterpret_cast<float4*>(p.Vt)[o] = make_float4(t[2][rr][c], t[2][rr][c + 1], t[2][rr][c + 2], t[2][rr][c + 3]);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float a = fabsf(t[0][rr][c + k]);
      // a NaN counts only as coordinate 0 (the sequential scan's start)
      const int j = j0 + c + k;
      if (j < p.d && (j == 0 || (kb < 0 ? a == a : a > best))) { best = a; kb = j; }
    }
    __syncthreads();
  }
  s_best[rr][part] = best;
  s_at[rr][part] = kb;
  __syncthreads();
  if (tid < kInitRows) {
    const int64_t pg = pg0 + tid;
    float b = 0.f;
    int at = -1;
    for (int q = 0; q < 8; ++q) {
      const int k = s_at[tid][q];
      const float v = s_best[tid][q];
      if (k >= 0 && (at < 0 || v > b || (v == b && k < at))) { b = v; at = k; }  // a NaN at 0 stays
    }
    const unsigned long long key =
        pg < p.P ? ((unsigned long long)__float_as_uint(b) << 32) | (0xffffffffu - (uint32_t)at) : 0ull;
    p.zkey[pg] = key;
    p.zkey[P2 + pg] = 0ull;
    p.oob[pg] = 0u;
    for (int k = 0; k < 2; ++k) {
      p.acc[k * P2 + pg] = 0u;
      p.idw[k * P2 + pg] = 0u;
      p.first[k * P2 + pg] = kNoNz;
    }
    if (p.dbg_phi && pg < p.P) p.dbg_phi[pg] = 0.f;
  }
  if (p.z_out) return;  // other blocks still read where the operands go: cl_operand_kernel
  __syncthreads();
  z_operands(p, tile, rq);
}

__global__ void __launch_bounds__(256) cl_operand_kernel(ClParams p) {
  z_operands(p, blockIdx.x / (kTM / kInitRows), blockIdx.x % (kTM / kInitRows));
}

// the blocked state back to the caller's rows
__global__ void __launch_bounds__(256) cl_unpack_kernel(ClParams p, float* __restrict__ Z, float* __restrict__ M,
                                                        float* __restrict__ V) {
  __shared__ float t[3][kInitRows][33];
  const int tile = blockIdx.x / (kTM / kInitRows), rq = blockIdx.x % (kTM / kInitRows);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t pg0 = (int64_t)tile * kTM + rq * kInitRows;
  const int rr = tid & 31, c = 4 * (tid >> 5);
  const size_t base = (size_t)tile * (p.d32 / 4) * kTM + rq * kInitRows + rr;
  for (int j0 = 32 * blockIdx.y; j0 < p.d32; j0 += 32 * gridDim.y) {
    const size_t o = base + (size_t)((j0 + c) / 4) * kTM;
    const float4 z = reinterpret_cast<const float4*>(p.Zt)[o], m = reinterpret_cast<const float4*>(p.Mt)[o],
                 v = reinterpret_cast<const float4*>(p.Vt)[o];
    t[0][rr][c] = z.x; t[0][rr][c + 1] = z.y; t[0][rr][c + 2] = z.z; t[0][rr][c + 3] = z.w;
    t[1][rr][c] = m.x; t[1][rr][c + 1] = m.y; t[1][rr][c + 2] = m.z; t[1][rr][c + 3] = m.w;
    t[2][rr][c] = v.x; t[2][rr][c + 1] = v.y; t[2][rr][c + 2] = v.z; t[2][rr][c + 3] = v.w;
    __syncthreads();
    for (int a = warp; a < kInitRows; a += 8) {
      const int64_t row = pg0 + a;
      const int j = j0 + lane;
      if (row < p.P && j < p.d) {
        Z[row * p.d + j] = t[0][a][lane];
        M[row * p.d + j] = t[1][a][lane];
        V[row * p.d + j] = t[2][a][lane];
      }
    }
    __syncthreads();
  }
}

int pad32(int x) { return (x + 31) / 32 * 32; }
int pad16(int x) { return (x + 15) / 16 * 16; }

constexpr int32_t kBiasSteps = 1 << 19;  // steps of a call: half of the step-by-step kernels' table, half its bytes
constexpr size_t kZAlign = 128;

// The z operands lie in the caller's M, V and Z where they fit: from the packing
// of the state to its unpacking these hold nothing that is needed.  (In the
// workspace they made it larger than that of the step-by-step kernels, by 31%
// at n = 2000 and P = 65536, and a server whose memory cap lay between refused
// the request.)  Where they do not fit, for a few hundred starts, the workspace has
// room for them.
struct ClShape {
  int R, d32, R32, tiles, ldi;
  size_t z_tile;   // bytes of a tile's z operands
  int z_fit;       // tiles that fit in each of the three arrays, at any address
  bool z_out;
};
ClShape cl_shape(int n, int d, int P, int32_t precision) {
  ClShape s{};
  s.R = n - d;
  s.d32 = pad32(d);
  s.R32 = s.R > 0 ? pad32(s.R) : 32;
  s.tiles = (int)mape_detail::ceil_div(P, kTM);
  s.ldi = pad16(d);
  const int per = precision == MAPE_PREC_FP8 ? 3 : precision == MAPE_PREC_BF16 ? 6 : 4;  // bytes a coordinate
  s.z_tile = (size_t)kTM * s.d32 * per;
  const size_t bytes = sizeof(float) * (size_t)P * d;
  s.z_fit = bytes > kZAlign ? (int)std::min<size_t>((bytes - kZAlign) / s.z_tile, (size_t)s.tiles) : 0;
  s.z_out = 3ll * s.z_fit >= s.tiles;
  return s;
}

struct ClCarved {
  ClShape sh;
  float *Zt, *Mt, *Vt;
  uint8_t *Zh, *S, *Bf, *Bg, *Bf8;
  int8_t *stage, *stage_map;
  unsigned long long* zkey;
  uint32_t *acc, *oob, *idw;
  int32_t *first, *hflags;
  float2* bias;
};

template <typename Carve>
void cl_carve(Carve& cv, const ClShape& sh, ClCarved* c) {
  const size_t P2 = (size_t)sh.tiles * kTM;
  ClCarved k{};
  k.sh = sh;
  auto take = [&](auto*& ptr, size_t count) {
    using T = std::remove_pointer_t<std::remove_reference_t<decltype(ptr)>>;
    if constexpr (std::is_same_v<Carve, mape_detail::Carver>) ptr = cv.template take<T>(count);
    else cv.template take<T>(count);
  };
  take(k.Zt, P2 * sh.d32);
  take(k.Mt, P2 * sh.d32);
  take(k.Vt, P2 * sh.d32);
  if (!sh.z_out) take(k.Zh, sh.z_tile * sh.tiles);
  take(k.S, P2 * sh.R32 * 2);
  take(k.stage, 2 * P2 * sh.ldi);
  take(k.stage_map, P2 * sh.R32);
  take(k.Bf, (size_t)sh.R32 * sh.d32 * 2);
  take(k.Bg, (size_t)sh.R32 * sh.d32 * 2);
  take(k.Bf8, (size_t)sh.R32 * sh.d32);
  take(k.zkey, 2 * P2);
  take(k.acc, 2 * P2);
  take(k.oob, P2);
  take(k.idw, 2 * P2);
  take(k.first, 2 * P2);
  take(k.hflags, (size_t)2);
  take(k.bias, (size_t)kBiasSteps);
  if (c) *c = k;
}

}  // namespace

namespace mape_detail {

// Blocks per cluster of a call, and their shared memory, by the tiles that run
// together (of the call, or of its whole batch).  More blocks per tile
// shorten a step (its latency is a part that stays and one that is shared), as
// long as all tiles run at once; clusters stay within a GPC, so that 15 of 8 blocks,
// 36 of 4 and 76 of 2 run with an SM per block, 36 of 8, 74 of 4 and 152 of 2
// with two blocks to an SM.  One tile more is a second wave: n = 487, 20
// steps, 36 tiles 0.50 ms with 8 and 4 blocks, 37 tiles 0.78 and 0.59; 73 tiles 0.65
// with 4, 76 tiles 0.99, 0.70 with 2.  Where the lines lie otherwise:
//  16 .. 36 tiles: 4 blocks with an SM each take 0.93 to 0.98 of the time of 8 with
//    two to an SM for n = 20 to 60, 1.02 to 1.09 for n = 100 to 2000;
//  .. 74 tiles: 2 blocks an SM each take 0.94 of the time of 4 for n = 20, 1.05 to
//    1.2 from n = 125 on;
//  77 .. 152 tiles, d > 1024: two waves of 4 blocks 4.6 ms against 5.0 with 2 (n =
//    2000, 128 tiles), 2.18 and 2.13 for n = 1000;
//  beyond: tiles wait for an SM anyway, and for small n the fewer blocks share a
//    tile the less is spent on barriers (512 tiles of n = 50, 200, 487, 700: 0.81,
//    1.33, 3.99, 5.96 ms with 1 block, 1.60, 2.17, 3.93, 5.54 with 4).
// False: the step-by-step kernels, where waves of 4 blocks leave the chip too
// empty for the gain of a step (1.2 at n = 2000 with full waves) to make up for
// it.  Collecting every step, BF16: n = 2000, 77, 101, 153 and 178 tiles 3.64, 4.20,
// 6.27 and 6.49 ms against 3.25, 3.95, 5.51 and 6.34, but 128 tiles 4.57 and 4.69; n =
// 1000, 153 tiles 3.02 and 2.79; n = 550 1.61 and 1.73.  Every second step: 75
// tiles 3.32 and 2.94, 101 3.76 and 3.67, 121 3.99 and 4.21.  More rows below the
// identity than coordinates (n = 1300, d = 120), 223 tiles: 2.99 and 2.63, FP8 2.95
// and 2.73.  FP8 is faster in clusters at the other sizes (n = 2000: 3.36, 3.77, 5.57
// against 3.44, 4.10, 5.70).
struct ClChoice {
  int C, dyn;
};
static bool cl_choose(const mape_extract_args* a, int64_t tiles, ClChoice* c) {
  const int n = a->n, d = a->d;
  if (tiles <= 15) *c = {8, kDynSmemOne};
  else if (tiles <= 36) *c = n <= 64 ? ClChoice{4, kDynSmemOne} : ClChoice{8, kDynSmem};
  else if (tiles <= 74 && n > 64) *c = {4, kDynSmem};
  else if (tiles <= 76 && d <= 1024) *c = {2, kDynSmemOne};
  else if (tiles <= 152 && d <= 1024) *c = {2, kDynSmem};
  else if (n <= 320) *c = {1, kDynSmem};
  else {
    *c = {4, kDynSmem};
    if (n <= 640) return true;
    if (n - d > d) return false;
    const bool often = a->precision == MAPE_PREC_BF16 && a->period == 1;
    if (a->precision == MAPE_PREC_FP8 || (!often && n <= 800)) return true;
    return 100 * tiles >= (often ? 84 : 76) * 74 * ceil_div(tiles, 74);
  }
  return true;
}

bool extract_cluster_takes(const mape_extract_args* a) { return a->d < a->n && a->T <= kBiasSteps; }

size_t extract_cluster_workspace(int32_t n, int32_t d, int32_t P, int32_t precision) {
  if (d >= n) return 0;
  Sizer s;
  cl_carve(s, cl_shape(n, d, P, precision), nullptr);
  return s.bytes();
}

static void cl_params(const ClCarved& c, const mape_extract_args* a, ClChoice choice, ClParams& p) {
  const ClShape& sh = c.sh;
  p = ClParams{};
  p.n = a->n; p.d = a->d; p.P = a->P; p.R = sh.R; p.d32 = sh.d32; p.R32 = sh.R32;
  p.tiles = sh.tiles; p.C = choice.C; p.dyn = choice.dyn; p.ldc = a->ldc; p.ldi = sh.ldi;
  p.Bf = c.Bf; p.Bf8 = c.Bf8; p.Bg = c.Bg; p.span = a->span; p.Zt = c.Zt; p.Mt = c.Mt; p.Vt = c.Vt;
  p.z_out = sh.z_out ? 1 : 0;
  if (sh.z_out) {
    float* const at[3] = {a->M, a->V, a->Z};
    for (int k = 0; k < 3; ++k)
      p.Zh[k] = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(at[k]) + kZAlign - 1) / kZAlign * kZAlign);
    p.z1 = std::min(sh.z_fit, sh.tiles);
    p.z2 = std::min(2 * sh.z_fit, sh.tiles);
  } else {
    p.Zh[0] = p.Zh[1] = p.Zh[2] = c.Zh;
    p.z1 = p.z2 = sh.tiles;
  }
  p.S = c.S; p.stage = c.stage; p.stage_map = c.stage_map; p.zkey = c.zkey; p.acc = c.acc;
  p.oob = c.oob; p.idw = c.idw; p.first = c.first; p.bias = c.bias;
  p.lambda1 = a->lambda1; p.lambda2 = a->lambda2; p.eps = a->eps;
  p.beta1 = (float)a->beta1; p.beta2 = (float)a->beta2;
  p.omb1 = (float)(1.0 - a->beta1); p.omb2 = (float)(1.0 - a->beta2);
  p.nterms = a->precision == MAPE_PREC_BF16 ? 2 : 1;
  p.f8 = a->precision == MAPE_PREC_FP8 ? 1 : 0;
  p.t0 = a->t0; p.T = a->T; p.period = a->period;
  p.cand = a->cand; p.cap = a->cand_cap; p.count = a->cand_count; p.flags = a->flags;
  p.dbg_phi = a->dbg_phi; p.dbg_grad = a->dbg_grad;
}

static int cl_pack(const ClParams& p, const mape_extract_args* a, int32_t* bad, cudaStream_t st) {
  MAPE_CUDA_TRY(cudaMemsetAsync(bad, 0, sizeof(int32_t), st));
  launch(cl_pack_b_kernel, (unsigned)ceil_div((int64_t)p.R32 * p.d32, 256), 256, 0, st, a->B, p.d, p.R, p.d32, p.R32,
         p.C, p.f8, const_cast<uint8_t*>(p.Bf), const_cast<uint8_t*>(p.Bf8), const_cast<uint8_t*>(p.Bg), bad, a->flags);
  MAPE_LAUNCH_CHECK();
  return MAPE_OK;
}

static int cl_setup(const ClCarved& c, const ClParams& p, const mape_extract_args* a, cudaStream_t st) {
  std::vector<float2> bc((size_t)a->T);
  for (int s = 0; s < a->T; ++s) {
    const double t = (double)a->t0 + s + 1;
    const double bc1 = 1.0 - std::pow(a->beta1, t), bc2 = 1.0 - std::pow(a->beta2, t);
    bc[s] = make_float2((float)((double)a->lr / bc1), (float)(1.0 / std::sqrt(bc2)));
  }
  MAPE_CUDA_TRY(cudaMemcpyAsync(c.bias, bc.data(), sizeof(float2) * bc.size(), cudaMemcpyHostToDevice, st));
  launch(cl_init_kernel, (unsigned)(p.tiles * (kTM / kInitRows)), 256, 0, st, p, (const float*)a->Z,
         (const float*)a->M, (const float*)a->V);
  if (p.z_out) launch(cl_operand_kernel, (unsigned)(p.tiles * (kTM / kInitRows)), 256, 0, st, p);
  MAPE_LAUNCH_CHECK();
  return MAPE_OK;
}

static int cl_unpack(const ClParams& p, const mape_extract_args* a, cudaStream_t st) {
  const unsigned gy = (unsigned)std::min<int64_t>(p.d32 / 32, std::max<int64_t>(1, 1216 / (p.tiles * (kTM / kInitRows))));
  launch(cl_unpack_kernel, dim3((unsigned)(p.tiles * (kTM / kInitRows)), gy), 256, 0, st, p, a->Z, a->M, a->V);
  MAPE_LAUNCH_CHECK();
  return MAPE_OK;
}

static int cl_attributes(bool batch) {
  const void* f = batch ? (const void*)cluster_batch_kernel : (const void*)cluster_kernel;
  MAPE_CUDA_TRY(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kDynSmemOne));
  return MAPE_OK;
}

template <typename... KArgs, typename... Args>
static int launch_clusters(void (*kernel)(KArgs...), int64_t clusters, int C, int dyn, cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(clusters * C));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = (size_t)dyn;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)C;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  MAPE_CUDA_TRY(cudaLaunchKernelEx(&cfg, kernel, args...));
  note_launch();
  return MAPE_OK;
}

// One call.  *general = true (and nothing done) when B has no identity top, or
// the step-by-step kernels are faster.
int extract_cluster(const mape_extract_args* a, cudaStream_t st, bool* general, Basis* basis) {
  *general = false;
  ClChoice choice;
  if (!extract_cluster_takes(a) || *basis == kBasisGeneral || !cl_choose(a, ceil_div(a->P, kTM), &choice)) {
    *general = true;
    return MAPE_OK;
  }
  Carver cv(a->workspace, a->workspace_bytes);
  ClCarved c;
  cl_carve(cv, cl_shape(a->n, a->d, a->P, a->precision), &c);
  if (!cv.ok) return MAPE_ERR_CAPACITY;
  int rc;
  if (*basis == kBasisUnknown) {
    std::vector<bool> ids;
    if ((rc = identity_tops(&a, 1, c.hflags, st, ids)) != MAPE_OK) return rc;
    *basis = ids[0] ? kBasisIdentity : kBasisGeneral;
  }
  if (*basis == kBasisGeneral) { *general = true; return MAPE_OK; }
  ClParams p;
  cl_params(c, a, choice, p);
  if ((rc = cl_pack(p, a, c.hflags + 1, st)) != MAPE_OK) return rc;
  int32_t h_bad = 0;
  MAPE_CUDA_TRY(cudaMemcpyAsync(&h_bad, c.hflags + 1, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
  MAPE_CUDA_TRY(cudaStreamSynchronize(st));
  if (h_bad) return MAPE_OK;  // flag 8 is set; nothing runs, nothing is collected
  if ((rc = cl_setup(c, p, a, st)) != MAPE_OK) return rc;
  if ((rc = cl_attributes(false)) != MAPE_OK) return rc;
  if ((rc = launch_clusters(cluster_kernel, p.tiles, p.C, p.dyn, st, p)) != MAPE_OK) return rc;
  return cl_unpack(p, a, st);
}

// Many calls (identity-topped, same T, t0, period and precision): the tiles of
// all calls with the same cluster size in one launch, the costliest tiles
// first; the (at most three) launches run side by side.
struct ClBatch {
  struct Class {
    int C = 0;
    int64_t first = 0, clusters = 0;
  };
  std::vector<Class> classes;
  ClParams* table = nullptr;
  int2* work = nullptr;
  std::vector<const mape_extract_args*> items;
  std::vector<ClParams> params;
  std::vector<bool> run;  // false: B not exact in BF16 (flag 8 set, nothing runs)
  std::vector<cudaStream_t> side;  // of the classes after the first, forked from and joined to the caller's
  cudaEvent_t fork = nullptr, join = nullptr;
  ~ClBatch() {
    if (fork) cudaEventDestroy(fork);
    if (join) cudaEventDestroy(join);
    for (cudaStream_t s : side) cudaStreamDestroy(s);  // released once its work has completed
  }
};

void extract_cluster_batch_free(ClBatch* b) { delete b; }

size_t extract_cluster_batch_workspace(const mape_extract_args* const* items, int count) {
  Sizer s;
  int64_t tiles = 0;
  for (int i = 0; i < count; ++i) tiles += ceil_div(items[i]->P, kTM);
  s.take<ClParams>((size_t)count);
  s.take<int2>((size_t)tiles);
  return s.bytes();
}

int extract_cluster_batch_prepare(const mape_extract_args* const* items, int count, void* ws, size_t ws_bytes,
                                  cudaStream_t st, ClBatch** out) {
  *out = nullptr;
  std::unique_ptr<ClBatch> plan(new ClBatch());
  plan->items.assign(items, items + count);
  plan->params.resize((size_t)count);
  plan->run.assign((size_t)count, true);
  Carver bc(ws, ws_bytes);
  plan->table = bc.take<ClParams>((size_t)count);
  int64_t tiles = 0;
  for (int i = 0; i < count; ++i) tiles += ceil_div(items[i]->P, kTM);
  plan->work = bc.take<int2>((size_t)tiles);
  if (!bc.ok) return MAPE_ERR_CAPACITY;
  std::vector<ClCarved> carved((size_t)count);
  int rc;
  for (int i = 0; i < count; ++i) {
    const mape_extract_args* a = items[i];
    Carver cv(a->workspace, a->workspace_bytes);
    cl_carve(cv, cl_shape(a->n, a->d, a->P, a->precision), &carved[i]);
    if (!cv.ok) return MAPE_ERR_CAPACITY;
    // by the tiles of the whole batch: 0.75 to 0.95 of the time of a rule by d
    // alone (8 blocks from 512 coordinates on, 4 from 256, else 2), which for 8
    // calls of n = 1000 and P = 16384 was slower than the step-by-step kernels
    // (22.3 ms against 20.9; 18.3 now)
    ClChoice choice;
    cl_choose(a, tiles, &choice);
    choice.dyn = kDynSmem;
    cl_params(carved[i], a, choice, plan->params[i]);
    if ((rc = cl_pack(plan->params[i], a, carved[i].hflags + 1, st)) != MAPE_OK) return rc;
  }
  std::vector<int32_t> bad((size_t)count, 0);
  for (int i = 0; i < count; ++i)
    MAPE_CUDA_TRY(cudaMemcpyAsync(&bad[i], carved[i].hflags + 1, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
  MAPE_CUDA_TRY(cudaStreamSynchronize(st));
  std::vector<int> order;  // by cost per tile, descending
  for (int i = 0; i < count; ++i) {
    plan->run[i] = bad[i] == 0;
    if (!plan->run[i]) continue;
    if ((rc = cl_setup(carved[i], plan->params[i], items[i], st)) != MAPE_OK) return rc;
    order.push_back(i);
  }
  std::stable_sort(order.begin(), order.end(), [&](int x, int y) {
    const ClParams &a = plan->params[x], &b = plan->params[y];
    return (int64_t)a.d32 * b.C > (int64_t)b.d32 * a.C;
  });
  std::vector<int2> work;
  for (int C = kMaxC; C >= 1; C >>= 1) {
    ClBatch::Class k;
    k.C = C;
    k.first = (int64_t)work.size();
    for (int i : order)
      if (plan->params[i].C == C)
        for (int t = 0; t < plan->params[i].tiles; ++t) work.push_back(make_int2(i, t));
    k.clusters = (int64_t)work.size() - k.first;
    if (k.clusters > 0) plan->classes.push_back(k);
  }
  MAPE_CUDA_TRY(cudaMemcpyAsync(plan->table, plan->params.data(), sizeof(ClParams) * count, cudaMemcpyHostToDevice, st));
  if (!work.empty())
    MAPE_CUDA_TRY(cudaMemcpyAsync(plan->work, work.data(), sizeof(int2) * work.size(), cudaMemcpyHostToDevice, st));
  MAPE_CUDA_TRY(cudaStreamSynchronize(st));
  if ((rc = cl_attributes(true)) != MAPE_OK) return rc;
  if (plan->classes.size() > 1) {
    MAPE_CUDA_TRY(cudaEventCreateWithFlags(&plan->fork, cudaEventDisableTiming));
    MAPE_CUDA_TRY(cudaEventCreateWithFlags(&plan->join, cudaEventDisableTiming));
    for (size_t k = 1; k < plan->classes.size(); ++k) {
      cudaStream_t s = nullptr;
      MAPE_CUDA_TRY(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking));
      plan->side.push_back(s);
    }
  }
  *out = plan.release();
  return MAPE_OK;
}

int extract_cluster_batch_enqueue(const ClBatch* plan, cudaStream_t st) {
  const size_t nc = plan->classes.size();
  int rc = MAPE_OK;
  if (nc > 1) MAPE_CUDA_TRY(cudaEventRecord(plan->fork, st));
  for (size_t k = 0; k < nc; ++k) {
    const auto& K = plan->classes[k];
    const cudaStream_t s = k == 0 ? st : plan->side[k - 1];
    if (k > 0) MAPE_CUDA_TRY(cudaStreamWaitEvent(s, plan->fork, 0));
    rc = launch_clusters(cluster_batch_kernel, K.clusters, K.C, kDynSmem, s, (const ClParams*)plan->table,
                         (const int2*)(plan->work + K.first), K.C);
    if (rc != MAPE_OK) return rc;
  }
  for (cudaStream_t s : plan->side) {
    MAPE_CUDA_TRY(cudaEventRecord(plan->join, s));
    MAPE_CUDA_TRY(cudaStreamWaitEvent(st, plan->join, 0));
  }
  for (size_t i = 0; i < plan->items.size(); ++i)
    if (plan->run[i] && (rc = cl_unpack(plan->params[i], plan->items[i], st)) != MAPE_OK) return rc;
  return MAPE_OK;
}

}  // namespace mape_detail
