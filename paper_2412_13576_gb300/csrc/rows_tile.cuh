// A tile of 32 int8 rows in shared memory, transposed: one 32-bit word holds a
// coordinate of four rows, eight words of a coordinate the tile's 32 rows.
// Eight lanes that take one coordinate each read a word and have four rows
// apiece, so an entry of a matrix over the coordinates is loaded once for 32
// rows; a warp works on four entries at a time.
//
// Word (c, q) (coordinate c, rows 4 q .. 4 q + 3) lies at byte tile_at(c) ^ (q << 4):
// four coordinates side by side, so that a thread that has transposed 4 x 4
// bytes writes 16 of them at once, and the eight q's of a coordinate in eight
// different 16-byte columns, turned by c / 16 so that the threads of a warp,
// 16 coordinates apart, write to different banks.
#pragma once
#include "common.cuh"

namespace {

constexpr int kTileRows = 32, kTileLanes = kTileRows / 4;

__host__ __device__ inline size_t tile_bytes(int n) { return (size_t)((n + 15) / 16) * 16 * kTileRows; }

__device__ __forceinline__ uint32_t tile_at(int c) {
  return (uint32_t)(c >> 2) * 128u + (uint32_t)(c & 3) * 4u + ((uint32_t)(c >> 4) & 7u) * 16u;
}

// product of the signed bytes r of two words: a dot product over bytes of which
// one side keeps only byte r (extracting both bytes and multiplying: 6% slower
// in the coefficients)
__device__ __forceinline__ int tile_product(int x, int y, int r) { return __dp4a(x & (int)(0xffu << (8 * r)), y, 0); }

// Rows k0 .. k0 + cnt - 1 of G (16-byte aligned rows, ldg a multiple of 16),
// zeros for the rest of the 32; kBiased: every byte + 128.  Entries past n are
// whatever the pitch holds.
template <bool kBiased>
__device__ __forceinline__ void stage_tile(const int8_t* __restrict__ G, int64_t k0, int cnt, int n, int ldg,
                                           char* __restrict__ tile) {
  const int pieces = (n + 15) / 16;
  const uint32_t bias = kBiased ? 0x80808080u : 0u;
  for (int u = threadIdx.x; u < pieces * kTileLanes; u += blockDim.x) {
    const int q = u / pieces, p = u - q * pieces;
    uint32_t v[4][4];  // [row][four coordinates]
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      uint4 x = make_uint4(0, 0, 0, 0);
      if (4 * q + r < cnt) x = *reinterpret_cast<const uint4*>(G + (k0 + 4 * q + r) * ldg + 16 * p);
      v[r][0] = x.x ^ bias;
      v[r][1] = x.y ^ bias;
      v[r][2] = x.z ^ bias;
      v[r][3] = x.w ^ bias;
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {  // coordinates 16 p + 4 j ..
      const uint32_t a = __byte_perm(v[0][j], v[1][j], 0x5140), b = __byte_perm(v[2][j], v[3][j], 0x5140);
      const uint32_t c = __byte_perm(v[0][j], v[1][j], 0x7362), d = __byte_perm(v[2][j], v[3][j], 0x7362);
      *reinterpret_cast<uint4*>(tile + (tile_at(16 * p + 4 * j) ^ ((uint32_t)q << 4))) =
          make_uint4(__byte_perm(a, b, 0x5410), __byte_perm(a, b, 0x7632), __byte_perm(c, d, 0x5410),
                     __byte_perm(c, d, 0x7632));
    }
  }
}

}  // namespace
