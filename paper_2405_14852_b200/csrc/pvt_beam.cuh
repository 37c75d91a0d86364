// Pieces of the fast scores on the tensor pipe that the beam search and the local search share: residuals of targets, in two
// halves each, against a codebook of up to 256 fp16 codewords (mma.sync, residuals as rows).
#pragma once

#include <cuda_fp16.h>

#include "pvt_internal.h"

namespace pvt {
namespace beam {

constexpr int kBsK = 256;  // codebooks are padded to this many codewords
constexpr float kPadHalfNorm = 3.0e38f;
constexpr float kInf = __builtin_huge_valf();

// A codebook: B fragments, word [tile][lane] = halves (c[column 8 tile + lane/4][2 (lane%4)], [.. + 1]); codeword k stands
// at column stage_column(k)
struct TensorStage {
  alignas(16) uint32_t b[kBsK / 8][32];
  alignas(8) float h[kBsK];  // ||c||^2/2 by column
};
__device__ __forceinline__ float min3(float a, float b, float c) {
  float d;
  asm("min.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
// D = A (16 x 16, rows = residuals) x B (16 x 8, columns = codewords) + C, fp16 operands, fp32 accumulation
__device__ __forceinline__ void mma_16x8x16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1, float c0,
                                            float c1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%10, %11, %10, %11};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(c0), "f"(c1));
}
// The power of two that brings the largest element (of non-negative bit pattern rbits) to [2^14, 2^15), and its inverse:
// both are normal numbers for every finite element, and halves of up to 2^-30 of it are not subnormal.  Elements below 2^-15
// get less (a score of 2^29 times a codeword's squared norm is finite).
__device__ __forceinline__ void half_scale(uint32_t rbits, float& sc, float& inv) {
  int e = 140 - (int)((rbits >> 23) & 0xffu);
  e = e > 29 ? 29 : e;
  sc = __uint_as_float((uint32_t)(e + 127) << 23);
  inv = __uint_as_float((uint32_t)(127 - e) << 23);
}
// x, y as the sum of two pairs of halves (22 significant bits)
__device__ __forceinline__ void split_halves(float x, float y, uint32_t& hi_bits, uint32_t& lo_bits) {
  const __half2 hi = __floats2half2_rn(x, y);
  const float2 back = __half22float2(hi);
  const __half2 lo = __floats2half2_rn(x - back.x, y - back.y);
  hi_bits = *reinterpret_cast<const uint32_t*>(&hi);
  lo_bits = *reinterpret_cast<const uint32_t*>(&lo);
}
// the same of three pairs: all bits
__device__ __forceinline__ void split_three_halves(float x, float y, uint32_t& hi_bits, uint32_t& mid_bits, uint32_t& lo_bits) {
  const __half2 hi = __floats2half2_rn(x, y);
  const float2 back = __half22float2(hi);
  hi_bits = *reinterpret_cast<const uint32_t*>(&hi);
  split_halves(x - back.x, y - back.y, mid_bits, lo_bits);
}

// Where codeword k stands among the columns of the tiles: the 32 codewords of a cell are what one thread sees of a
// residual, columns 2 q and 2 q + 1 of sixteen tiles (q = lane % 4).
__device__ __forceinline__ int stage_column(int k) {
  const int cell = k >> 5, i = k & 31;
  return 8 * (16 * (cell & 1) + (i >> 1)) + 2 * (cell >> 1) + (i & 1);
}

// The fast scores ||r - c||^2/2 of 32 residuals, the lane's in r[lane], those of lanes 0..15 against one codebook, of lanes
// 16..31 against another (or the same): the lane's minimum of each of eight cells of 32 adjacent codewords (rho =
// ||r||^2/2 of its residual; infinity where it is not active).  Returns what the halves add to the margin of a score.
// The margins take a sum of the tensor pipe to be off by no more than 26 u (||r|| + ||c||)^2, u = 2^-24.  How the tensor cores
// add is not documented, so that this is an assumption; the largest errors against binary64 were 3.5 to 7.1 u of ||c||^2/2 +
// ||r|| ||c|| over 4 million scores each of vectors as the layers have them, 16 times larger and smaller, and of mixed sizes.
__device__ __forceinline__ float tensor_minima(const TensorStage& st0, const TensorStage& st1, const float (*wr)[8],
                                               float (*wmin)[8], float rho, bool active, float smax, float (&sub_min)[8]) {
  const uint32_t lane = threadIdx.x & 31;
  // The 32 residuals are the rows of two 16-row A tiles, each row [ -hi(2^e r) | -lo(2^e r) ] in fp16 (hi + lo keeps 22
  // significant bits of r, or all bits above 2^-25 in scaled units); the columns of B are the codewords, [ c | c ]; C
  // starts at 2^e ||c||^2/2.  e is common to the residuals: the largest element becomes [2^14, 2^15).  A thread holds
  // elements 2 qd, 2 qd + 1 of rows g8, g8 + 8 of each tile.
  const uint32_t g8 = lane >> 2, qd = lane & 3u;
  float2 nr[4];
  float rmax = 0.0f;
#pragma unroll
  for (int r4 = 0; r4 < 4; ++r4) {
    nr[r4] = *reinterpret_cast<const float2*>(&wr[16 * (r4 >> 1) + 8 * (r4 & 1) + g8][2 * qd]);
    rmax = fmaxf(rmax, fmaxf(fabsf(nr[r4].x), fabsf(nr[r4].y)));
  }
  const uint32_t rbits = __reduce_max_sync(0xffffffffu, __float_as_uint(rmax));  // non-negative floats order as u32
  float sc, inv;
  half_scale(rbits, sc, inv);
  uint32_t a[2][4];
#pragma unroll
  for (int r4 = 0; r4 < 4; ++r4) split_halves(nr[r4].x * -sc, nr[r4].y * -sc, a[r4 >> 1][r4 & 1], a[r4 >> 1][2 + (r4 & 1)]);
  // a cell is what one thread sees of a residual in half the tiles: no exchange between the threads (with cells of 32
  // adjacent columns, two exchanges per cell and row: 11008x4096 k = 56360 two codebooks 1.8 us more, three 4.8 us)
  float m[4][2];
#pragma unroll
  for (int half = 0; half < 2; ++half) {
    float x[4] = {kInf, kInf, kInf, kInf};
#pragma unroll 4
    for (int n = 0; n < 16; ++n) {
      const int nt = 16 * half + n;
      const uint32_t b0 = st0.b[nt][lane], b1 = st1.b[nt][lane];
      const float2 h0 = *reinterpret_cast<const float2*>(&st0.h[8 * nt + 2 * qd]);
      const float2 h1 = *reinterpret_cast<const float2*>(&st1.h[8 * nt + 2 * qd]);
      float d0[4], d1[4];
      mma_16x8x16(d0, a[0], b0, b0, h0.x * sc, h0.y * sc);
      mma_16x8x16(d1, a[1], b1, b1, h1.x * sc, h1.y * sc);
      x[0] = min3(x[0], d0[0], d0[1]);
      x[1] = min3(x[1], d0[2], d0[3]);
      x[2] = min3(x[2], d1[0], d1[1]);
      x[3] = min3(x[3], d1[2], d1[3]);
    }
#pragma unroll
    for (int r4 = 0; r4 < 4; ++r4) m[r4][half] = x[r4];
  }
#pragma unroll
  for (int r4 = 0; r4 < 4; ++r4)
    *reinterpret_cast<float2*>(&wmin[16 * (r4 >> 1) + 8 * (r4 & 1) + g8][2 * qd]) = make_float2(m[r4][0], m[r4][1]);
  __syncwarp();
  const float4 ma = *reinterpret_cast<const float4*>(&wmin[lane][0]);
  const float4 mb = *reinterpret_cast<const float4*>(&wmin[lane][4]);
  const float mm[8] = {ma.x, ma.y, ma.z, ma.w, mb.x, mb.y, mb.z, mb.w};
#pragma unroll
  for (int sub = 0; sub < 8; ++sub) sub_min[sub] = active ? __fmaf_rn(mm[sub], inv, rho) : kInf;
  // the halves' absolute rounding floor (2^-25 per element in scaled units), doubled, with a factor 4 to spare
  return 4.76837158203125e-7f /* 2^-21 */ * inv * smax;
}

}  // namespace beam
}  // namespace pvt
