// Beam search of the V step for two to four additive codebooks (Appendix C: the code combination is found by beam
// search; Appendix J: 8-bit codebooks, group size 8, beam size 8, target = gradient-updated dequantised weight; Eq. 8
// for the target; Lemma 3.3 for keeping the previous tuple in the pool).
//
//   stage m (m = 1..M): each kept partial tuple (one empty tuple before stage 1) is extended by every codeword of
//     codebook m; the score of an extension is ||t - c^1 - ... - c^m||^2;
//   after stages 1..M-1 the `beam` smallest extensions under (score, tuple) are kept;
//   the result is the smallest member of the last stage's extensions and the previous tuple.
//
// A warp handles four targets at a time; the codebooks live in shared memory; three or four CTAs (24 or 32 warps) share an
// SM.
//   stage 1 (four targets side by side): fast scores ||c1||^2/2 - <t, c1>, on the tensor pipe for fp16 codebooks (mma.sync,
//            the codewords as rows); a thread keeps the minima of cells of four codewords, 64 per target, and goes on as a
//            stage in the middle.  Binary32 codebooks: one target after the other, 256 scores on the FP32 pipe, 8 per lane,
//            of which the `beam` smallest are extracted with warp-wide minima on (score bits | code) keys.
//   further stages (four targets x eight kept tuples = 32 residuals, one per lane): fast scores
//            ||r||^2/2 + ||c||^2/2 - <r, c> of all residuals against all codewords, on the tensor pipe for fp16
//            codebooks (mma.sync, the residuals as rows), on the FP32 pipe otherwise; only the minimum of each
//            (residual, 32 codewords) cell is kept: 64 cells per target.
//   a stage in the middle: the `beam`-th smallest of a target's 64 cell minima bounds its `beam`-th smallest score, so
//            only cells within the rounding margin of it -- usually `beam` of them -- are scored again, a codeword per
//            lane; what is within the margin goes on a short list, of which the `beam` smallest are kept.
//   last stage: cells within the margin of the smallest are revisited, and what is within the margin gets its
//            binary64 distance.
// Fast scores are binary32.  Every decision they cannot settle within twice their rounding-error bound (membership of
// the beam, the final argmin) is taken on binary64 distances accumulated in index order (the residual carried through
// the codebooks in order), so the result is the argmin of (distance, tuple) over the pool exactly as defined.
// What bounds it: issue slots and shared memory, busy two thirds of the time, and between them the dependences of one target's
// chain (sort, minima over eight lanes, acceptance), which six to eight warps per scheduler do not hide.  A step of an
// 11008 x 4096 layer, k = 56 360, two / three fp16 codebooks of 256: 151 / 227 us, of which the search is 58 / 140 (four
// codebooks 223 by itself).  Stage 1 in two halves on one scale for the four targets, with a margin for residuals: 155 / 229
// and 62 / 140 (232); where one target in four is 1024 times larger than the others 76 instead of 58, with 2^20 times 1811
// instead of 787 (a stage 1 in binary32, one target after the other, 72 and 802).  When a step was 160.5 / 233.4: with stage 1
// of fp16 codebooks one target after the other on the FP32 pipe 169.3 / 236.1; with the binary64 decisions of choose_exact
// inlined 160.4 / 238.2 (spills).  Before all that, a warp per target, with two passes over all extensions in every stage and
// every decision in binary64: 415 / 522 us for three / four codebooks by themselves, 992 us for three of binary32.
#include <cuda_fp16.h>

#include "pvt_internal.h"

namespace pvt {

// header + the image of the codebooks (at most four binary32 codebooks: under 76 KiB)
size_t encode_beam_workspace_bytes() { return kWsHeaderBytes + 77824; }

namespace {

constexpr int kBsThreads = 256;
constexpr int kBsK = 256;  // codebooks are padded to this many codewords
constexpr float kPadHalfNorm = 3.0e38f;
constexpr float kInf = __builtin_huge_valf();
constexpr int kBsWarps = kBsThreads / 32;
// Resident CTAs per SM the kernel is compiled for (registers) and launched as: four for two fp16 codebooks (563609 / 56360 /
// 32768 targets 469 / 58.1 / 42.1 us, with three 487 / 59.8 / 43.3; 20011, where a warp has one group or two, 31.0 and 29.1;
// two of binary32 106 and 105), three otherwise (three / four fp16 codebooks 140 / 223 us, with four 142 / 234: spills).
constexpr int beam_ctas_per_sm(int M, bool tc) { return M == 2 && tc ? 4 : 3; }
constexpr int kBsGroup = 4;      // targets per warp iteration: 4 targets x 8 kept tuples = 32 lanes
constexpr int kBsList = 32;      // extensions per target that a middle stage's list holds
constexpr long long kInfBits = 0x7ff0000000000000ll;

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

// The fast scores ||r - c||^2/2 of 32 residuals, the lane's in r[lane], against a codebook: the lane's minimum of each of
// eight cells of 32 adjacent codewords (rho = ||r||^2/2 of its residual; infinity where it is not active).  Returns what the
// halves add to the margin of a score.
// The margins take a sum of the tensor pipe to be off by no more than 26 u (||r|| + ||c||)^2, u = 2^-24.  How the tensor cores
// add is not documented, so that this is an assumption; the largest errors against binary64 were 3.5 to 7.1 u of ||c||^2/2 +
// ||r|| ||c|| over 4 million scores each of vectors as the layers have them, 16 times larger and smaller, and of mixed sizes.
__device__ __forceinline__ float tensor_minima(const TensorStage& st, const float (*wr)[8], float (*wmin)[8], float rho,
                                               bool active, float smax, float (&sub_min)[8]) {
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
      const uint32_t b = st.b[nt][lane];
      const float2 h = *reinterpret_cast<const float2*>(&st.h[8 * nt + 2 * qd]);
      float d0[4], d1[4];
      mma_16x8x16(d0, a[0], b, b, h.x * sc, h.y * sc);
      mma_16x8x16(d1, a[1], b, b, h.x * sc, h.y * sc);
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

struct BeamParams {
  const float* W;
  const float* g;
  const float* scale;
  const uint32_t* idx;
  uint64_t k, G;
  FastDiv gpr;
  float eta;
  const void* books;
  uint32_t K, beam;
  uint8_t* codes;  // M adjacent bytes per group
  WeightsOut out;
  float* err_out;
  uint32_t* status;
};

// Everything the kernel derives from the codebooks, in the byte order it has in shared memory.  One small kernel writes
// it once per call into the workspace; every CTA of the search fetches it with a single bulk copy (cp.async.bulk,
// completion on an mbarrier; no multicast).
// The first codebook.  A cell of stage 1 is four adjacent codewords, what one thread sees of a target in two tiles; cell
// 8 g + c, codeword x of it (0..3) is row g + 8 (x % 2) of tile 2 c + x / 2.
template <bool TC>
struct FirstImage;
template <>
struct FirstImage<true> {  // tensor pipe: A fragments, [tile][lane] = halves (c[row][2 (lane%4)], [.. + 1]), rows lane/4, + 8
  uint2 a[kBsK / 16][32];
  float2 h2[kBsK / 16][8];  // ||c||^2/2 of rows g, g + 8
  float h[kBsK];            // the same by codeword
};
template <>
struct FirstImage<false> {  // FP32 pipe
  uint64_t p1[4][8][32];  // (c1[l+64q][i], c1[l+64q+32][i])
  uint64_t h1[4][32];     // (||c1||^2/2) pairs in the same order
};
template <bool TC>
struct StageImage;
template <>
struct StageImage<true> : TensorStage {};
template <>
struct StageImage<false> {  // FP32 pipe
  alignas(16) float x[kBsK / 2][16];  // pair p holds (c[2p][0], c[2p+1][0], c[2p][1], ...)
  alignas(8) float h[kBsK];           // ||c||^2/2 (in pairs, too)
};
template <int M, bool TC>
struct BeamImage {
  alignas(16) float c[M][kBsK][8];
  alignas(16) FirstImage<TC> first;
  StageImage<TC> st[M - 1];
  float smax[4];                      // largest norm per codebook
};

struct BeamScratch {  // per warp
  alignas(16) float r[32][8];                  // residuals, one per lane
  union {
    alignas(16) float wmin[32][8];             // cell minima on their way to the lanes that own the residuals
    alignas(8) uint2 list[kBsGroup][kBsList];  // a middle stage's extensions within the margin: score bits, tuple
  };
  alignas(16) float t[kBsGroup][8];            // the targets of the group
  alignas(16) uint32_t kept[kBsGroup][8];      // their kept tuples: code of codebook q in bits [31 - 8 q : 24 - 8 q]
  uint8_t cells[kBsGroup][64];                 // stage 1: a target's cells within the margin
};
template <int M, bool TC, bool WRITE>
struct BeamSmem {
  BeamImage<M, TC> img;
  BeamScratch w[kBsWarps];
  float scale[WRITE ? kBsWarps : 1][kBsGroup];  // of the targets' rows
  alignas(8) uint64_t img_bar;  // completion of the image copy
};

__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
// the same with the roles exchanged, rows = codewords, columns = targets: both K halves of A are the codeword; C = 0
__device__ __forceinline__ void mma_codeword_rows(float (&d)[4], uint2 a, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %4, %5}, {%6, %7}, "
      "{%8, %8, %8, %8};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a.x), "r"(a.y), "r"(b0), "r"(b1), "f"(0.0f));
}
// largest magnitude; not a number if one of them is not
__device__ __forceinline__ float max_abs3(float a, float b, float c) {
  float d;
  asm("max.NaN.abs.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  return (uint64_t)__float_as_uint(lo) | ((uint64_t)__float_as_uint(hi) << 32);
}
__device__ __forceinline__ float lo_of(uint64_t v) { return __uint_as_float((uint32_t)v); }
__device__ __forceinline__ float hi_of(uint64_t v) { return __uint_as_float((uint32_t)(v >> 32)); }
// order-preserving map binary32 -> u32
__device__ __forceinline__ uint32_t ord(float f) {
  const uint32_t b = __float_as_uint(f);
  return b ^ ((b >> 31) ? 0xffffffffu : 0x80000000u);
}
__device__ __forceinline__ float unord(uint32_t o) {
  return __uint_as_float(o ^ ((o >> 31) ? 0x80000000u : 0xffffffffu));
}

// ||t - c_1 - ... - c_n||^2 in binary64: the residual through the codebooks in order, the terms in element order;
// code q of the tuple sits in bits [31 - 8 q : 24 - 8 q]
template <int N>
__device__ __forceinline__ double exact_tuple(const float* t, const float (*books)[kBsK][8], uint32_t key) {
  double d = 0.0;
#pragma unroll
  for (int half = 0; half < 2; ++half) {
    const float4 tt = *reinterpret_cast<const float4*>(t + 4 * half);
    double e0 = (double)tt.x, e1 = (double)tt.y, e2 = (double)tt.z, e3 = (double)tt.w;
#pragma unroll
    for (int m = 0; m < N; ++m) {
      const float4 c = *reinterpret_cast<const float4*>(&books[m][(key >> (24 - 8 * m)) & 0xffu][4 * half]);
      e0 = __dsub_rn(e0, (double)c.x);
      e1 = __dsub_rn(e1, (double)c.y);
      e2 = __dsub_rn(e2, (double)c.z);
      e3 = __dsub_rn(e3, (double)c.w);
    }
    d = __dadd_rn(d, __dmul_rn(e0, e0));
    d = __dadd_rn(d, __dmul_rn(e1, e1));
    d = __dadd_rn(d, __dmul_rn(e2, e2));
    d = __dadd_rn(d, __dmul_rn(e3, e3));
  }
  return d;
}
// the same for the first n codes of a tuple (rarely needed: not inlined)
__device__ __noinline__ double exact_partial(const float* t, const float (*books)[kBsK][8], uint32_t key, int n) {
  double d = 0.0;
#pragma unroll 1
  for (int i = 0; i < 8; ++i) {
    double e = (double)t[i];
#pragma unroll 1
    for (int m = 0; m < n; ++m) e = __dsub_rn(e, (double)books[m][(key >> (24 - 8 * m)) & 0xffu][i]);
    d = __dadd_rn(d, __dmul_rn(e, e));
  }
  return d;
}
// ||t - c||^2 in binary64, the operations of the definition in index order
__device__ __forceinline__ double exact1(const float* t, const float* c) {
  double d = 0.0;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const double e = __dsub_rn((double)t[i], (double)c[i]);
    d = __dadd_rn(d, __dmul_rn(e, e));
  }
  return d;
}

// ---- PTX helpers of the image copy ----------------------------------------------------------------------------
constexpr uint32_t kBsMaxSpins = 1u << 22;  // polls after which the wait for the image gives up
__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ bool mbar_try_wait0(uint32_t bar) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar)
      : "memory");
  return ok != 0;
}
// One bulk copy global -> shared of the whole image (16-byte aligned on both sides, a multiple of 16 bytes),
// issued by one thread; every thread then waits, a bounded number of polls, for its completion.  Returns false
// (after recording PVT_DEV_WAIT_EXPIRED) if the copy has not landed by then: the CTA must leave without reading it.
__device__ __forceinline__ bool fetch_image(void* dst, const void* src, uint32_t bytes, uint64_t* bar, uint32_t* status) {
  const uint32_t b = smem_addr(bar);
  if (threadIdx.x == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(b));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(b), "r"(bytes) : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_addr(dst)),
                 "l"(src), "r"(bytes), "r"(b)
                 : "memory");
  }
  __syncthreads();  // the barrier is initialised before anybody polls it
  bool ok = false;
  for (uint32_t spin = 0; spin < kBsMaxSpins && !ok; ++spin) {
    ok = mbar_try_wait0(b);
    if (!ok && spin > 4096) __nanosleep(64);
  }
  if (!ok) atomicOr(status, PVT_DEV_WAIT_EXPIRED);
  // everybody agrees (a thread that gave up makes the whole CTA leave)
  return __syncthreads_and(ok) != 0;
}

// ---- the codebook image: a block per codebook, a codeword per thread (K <= 256 = block size); a trip to memory, a few
// stores (one block for all codebooks, an element per load: a step of 11008x4096 with two / three of them 2.1 / 4.0 us more)
template <int M, bool TC>
__global__ void __launch_bounds__(kBsThreads) beam_image_kernel(const BeamParams p, BeamImage<M, TC>* img) {
  __shared__ float red[kBsWarps];
  pdl_trigger();
  pdl_wait();
  BeamImage<M, TC>& sm = *img;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, m = blockIdx.x;
  const bool real = (uint32_t)tid < p.K;
  alignas(16) uint32_t raw[TC ? 4 : 8] = {};  // the codeword as it lies in memory
  if (real) {
    const uint4* from = reinterpret_cast<const uint4*>(p.books) + ((size_t)m * p.K + tid) * (TC ? 1 : 2);
#pragma unroll
    for (int i = 0; i < (TC ? 1 : 2); ++i) reinterpret_cast<uint4*>(raw)[i] = from[i];
  }
  float c[8], n2 = 0.0f;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    if (TC) {
      const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&raw[i / 2]));
      c[i] = i & 1 ? f.y : f.x;
    } else {
      c[i] = __uint_as_float(raw[i % (TC ? 4 : 8)]);
    }
    n2 = __fmaf_rn(c[i], c[i], n2);
  }
  reinterpret_cast<float4*>(&sm.c[m][tid][0])[0] = make_float4(c[0], c[1], c[2], c[3]);
  reinterpret_cast<float4*>(&sm.c[m][tid][0])[1] = make_float4(c[4], c[5], c[6], c[7]);
  const float h = real ? 0.5f * n2 : kPadHalfNorm;
  if (m == 0) {
    if constexpr (TC) {
      const int cell = tid >> 2, x = tid & 3, row = cell >> 3, tile = 2 * (cell & 7) + (x >> 1), lower = x & 1;
#pragma unroll
      for (int qq = 0; qq < 4; ++qq) reinterpret_cast<uint32_t*>(&sm.first.a[tile][4 * row + qq])[lower] = raw[qq];
      reinterpret_cast<float*>(&sm.first.h2[tile][row])[lower] = h;
      sm.first.h[tid] = h;
    } else {
      // codeword tid = l + 32*jj, jj = 2q + half
      const int jj = tid >> 5, q = jj >> 1, half = jj & 1;
      float* p1f = reinterpret_cast<float*>(&sm.first.p1[0][0][0]);
#pragma unroll
      for (int i = 0; i < 8; ++i) p1f[(((q * 8 + i) * 32) + lane) * 2 + half] = c[i];
      reinterpret_cast<float*>(&sm.first.h1[0][0])[(q * 32 + lane) * 2 + half] = h;
    }
  } else {
    StageImage<TC>& st = sm.st[m - 1];
    if constexpr (TC) {
      const int at = stage_column(tid);
      *reinterpret_cast<uint4*>(&st.b[at >> 3][4 * (at & 7)]) = make_uint4(raw[0], raw[1], raw[2], raw[3]);
      st.h[at] = h;
    } else {
#pragma unroll
      for (int i = 0; i < 8; ++i) st.x[tid >> 1][2 * i + (tid & 1)] = c[i];
      st.h[tid] = h;
    }
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) n2 = fmaxf(n2, __shfl_xor_sync(0xffffffffu, n2, o));
  if (lane == 0) red[warp] = n2;
  __syncthreads();
  if (tid == 0) {
    float a = 0.0f;
    for (int w = 0; w < kBsWarps; ++w) a = fmaxf(a, red[w]);
    sm.smax[m] = sqrtf(a);
  }
}

// compare-exchange network of eight keys (19 exchanges), of four (5)
#define PVT_CE(a, b)                          \
  {                                           \
    const uint32_t lo_ = min(key[a], key[b]); \
    key[b] = max(key[a], key[b]);             \
    key[a] = lo_;                             \
  }
__device__ __forceinline__ void sort8(uint32_t (&key)[8]) {
  PVT_CE(0, 2) PVT_CE(1, 3) PVT_CE(4, 6) PVT_CE(5, 7)
  PVT_CE(0, 4) PVT_CE(1, 5) PVT_CE(2, 6) PVT_CE(3, 7)
  PVT_CE(0, 1) PVT_CE(2, 3) PVT_CE(4, 5) PVT_CE(6, 7)
  PVT_CE(2, 4) PVT_CE(3, 5)
  PVT_CE(1, 4) PVT_CE(3, 6)
  PVT_CE(1, 2) PVT_CE(3, 4) PVT_CE(5, 6)
}
__device__ __forceinline__ void sort4(uint32_t (&key)[4]) {
  PVT_CE(0, 1) PVT_CE(2, 3) PVT_CE(0, 2) PVT_CE(1, 3) PVT_CE(1, 2)
}
#undef PVT_CE
// The eight lanes of a target: adjacent ones (S = 1, lane = 8 target + member), or every fourth (S = 4, lane = target +
// 4 member: as the tensor pipe leaves stage 1).  Minimum over them:
template <int S = 1>
__device__ __forceinline__ uint32_t team_min(uint32_t v) {
#pragma unroll
  for (int o = S; o < 8 * S; o <<= 1) v = min(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
// of a warp-wide ballot, the target's bits; and those of its members before this one
template <int S>
__device__ __forceinline__ uint32_t team_bits(uint32_t ballot) {
  const uint32_t lane = threadIdx.x & 31;
  return S == 1 ? (ballot >> (lane & 24u)) & 0xffu : (ballot >> (lane & 3u)) & 0x11111111u;
}
template <int S>
__device__ __forceinline__ uint32_t bits_before(uint32_t bits) {
  const uint32_t lane = threadIdx.x & 31;
  return bits & ((1u << (S == 1 ? lane & 7u : lane & 28u)) - 1u);
}
// drops the head of the sorted list if it is `head` (keys are distinct where they matter)
template <int N>
__device__ __forceinline__ void pop_if(uint32_t (&key)[N], uint32_t head) {
  const bool own = key[0] == head;
#pragma unroll
  for (int i = 0; i < N - 1; ++i) key[i] = own ? key[i + 1] : key[i];
  key[N - 1] = own ? 0xffffffffu : key[N - 1];
}
// lexicographic minimum of (distance, tuple) over the eight lanes of a target
template <int S = 1>
__device__ __forceinline__ void team_min_exact(double& d, uint32_t& key) {
#pragma unroll
  for (int o = S; o < 8 * S; o <<= 1) {
    const double od = __shfl_xor_sync(0xffffffffu, d, o);
    const uint32_t ok = __shfl_xor_sync(0xffffffffu, key, o);
    if (od < d || (od == d && ok < key)) {
      d = od;
      key = ok;
    }
  }
}

// The `keep` smallest of a target's extensions under (binary64 distance, tuple), the one of member `b`: of the n_list listed
// ones (unsure), or of all (more than the list holds).  Seldom needed: not inlined.
template <int S>
__device__ __noinline__ uint32_t choose_exact(const uint2* list, uint32_t n_list, uint32_t b, uint32_t keep, bool unsure,
                                              bool all, const float* t, const float (*books)[kBsK][8], int codes,
                                              const uint32_t* kept, uint32_t before, uint32_t K) {
  constexpr uint32_t kFull = 0xffffffffu;
  uint32_t next = 0;
  if (__any_sync(kFull, unsure)) {
    double ed[4];
    uint32_t ek[4];
#pragma unroll 1
    for (int i = 0; i < 4; ++i) {
      const uint32_t at = 8 * i + b;
      ek[i] = at < n_list ? list[at].y : kFull;
      ed[i] = unsure && ek[i] != kFull ? exact_partial(t, books, ek[i], codes) : __longlong_as_double(kInfBits);
    }
    for (uint32_t r = 0; r < keep; ++r) {
      double d = ed[0];
      uint32_t k = ek[0];
      for (int i = 1; i < 4; ++i)
        if (ed[i] < d || (ed[i] == d && ek[i] < k)) d = ed[i], k = ek[i];
      team_min_exact<S>(d, k);
      if (unsure && b == r) next = k;
      for (int i = 0; i < 4; ++i)
        if (ek[i] == k) ed[i] = __longlong_as_double(kInfBits), ek[i] = kFull;
    }
  }
  if (__any_sync(kFull, all)) {
    double ld = -1.0;  // the (distance, tuple) taken last
    uint32_t lk = 0;
    for (uint32_t r = 0; r < keep; ++r) {
      double d = __longlong_as_double(kInfBits);
      uint32_t k = kFull;
      for (uint32_t e = b; e < before * K; e += 8) {
        if (!all) break;
        const uint32_t key2 = (codes > 1 ? kept[e / K] : 0u) | ((e % K) << (32 - 8 * codes));
        const double x = exact_partial(t, books, key2, codes);
        const bool later = x > ld || (x == ld && (key2 > lk || r == 0));
        if (later && (x < d || (x == d && key2 < k))) d = x, k = key2;
      }
      __syncwarp();
      team_min_exact<S>(d, k);
      if (all && b == r) next = k;
      ld = d;
      lk = k;
    }
  }
  return next;
}
// The `keep` smallest of a target's listed extensions under (score, tuple), n_list of them (more than kBsList: the list is
// not complete): the one of member `b`.  Scores decide where exactly `keep` lie within the margin, otherwise binary64.
// `before` tuples were kept before the stage; with its codeword a tuple has `codes` codes.
template <int S>
__device__ __forceinline__ uint32_t choose_kept(const uint2* list, uint32_t n_list, uint32_t b, uint32_t keep, float margin,
                                                bool target, const float* t, const float (*books)[kBsK][8], int codes,
                                                const uint32_t* kept, uint32_t before, uint32_t K) {
  constexpr uint32_t kFull = 0xffffffffu;
  // eight lanes per target, up to four entries each
  float es[4];
  uint32_t key[4];
  const bool all = n_list > (uint32_t)kBsList;  // many equal extensions: every one of them gets its distance
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint32_t at = 8 * i + b;
    const bool have = at < n_list && !all;
    es[i] = have ? __uint_as_float(list[at].x) : kInf;
    key[i] = have ? (ord(es[i]) & ~31u) | at : kFull;
  }
  sort4(key);
  uint32_t pick = kFull, last = 0;  // the list entry that becomes kept tuple b
  for (uint32_t r = 0; r < keep; ++r) {
    last = team_min<S>(key[0]);
    if (b == r) pick = last & 31u;
    pop_if(key, last);
  }
  // exactly `keep` entries up to the last one's bucket plus the margin: provably the exact ones
  const float sure = unord(last | 31u) + margin;
  uint32_t near = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) near += es[i] <= sure && 8 * i + b < n_list;
#pragma unroll
  for (int o = S; o < 8 * S; o <<= 1) near += __shfl_xor_sync(kFull, near, o);
  uint32_t next = b < keep && pick < n_list ? list[pick].y : 0u;
  const bool unsure = target && !all && near != keep;
  if (__any_sync(kFull, unsure || (target && all))) {
    const uint32_t exact = choose_exact<S>(list, n_list, b, keep, unsure, target && all, t, books, codes, kept, before, K);
    if (unsure || (target && all)) next = exact;
  }
  return next;
}
// A limit that the list of more extensions than it holds (one target in fifty) is collected again with: the keep-th
// smallest of those it holds, plus the margin.  Equal scores in that number are left to choose_kept.
template <int S>
__device__ __forceinline__ float lower_limit(const uint2* list, bool over, uint32_t b, uint32_t keep, float margin) {
  uint32_t key[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) key[i] = over ? (ord(__uint_as_float(list[8 * i + b].x)) & ~31u) | (8 * i + b) : 0xffffffffu;
  sort4(key);
  uint32_t last = 0;
  for (uint32_t r = 0; r < keep; ++r) {
    last = team_min<S>(key[0]);
    pop_if(key, last);
  }
  return unord(last | 31u) + margin;
}
// The limit up to which fast scores matter: the keep-th smallest of a target's 64 cell minima (keep different extensions
// score no more than that), plus the margin; without a limit if there are fewer cells, or padding among them
template <int S>
__device__ __forceinline__ float kept_limit(const float (&cell_min)[8], uint32_t b, uint32_t keep, float margin) {
  uint32_t key[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) key[c] = (ord(cell_min[c]) & ~63u) | (b * 8 + c);
  sort8(key);
  uint32_t last = 0;
  for (uint32_t r = 0; r < keep; ++r) {
    last = team_min<S>(key[0]);
    pop_if(key, last);
  }
  return last >= ord(1.0e38f) ? kInf : unord(last | 63u) + margin;
}

// One further stage's fast scores for the lane's residual (target my_q, kept tuple my_b; rho = ||r||^2/2): the minimum
// of each of eight cells of 32 codewords.  The residuals of all lanes are in w.r.  Returns what the tensor path adds to the
// margin.
template <bool TC>
__device__ __forceinline__ float stage_minima(const StageImage<TC>& st, BeamScratch& w, const float (&r)[8], float rho,
                                              bool active, float smax, float (&sub_min)[8]) {
  if constexpr (TC) {
    return tensor_minima(st, w.r, w.wmin, rho, active, smax, sub_min);
  } else {
    uint64_t nrd[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) nrd[i] = pack2(-r[i], -r[i]);
    const uint64_t rho2 = pack2(rho, rho);
#pragma unroll
    for (int sub = 0; sub < 8; ++sub) {
      float cmin = kInf;
      const ulonglong2* vals = reinterpret_cast<const ulonglong2*>(&st.x[0][0]) + sub * 16 * 4;
      const uint64_t* norms = reinterpret_cast<const uint64_t*>(&st.h[0]) + sub * 16;
#pragma unroll 4
      for (int pr = 0; pr < 16; ++pr) {
        const ulonglong2 q0 = vals[4 * pr], q1 = vals[4 * pr + 1], q2 = vals[4 * pr + 2], q3 = vals[4 * pr + 3];
        uint64_t acc = add2(norms[pr], rho2);
        acc = fma2(nrd[0], q0.x, acc);
        acc = fma2(nrd[1], q0.y, acc);
        acc = fma2(nrd[2], q1.x, acc);
        acc = fma2(nrd[3], q1.y, acc);
        acc = fma2(nrd[4], q2.x, acc);
        acc = fma2(nrd[5], q2.y, acc);
        acc = fma2(nrd[6], q3.x, acc);
        acc = fma2(nrd[7], q3.y, acc);
        cmin = min3(cmin, lo_of(acc), hi_of(acc));
      }
      sub_min[sub] = active ? cmin : kInf;
    }
    return 0.0f;
  }
}

// The target's 64 (kept tuple, cell) flags from its lanes' eight: byte b belongs to kept tuple b.
__device__ __forceinline__ uint64_t team_flags(uint32_t mine, uint32_t my_b) {
  uint32_t lo = my_b < 4 ? mine << (8 * my_b) : 0u, hi = my_b >= 4 ? mine << (8 * (my_b - 4)) : 0u;
#pragma unroll
  for (int o = 1; o < 8; o <<= 1) {
    lo |= __shfl_xor_sync(0xffffffffu, lo, o);
    hi |= __shfl_xor_sync(0xffffffffu, hi, o);
  }
  return ((uint64_t)hi << 32) | lo;
}

// WRITE: the weights of the re-encoded groups are written as well.
template <int M, bool TC, bool WRITE>
__global__ void __launch_bounds__(kBsThreads, beam_ctas_per_sm(M, TC)) encode_beam_kernel(const BeamParams p,
                                                                               const BeamImage<M, TC>* image) {
  extern __shared__ __align__(16) unsigned char beam_smem[];
  BeamSmem<M, TC, WRITE>& smem = *reinterpret_cast<BeamSmem<M, TC, WRITE>*>(beam_smem);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  pdl_trigger();
  pdl_wait();
  if (!fetch_image(&smem.img, image, (uint32_t)sizeof(BeamImage<M, TC>), &smem.img_bar, p.status)) return;
  const BeamImage<M, TC>& sm = smem.img;
  BeamScratch& w = smem.w[warp];
  const float s1max = sm.smax[0];
  float sall_books = 0.0f;
#pragma unroll
  for (int m = 0; m < M; ++m) sall_books += sm.smax[m];

  const uint64_t nwarps = (uint64_t)gridDim.x * kBsWarps;
  const uint64_t n_groups = (p.k + kBsGroup - 1) / kBsGroup;
  const uint32_t my_q = (uint32_t)lane >> 3, my_b = (uint32_t)lane & 7u;
  constexpr uint32_t kFull = 0xffffffffu;

  for (uint64_t gi = (uint64_t)blockIdx.x * kBsWarps + warp; gi < n_groups; gi += nwarps) {
    uint32_t B = p.beam < p.K ? p.beam : p.K;  // tuples kept after the stage
    // what this lane needs of its own target (target my_q of the group)
    uint32_t my_j = kFull, my_prev = 0;
    float my_sall = 0.0f;

    // the four targets of the group, one element per lane (lane = 8 * target + element): index, W, g, row scale
    // and previous tuple are fetched for all four at once, one fma and one division per lane (binary32)
    uint32_t lane_j = kFull, lane_prev = 0;
    {
      const uint64_t n_mine = gi * kBsGroup + my_q;
      if (n_mine < p.k) lane_j = p.idx[n_mine];
      float tv = 0.0f;
      if (lane_j < p.G) {
        const float wv = p.W[(size_t)lane_j * 8 + my_b], gv = p.g[(size_t)lane_j * 8 + my_b];
        const float sc = p.scale[fast_div(lane_j, p.gpr)];
        if (M == 2) {
          const uint32_t both = reinterpret_cast<const uint16_t*>(p.codes)[lane_j];
          lane_prev = (both << 24) | ((both >> 8) << 16);
        } else {
#pragma unroll
          for (int m = 0; m < M; ++m) lane_prev |= (uint32_t)p.codes[(size_t)lane_j * M + m] << (24 - 8 * m);
        }
        tv = __fdiv_rn(__fmaf_rn(-p.eta, gv, wv), sc);
        if (WRITE && my_b == 0) smem.scale[warp][my_q] = sc;
      }
      w.t[my_q][my_b] = tv;
    }
    __syncwarp();

    if constexpr (TC) {
      // ---- stage 1 on the tensor pipe, the four targets side by side: lane = target q + 4 part.  The columns of B are the
      // targets, split in three halves, which keep every bit: [ -hi | 0 ] in an even column, [ -mid | -lo ] in the next, each
      // target on a scale of its own.  A thread gets both sums of one target and adds the codeword's half norm.
      const uint32_t q = (uint32_t)lane & 3u, part = (uint32_t)lane >> 2;
      const uint64_t n = gi * kBsGroup + q;
      const uint32_t j = __shfl_sync(kFull, lane_j, 8 * q);
      const bool target = j < p.G;
      if (n < p.k && !target && part == 0) atomicOr(p.status, PVT_DEV_BAD_INDEX);
      const float* tq = &w.t[q][0];
      float sr[8], tnorm, top;
      {
        const float4 ta = *reinterpret_cast<const float4*>(tq), tb = *reinterpret_cast<const float4*>(tq + 4);
        sr[0] = ta.x, sr[1] = ta.y, sr[2] = ta.z, sr[3] = ta.w, sr[4] = tb.x, sr[5] = tb.y, sr[6] = tb.z, sr[7] = tb.w;
        float nt2 = 0.0f;
#pragma unroll
        for (int i = 0; i < 8; ++i) nt2 = fmaf(sr[i], sr[i], nt2);
        tnorm = sqrtf(nt2);
        top = max_abs3(max_abs3(sr[0], sr[1], sr[2]), max_abs3(sr[3], sr[4], sr[5]), max_abs3(sr[6], sr[7], sr[7]));
      }
      const bool search = target && top < kInf;  // (no codeword is near a target that is not finite)
      my_j = lane_j < p.G ? lane_j : kFull;
      my_prev = lane_prev;
      my_sall = __shfl_sync(kFull, tnorm, my_q) + sall_books;
      float sc, inv, cell_min[8];
      half_scale(__float_as_uint(top), sc, inv);
      {
        const uint32_t column = part >> 1;  // the target of this lane's column
        const float2 x = *reinterpret_cast<const float2*>(&w.t[column][2 * q]);
        const float neg = -__shfl_sync(kFull, sc, column);
        uint32_t hi, mid, lo;
        split_three_halves(x.x * neg, x.y * neg, hi, mid, lo);
        const uint32_t b0 = part & 1u ? mid : hi, b1 = part & 1u ? lo : 0u;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          float d0[4], d1[4];
          const float2 h0 = sm.first.h2[2 * c][part], h1 = sm.first.h2[2 * c + 1][part];
          mma_codeword_rows(d0, sm.first.a[2 * c][lane], b0, b1);
          mma_codeword_rows(d1, sm.first.a[2 * c + 1][lane], b0, b1);
          const float s0 = __fmaf_rn(d0[0], inv, __fmaf_rn(d0[1], inv, h0.x));
          const float s1 = __fmaf_rn(d0[2], inv, __fmaf_rn(d0[3], inv, h0.y));
          const float s2 = __fmaf_rn(d1[0], inv, __fmaf_rn(d1[1], inv, h1.x));
          const float s3 = __fmaf_rn(d1[2], inv, __fmaf_rn(d1[3], inv, h1.y));
          cell_min[c] = target ? min3(fminf(s0, s1), s2, s3) : kInf;
        }
      }
      // Twice the rounding-error bound of a fast score with a factor 2 to spare, as for binary32 below; then what binary64
      // distances, which decide, are off (2^-53 of at most twelve terms of (||t|| + ||c||)^2; it counts for targets 2^18
      // times larger than codewords), and what subnormal halves are.  How the tensor cores add is not documented: that these
      // sums are off by no more than a chain of fused multiply-adds in binary32 (16.1 u (||c||^2/2 + ||t|| ||c||), u = 2^-24)
      // is an assumption.  What supports it: over 4 million scores each of targets and codewords as the layers have them,
      // targets 16 times larger and smaller, one of four 1024 times larger, targets next to codewords, elements and codewords
      // of mixed sizes, the largest errors against binary64 were 2.5 to 5.1 u of that sum of magnitudes (the chain: 3.6 to
      // 8.3), their root mean squares 0.30 to 0.94 u (0.31 to 1.32), the chain's larger in each.  (Two halves, on one
      // scale for the four targets: up to 2000 u beside the larger one; 1.7 times the chain's root mean square for targets 16
      // times larger.)
      const float reach = tnorm + s1max;
      const float margin = 3.8146973e-6f /* 2^-18 */ * (0.5f * s1max * s1max + tnorm * s1max) +
                           (3.5527137e-15f /* 2^-48 */ * reach) * reach +
                           4.76837158203125e-7f /* 2^-21 */ * inv * s1max + 1e-30f;
      // Scores and margin of a target of large elements (from 2^64 on the margin) may be infinite and the limit then not a
      // number: what is not above the limit is within it, so that binary64 decides between all codewords.
      float limit = kept_limit<4>(cell_min, part, B, margin);
      uint32_t n_list = 0;  // the same in the target's eight lanes
#pragma unroll 1
      for (int pass = 0;; ++pass) {
        // the cells within the limit, eight at a time, one per lane, four codewords each
        uint32_t hits = 0;
#pragma unroll
        for (int c = 0; c < 8; ++c) hits |= search && !(cell_min[c] > limit) ? 1u << c : 0u;
        uint32_t at = __popc(hits), total;
        {
          const uint32_t mine = at;
#pragma unroll
          for (int o = 4; o < 32; o <<= 1) {
            const uint32_t up = __shfl_up_sync(kFull, at, o);
            if (lane >= o) at += up;
          }
          total = __shfl_sync(kFull, at, 28 + q);
          at -= mine;
        }
        for (uint32_t m = hits; m; m &= m - 1) w.cells[q][at++] = (uint8_t)(8 * part + __ffs(m) - 1);
        __syncwarp();
        n_list = 0;
        for (uint32_t base = 0; __any_sync(kFull, base < total); base += 8) {
          const bool work = base + part < total;
          const uint32_t cell = work ? w.cells[q][base + part] : 0u;
#pragma unroll
          for (uint32_t c = 0; c < 4; ++c) {
            const uint32_t k1 = 4 * cell + ((c + part) & 3u);  // (the lanes begin at different ones: fewer bank conflicts)
            const float4 ca = *reinterpret_cast<const float4*>(&sm.c[0][k1][0]);
            const float4 cb = *reinterpret_cast<const float4*>(&sm.c[0][k1][4]);
            const float cv[8] = {ca.x, ca.y, ca.z, ca.w, cb.x, cb.y, cb.z, cb.w};
            float s1 = sm.first.h[k1];
#pragma unroll
            for (int i = 0; i < 8; ++i) s1 = __fmaf_rn(-sr[i], cv[i], s1);
            const bool in = work && !(s1 > limit) && k1 < p.K;
            const uint32_t who = team_bits<4>(__ballot_sync(kFull, in));
            const uint32_t to = n_list + __popc(bits_before<4>(who));
            if (in && to < (uint32_t)kBsList) w.list[q][to] = make_uint2(__float_as_uint(s1), k1 << 24);
            n_list += __popc(who);
          }
        }
        __syncwarp();
        const bool over = n_list > (uint32_t)kBsList;
        if (pass == 3 || !__any_sync(kFull, over)) break;
        const float lower = lower_limit<4>(w.list[q], over, part, B, margin);
        const bool again = over && lower < limit;
        if (!__any_sync(kFull, again)) break;
        if (again) limit = lower;
        __syncwarp();
      }
      const uint32_t next = choose_kept<4>(w.list[q], n_list, part, B, margin, target, tq, sm.c, 1, nullptr, 1, p.K);
      if (target) w.kept[q][part] = next;
    } else {
      // ---- stage 1, one target after the other, the whole warp on each
#pragma unroll 1
      for (uint32_t q = 0; q < (uint32_t)kBsGroup; ++q) {
        const uint64_t n = gi * kBsGroup + q;
        if (n >= p.k) break;
        const uint32_t j = __shfl_sync(kFull, lane_j, 8 * q);
        const uint32_t prev = __shfl_sync(kFull, lane_prev, 8 * q);
        if (j >= p.G) {
          if (lane == 0) atomicOr(p.status, PVT_DEV_BAD_INDEX);
          continue;
        }
        float t[8];
        {
          const float4 ta = *reinterpret_cast<const float4*>(&w.t[q][0]);
          const float4 tb = *reinterpret_cast<const float4*>(&w.t[q][4]);
          t[0] = ta.x, t[1] = ta.y, t[2] = ta.z, t[3] = ta.w, t[4] = tb.x, t[5] = tb.y, t[6] = tb.z, t[7] = tb.w;
        }
        float nt2 = 0.0f;
#pragma unroll
        for (int i = 0; i < 8; ++i) nt2 = fmaf(t[i], t[i], nt2);
        const float tnorm = sqrtf(nt2);
        // twice the rounding-error bound of the fast score (factor >= 2 to spare), u = 2^-24:
        //   |score1_fl - score1| <= 16.1 u (||c1||^2/2 + ||t|| ||c1||)
        // and what binary64 distances, which decide, are off
        const float reach1 = tnorm + s1max;
        const float margin1 = 3.8146973e-6f /* 2^-18 */ * (0.5f * s1max * s1max + tnorm * s1max) +
                              (3.5527137e-15f /* 2^-48 */ * reach1) * reach1 + 1e-30f;

        // 256 scores, 8 per lane
        float f[8];
        {
          uint64_t acc[4];
#pragma unroll
          for (int qq = 0; qq < 4; ++qq) acc[qq] = sm.first.h1[qq][lane];
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const uint64_t ntd = pack2(-t[i], -t[i]);
#pragma unroll
            for (int qq = 0; qq < 4; ++qq) acc[qq] = fma2(ntd, sm.first.p1[qq][i][lane], acc[qq]);
          }
#pragma unroll
          for (int qq = 0; qq < 4; ++qq) {
            f[2 * qq] = lo_of(acc[qq]);
            f[2 * qq + 1] = hi_of(acc[qq]);
          }
        }
        // extract the B smallest (score truncated to 24 bits | code): a first guess of the beam.  Every lane sorts
        // its eight keys once; a round is then one warp minimum of the lanes' heads and a shift of the winning lane's list.
        uint32_t key[8];
#pragma unroll
        for (int jj = 0; jj < 8; ++jj) key[jj] = (ord(f[jj]) & 0xffffff00u) | (uint32_t)(lane + 32 * jj);
        sort8(key);
        uint32_t beam_code[8];
        uint32_t last = 0;  // the key extracted last
#pragma unroll
        for (int b = 0; b < 8; ++b) {
          beam_code[b] = 0;
          if ((uint32_t)b < B) {
            last = __reduce_min_sync(kFull, key[0]);
            beam_code[b] = last & 0xffu;
            pop_if(key, last);  // keys are distinct: they end in the code
          }
        }
        // is that guess provably the exact beam?  theta = an upper bound of the scores in the guess (the top of the
        // truncation bucket of the key extracted last); every member of the exact beam scores <= theta + margin1; if
        // exactly B codewords do, they are the guess and the exact beam at once.
        {
          uint32_t cnt = 0;
          const float theta = unord(last | 0xffu);
          const float limit1 = theta + margin1;
          uint32_t member = 0;
#pragma unroll
          for (int jj = 0; jj < 8; ++jj) {
            const bool in = f[jj] <= limit1 && (uint32_t)(lane + 32 * jj) < p.K;
            member |= in ? (1u << jj) : 0u;
            cnt += in;
          }
          cnt = __reduce_add_sync(kFull, cnt);
          if (cnt != B) {
            // undecided: order the shortlisted codewords by (binary64 distance, code)
            for (uint32_t b = 0; b < B; ++b) {
              double ld = __longlong_as_double(kInfBits);
              uint32_t lk = kFull;
#pragma unroll
              for (int jj = 0; jj < 8; ++jj) {
                if (member & (1u << jj)) {
                  const uint32_t kap = lane + 32 * jj;
                  const double d = exact1(t, sm.c[0][kap]);
                  if (d < ld || (d == ld && kap < lk)) {
                    ld = d;
                    lk = kap;
                  }
                }
              }
              // warp-wide lexicographic minimum of (ld, lk); distances are >= 0 so their bits order like u64
              const uint64_t bits = (uint64_t)__double_as_longlong(ld);
              const uint32_t hi = (uint32_t)(bits >> 32), lo = (uint32_t)bits;
              const uint32_t mhi = __reduce_min_sync(kFull, hi);
              const uint32_t mlo = __reduce_min_sync(kFull, hi == mhi ? lo : kFull);
              const uint32_t mk = __reduce_min_sync(kFull, (hi == mhi && lo == mlo) ? lk : kFull);
              const uint32_t chosen = mk < (uint32_t)kBsK ? mk : 0u;
#pragma unroll
              for (int bb = 0; bb < 8; ++bb)
                if ((uint32_t)bb == b) beam_code[bb] = chosen;
              if ((chosen & 31u) == (uint32_t)lane) member &= ~(1u << (chosen >> 5));
            }
          }
        }
        // hand the beam to the lanes of the further stages
        if (lane == 0) {
          *reinterpret_cast<uint4*>(&w.kept[q][0]) =
              make_uint4(beam_code[0] << 24, beam_code[1] << 24, beam_code[2] << 24, beam_code[3] << 24);
          *reinterpret_cast<uint4*>(&w.kept[q][4]) =
              make_uint4(beam_code[4] << 24, beam_code[5] << 24, beam_code[6] << 24, beam_code[7] << 24);
        }
        if (my_q == q) {
          my_j = j;
          my_prev = prev;
          my_sall = tnorm + sall_books;
        }
      }
    }
    __syncwarp();

    // ---- further stages: lane = (target my_q, kept tuple my_b)
    double bd = __longlong_as_double(kInfBits);  // the best extension of the last stage: distance and tuple
    uint32_t bk = kFull;
#pragma unroll
    for (int m = 1; m < M; ++m) {
      const bool active = my_j != kFull && my_b < B;
      const StageImage<TC>& st = sm.st[m - 1];
      float r[8], rho = 0.0f;
      {
        const float4 ta = *reinterpret_cast<const float4*>(&w.t[my_q][0]);
        const float4 tb = *reinterpret_cast<const float4*>(&w.t[my_q][4]);
        r[0] = ta.x, r[1] = ta.y, r[2] = ta.z, r[3] = ta.w, r[4] = tb.x, r[5] = tb.y, r[6] = tb.z, r[7] = tb.w;
        const uint32_t tuple = active ? w.kept[my_q][my_b] : 0u;  // (that of a skipped target was never written)
#pragma unroll
        for (int q = 0; q < m; ++q) {
          const float* c = &sm.c[q][(tuple >> (24 - 8 * q)) & 0xffu][0];
          const float4 ca = *reinterpret_cast<const float4*>(c), cb = *reinterpret_cast<const float4*>(c + 4);
          const float cv[8] = {ca.x, ca.y, ca.z, ca.w, cb.x, cb.y, cb.z, cb.w};
#pragma unroll
          for (int i = 0; i < 8; ++i) r[i] = __fsub_rn(r[i], cv[i]);
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          r[i] = active ? r[i] : 0.0f;
          rho = __fmaf_rn(r[i], r[i], rho);
        }
        rho = __fmul_rn(0.5f, rho);
        *reinterpret_cast<float4*>(&w.r[lane][0]) = make_float4(r[0], r[1], r[2], r[3]);
        *reinterpret_cast<float4*>(&w.r[lane][4]) = make_float4(r[4], r[5], r[6], r[7]);
      }
      __syncwarp();
      float sub_min[8];
      // twice the rounding-error bound of a fast score, with a factor 2 to spare (u = 2^-24; R = the target's largest
      // residual, C = the largest codeword, S = the target plus the largest codeword of every codebook): 26 u (R + C)^2
      // for its evaluation, (M - 1) u S (R + C) for the residual's own roundings
      float rho_max = rho;
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) rho_max = fmaxf(rho_max, __shfl_xor_sync(kFull, rho_max, o));
      const float reach = sqrtf(2.0f * rho_max) + sm.smax[m];
      const float margin = (7.6293945e-6f /* 2^-17 */ * reach + 9.5367432e-7f /* 2^-20 */ * my_sall) * reach + 1e-30f +
                           stage_minima<TC>(st, w, r, rho, active, sm.smax[m], sub_min);

      // the limit up to which fast scores matter: the smallest score, or the keep-th smallest cell minimum (keep
      // different extensions score no more than that), plus the margin
      const uint32_t keep = m == M - 1 ? 1u : (p.beam < B * p.K ? p.beam : B * p.K);
      float limit;
      if (m == M - 1) {
        float gmin = sub_min[0];
#pragma unroll
        for (int sub = 1; sub < 8; ++sub) gmin = fminf(gmin, sub_min[sub]);
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) gmin = fminf(gmin, __shfl_xor_sync(kFull, gmin, o));
        limit = gmin + margin;
      } else {
        limit = kept_limit<1>(sub_min, my_b, keep, margin);
      }
      auto flag_cells = [&]() {
        uint32_t hits = 0;
#pragma unroll
        for (int sub = 0; sub < 8; ++sub) hits |= (active && sub_min[sub] <= limit) ? (1u << sub) : 0u;
        return team_flags(hits, my_b);
      };
      uint64_t flags = flag_cells();
      uint32_t n_list = 0;  // the same in the target's eight lanes
      __syncwarp();         // the cell minima have been read: the list takes their place

      // Revisit the flagged cells one after the other, four codewords per lane, the four targets of the group side by
      // side.  (The fast score is evaluated again here, in another order: both evaluations lie within half the margin
      // of the true score, so what the definition selects passes both tests.)
#pragma unroll 1
      for (int pass = 0;; ++pass) {
        while (__any_sync(kFull, flags != 0)) {
          const bool work = flags != 0;
          const uint32_t pos = work ? (uint32_t)__ffsll((long long)flags) - 1u : 0u;
          flags &= flags - 1;
          const uint32_t hb = pos >> 3, hsub = pos & 7u;
          const uint32_t tuple = work ? w.kept[my_q][hb] : 0u;
          float sr[8], srho = 0.0f;
          {
            const float4 ra = *reinterpret_cast<const float4*>(&w.r[8 * my_q + hb][0]);
            const float4 rb = *reinterpret_cast<const float4*>(&w.r[8 * my_q + hb][4]);
            sr[0] = ra.x, sr[1] = ra.y, sr[2] = ra.z, sr[3] = ra.w, sr[4] = rb.x, sr[5] = rb.y, sr[6] = rb.z, sr[7] = rb.w;
          }
#pragma unroll
          for (int i = 0; i < 8; ++i) srho = __fmaf_rn(sr[i], sr[i], srho);
          srho = __fmul_rn(0.5f, srho);
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const uint32_t k2 = hsub * 32u + 8u * c + my_b;
            const float4 ca = *reinterpret_cast<const float4*>(&sm.c[m][k2][0]);
            const float4 cb = *reinterpret_cast<const float4*>(&sm.c[m][k2][4]);
            const float cv[8] = {ca.x, ca.y, ca.z, ca.w, cb.x, cb.y, cb.z, cb.w};
            float s2 = __fadd_rn(st.h[TC ? stage_column(k2) : k2], srho);
#pragma unroll
            for (int i = 0; i < 8; ++i) s2 = __fmaf_rn(-sr[i], cv[i], s2);
            const bool in = work && s2 <= limit && k2 < p.K;
            const uint32_t key = tuple | (k2 << (24 - 8 * m));
            if (m == M - 1) {
              if (in) {
                const double d = exact_tuple<M>(w.t[my_q], sm.c, key);
                if (d < bd || (d == bd && key < bk)) {
                  bd = d;
                  bk = key;
                }
              }
            } else {
              const uint32_t who = team_bits<1>(__ballot_sync(kFull, in));
              const uint32_t at = n_list + __popc(bits_before<1>(who));
              if (in && at < (uint32_t)kBsList) w.list[my_q][at] = make_uint2(__float_as_uint(s2), key);
              n_list += __popc(who);
            }
          }
        }
        if (m == M - 1) break;
        const bool over = n_list > (uint32_t)kBsList;
        if (pass == 3 || !__any_sync(kFull, over)) break;
        __syncwarp();
        const float lower = lower_limit<1>(w.list[my_q], over, my_b, keep, margin);
        const bool again = over && lower < limit;
        if (!__any_sync(kFull, again)) break;
        if (again) {
          limit = lower;
          n_list = 0;
        }
        flags = flag_cells();
        if (!again) flags = 0;
        __syncwarp();
      }
      if (m < M - 1) {
        __syncwarp();
        const bool target = my_j != kFull;
        const uint32_t next = choose_kept<1>(w.list[my_q], n_list, my_b, keep, margin, target, w.t[my_q], sm.c, m + 1,
                                             w.kept[my_q], B, p.K);
        __syncwarp();  // everybody has read the tuples that are replaced now
        if (target) w.kept[my_q][my_b] = next;
        B = keep;
        __syncwarp();
      }
    }
    if (my_b == 0 && my_j != kFull) {  // the previous tuple joins the pool
      bool ok = true;
#pragma unroll
      for (int m = 0; m < M; ++m) ok &= ((my_prev >> (24 - 8 * m)) & 0xffu) < p.K;
      if (ok) {
        const double d = exact_tuple<M>(w.t[my_q], sm.c, my_prev);
        if (d < bd || (d == bd && my_prev < bk)) {
          bd = d;
          bk = my_prev;
        }
      } else {
        atomicOr(p.status, PVT_DEV_BAD_CODE);
      }
    }
    __syncwarp();
    team_min_exact(bd, bk);
    // each lane an element of the group's weights, as dequantisation forms it
    if (WRITE && my_j != kFull && bd < __longlong_as_double(kInfBits)) {
      float v = sm.c[0][bk >> 24][my_b];
#pragma unroll
      for (int m = 1; m < M; ++m) v = __fadd_rn(v, sm.c[m][(bk >> (24 - 8 * m)) & 0xffu][my_b]);
      const float x = __fmul_rn(smem.scale[warp][my_q], v);
      if (p.out.f16)
        reinterpret_cast<__half*>(p.out.W_hat)[(size_t)my_j * 8 + my_b] = __float2half_rn(x);
      else
        reinterpret_cast<float*>(p.out.W_hat)[(size_t)my_j * 8 + my_b] = x;
    }
    if (my_b == 0 && my_j != kFull) {
      if (bd < __longlong_as_double(kInfBits)) {
        if (M == 2) {
          reinterpret_cast<uint16_t*>(p.codes)[my_j] = (uint16_t)((bk >> 24) | ((bk >> 8) & 0xff00u));
        } else {
#pragma unroll
          for (int m = 0; m < M; ++m) p.codes[(size_t)my_j * M + m] = (uint8_t)(bk >> (24 - 8 * m));
        }
        if (p.err_out) p.err_out[gi * kBsGroup + my_q] = (float)bd;
      } else {
        atomicOr(p.status, PVT_DEV_INTERNAL);  // non-finite target: no distance compares below infinity
      }
    }
    __syncwarp();  // the group's scratch is rewritten by the next iteration
  }
}

template <int M, bool TC, bool WRITE>
cudaError_t launch_beam(const BeamParams& p, unsigned char* image_at, int sm_count, cudaStream_t stream) {
  using Image = BeamImage<M, TC>;
  static_assert(sizeof(Image) % 16 == 0, "the bulk copy moves multiples of 16 bytes");
  static_assert(sizeof(Image) <= 77824, "the workspace reserves 76 KiB for the image");
  constexpr size_t smem = sizeof(BeamSmem<M, TC, WRITE>);
  cudaError_t err = allow_smem<encode_beam_kernel<M, TC, WRITE>>();
  if (err != cudaSuccess) return err;
  Image* image = reinterpret_cast<Image*>(image_at);
  timing_begin(kKernEncodeAux, stream);
  err = launch_dependent(beam_image_kernel<M, TC>, M, kBsThreads, 0, stream, p, image);
  timing_end(kKernEncodeAux, stream);
  if (err != cudaSuccess) return err;
  constexpr uint64_t fit = (228 * 1024) / (smem + 1024);
  constexpr uint64_t bound = beam_ctas_per_sm(M, TC), per_sm = fit < bound ? fit : bound;  // persistent: the resident CTAs
  const uint64_t groups = (p.k + kBsGroup - 1) / kBsGroup, want = (groups + kBsWarps - 1) / kBsWarps;
  const uint64_t most = per_sm * (uint64_t)sm_count;
  timing_begin(kKernEncodeMain, stream);
  err = launch_dependent(encode_beam_kernel<M, TC, WRITE>, (unsigned)(want < most ? want : most), kBsThreads, smem, stream, p,
                         (const Image*)image);
  count_launches(2);
  timing_end(kKernEncodeMain, stream);
  return err;
}

template <int M>
cudaError_t launch_type(const pvt_layer& L, const BeamParams& p, unsigned char* image, int sm_count, cudaStream_t stream) {
  if (L.codebook_dtype == PVT_F16)
    return p.out.W_hat ? launch_beam<M, true, true>(p, image, sm_count, stream)
                       : launch_beam<M, true, false>(p, image, sm_count, stream);
  return p.out.W_hat ? launch_beam<M, false, true>(p, image, sm_count, stream)
                     : launch_beam<M, false, false>(p, image, sm_count, stream);
}

}  // namespace

cudaError_t launch_encode_beam(const pvt_layer& L, uint64_t G, const uint32_t* idx, uint64_t k, float* err_out,
                             WeightsOut out, void* ws, int sm_count, cudaStream_t stream) {
  BeamParams p;
  p.W = L.W;
  p.g = L.g;
  p.scale = L.scale;
  p.idx = idx;
  p.k = k;
  p.G = G;
  p.gpr = make_fast_div((uint32_t)(L.cols / kGroupDim));
  p.eta = L.eta;
  p.books = L.codebooks;
  p.K = (uint32_t)L.codebook_size;
  p.beam = (uint32_t)L.beam;
  p.codes = static_cast<uint8_t*>(L.codes);
  p.out = out;
  p.err_out = err_out;
  p.status = static_cast<uint32_t*>(ws);
  unsigned char* image = static_cast<unsigned char*>(ws) + kWsHeaderBytes;
  switch (L.num_codebooks) {
    case 2: return launch_type<2>(L, p, image, sm_count, stream);
    case 3: return launch_type<3>(L, p, image, sm_count, stream);
    default: return launch_type<4>(L, p, image, sm_count, stream);
  }
}

}  // namespace pvt
