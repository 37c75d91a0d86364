// Local search over single-code changes (Appendix D) for the groups of a subspace, started from the codes
// that are stored -- typically right after pvt_vstep_encode, whose beam search is a heuristic for two
// codebooks.  A move replaces one code of the group's tuple by the value that lowers ||t - sum_m C_m[b_m]||^2
// most (the neighbour that is smallest under (error, tuple)), and is taken only if the error strictly drops.
//
// Every error that decides is the binary64 sum the final decision of the search kernels uses (residual through the codebooks
// in order, terms added in element order), so the moves are decided on exact values and the error can only fall.
//
// Every neighbour is tried in binary32 first (M*K*16 operations per target), which says what may be below an error.
// Two to four fp16 codebooks: a warp takes sixteen targets, a lane a target and a codebook, and finds which targets have a
// neighbour within the limit at all: after a beam search few or none.  Only those are searched, each by a whole warp.  After a
// beam search, 20011 targets of 2x251 / 200000 of 2x256 / 56360 of 4x256: 23 / 91 / 80 us, bound by the issue of packed
// arithmetic (a warp per target: 35 / 241 / 188; with the filter on the tensor pipe, targets in two halves: 21 / 63 / 86, but
// its scores were less exact than binary32 distances).  From random codes, where every target is searched, 86 / 674 / 640
// (a warp per target 138 / 1203 / 1345): the filter ends once every target has a neighbour, and the search evaluates in
// binary64 only what may be as near as the nearest neighbour.  Three blocks per SM: two 87 / 654 / 773, four 101 / 692 / 787.
// Others: a warp per target; bound by the issue of the binary32 operations and of the conversions around them.
#include <cuda_fp16.h>

#include "pvt_internal.h"

namespace pvt {
namespace {

constexpr int kRfThreads = 256;
constexpr int kRfSmemCodewords = 512;  // M*K up to this many codewords are staged in shared memory as binary32

struct RefineParams {
  const float* W;
  const float* g;
  const float* scale;
  const void* books;
  void* codes;
  const uint32_t* idx;
  uint64_t k, G;
  uint32_t gpr, K;
  float eta;
  int max_moves;
  float* err_out;
  uint32_t* moves_out;
  uint32_t* status;
};

// codeword `row` of a codebook in global or shared memory
template <bool CB_F16>
__device__ __forceinline__ void codeword_at(const void* books, uint32_t row, float c[8]) {
  if (CB_F16) {
    const uint4 raw = reinterpret_cast<const uint4*>(books)[row];
    const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w[i]));
      c[2 * i] = f.x;
      c[2 * i + 1] = f.y;
    }
  } else {
    const float4* src = reinterpret_cast<const float4*>(books) + 2 * (size_t)row;
    const float4 lo = src[0], hi = src[1];
    c[0] = lo.x, c[1] = lo.y, c[2] = lo.z, c[3] = lo.w, c[4] = hi.x, c[5] = hi.y, c[6] = hi.z, c[7] = hi.w;
  }
}

// ||t - c_1 - ... - c_M||^2 with the residual carried in binary64 through the codebooks in order and the terms
// added in element order; cw[m] = the codeword of codebook m
template <int M>
__device__ __forceinline__ double tuple_error(const float t[8], const float (*cw)[8]) {
  double d = 0.0;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    double e = (double)t[i];
#pragma unroll
    for (int m = 0; m < M; ++m) e = __dsub_rn(e, (double)cw[m][i]);
    d = __dadd_rn(d, __dmul_rn(e, e));
  }
  return d;
}

// target of the search (Eq. 8 in the scaled space): one fma and one division per element, binary32
__device__ __forceinline__ void target_of(const RefineParams& p, uint32_t j, float t[8]) {
  const float4* W4 = reinterpret_cast<const float4*>(p.W) + 2 * (size_t)j;
  const float4* g4 = reinterpret_cast<const float4*>(p.g) + 2 * (size_t)j;
  const float4 w0 = W4[0], w1 = W4[1], g0 = g4[0], g1 = g4[1];
  const float s = p.scale[j / p.gpr], ne = -p.eta;
  const float w[8] = {w0.x, w0.y, w0.z, w0.w, w1.x, w1.y, w1.z, w1.w};
  const float gg[8] = {g0.x, g0.y, g0.z, g0.w, g1.x, g1.y, g1.z, g1.w};
#pragma unroll
  for (int i = 0; i < 8; ++i) t[i] = __fdiv_rn(__fmaf_rn(ne, gg[i], w[i]), s);
}
// the group's codes; whether all of them are codes
template <int M, bool CODE_U16>
__device__ __forceinline__ bool codes_of(const RefineParams& p, uint32_t j, uint32_t (&b)[M]) {
  if (M == 1) {
    b[0] = CODE_U16 ? reinterpret_cast<const uint16_t*>(p.codes)[j] : reinterpret_cast<const uint8_t*>(p.codes)[j];
  } else {
    const uint8_t* c = reinterpret_cast<const uint8_t*>(p.codes) + (size_t)j * M;
#pragma unroll
    for (int m = 0; m < M; ++m) b[m] = c[m];
  }
  bool ok = true;
#pragma unroll
  for (int m = 0; m < M; ++m) ok = ok && b[m] < p.K;
  return ok;
}

// Two binary32 values in one register pair (packed arithmetic rounds each as the scalar one does)
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  return (uint64_t)__float_as_uint(lo) | ((uint64_t)__float_as_uint(hi) << 32);
}
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}

// Only a neighbour below a known error d matters, and binary32 says which may be: with r the target less the other codewords,
// each difference rounded, the root of ||r - c||^2 is off by no more than 2^-24 of r's and its intermediates' norms (rr: the
// sum of their squares) and of itself.  What is not above the limit of d's root may be below d (so for NaN).
__device__ __forceinline__ float rounding_of(float rr) { return 2.384185791015625e-7f /* 2^-22 */ * sqrtf(rr); }
__device__ __forceinline__ float limit_of(float root, float off) {
  root += off;
  return fmaf(root * root, 1.000003814697265625f /* 1 + 2^-18 */, 1e-36f);
}

// target less the codewords of all codebooks but m
template <int M>
__device__ __forceinline__ void residual_of(const float (&t)[8], const float (&cw)[M][8], uint32_t m, float (&r)[8],
                                            float& rr) {
  rr = 0.0f;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    r[i] = t[i];
#pragma unroll
    for (int o = 0; o < M; ++o) {
      if ((uint32_t)o == m) continue;
      r[i] -= cw[o][i];
      rr = fmaf(r[i], r[i], rr);
    }
  }
}

// The codebooks as a search goes through them, kWide adjacent codewords per lane and step
template <bool CB_F16>
struct Plain {  // one, as it lies in global or shared memory
  static constexpr int kWide = 1;
  const void* books;
  uint32_t K;
  __device__ __forceinline__ void codeword(uint32_t m, uint32_t q, float c[8]) const {
    codeword_at<CB_F16>(books, m * K + q, c);
  }
  __device__ __forceinline__ void distances(uint32_t m, uint32_t q, const float (&r)[8], float (&fast)[1]) const {
    float c[8];
    codeword(m, q, c);
    fast[0] = 0.0f;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float x = r[i] - c[i];
      fast[0] = fmaf(x, x, fast[0]);
    }
  }
};
constexpr int kRfPairs = 128;      // a codebook of up to 256 codewords
constexpr int kRfPairFloats = 20;  // a pair's 16 values and a gap: eight lanes that read adjacent pairs meet no bank twice
struct Pairs {  // two, in shared memory as binary32: codewords 2 p and 2 p + 1, element by element
  static constexpr int kWide = 2;
  const float (*pair)[kRfPairs][kRfPairFloats];
  __device__ __forceinline__ void codeword(uint32_t m, uint32_t q, float c[8]) const {
#pragma unroll
    for (int i = 0; i < 8; ++i) c[i] = pair[m][q >> 1][2 * i + (q & 1u)];
  }
  __device__ __forceinline__ void distances(uint32_t m, uint32_t q, const float (&r)[8], float (&fast)[2]) const {
    const ulonglong2* at = reinterpret_cast<const ulonglong2*>(&pair[m][q >> 1][0]);
    uint64_t sum = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const ulonglong2 c = at[i];
      const uint64_t x = sub2(pack2(r[2 * i], r[2 * i]), c.x), y = sub2(pack2(r[2 * i + 1], r[2 * i + 1]), c.y);
      sum = fma2(x, x, sum);
      sum = fma2(y, y, sum);
    }
    fast[0] = __uint_as_float((uint32_t)sum);
    fast[1] = __uint_as_float((uint32_t)(sum >> 32));
  }
};

// The moves of target n (group j) from codes b, codewords cw on, by the whole warp; writes what the call returns for it
template <int M, bool CODE_U16, class Books>
__device__ __forceinline__ void climb(const RefineParams& p, const Books& books, uint64_t n, uint32_t j, const float (&t)[8],
                                      uint32_t (&b)[M], float (&cw)[M][8]) {
  const uint32_t K = p.K;
  const int lane = threadIdx.x & 31;
  double d_cur = tuple_error<M>(t, cw);
  uint32_t moves = 0;
  while (moves < (uint32_t)p.max_moves) {
    float root = sqrtf((float)d_cur);  // no neighbour matters whose distance has a larger one
    float least[M], off[M];            // of the lane's neighbours by codebook
    if constexpr (Books::kWide > 1) {
      // No more is to be evaluated than what may be as near as the nearest neighbour of all: a pass over the codebooks finds
      // that one's binary32 distance.  (Everything below the current error: from random codes 1033 us for 200000 targets of
      // 2x256, two thirds of it the conversions to binary64; now 674.)
      float nearest = __int_as_float(0x7f800000), off_most = 0.0f;
#pragma unroll
      for (int m = 0; m < M; ++m) {
        float r[8], rr;
        residual_of<M>(t, cw, m, r, rr);
        off[m] = rounding_of(rr);
        least[m] = __int_as_float(0x7f800000);
        for (uint32_t q0 = Books::kWide * lane; q0 < K; q0 += 32 * Books::kWide) {
          float fast[Books::kWide];
          books.distances((uint32_t)m, q0, r, fast);
#pragma unroll
          for (int w = 0; w < Books::kWide; ++w) least[m] = q0 + w == b[m] ? least[m] : fminf(least[m], fast[w]);
        }
        nearest = fminf(nearest, least[m]);
        off_most = fmaxf(off_most, off[m]);
      }
      if (!__any_sync(0xffffffffu, !(nearest > limit_of(root, off_most)))) break;
      nearest = __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(nearest)));  // non-negative: ordered like u32
      root = fminf(root, (sqrtf(nearest) + off_most) * 1.0000019073486328125f /* 1 + 2^-19 */);
    }
    // best neighbour of this lane under (error, tuple); a neighbour is named by (codebook changed, new code)
    double ld = __longlong_as_double(0x7ff0000000000000ll);
    uint32_t lm = 0, lq = 0;
    bool lhave = false;
    auto tuple_less = [&](uint32_t m1, uint32_t q1, uint32_t m2, uint32_t q2) {
      // lexicographic order of the two neighbours' tuples (both differ from the current tuple in one place)
#pragma unroll
      for (int m = 0; m < M; ++m) {
        const uint32_t x = (uint32_t)m == m1 ? q1 : b[m], y = (uint32_t)m == m2 ? q2 : b[m];
        if (x != y) return x < y;
      }
      return false;
    };
#pragma unroll
    for (int m = 0; m < M; ++m) {
      if (Books::kWide > 1 && !__any_sync(0xffffffffu, !(least[m] > limit_of(root, off[m])))) continue;
      float keep[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) keep[i] = cw[m][i];
      float r[8], rr;
      residual_of<M>(t, cw, m, r, rr);
      const float limit = limit_of(root, rounding_of(rr));
      for (uint32_t q0 = Books::kWide * lane; q0 < K; q0 += 32 * Books::kWide) {
        float fast[Books::kWide];
        books.distances((uint32_t)m, q0, r, fast);
#pragma unroll
        for (int w = 0; w < Books::kWide; ++w) {
          const uint32_t q = q0 + w;
          if (fast[w] > limit || q == b[m] || q >= K) continue;  // (not so for NaN)
          books.codeword((uint32_t)m, q, cw[m]);
          const double d = tuple_error<M>(t, cw);
          if (!lhave || d < ld || (d == ld && tuple_less((uint32_t)m, q, lm, lq))) {
            ld = d;
            lm = (uint32_t)m;
            lq = q;
            lhave = true;
          }
        }
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) cw[m][i] = keep[i];
    }
    // warp-wide minimum of (error, tuple); errors are >= 0, so their bits order like u64
    const uint64_t bits = (uint64_t)__double_as_longlong(ld);
    const uint32_t hi = (uint32_t)(bits >> 32), lo = (uint32_t)bits;
    const uint32_t mhi = __reduce_min_sync(0xffffffffu, hi);
    const uint32_t mlo = __reduce_min_sync(0xffffffffu, hi == mhi ? lo : 0xffffffffu);
    const bool tied = lhave && hi == mhi && lo == mlo;
    // among the lanes that hold the minimum error: the smallest tuple, codebook by codebook
    uint32_t alive_mask = __ballot_sync(0xffffffffu, tied);
    if (alive_mask == 0 || !(__longlong_as_double((long long)(((uint64_t)mhi << 32) | mlo)) < d_cur)) break;
    bool mine = tied;
#pragma unroll
    for (int m = 0; m < M; ++m) {
      const uint32_t x = mine ? ((uint32_t)m == lm ? lq : b[m]) : 0xffffffffu;
      const uint32_t mx = __reduce_min_sync(0xffffffffu, x);
      mine = mine && x == mx;
    }
    const int winner = __ffs(__ballot_sync(0xffffffffu, mine)) - 1;  // exactly one lane (tuples are distinct)
    const uint32_t wm = __shfl_sync(0xffffffffu, lm, winner), wq = __shfl_sync(0xffffffffu, lq, winner);
#pragma unroll
    for (int m = 0; m < M; ++m)
      if ((uint32_t)m == wm) {
        b[m] = wq;
        books.codeword((uint32_t)m, wq, cw[m]);
      }
    d_cur = __longlong_as_double((long long)(((uint64_t)mhi << 32) | mlo));
    ++moves;
  }
  if (lane == 0) {
    if (moves) {
      if (M == 1) {
        if (CODE_U16)
          reinterpret_cast<uint16_t*>(p.codes)[j] = (uint16_t)b[0];
        else
          reinterpret_cast<uint8_t*>(p.codes)[j] = (uint8_t)b[0];
      } else {
        uint8_t* c = reinterpret_cast<uint8_t*>(p.codes) + (size_t)j * M;
#pragma unroll
        for (int m = 0; m < M; ++m) c[m] = (uint8_t)b[m];
      }
    }
    if (p.err_out) p.err_out[n] = (float)d_cur;
    if (p.moves_out) p.moves_out[n] = moves;
  }
}

template <int M, bool CB_F16, bool CODE_U16, bool STAGED>
__global__ void __launch_bounds__(kRfThreads, M <= 2 ? 4 : 2) refine_kernel(const RefineParams p) {
  __shared__ __align__(16) float sh_book[STAGED ? kRfSmemCodewords * 8 : 8];
  const uint32_t K = p.K;
  pdl_trigger();
  pdl_wait();
  if (STAGED) {
    for (uint32_t row = threadIdx.x; row < M * K; row += kRfThreads) {
      float c[8];
      codeword_at<CB_F16>(p.books, row, c);
#pragma unroll
      for (int i = 0; i < 8; ++i) sh_book[row * 8 + i] = c[i];
    }
    __syncthreads();
  }
  const Plain<!STAGED && CB_F16> books{STAGED ? (const void*)sh_book : p.books, K};
  const int lane = threadIdx.x & 31;
  // persistent blocks: the codebooks are staged once per block, not once per eight targets
  for (uint64_t n = (uint64_t)blockIdx.x * (kRfThreads / 32) + (threadIdx.x >> 5); n < p.k;
       n += (uint64_t)gridDim.x * (kRfThreads / 32)) {
    const uint32_t j = p.idx[n];
    if (j >= p.G) {
      if (lane == 0 && p.status) atomicOr(p.status, PVT_DEV_BAD_INDEX);
      continue;
    }
    float t[8];
    target_of(p, j, t);
    uint32_t b[M];
    const bool ok = codes_of<M, CODE_U16>(p, j, b);
    if (!ok) {
      if (lane == 0 && p.status) atomicOr(p.status, PVT_DEV_BAD_CODE);
      continue;
    }
    float cw[M][8];
#pragma unroll
    for (int m = 0; m < M; ++m) books.codeword((uint32_t)m, b[m], cw[m]);
    climb<M, CODE_U16>(p, books, n, j, t, b, cw);
  }
}

// ---- two to four fp16 codebooks: sixteen targets per warp
constexpr int kRfGroup = 16;
template <int M>
struct RefineSmem {
  alignas(16) float pair[M][kRfPairs][kRfPairFloats];
  uint32_t n_better, next;  // targets of the trip that have a neighbour to be looked at: their places; the next one to search
  uint8_t better[kRfThreads / 32 * kRfGroup];
  uint32_t found[kRfThreads / 32];  // those of a group that several warps share
};

template <int M>
__device__ __forceinline__ void climb_target(const RefineParams& p, const Pairs books, uint64_t n, uint32_t j) {
  float t[8], cw[M][8];
  uint32_t b[M];
  target_of(p, j, t);
  codes_of<M, false>(p, j, b);
#pragma unroll
  for (int m = 0; m < M; ++m) books.codeword((uint32_t)m, b[m], cw[m]);
  climb<M, false>(p, books, n, j, t, b, cw);
}

template <int M>
__global__ void __launch_bounds__(kRfThreads, 3) refine_group_kernel(const RefineParams p) {
  __shared__ RefineSmem<M> sm;
  constexpr uint32_t kFull = 0xffffffffu;
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, K = p.K;
  pdl_trigger();
  pdl_wait();
  // a codeword of every codebook per thread
  static_assert(kRfThreads == 2 * kRfPairs, "");
#pragma unroll
  for (int m = 0; m < M; ++m) {
    float c[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) c[i] = 1.0e30f;  // (beyond the codebook: at no distance that counts)
    if (tid < K) codeword_at<true>(p.books, m * K + tid, c);
#pragma unroll
    for (int i = 0; i < 8; ++i) sm.pair[m][tid >> 1][2 * i + (tid & 1u)] = c[i];
  }
  const Pairs books{sm.pair};
  const uint32_t half = lane >> 4;  // lane = target + 16 half: of two codebooks at a time the half's
  const uint64_t groups = (p.k + kRfGroup - 1) / kRfGroup;
  // A trip of the block: `per` groups, each by `parts` warps that share the codewords, then the targets that are to be
  // searched, by all warps.  (One warp per group: 3000 targets of 2x256 after a beam search 12.5 us, now 10.5.)
  const uint32_t share = (uint32_t)((groups + gridDim.x - 1) / gridDim.x);
  const uint32_t per = share < kRfThreads / 32 ? share : kRfThreads / 32;
  const uint32_t parts = per > 4 ? 1 : per > 2 ? 2 : per > 1 ? 4 : 8, own_group = warp / parts, part = warp % parts;
  const uint32_t steps = (K + 15) / 16, q_lo = 16 * (steps * part / parts), q_hi = 16 * (steps * (part + 1) / parts);
  for (uint64_t g0 = (uint64_t)blockIdx.x * per; g0 < groups; g0 += (uint64_t)gridDim.x * per) {
    if (tid == 0) sm.n_better = sm.next = 0;
    if (tid < kRfThreads / 32) sm.found[tid] = 0;
    __syncthreads();
    const uint64_t gi = g0 + own_group, n = gi * kRfGroup + (lane & 15u);
    uint32_t who = 0;  // the group's targets that are to be searched
    bool active = false;
    double d_cur = 0.0;
    if (own_group < per && gi < groups) {
      uint32_t j = kFull, b[M];
      float t[8] = {}, cw[M][8];
      if (n < p.k) {
        j = p.idx[n];
        uint32_t wrong = 0;
        if (j < p.G) {
          target_of(p, j, t);
          active = codes_of<M, false>(p, j, b);
          if (!active) wrong = PVT_DEV_BAD_CODE;
        } else {
          wrong = PVT_DEV_BAD_INDEX;
        }
        if (wrong && half == 0 && part == 0 && p.status) atomicOr(p.status, wrong);
      }
#pragma unroll
      for (int m = 0; m < M; ++m) {
        if (!active) b[m] = 0;
        books.codeword((uint32_t)m, b[m], cw[m]);
      }
      d_cur = tuple_error<M>(t, cw);
      // The search's own test of every neighbour, the operations in the same order: a target of which no code but the stored
      // ones is within the limit stays as it is.
      uint32_t done = __ballot_sync(kFull, !active || p.max_moves == 0);  // targets that are decided
#pragma unroll
      for (int m0 = 0; m0 < M; m0 += 2) {
        const bool last = m0 + 1 == M;  // an odd codebook: nothing for the upper half
        const uint32_t m = m0 + (last ? 0 : half);
        float r[8], rr;
        uint32_t own = 0;
        residual_of<M>(t, cw, m, r, rr);
#pragma unroll
        for (int o = 0; o < M; ++o) own = (uint32_t)o == m ? b[o] : own;
        const float limit = active && !(last && half) ? limit_of(sqrtf((float)d_cur), rounding_of(rr)) : -1.0f;
        float fast[2];
        books.distances(m, own & ~1u, r, fast);
        // codes within the limit, not counting the stored one
        int within = own < q_lo || own >= q_hi || (own & 1u ? fast[1] : fast[0]) > limit ? 0 : -1;
        for (uint32_t q0 = q_lo; q0 < q_hi && done != kFull; q0 += 16) {
#pragma unroll
          for (uint32_t i = 0; i < 16; i += 2) {
            books.distances(m, q0 + i, r, fast);
            within += fast[0] > limit ? 0 : 1;
            within += fast[1] > limit ? 0 : 1;
          }
          const uint32_t found = __ballot_sync(kFull, within > 0);
          who |= found | found >> 16 | found << 16;
          done |= who;
        }
      }
    }
    if (parts > 1) {
      if (lane == 0 && who) atomicOr(&sm.found[own_group], who);
      __syncthreads();
      who = sm.found[own_group];
    }
    if (active && part == 0 && half == 0) {
      if ((who >> lane) & 1u) {
        sm.better[atomicAdd(&sm.n_better, 1u)] = (uint8_t)(kRfGroup * own_group + lane);
      } else {
        if (p.err_out) p.err_out[n] = (float)d_cur;
        if (p.moves_out) p.moves_out[n] = 0;
      }
    }
    __syncthreads();
    while (true) {
      uint32_t i = 0;
      if (lane == 0) i = atomicAdd(&sm.next, 1u);
      i = __shfl_sync(kFull, i, 0);
      if (i >= sm.n_better) break;
      const uint64_t n = g0 * kRfGroup + sm.better[i];
      climb_target<M>(p, books, n, p.idx[n]);
    }
    __syncthreads();
  }
}

template <int M>
cudaError_t launch_groups(const RefineParams& p, cudaStream_t stream) {
  constexpr auto kernel = refine_group_kernel<M>;
  uint64_t most = 0;
  const cudaError_t e = resident_blocks<kernel>(kRfThreads, device_sm_count(), &most);
  if (e != cudaSuccess) return e;
  // as many blocks as are resident, if there is a group for each: few groups per block leave warps for the search
  const uint64_t want = (p.k + kRfGroup - 1) / kRfGroup;
  count_launches(1);
  return launch_dependent(kernel, (unsigned)(want < most ? want : most), kRfThreads, 0, stream, p);
}

template <int M, bool CB_F16, bool CODE_U16, bool STAGED>
cudaError_t launch_resident(const RefineParams& p, cudaStream_t stream) {
  constexpr auto kernel = refine_kernel<M, CB_F16, CODE_U16, STAGED>;
  const uint64_t want = (p.k + kRfThreads / 32 - 1) / (kRfThreads / 32);
  uint64_t most = 0;
  const cudaError_t e = resident_blocks<kernel>(kRfThreads, device_sm_count(), &most);
  if (e != cudaSuccess) return e;
  // Staged codebooks: the resident blocks and no more, since each further wave stages them again (20011 targets of 2x251 in
  // binary32 33.2 us, with twice as many blocks 35.2).  Nothing staged: a second wave evens out the first (56360 targets of
  // 1x4096 310 us, without it 327).
  if (!STAGED) most *= 2;
  count_launches(1);
  return launch_dependent(kernel, (unsigned)(want < most ? want : most), kRfThreads, 0, stream, p);
}

template <int M, bool CB_F16, bool CODE_U16>
cudaError_t launch_staged(const RefineParams& p, cudaStream_t stream) {
  if ((uint64_t)M * p.K <= (uint64_t)kRfSmemCodewords) return launch_resident<M, CB_F16, CODE_U16, true>(p, stream);
  return launch_resident<M, CB_F16, CODE_U16, false>(p, stream);
}

}  // namespace

cudaError_t launch_refine(const pvt_layer& L, uint64_t G, const uint32_t* idx, uint64_t k, int max_moves,
                          float* err_out, uint32_t* moves_out, uint32_t* status, cudaStream_t stream) {
  RefineParams p;
  p.W = L.W;
  p.g = L.g;
  p.scale = L.scale;
  p.books = L.codebooks;
  p.codes = L.codes;
  p.idx = idx;
  p.k = k;
  p.G = G;
  p.gpr = (uint32_t)(L.cols / kGroupDim);
  p.K = (uint32_t)L.codebook_size;
  p.eta = L.eta;
  p.max_moves = max_moves;
  p.err_out = err_out;
  p.moves_out = moves_out;
  p.status = status;
  const bool f16 = L.codebook_dtype == PVT_F16, u16 = L.code_dtype == PVT_U16;
  timing_begin(kKernRefine, stream);
  cudaError_t e;
  if (L.num_codebooks == 2)
    e = f16 ? launch_groups<2>(p, stream) : launch_staged<2, false, false>(p, stream);
  else if (L.num_codebooks == 3)
    e = f16 ? launch_groups<3>(p, stream) : launch_staged<3, false, false>(p, stream);
  else if (L.num_codebooks == 4)
    e = f16 ? launch_groups<4>(p, stream) : launch_staged<4, false, false>(p, stream);
  else if (f16)
    e = u16 ? launch_staged<1, true, true>(p, stream) : launch_staged<1, true, false>(p, stream);
  else
    e = u16 ? launch_staged<1, false, true>(p, stream) : launch_staged<1, false, false>(p, stream);
  timing_end(kKernRefine, stream);
  return e;
}

}  // namespace pvt
