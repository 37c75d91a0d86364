// Exhaustive nearest-codeword search of the V step for one codebook of at most 1024 codewords (below 1024 for fp16: from
// there on the tensor engine takes them), groups of 8 (Appendix C / Appendix J: all
// codewords of the codebook are tried; Appendix D: the score ||c||^2 - 2 <t, c>; Eq. 8 for the target).
//
// One kernel does all of it.  The codebook is expanded into shared memory by every CTA (pairs of codewords interleaved
// for fma.rn.f32x2, half squared norms beside them); a team of eight lanes takes one or two targets, each lane every
// eighth pair of codewords.  A lane keeps its smallest pair score, the pair, and its second smallest; the team's
// minimum plus twice the rounding-error bound of the scores says which pairs can hold the nearest codeword.  Those --
// nearly always one -- get their binary64 distance sum (t_i - c_i)^2 (index order), and the argmin of (distance, code)
// is written.  A lane with two pairs within the margin goes through all of its codewords in binary64.
//
// What bounds it: the FP32 pipe for many targets (8 packed FMAs per pair of codewords and target against 7 other
// instructions with two targets per team), one chain of latencies for few.  Two targets per team when there are enough
// of them to fill the machine, else one.  256
// codewords, 8192 / 2 million targets: 10 / 448 us; 1000 codewords, 20000 / 500000 targets: 34 / 295 us.  (Expansion,
// search with codebook slices and rescoring as kernels of their own: 37 / 690 and 39 / 362 us.)  The bound on the
// codebook: with 2048 codewords an SM holds too few warps, and the kernels of their own are faster (130 against 137 us
// for 100000 targets, 880 against 1180 us for 4096 codewords and 500000 targets).
#include <cuda_fp16.h>

#include "pvt_encode_m1.cuh"

namespace pvt {

using namespace m1;

namespace {

constexpr int kSmThreads = 256;
constexpr float kPadHalfNorm = 3.0e38f;  // half norm of padding codewords: never near a minimum
constexpr uint32_t kFull = 0xffffffffu;

__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  return (uint64_t)__float_as_uint(lo) | ((uint64_t)__float_as_uint(hi) << 32);
}

__host__ __device__ constexpr uint32_t small_blocks(uint32_t K) { return (K + 15) / 16; }  // 16 codewords: a pair per lane
__host__ __device__ constexpr size_t small_smem_bytes(uint32_t K) { return (size_t)small_blocks(K) * (512 + 64); }

// What a search leaves besides the codes: kCodes nothing, kWeights the groups' weights, kStep those (if anywhere) and the list
// of groups, which are all.
enum SmallOut { kCodes, kWeights, kStep };

// kStep: every group is a target (no list to read), and the team that found a group's codeword writes its weights too, so
// that a step is one kernel in place of three.  256 x 256 weights, 256 fp32 codewords: 10.2 -> 7.0 us per step, the first
// on new buffers 29 -> 24.
template <bool CB_F16, int TT, SmallOut OUT>
__global__ void __launch_bounds__(kSmThreads, 4) encode_m1_small_kernel(const EncM1Params p, uint32_t* idx_out) {
  // [block of 16 codewords][piece q of 4][lane of 8]: (c[2l][2q], c[2l+1][2q], c[2l][2q+1], c[2l+1][2q+1])
  extern __shared__ __align__(16) float sm_vals[];
  __shared__ uint32_t sm_n2max;
  const uint32_t K = p.K, n_blocks = small_blocks(K);
  float* norms = sm_vals + (size_t)n_blocks * 128;  // [block][lane][2]
  const uint32_t tid = threadIdx.x, l = tid & 7u, team = tid >> 3, n_teams = kSmThreads / 8;
  if (tid == 0) sm_n2max = 0;
  __syncthreads();
  pdl_trigger();
  pdl_wait();
  {
    uint32_t n2bits = 0;
    for (uint32_t kappa = tid; kappa < n_blocks * 16; kappa += kSmThreads) {
      float c[8], n2 = 0.0f;
#pragma unroll
      for (int i = 0; i < 8; ++i) c[i] = 0.0f;
      if (kappa < K) {
        load_codeword<CB_F16, 8>(p.book, kappa, c);
#pragma unroll
        for (int i = 0; i < 8; ++i) n2 = __fmaf_rn(c[i], c[i], n2);
        n2bits = max(n2bits, __float_as_uint(n2));  // non-negative floats order like their bits
      }
      const uint32_t block = kappa >> 4, pair = (kappa >> 1) & 7u, half = kappa & 1u;
#pragma unroll
      for (int i = 0; i < 8; ++i) sm_vals[block * 128 + (i >> 1) * 32 + pair * 4 + (i & 1) * 2 + half] = c[i];
      norms[block * 16 + pair * 2 + half] = kappa < K ? __fmul_rn(0.5f, n2) : kPadHalfNorm;
    }
    n2bits = __reduce_max_sync(kFull, n2bits);
    if ((tid & 31u) == 0) atomicMax(&sm_n2max, n2bits);
  }
  __syncthreads();
  const float n2max = __uint_as_float(sm_n2max);

  const uint64_t per_cta = (uint64_t)n_teams * TT, n_tiles = (p.k + per_cta - 1) / per_cta;
  for (uint64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
    uint32_t j[TT];
    float mine[TT], row_scale[TT];  // element l of the target, the scale of its row
    uint64_t nt[TT][8];
    float best[TT], second[TT];
    uint32_t at[TT];
    float nt2[TT];
#pragma unroll
    for (int tt = 0; tt < TT; ++tt) {
      const uint64_t n = tile * per_cta + (uint64_t)tt * n_teams + team;
      j[tt] = n < p.k ? (OUT == kStep ? (uint32_t)n : p.idx[n]) : kFull;
      mine[tt] = 0.0f;
    }
#pragma unroll
    for (int tt = 0; tt < TT; ++tt) {
      if (j[tt] < p.G) {
        const float w = p.W[(size_t)j[tt] * 8 + l], gg = p.g[(size_t)j[tt] * 8 + l];
        row_scale[tt] = p.scale[fast_div(j[tt], p.gpr_div)];
        mine[tt] = __fdiv_rn(__fmaf_rn(-p.eta, gg, w), row_scale[tt]);
      }
      nt2[tt] = 0.0f;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float t = __shfl_sync(kFull, mine[tt], i, 8);
        nt2[tt] = fmaf(t, t, nt2[tt]);
        nt[tt][i] = pack2(-t, -t);
      }
      best[tt] = second[tt] = __uint_as_float(0x7f800000u);
      at[tt] = 0;
    }
    const ulonglong2* vals = reinterpret_cast<const ulonglong2*>(sm_vals) + l;
    const uint64_t* hn = reinterpret_cast<const uint64_t*>(norms) + l;
#pragma unroll 2
    for (uint32_t b = 0; b < n_blocks; ++b) {
      const ulonglong2 q0 = vals[32 * b], q1 = vals[32 * b + 8], q2 = vals[32 * b + 16], q3 = vals[32 * b + 24];
      const uint64_t h = hn[8 * b];
#pragma unroll
      for (int tt = 0; tt < TT; ++tt) {
        uint64_t acc = h;
        acc = fma2(nt[tt][0], q0.x, acc);
        acc = fma2(nt[tt][1], q0.y, acc);
        acc = fma2(nt[tt][2], q1.x, acc);
        acc = fma2(nt[tt][3], q1.y, acc);
        acc = fma2(nt[tt][4], q2.x, acc);
        acc = fma2(nt[tt][5], q2.y, acc);
        acc = fma2(nt[tt][6], q3.x, acc);
        acc = fma2(nt[tt][7], q3.y, acc);
        const float m = fminf(__uint_as_float((uint32_t)acc), __uint_as_float((uint32_t)(acc >> 32)));
        second[tt] = fminf(second[tt], fmaxf(m, best[tt]));
        at[tt] = m < best[tt] ? b : at[tt];
        best[tt] = fminf(best[tt], m);
      }
    }
#pragma unroll
    for (int tt = 0; tt < TT; ++tt) {
      float least = best[tt];
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) least = fminf(least, __shfl_xor_sync(kFull, least, o));
      // twice the rounding-error bound of the fast score, with a factor 2 to spare:
      // |score_fl - score| <= 16.1 u (||c||^2/2 + ||t|| ||c||), u = 2^-24
      const float limit = least + 3.8146973e-6f /* 2^-18 */ * (0.5f * n2max + sqrtf(nt2[tt] * n2max)) + 1e-30f;
      const bool real = j[tt] < p.G;
      // a score that is no number (a target or codeword that is not finite) leaves every pair to the exact distances
      const bool odd = !(least <= 1e38f) || !(limit == limit);
      uint32_t lo = at[tt], hi = at[tt] + 1;  // blocks this lane looks at again
      if (odd || second[tt] <= limit)
        lo = 0, hi = n_blocks;
      else if (!(best[tt] <= limit))
        hi = lo;
      double d_best = __longlong_as_double(0x7ff0000000000000ll);
      uint32_t code = kFull;
      float t[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) t[i] = -__uint_as_float((uint32_t)nt[tt][i]);
      for (uint32_t b = real ? lo : hi; b < hi; ++b) {
        const float4* v = reinterpret_cast<const float4*>(sm_vals) + 32 * b + l;
        double d0 = 0.0, d1 = 0.0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float4 c = v[8 * q];
          double e = __dsub_rn((double)t[2 * q], (double)c.x);
          d0 = __dadd_rn(d0, __dmul_rn(e, e));
          e = __dsub_rn((double)t[2 * q + 1], (double)c.z);
          d0 = __dadd_rn(d0, __dmul_rn(e, e));
          e = __dsub_rn((double)t[2 * q], (double)c.y);
          d1 = __dadd_rn(d1, __dmul_rn(e, e));
          e = __dsub_rn((double)t[2 * q + 1], (double)c.w);
          d1 = __dadd_rn(d1, __dmul_rn(e, e));
        }
        const uint32_t kappa = 16 * b + 2 * l;
        if (kappa < K && (d0 < d_best || (d0 == d_best && kappa < code))) d_best = d0, code = kappa;
        if (kappa + 1 < K && (d1 < d_best || (d1 == d_best && kappa + 1 < code))) d_best = d1, code = kappa + 1;
      }
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) {
        const double od = __shfl_xor_sync(kFull, d_best, o);
        const uint32_t oc = __shfl_xor_sync(kFull, code, o);
        if (od < d_best || (od == d_best && oc < code)) d_best = od, code = oc;
      }
      const uint64_t n = tile * per_cta + (uint64_t)tt * n_teams + team;
      if (l == 0 && n < p.k) {
        if (!real) {
          atomicOr(p.status, PVT_DEV_BAD_INDEX);
        } else if (code < K) {
          if (p.code_u16)
            reinterpret_cast<uint16_t*>(p.codes)[j[tt]] = (uint16_t)code;
          else
            reinterpret_cast<uint8_t*>(p.codes)[j[tt]] = (uint8_t)code;
          if (p.err_out) p.err_out[n] = (float)d_best;
        } else {
          atomicOr(p.status, PVT_DEV_INTERNAL);  // non-finite target: no distance compares below infinity
        }
        if (OUT == kStep) idx_out[n] = (uint32_t)n;
      }
      if (OUT != kCodes && p.out.W_hat && real) {  // element l, as dequantisation forms it
        uint32_t kappa = code;
        if (kappa >= K) {  // the stored code stays
          kappa = p.code_u16 ? reinterpret_cast<const uint16_t*>(p.codes)[j[tt]]
                             : reinterpret_cast<const uint8_t*>(p.codes)[j[tt]];
          if (kappa >= K) kappa = 0;
        }
        const float c = sm_vals[(kappa >> 4) * 128 + (l >> 1) * 32 + ((kappa >> 1) & 7u) * 4 + (l & 1u) * 2 + (kappa & 1u)];
        const float w = __fmul_rn(row_scale[tt], c);
        if (p.out.f16)
          reinterpret_cast<__half*>(p.out.W_hat)[(size_t)j[tt] * 8 + l] = __float2half_rn(w);
        else
          reinterpret_cast<float*>(p.out.W_hat)[(size_t)j[tt] * 8 + l] = w;
      }
    }
  }
}

template <bool CB_F16, int TT, SmallOut OUT>
cudaError_t launch_small(const EncM1Params& p, uint32_t* idx_out, int sm_count, cudaStream_t stream) {
  const size_t smem = small_smem_bytes(p.K);
  const cudaError_t err = allow_smem<encode_m1_small_kernel<CB_F16, TT, OUT>>();
  if (err != cudaSuccess) return err;
  const uint64_t per_cta = kSmThreads / 8 * TT, tiles = (p.k + per_cta - 1) / per_cta;
  constexpr uint64_t kMost = 1024 / kSmThreads;  // 64 registers a thread
  const uint64_t fit = (228 * 1024) / (smem + 2048), per_sm = fit < kMost ? fit : kMost;
  const uint64_t resident = per_sm * (uint64_t)sm_count;
  timing_begin(kKernEncodeMain, stream);
  const cudaError_t e = launch_dependent(encode_m1_small_kernel<CB_F16, TT, OUT>,
                                         (unsigned)(tiles < resident ? tiles : resident), kSmThreads, smem, stream, p,
                                         idx_out);
  timing_end(kKernEncodeMain, stream);
  count_launches(1);
  return e;
}

template <SmallOut OUT>
cudaError_t launch_kind(const pvt_layer& L, uint64_t G, const uint32_t* idx, uint64_t k, float* err_out, void* ws,
                        WeightsOut out, uint32_t* idx_out, int sm_count, cudaStream_t stream) {
  EncM1Params p = {};
  p.W = L.W;
  p.g = L.g;
  p.scale = L.scale;
  p.idx = idx;
  p.k = k;
  p.G = G;
  p.gpr_div = make_fast_div((uint32_t)(L.cols / kGroupDim));
  p.eta = L.eta;
  p.K = (uint32_t)L.codebook_size;
  p.book = L.codebooks;
  p.codes = L.codes;
  p.code_u16 = L.code_dtype == PVT_U16;
  p.out = out;
  p.err_out = err_out;
  p.status = static_cast<uint32_t*>(ws);
  const bool two = k >= (uint64_t)sm_count * 256;  // otherwise one target per team keeps more SMs busy
  if (L.codebook_dtype == PVT_F16)
    return two ? launch_small<true, 2, OUT>(p, idx_out, sm_count, stream)
               : launch_small<true, 1, OUT>(p, idx_out, sm_count, stream);
  return two ? launch_small<false, 2, OUT>(p, idx_out, sm_count, stream)
             : launch_small<false, 1, OUT>(p, idx_out, sm_count, stream);
}

}  // namespace

cudaError_t launch_encode_m1_small(const pvt_layer& L, uint64_t G, const uint32_t* idx, uint64_t k, float* err_out,
                                   WeightsOut out, void* ws, int sm_count, cudaStream_t stream) {
  return out.W_hat ? launch_kind<kWeights>(L, G, idx, k, err_out, ws, out, nullptr, sm_count, stream)
                   : launch_kind<kCodes>(L, G, idx, k, err_out, ws, out, nullptr, sm_count, stream);
}

cudaError_t launch_step_m1_small(const pvt_layer& L, uint64_t G, uint32_t* idx_out, WeightsOut out, void* ws, int sm_count,
                                 cudaStream_t stream) {
  return launch_kind<kStep>(L, G, nullptr, G, nullptr, ws, out, idx_out, sm_count, stream);
}

}  // namespace pvt
