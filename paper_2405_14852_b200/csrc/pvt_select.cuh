// The first pass of the selection: what it takes and computes, for the kernels that contain it.
#pragma once

#include "pvt_internal.h"

namespace pvt {
namespace select {

// Keys: n_j = ||eta * g_j||^2 in binary32: u = eta*g_i rounded once, acc = fma(u, u, acc)
// in index order from 0.  Non-negative, so the bit pattern orders like the value.

// ---- random subspace rules (appendix on small-scale experiments: subspaces drawn uniformly at random, or at
// random in proportion to the size of the gradient entries) --------------------------------------------------
// Every group gets the first output word of Philox-4x32 with 10 rounds (Salmon et al., SC 2011) at counter
// (j mod 2^32, j div 2^32, 0, 0) under the key (seed mod 2^32, seed div 2^32).
__device__ __forceinline__ uint32_t philox_first_word(uint64_t j, uint64_t seed) {
  uint32_t c0 = (uint32_t)j, c1 = (uint32_t)(j >> 32), c2 = 0u, c3 = 0u;
  uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
#pragma unroll
  for (int round = 0; round < 10; ++round) {
    const uint32_t h0 = __umulhi(0xD2511F53u, c0), l0 = 0xD2511F53u * c0;
    const uint32_t h1 = __umulhi(0xCD9E8D57u, c2), l1 = 0xCD9E8D57u * c2;
    const uint32_t n0 = h1 ^ c1 ^ k0, n2 = h0 ^ c3 ^ k1;
    c0 = n0; c1 = l1; c2 = n2; c3 = l0;
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
  return c0;
}

// E = -ln((r + 1/2) 2^-32) by a fixed sequence of binary64 operations (each rounded once, none contracted):
// r + 1/2 = m 2^e, m in [1, 2), m halved and e raised when m > sqrt 2; z = (m - 1)/(m + 1);
// p = 1 + z^2/3 + ... + z^20/21 by Horner's rule, one fused operation per coefficient; E = fma(32 - e, ln 2, -(2z p)).
__device__ __forceinline__ double neglog_u32(uint32_t r) {
  int e = r ? 31 - __clz((int)r) : -1;
  // (r + 1/2) 2^-e, exact: the significand of r + 1/2 with the exponent field set to that of 1.0
  const double x = __dadd_rn((double)r, 0.5);
  double m = __longlong_as_double((__double_as_longlong(x) & 0x000fffffffffffffll) | 0x3ff0000000000000ll);
  if (m > 1.4142135623730951) {
    m = __dmul_rn(m, 0.5);
    e = e + 1;
  }
  const double z = __ddiv_rn(__dadd_rn(m, -1.0), __dadd_rn(m, 1.0)), z2 = __dmul_rn(z, z);
  double p = 1.0 / 21.0;
#pragma unroll
  for (int d = 19; d >= 1; d -= 2) p = __fma_rn(p, z2, 1.0 / (double)d);
  const double lnm = __dmul_rn(__dmul_rn(2.0, z), p);
  return __fma_rn((double)(32 - e), 0.6931471805599453, -lnm);
}

template <int DG>
__device__ __forceinline__ float norm_of(const float* v, float eta) {
  float acc = 0.0f;
#pragma unroll
  for (int i = 0; i < DG; ++i) {
    const float u = __fmul_rn(eta, v[i]);
    acc = __fmaf_rn(u, u, acc);
  }
  return acc;
}

// What the first pass computes per group (everything after the keys is the same top-k):
//   kKeyNorm          key = squared update norm (the greedy rule of the V step)
//   kKeyNormBuffer    the same, and the straight-through buffer takes the step: buffer = fma(-eta, g, buffer)
//   kKeyUniform       key = the top 24 bits of the group's random word, as a binary32 number
//   kKeyProportional  key = (float)(norm / E), E the exponential clock of the group's random word
enum KeyMode { kKeyNorm = 0, kKeyNormBuffer = 1, kKeyUniform = 2, kKeyProportional = 3 };

struct SelParams {
  const float* g;
  float* buffer;
  uint64_t G, k, seed;
  uint32_t words;        // words of 32 groups per CTA of passes 2 and 3
  float eta;
  uint32_t* idx_out;
  uint32_t* status;
  uint32_t* keys;        // [G]
  uint2* masks;          // per word of 32 groups: above the threshold bin, inside it (pass 3: above, equal the threshold)
  uint32_t* hist0;       // sum over the CTAs: key bits [30:18]
  uint32_t* hist1;       // members of the threshold bin: key bits [17:9]
  uint32_t* fine;        // members of the threshold bin: key bits [17:0]
  uint32_t* state;       // [0] threshold bin, [1] keys still to be taken from it, [2] ticket
  uint64_t* counts;      // per CTA of the last pass: ready << 63 | equal << 31 | greater
};

template <int DG, int MODE>
constexpr int kKeyGroups = (DG == 16 ? 2 : 4) / (MODE == kKeyNormBuffer ? 2 : 1);  // groups in flight per thread

// the pass, shared by the first `blocks` blocks of kNormThreads
template <int DG, int MODE, int U = kKeyGroups<DG, MODE>>
__device__ __forceinline__ void keys_pass(const SelParams& p, uint32_t* hist, uint32_t blocks) {
  const uint32_t tid = threadIdx.x;
  const bool wide = ((reinterpret_cast<uintptr_t>(p.g) |
                      (MODE == kKeyNormBuffer ? reinterpret_cast<uintptr_t>(p.buffer) : 0)) & 31u) == 0;
  const uint64_t stride = (uint64_t)blocks * (U * kNormThreads);
  for (uint64_t j0 = (uint64_t)blockIdx.x * (U * kNormThreads) + tid; j0 < p.G; j0 += stride) {
    float v[U][DG];
    if (MODE != kKeyUniform) {
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const uint64_t j = j0 + u * kNormThreads;
        if (j < p.G) {
#pragma unroll
          for (int part = 0; part < DG / 8; ++part) load8(p.g + j * DG + 8 * part, wide, &v[u][8 * part]);
        }
      }
    }
    if (MODE == kKeyNormBuffer) {  // the straight-through buffer takes the step of every weight (Appendix E)
      float b[U][DG];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const uint64_t j = j0 + u * kNormThreads;
        if (j < p.G) {
#pragma unroll
          for (int part = 0; part < DG / 8; ++part) load8(p.buffer + j * DG + 8 * part, wide, &b[u][8 * part]);
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const uint64_t j = j0 + u * kNormThreads;
        if (j < p.G) {
#pragma unroll
          for (int i = 0; i < DG; ++i) b[u][i] = __fmaf_rn(-p.eta, v[u][i], b[u][i]);
#pragma unroll
          for (int part = 0; part < DG / 8; ++part) store8(p.buffer + j * DG + 8 * part, wide, &b[u][8 * part]);
        }
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const uint64_t j = j0 + u * kNormThreads;
      if (j < p.G) {
        uint32_t key;
        if (MODE == kKeyUniform) {
          key = __float_as_uint((float)(philox_first_word(j, p.seed) >> 8));
        } else {
          const float acc = norm_of<DG>(v[u], p.eta);
          key = __float_as_uint(acc);
          if (MODE == kKeyProportional)
            key = acc > 0.0f ? __float_as_uint(__double2float_rn(
                                   __ddiv_rn((double)acc, neglog_u32(philox_first_word(j, p.seed)))))
                             : 0u;
        }
        p.keys[j] = key;
        atomicAdd(&hist[key >> 18], 1u);
      }
    }
  }
  __syncthreads();
  for (uint32_t i = tid; i < kSelBins0; i += kNormThreads)
    if (hist[i]) atomicAdd(&p.hist0[i], hist[i]);
}

}  // namespace select

// that pass and the dequantisation of all groups from their present codes in one kernel
cudaError_t launch_keys_dequant(const select::SelParams& p, const pvt_layer& L, void* W_hat, int32_t out_dtype, int sm_count,
                                cudaStream_t stream);

}  // namespace pvt
