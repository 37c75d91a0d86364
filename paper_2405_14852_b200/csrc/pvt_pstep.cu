// The part of the P step that shares its inputs with the V step (Algorithm 3, P-step lines:
// grad_codebooks = backprop(grad_phi); codebooks = adam(grad_codebooks); Section 3.4 and Appendix J for Adam
// and its betas).
//
// backprop is the chain rule through dequantize_weights, W_hat[r, 8c + i] = s_r * v_{j,i} with
// v_j = sum_m C_m[b_{j,m}] (the binary32 sum that dequantisation forms):
//     grad_codebooks[m][kappa][i] = sum over groups j with b_{j,m} = kappa of  s_{r(j)} * g[j][i]
//     grad_scale[r]               = sum over groups j of row r and over i of   g[j][i] * v_{j,i}
// Every product of two binary32 numbers is exact in binary64 and the sums are accumulated in binary64 with
// atomic adds, so the result differs from a sequential sum only by the order of binary64 roundings.
//
// One streaming pass over g.  Small codebooks (M K <= 1024 codewords) are accumulated in shared memory per CTA and
// flushed once; large ones go straight to the L2.  Scale gradients are summed over a warp first when the warp lies inside
// one row.
#include <cuda_fp16.h>

#include "pvt_internal.h"

namespace pvt {
namespace {

constexpr int kPsThreads = 256;
constexpr size_t kPsMaxSmem = 227 * 1024;
// M K up to here: sums in shared memory, above it in the L2.  Shared memory slows down with the codewords that a tile is
// sorted into, the L2 speeds up with the codewords that its reductions spread over.  4096 x 4096, one fp16 codebook of
// 512 / 1024 / 1500 / 1944 codewords: 59 / 89 / 99 / 114 us in shared memory, 163 / 115 / 70 / 59 us in the L2;
// four codebooks of 256 (the most that several codebooks have): 161 and 470 us.
constexpr int kPsSmallBins = 1024;

__device__ __forceinline__ void red_add_f64(double* p, double v) {
  asm volatile("red.global.add.f64 [%0], %1;" ::"l"(p), "d"(v) : "memory");
}

// v = the codeword of a group (codebooks added left to right, each sum rounded once), from global or shared memory
template <int M, bool CB_F16, int DG>
__device__ __forceinline__ void group_codeword(const uint4* book, const uint32_t (&b)[M], uint32_t K, float (&v)[DG]) {
#pragma unroll
  for (int m = 0; m < M; ++m) {
    const uint4* row = book + (size_t)(m * K + b[m]) * (DG / (CB_F16 ? 8 : 4));
    float c[DG];
#pragma unroll
    for (int part = 0; part < DG / (CB_F16 ? 8 : 4); ++part) {
      const uint4 raw = row[part];
      const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (CB_F16) {
          const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w[i]));
          c[8 * part + 2 * i] = f.x;
          c[8 * part + 2 * i + 1] = f.y;
        } else {
          c[4 * part + i] = __uint_as_float(w[i]);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < DG; ++i) v[i] = m == 0 ? c[i] : __fadd_rn(v[i], c[i]);
  }
}

template <int M, bool CODE_U16>
__device__ __forceinline__ void group_codes(const void* codes, uint64_t j, uint32_t (&b)[M]) {
  if (!CODE_U16 && M == 2) {
    const uint32_t both = reinterpret_cast<const uint16_t*>(codes)[j];
    b[0] = both & 0xffu;
    b[M - 1] = both >> 8;
  } else {
#pragma unroll
    for (int m = 0; m < M; ++m)
      b[m] = CODE_U16 ? reinterpret_cast<const uint16_t*>(codes)[j * M + m] : reinterpret_cast<const uint8_t*>(codes)[j * M + m];
  }
}

// sum over i of g_i v_i: the products are exact, one rounding each as for a sum
template <int DG>
__device__ __forceinline__ double dot_exact(const double (&g)[DG], const float (&v)[DG]) {
  double d = g[0] * (double)v[0];
#pragma unroll
  for (int i = 1; i < DG; ++i) d = __fma_rn(g[i], (double)v[i], d);
  return d;
}

// the exact products s * g of a group as one row of doubles; lanes start at different pieces (no bank conflict)
template <int DG>
__device__ __forceinline__ void put_products(double* row, uint32_t lane, double s, const double (&g)[DG]) {
  double2* dst = reinterpret_cast<double2*>(row);
#pragma unroll
  for (int q = 0; q < DG / 2; q += 2) {
    const double2 lo = make_double2(s * g[2 * q], s * g[2 * q + 1]), hi = make_double2(s * g[2 * q + 2], s * g[2 * q + 3]);
    const uint32_t first = (lane >> 1) & 1u;
    dst[q + first] = first ? hi : lo;
    dst[q + (first ^ 1u)] = first ? lo : hi;
  }
}

// The sums start at zero.  (Two fills by the driver instead, and the sums launched behind them the plain way: gradient, both
// updates and dequantisation of 4096x4096 1x16 72.8 us for 65.3.)
__global__ void __launch_bounds__(kPsThreads) pstep_clear_kernel(double* books, uint64_t n_books, double* scale,
                                                                 uint64_t n_scale) {
  pdl_trigger();
  pdl_wait();
  const uint64_t stride = (uint64_t)gridDim.x * kPsThreads;
  for (uint64_t i = (uint64_t)blockIdx.x * kPsThreads + threadIdx.x; i < n_books + n_scale; i += stride) {
    if (i < n_books)
      books[i] = 0.0;
    else
      scale[i - n_books] = 0.0;
  }
}

// Large codebooks: one reduction per element in the L2.  A lane takes a group: its 32 bytes of g, its codeword, its
// share of the scale's gradient; the products then change places through shared memory so that the DG elements of a
// group are added by DG adjacent lanes: an L2 slice takes the four binary64 values of a sector that one instruction
// brings as one operation.  4096 x 4096: 48 us; with four elements of a group in a thread, four instructions to
// the same sector, 107 us; with a lane per element from the start (three conversions and a codeword load per
// element) 59 us.
template <int M, bool CB_F16, bool CODE_U16, int DG>
__global__ void __launch_bounds__(kPsThreads) pstep_grad_kernel(const float* g, const float* scale, const void* codes,
                                                                 const void* codebooks, uint64_t G, FastDiv gpr, uint32_t K,
                                                                 double* grad_books, double* grad_scale, uint32_t* status) {
  __shared__ __align__(16) double sh_prod[kPsThreads / 32][32][DG];
  constexpr uint32_t kFull = 0xffffffffu;
  constexpr int PER = 32 / DG;  // groups per instruction of the reductions
  pdl_trigger();
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, sub = lane / DG, e = lane % DG;
  const bool wide = (reinterpret_cast<uintptr_t>(g) & 31u) == 0;
  const uint64_t stride = 32 * (uint64_t)gridDim.x * (kPsThreads / 32);
  uint64_t j0 = 32 * ((uint64_t)blockIdx.x * (kPsThreads / 32) + warp);
  float gv[DG];
  uint32_t b[M];
  pdl_wait();
  auto fetch = [&](uint64_t at) {
#pragma unroll
    for (int i = 0; i < DG; ++i) gv[i] = 0.0f;
#pragma unroll
    for (int m = 0; m < M; ++m) b[m] = 0;
    if (at + lane < G) {
#pragma unroll
      for (int part = 0; part < DG / 8; ++part) load8(g + (at + lane) * DG + 8 * part, wide, &gv[8 * part]);
      group_codes<M, CODE_U16>(codes, at + lane, b);
    }
  };
  fetch(j0);
  for (; j0 < G; j0 += stride) {
    const bool mine = j0 + lane < G;
    const uint32_t row = mine ? fast_div((uint32_t)(j0 + lane), gpr) : kFull;
    const double s = mine ? (double)scale[row] : 0.0;
    bool bad = false;
#pragma unroll
    for (int m = 0; m < M; ++m) bad |= b[m] >= K;
    if (bad && status) atomicOr(status, PVT_DEV_BAD_CODE);
    const bool ok = mine && !bad;  // a group with a bad code contributes nothing
    double gd[DG];
#pragma unroll
    for (int i = 0; i < DG; ++i) gd[i] = (double)gv[i];
    uint32_t code[M];
#pragma unroll
    for (int m = 0; m < M; ++m) code[m] = b[m];
    double ds = 0.0;
    if (grad_scale && ok) {
      float v[DG];
      group_codeword<M, CB_F16, DG>(reinterpret_cast<const uint4*>(codebooks), code, K, v);
      ds = dot_exact<DG>(gd, v);
    }
    put_products<DG>(sh_prod[warp][lane], lane, s, gd);
    __syncwarp();
    fetch(j0 + stride);  // beside the reductions
    const uint32_t use = __ballot_sync(kFull, ok);
#pragma unroll
    for (int u = 0; u < DG; ++u) {
      const int src = PER * u + sub;
      const double p = sh_prod[warp][src][e];
#pragma unroll
      for (int m = 0; m < M; ++m) {
        const uint32_t c = __shfl_sync(kFull, code[m], src);
        if ((use >> src) & 1u) red_add_f64(grad_books + ((size_t)m * K + c) * DG + e, p);
      }
    }
    __syncwarp();
    if (grad_scale) {
      // a warp that lies inside one row adds its contributions with one reduction
      const uint32_t row0 = __shfl_sync(kFull, row, 0);
      if (__all_sync(kFull, row == row0)) {
#pragma unroll
        for (int o = 16; o; o >>= 1) ds = __dadd_rn(ds, __shfl_xor_sync(kFull, ds, o));
        if (lane == 0) red_add_f64(grad_scale + row0, ds);
      } else if (ok) {
        red_add_f64(grad_scale + row, ds);
      }
    }
  }
}


// Small codebooks: the sums stay in shared memory.  A CTA takes tiles of 1024 groups.  Per tile it stages the exact
// products s * g, sorts the tile's (codebook, code) pairs by counting (integer shared-memory atomics hand out the
// slots) and lets the team of four lanes that owns a pair, two elements each, add up its products in registers.
// The next tile's loads are in flight meanwhile.  What bounds it is shared memory (its pipe 71 % busy, 66 % of the cycles
// with a wavefront of it): products, lists, counters and codewords, and the rows of products in sorted order.
// 11008 x 4096, codes as a search leaves them, two / four codebooks of 256: 195 / 416 us, in the L2 843 / 1101 us.  With
// uniformly random codes 166 / 332 us; there tiles of 512 groups with no loads ahead took 283 us for two codebooks.
constexpr int kPsSmallThreads = 512;
constexpr int kPsTile = 1024;
constexpr int kPsTeams = kPsSmallThreads / 4;

template <int M, bool CB_F16>
constexpr size_t small_smem(uint32_t K) {
  const uint32_t bins = (M * K + kPsSmallThreads - 1) / kPsSmallThreads * kPsSmallThreads;
  return (sizeof(double) * 8 + (CB_F16 ? 16 : 32)) * M * (size_t)K + sizeof(double) * 8 * kPsTile + sizeof(uint32_t) * (bins + 32) + sizeof(uint16_t) * M * kPsTile;
}

template <int M, bool CB_F16, bool CODE_U16>
__global__ void __launch_bounds__(kPsSmallThreads, 2) pstep_grad_small_kernel(const float* __restrict__ g,
                                                                              const float* __restrict__ scale,
                                                                              const void* __restrict__ codes,
                                                                              const void* __restrict__ codebooks,
                                                                              uint64_t G, FastDiv gpr, uint32_t K,
                                                                              double* __restrict__ grad_books,
                                                                              double* __restrict__ grad_scale,
                                                                              uint32_t* status) {
  extern __shared__ __align__(16) unsigned char ps_smem[];
  constexpr uint32_t kFull = 0xffffffffu;
  pdl_trigger();
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t n_bins = M * K, per = (n_bins + kPsSmallThreads - 1) / kPsSmallThreads;
  double* acc = reinterpret_cast<double*>(ps_smem);              // [M K][8]
  double* prod = acc + (size_t)n_bins * 8;                       // [tile][8]: the exact products s * g
  uint4* book = reinterpret_cast<uint4*>(prod + kPsTile * 8);    // [M K]: the codebooks
  uint32_t* bin = reinterpret_cast<uint32_t*>(book + (size_t)n_bins * (CB_F16 ? 1 : 2));  // [M K, padded]: counts, then starts
  uint32_t* part = bin + per * kPsSmallThreads + 1;              // [31]
  uint16_t* list = reinterpret_cast<uint16_t*>(part + 31);       // [M tile]: the groups by (codebook, code)
  for (uint32_t i = tid; i < n_bins * 8; i += kPsSmallThreads) acc[i] = 0.0;
  constexpr uint32_t kRowPieces = CB_F16 ? 1 : 2;
  if (grad_scale) {
    for (uint32_t i = tid; i < n_bins * kRowPieces; i += kPsSmallThreads)
      book[i] = __ldg(reinterpret_cast<const uint4*>(codebooks) + i);
  }
  const uint64_t n_tiles = (G + kPsTile - 1) / kPsTile;
  const bool wide = (reinterpret_cast<uintptr_t>(g) & 31u) == 0;
  constexpr uint32_t kIter = kPsTile / kPsSmallThreads, kRun = 32 * kIter;  // groups of a thread, of a warp
  const uint32_t slot0 = warp * kRun + lane;
  float gv[kIter][8];
  uint32_t b[kIter][M];
  auto fetch = [&](uint64_t tile) {  // all loads of a tile, before the first use and beside the walk of the tile before it
#pragma unroll
    for (uint32_t it = 0; it < kIter; ++it) {
      const uint64_t j = tile * kPsTile + slot0 + 32 * it;
#pragma unroll
      for (int i = 0; i < 8; ++i) gv[it][i] = 0.0f;
#pragma unroll
      for (int m = 0; m < M; ++m) b[it][m] = 0;
      if (j < G) {
        load8(g + j * 8, wide, gv[it]);
        group_codes<M, CODE_U16>(codes, j, b[it]);
      }
    }
  };
  fetch(blockIdx.x);
  for (uint64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
    const uint64_t j0 = tile * kPsTile;
    const uint32_t n_here = (uint32_t)(G - j0 < (uint64_t)kPsTile ? G - j0 : (uint64_t)kPsTile);
    for (uint32_t i = tid; i < per * kPsSmallThreads; i += kPsSmallThreads) bin[i] = 0;
    __syncthreads();  // (the previous tile has been consumed, too)
    // rows of the warp's first and last group: usually the same, and then one scale and one sum serve all iterations
    const uint32_t w_lo = warp * kRun, w_hi = min(w_lo + kRun, n_here);
    const uint32_t row_lo = w_lo < n_here ? fast_div((uint32_t)(j0 + w_lo), gpr) : 0u;
    const uint32_t row_hi = w_lo < n_here ? fast_div((uint32_t)(j0 + w_hi - 1), gpr) : 0u;
    const bool one_row = row_lo == row_hi;
    const double s_row = (double)__ldg(scale + row_lo);
    double ds = 0.0;
    uint32_t rank[kIter][M];  // slot of the pair within its bin
#pragma unroll
    for (uint32_t it = 0; it < kIter; ++it) {
      const uint32_t slot = slot0 + 32 * it;
      const bool valid = slot < n_here;
      bool bad = false;
#pragma unroll
      for (int m = 0; m < M; ++m) {
        if (b[it][m] >= K) {
          bad = true;
          b[it][m] = 0;
        }
        if (valid) rank[it][m] = atomicAdd(&bin[m * K + b[it][m]], 1u);
      }
      if (bad && status) atomicOr(status, PVT_DEV_BAD_CODE);
      const uint32_t row = one_row || !valid ? row_lo : fast_div((uint32_t)(j0 + slot), gpr);
      const double sd = bad ? 0.0 : one_row ? s_row : (double)__ldg(scale + row);  // a bad code's group contributes nothing
      double gd[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) gd[i] = (double)gv[it][i];
      put_products<8>(&prod[slot * 8], lane, sd, gd);
      if (grad_scale) {
        double d = 0.0;
        if (valid && !bad) {
          float v[8];
          group_codeword<M, CB_F16, 8>(book, b[it], K, v);
          d = dot_exact<8>(gd, v);
        }
        if (one_row)
          ds = __dadd_rn(ds, d);
        else if (valid)
          red_add_f64(grad_scale + row, d);
      }
    }
    if (grad_scale && one_row) {
#pragma unroll
      for (int o = 16; o; o >>= 1) ds = __dadd_rn(ds, __shfl_xor_sync(kFull, ds, o));
      if (lane == 0 && w_lo < n_here) red_add_f64(grad_scale + row_lo, ds);
    }
    __syncthreads();
    // starts of the bins: every thread owns `per` adjacent ones
    {
      uint32_t sum = 0;
      for (uint32_t i = 0; i < per; ++i) sum += bin[tid * per + i];
      uint32_t incl = sum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t up = __shfl_up_sync(kFull, incl, o);
        if (lane >= (uint32_t)o) incl += up;
      }
      if (lane == 31) part[warp] = incl;
      __syncthreads();
      const uint32_t before = __reduce_add_sync(kFull, lane < warp ? part[lane] : 0u);
      uint32_t run = before + incl - sum;
      for (uint32_t i = 0; i < per; ++i) {
        const uint32_t c = bin[tid * per + i];
        bin[tid * per + i] = run;
        run += c;
      }
      if (tid == kPsSmallThreads - 1) bin[tid * per + per] = run;
    }
    __syncthreads();
#pragma unroll
    for (uint32_t it = 0; it < kIter; ++it) {
      const uint32_t slot = slot0 + 32 * it;
      if (slot < n_here) {
#pragma unroll
        for (int m = 0; m < M; ++m) list[bin[m * K + b[it][m]] + rank[it][m]] = (uint16_t)slot;
      }
    }
    __syncthreads();
    fetch(tile + gridDim.x);
    // a team of four lanes, two elements each, owns every (codebook, code) pair
    {
      const double2* rows = reinterpret_cast<const double2*>(prod) + (tid & 3u);
      for (uint32_t c = tid >> 2; c < n_bins; c += kPsTeams) {
        uint32_t i = bin[c];
        const uint32_t end = bin[c + 1];
        if (i == end) continue;
        double2* at = reinterpret_cast<double2*>(acc) + 4 * c + (tid & 3u);
        double2 sum = *at;
        do {
          const double2 x = rows[4 * (uint32_t)list[i]];
          sum.x = __dadd_rn(sum.x, x.x);
          sum.y = __dadd_rn(sum.y, x.y);
        } while (++i < end);
        *at = sum;
      }
    }
    __syncthreads();
  }
  __syncthreads();
  for (uint32_t i = tid; i < n_bins * 8; i += kPsSmallThreads)
    if (acc[i] != 0.0) red_add_f64(grad_books + i, acc[i]);
}

template <int M, bool CB_F16, bool CODE_U16>
cudaError_t launch_grad_small(const pvt_layer& L, uint64_t G, double* grad_books, double* grad_scale, uint32_t* status,
                              int sm_count, cudaStream_t stream) {
  const uint32_t K = (uint32_t)L.codebook_size;
  const size_t smem = small_smem<M, CB_F16>(K);
  const cudaError_t e = allow_smem<pstep_grad_small_kernel<M, CB_F16, CODE_U16>>();
  if (e != cudaSuccess) return e;
  const uint64_t tiles = (G + kPsTile - 1) / kPsTile, cap = (uint64_t)sm_count * (smem <= 112 * 1024 ? 2 : 1);
  pstep_grad_small_kernel<M, CB_F16, CODE_U16><<<(unsigned)(tiles < cap ? tiles : cap), kPsSmallThreads, smem, stream>>>(
      L.g, L.scale, L.codes, L.codebooks, G, make_fast_div((uint32_t)(L.cols / kGroupDim)), K, grad_books, grad_scale,
      status);
  return cudaGetLastError();
}

template <int M, bool CB_F16, bool CODE_U16, int DG>
cudaError_t launch_grad_large(const pvt_layer& L, uint64_t G, double* grad_books, double* grad_scale, uint32_t* status,
                              int sm_count, cudaStream_t stream) {
  const uint64_t want = (G + kPsThreads - 1) / kPsThreads, cap = (uint64_t)sm_count * 8;
  return launch_dependent(pstep_grad_kernel<M, CB_F16, CODE_U16, DG>, (unsigned)(want < cap ? want : cap), kPsThreads, 0, stream,
                          L.g, L.scale, (const void*)L.codes, L.codebooks, G, make_fast_div((uint32_t)(L.cols / DG)),
                          (uint32_t)L.codebook_size, grad_books, grad_scale, status);
}

template <int M, bool CB_F16, bool CODE_U16>
cudaError_t launch_grad(const pvt_layer& L, uint64_t G, double* grad_books, double* grad_scale, uint32_t* status,
                        int sm_count, cudaStream_t stream) {
  if (L.group_dim == 16) {  // groups of 16 weights: one codebook
    if constexpr (M == 1)
      return launch_grad_large<1, CB_F16, CODE_U16, 16>(L, G, grad_books, grad_scale, status, sm_count, stream);
  }
  static_assert(small_smem<M, CB_F16>(kPsSmallBins / M) <= kPsMaxSmem, "a block holds every small codebook's sums");
  if ((uint32_t)M * (uint32_t)L.codebook_size <= (uint32_t)kPsSmallBins)
    return launch_grad_small<M, CB_F16, CODE_U16>(L, G, grad_books, grad_scale, status, sm_count, stream);
  return launch_grad_large<M, CB_F16, CODE_U16, 8>(L, G, grad_books, grad_scale, status, sm_count, stream);
}

// One Adam update, binary32, each operation rounded once, in the order stated in pvt.h.
__global__ void __launch_bounds__(256) adam_kernel(float* param, __half* param_f16, const double* grad, float* exp_avg,
                                                    float* exp_avg_sq, uint64_t n, float lr, float beta1, float beta2,
                                                    float eps, float bias1, float bias2) {
  pdl_trigger();
  pdl_wait();
  const float omb1 = __fsub_rn(1.0f, beta1), omb2 = __fsub_rn(1.0f, beta2);
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
    const float gr = __double2float_rn(grad[i]);
    const float m = __fmaf_rn(beta1, exp_avg[i], __fmul_rn(omb1, gr));
    const float v = __fmaf_rn(beta2, exp_avg_sq[i], __fmul_rn(__fmul_rn(omb2, gr), gr));
    exp_avg[i] = m;
    exp_avg_sq[i] = v;
    const float num = __fmul_rn(lr, __fdiv_rn(m, bias1));
    const float den = __fadd_rn(__fsqrt_rn(__fdiv_rn(v, bias2)), eps);
    const float p = __fsub_rn(param[i], __fdiv_rn(num, den));
    param[i] = p;
    if (param_f16) param_f16[i] = __float2half_rn(p);
  }
}

// Adam-normalised update direction of the V step (Section 3.4): moments as in Adam, u = (m / bias1) /
// (sqrt(v / bias2) + eps), binary32, each operation rounded once.
// Bound by HBM, three arrays read and three written.  Eight elements, 32 bytes of each, per thread and trip: 5120x5120
// 106 us (16 bytes: 113).
__global__ void __launch_bounds__(256) adam_direction_kernel(const float* grad, float* exp_avg, float* exp_avg_sq,
                                                              float* dir, uint64_t n4, float beta1, float beta2, float eps,
                                                              float bias1, float bias2) {
  pdl_trigger();
  pdl_wait();
  const float omb1 = __fsub_rn(1.0f, beta1), omb2 = __fsub_rn(1.0f, beta2);
  auto one = [&](float gr, float& m, float& v) {
    m = __fmaf_rn(beta1, m, __fmul_rn(omb1, gr));
    v = __fmaf_rn(beta2, v, __fmul_rn(__fmul_rn(omb2, gr), gr));
    return __fdiv_rn(__fdiv_rn(m, bias1), __fadd_rn(__fsqrt_rn(__fdiv_rn(v, bias2)), eps));
  };
  const bool wide = ((reinterpret_cast<uintptr_t>(grad) | reinterpret_cast<uintptr_t>(exp_avg) |
                      reinterpret_cast<uintptr_t>(exp_avg_sq) | reinterpret_cast<uintptr_t>(dir)) & 31u) == 0;
  const uint64_t n8 = n4 / 2;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n8; i += (uint64_t)gridDim.x * blockDim.x) {
    float g[8], m[8], v[8];
    load8(grad + 8 * i, wide, g);
    load8(exp_avg + 8 * i, wide, m);
    load8(exp_avg_sq + 8 * i, wide, v);
#pragma unroll
    for (int q = 0; q < 8; ++q) g[q] = one(g[q], m[q], v[q]);
    store8(exp_avg + 8 * i, wide, m);
    store8(exp_avg_sq + 8 * i, wide, v);
    store8(dir + 8 * i, wide, g);
  }
  if ((n4 & 1) && blockIdx.x == 0 && threadIdx.x < 4) {  // the last four
    const uint64_t i = 8 * n8 + threadIdx.x;
    float m = exp_avg[i], v = exp_avg_sq[i];
    dir[i] = one(grad[i], m, v);
    exp_avg[i] = m;
    exp_avg_sq[i] = v;
  }
}

}  // namespace

cudaError_t launch_adam_direction(const float* grad, float* exp_avg, float* exp_avg_sq, float* dir, uint64_t n,
                                  float beta1, float beta2, float eps, float bias1, float bias2, int sm_count,
                                  cudaStream_t stream) {
  timing_begin(kKernAdam, stream);
  const uint64_t n4 = n / 4, want = (n4 / 2 + 255) / 256, cap = (uint64_t)sm_count * 8;
  const cudaError_t err =
      launch_dependent(adam_direction_kernel, (unsigned)(want < 1 ? 1 : want < cap ? want : cap), 256, 0, stream, grad,
                       exp_avg, exp_avg_sq, dir, n4, beta1, beta2, eps, bias1, bias2);
  count_launches(1);
  timing_end(kKernAdam, stream);
  return err;
}

cudaError_t launch_pstep_grad(const pvt_layer& L, uint64_t G, double* grad_books, double* grad_scale, uint32_t* status,
                              int sm_count, cudaStream_t stream) {
  const uint64_t n_books = (uint64_t)L.num_codebooks * (uint64_t)L.codebook_size * (uint64_t)L.group_dim;
  const uint64_t n_scale = grad_scale ? (uint64_t)L.rows : 0, want = (n_books + n_scale + kPsThreads - 1) / kPsThreads;
  const uint64_t most = (uint64_t)sm_count * 8;
  cudaError_t err = launch_dependent(pstep_clear_kernel, (unsigned)(want < most ? want : most), kPsThreads, 0, stream, grad_books,
                                     n_books, grad_scale, n_scale);
  if (err != cudaSuccess) return err;
  count_launches(1);
  timing_begin(kKernPstepGrad, stream);
  const bool f16 = L.codebook_dtype == PVT_F16, u16 = L.code_dtype == PVT_U16;
  if (L.num_codebooks == 1) {
    if (f16)
      err = u16 ? launch_grad<1, true, true>(L, G, grad_books, grad_scale, status, sm_count, stream)
                : launch_grad<1, true, false>(L, G, grad_books, grad_scale, status, sm_count, stream);
    else
      err = u16 ? launch_grad<1, false, true>(L, G, grad_books, grad_scale, status, sm_count, stream)
                : launch_grad<1, false, false>(L, G, grad_books, grad_scale, status, sm_count, stream);
  } else if (L.num_codebooks == 2) {
    if (f16)
      err = u16 ? launch_grad<2, true, true>(L, G, grad_books, grad_scale, status, sm_count, stream)
                : launch_grad<2, true, false>(L, G, grad_books, grad_scale, status, sm_count, stream);
    else
      err = u16 ? launch_grad<2, false, true>(L, G, grad_books, grad_scale, status, sm_count, stream)
                : launch_grad<2, false, false>(L, G, grad_books, grad_scale, status, sm_count, stream);
  } else if (L.num_codebooks == 3) {  // three and four codebooks: one-byte codes
    err = f16 ? launch_grad<3, true, false>(L, G, grad_books, grad_scale, status, sm_count, stream)
              : launch_grad<3, false, false>(L, G, grad_books, grad_scale, status, sm_count, stream);
  } else {
    err = f16 ? launch_grad<4, true, false>(L, G, grad_books, grad_scale, status, sm_count, stream)
              : launch_grad<4, false, false>(L, G, grad_books, grad_scale, status, sm_count, stream);
  }
  count_launches(1);
  timing_end(kKernPstepGrad, stream);
  return err;
}

cudaError_t launch_adam(float* param, void* param_f16, const double* grad, float* exp_avg, float* exp_avg_sq,
                        uint64_t n, float lr, float beta1, float beta2, float eps, float bias1, float bias2,
                        int sm_count, cudaStream_t stream) {
  timing_begin(kKernAdam, stream);
  const uint64_t want = (n + 255) / 256, cap = (uint64_t)sm_count * 8;
  const cudaError_t err =
      launch_dependent(adam_kernel, (unsigned)(want < cap ? want : cap), 256, 0, stream, param,
                       reinterpret_cast<__half*>(param_f16), grad, exp_avg, exp_avg_sq, n, lr, beta1, beta2, eps, bias1, bias2);
  count_launches(1);
  timing_end(kKernAdam, stream);
  return err;
}

}  // namespace pvt
