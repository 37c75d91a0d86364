// dequantize_weights (Algorithm 3, first line): W_hat = s_row * sum_m C_m[b_m] for
// every weight group.  Streaming kernel, persistent grid: one thread per 16 bytes of the
// result, two of them in flight per thread, codes read coalesced, codewords gathered from
// the L2-resident codebook (small ones are first copied to shared memory), and a
// warp's stores contiguous: 512 bytes per instruction.
//
// Arithmetic per element, binary32, each step rounded once: v = c1 (+ c2);
// w = s * v; fp16 output = round-to-nearest-even of w.
#include <cuda_fp16.h>

#include "pvt_select.cuh"

namespace pvt {
namespace {

constexpr int kDqThreads = 256;
constexpr int kDqUnroll = 2;  // pieces of 16 result bytes in flight per thread (5120x5120 2x8 fp16 14.0 us; four 14.8, eight 19.8)
// Codebooks of up to this size are staged in shared memory: two to four always (256 codewords each at most), one if it is
// small.  No more than that is reserved, for it costs resident blocks (32 KB for all: 11008x4096 2x8 39 us after the
// search instead of 32).
__host__ __device__ constexpr int staged_bytes(int M, int cw_bytes) { return M == 1 ? 8192 : M * 256 * cw_bytes; }

// elements EL*part .. EL*part+EL-1 of one codeword of EL*PARTS elements, widened to binary32
template <bool CB_F16, int EL, int PARTS>
__device__ __forceinline__ void load_part(const void* book, uint32_t code, uint32_t part, float* v) {
  const size_t at = PARTS * (size_t)code + part;
  if (CB_F16) {
    uint32_t raw[EL / 2];
    if (EL == 8)
      *reinterpret_cast<uint4*>(raw) = reinterpret_cast<const uint4*>(book)[at];
    else
      *reinterpret_cast<uint2*>(raw) = reinterpret_cast<const uint2*>(book)[at];
#pragma unroll
    for (int i = 0; i < EL / 2; ++i) {
      const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&raw[i]));
      v[2 * i] = f.x;
      v[2 * i + 1] = f.y;
    }
  } else {
#pragma unroll
    for (int i = 0; i < EL / 4; ++i) {
      const float4 a = reinterpret_cast<const float4*>(book)[at * (EL / 4) + i];
      v[4 * i] = a.x, v[4 * i + 1] = a.y, v[4 * i + 2] = a.z, v[4 * i + 3] = a.w;
    }
  }
}

// 16 result bytes per thread, eight fp16 or four fp32 weights: DG / EL threads per group.
// Bound by the stores where the codebook is in shared memory; a codebook of 2^16 codewords is gathered from L2 at no
// more than one group per cycle and SM, since each lane's codeword is another line.  (fp16 results with four weights per
// thread: 11008x4096 3x8 43.5 us instead of 29.8, 5120x5120 2x8 19.6 instead of 14.7.  fp32 results with eight:
// 11008x4096 2x8 45 us instead of 31.7, 32 bytes per lane are stored more slowly.)
// the share of block `block` of so many blocks of THREADS threads; `staged`: shared memory for the codebooks
template <int M, bool CB_F16, bool CODE_U16, bool OUT_F16, bool SMEM_BOOK, int DG, int THREADS, int UNROLL>
__device__ __forceinline__ void dequant_share(const void* codebooks, const void* codes, const float* scale, uint64_t G,
                                              FastDiv gpr, uint32_t K, void* __restrict__ W_hat, uint32_t* status,
                                              unsigned char* staged, uint32_t block, uint32_t blocks) {
  constexpr int EL = OUT_F16 ? 8 : 4, PARTS = DG / EL;
  constexpr int kCwBytes = (CB_F16 ? 2 : 4) * DG;
  const void* book = codebooks;
  if (SMEM_BOOK) {
    const uint4* src = reinterpret_cast<const uint4*>(codebooks);
    uint4* dst = reinterpret_cast<uint4*>(staged);
    const int n16 = M * K * kCwBytes / 16;
    for (int i = threadIdx.x; i < n16; i += THREADS) dst[i] = src[i];
    __syncthreads();
    book = staged;
  }
  // UNROLL parts per thread and iteration, a block apart, all their loads issued
  // before the first use: the code -> codeword -> store chain of one group is two
  // dependent memory round trips, so several must be in flight per thread; the codes
  // and scales of the next iteration are asked for ahead of this one's stores (with the
  // loads behind the stores 11008x4096 2x8 fp32 takes 9 us more)
  const uint64_t H = (uint64_t)PARTS * G;
  const uint64_t stride = (uint64_t)blocks * (THREADS * UNROLL);
  uint32_t b[UNROLL][M];
  float s[UNROLL];
  auto fetch = [&](uint64_t base) {
#pragma unroll
    for (int u = 0; u < UNROLL; ++u) {
      const uint64_t h = base + (uint64_t)u * THREADS + threadIdx.x;
      const uint32_t j = (uint32_t)(h / PARTS);
      s[u] = 0.0f;
#pragma unroll
      for (int m = 0; m < M; ++m) b[u][m] = 0;
      if (h < H) {
        if (CODE_U16) {
          const uint16_t* c = reinterpret_cast<const uint16_t*>(codes) + (size_t)j * M;
#pragma unroll
          for (int m = 0; m < M; ++m) b[u][m] = c[m];
        } else if (M % 2 == 0) {  // two adjacent bytes at a time
          const uint16_t* c = reinterpret_cast<const uint16_t*>(codes) + (size_t)j * (M / 2);
#pragma unroll
          for (int m = 0; m < M; m += 2) {
            const uint16_t both = c[m / 2];
            b[u][m] = both & 0xffu;
            b[u][(m + 1) % M] = both >> 8;
          }
        } else {
          const uint8_t* c = reinterpret_cast<const uint8_t*>(codes) + (size_t)j * M;
#pragma unroll
          for (int m = 0; m < M; ++m) b[u][m] = c[m];
        }
        s[u] = scale[fast_div(j, gpr)];  // row of group j (G < 2^32)
      }
    }
  };
  uint64_t base = (uint64_t)block * (THREADS * UNROLL);
  fetch(base);
  for (; base < H; base += stride) {
    bool bad = false;
#pragma unroll
    for (int u = 0; u < UNROLL; ++u) {
#pragma unroll
      for (int m = 0; m < M; ++m) {
        if (b[u][m] >= K) {
          bad = true;
          b[u][m] = 0;
        }
      }
    }
    if (bad && status) atomicOr(status, PVT_DEV_BAD_CODE);
    float v[UNROLL][EL], row_scale[UNROLL];
#pragma unroll
    for (int u = 0; u < UNROLL; ++u)
      load_part<CB_F16, EL, PARTS>(book, b[u][0], threadIdx.x % PARTS, v[u]);
#pragma unroll
    for (int m = 1; m < M; ++m) {  // codebooks added left to right, each sum rounded once
#pragma unroll
      for (int u = 0; u < UNROLL; ++u) {
        float v2[EL];
        load_part<CB_F16, EL, PARTS>(book, m * K + b[u][m], threadIdx.x % PARTS, v2);
#pragma unroll
        for (int i = 0; i < EL; ++i) v[u][i] = __fadd_rn(v[u][i], v2[i]);
      }
    }
#pragma unroll
    for (int u = 0; u < UNROLL; ++u) row_scale[u] = s[u];
    fetch(base + stride);
#pragma unroll
    for (int u = 0; u < UNROLL; ++u) {
      const uint64_t h = base + (uint64_t)u * THREADS + threadIdx.x;
      if (h >= H) continue;
#pragma unroll
      for (int i = 0; i < EL; ++i) v[u][i] = __fmul_rn(row_scale[u], v[u][i]);
      uint32_t w[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (OUT_F16) {
          const __half2 two = __floats2half2_rn(v[u][2 * i % EL], v[u][(2 * i + 1) % EL]);
          w[i] = *reinterpret_cast<const uint32_t*>(&two);
        } else {
          w[i] = __float_as_uint(v[u][i]);
        }
      }
      __stcs(reinterpret_cast<uint4*>(W_hat) + h, make_uint4(w[0], w[1], w[2], w[3]));
    }
  }
}

template <int M, bool CB_F16, bool CODE_U16, bool OUT_F16, bool SMEM_BOOK, int DG>
__global__ void __launch_bounds__(kDqThreads) dequant_kernel(const void* codebooks, const void* codes, const float* scale,
                                                              uint64_t G, FastDiv gpr, uint32_t K, void* __restrict__ W_hat,
                                                              uint32_t* status) {
  __shared__ __align__(16) unsigned char sh_book[SMEM_BOOK ? staged_bytes(M, (CB_F16 ? 2 : 4) * DG) : 16];
  pdl_wait();
  dequant_share<M, CB_F16, CODE_U16, OUT_F16, SMEM_BOOK, DG, kDqThreads, kDqUnroll>(
      codebooks, codes, scale, G, gpr, K, W_hat, status, sh_book, blockIdx.x, gridDim.x);
}

struct DequantIn {
  const void *codebooks, *codes;
  const float* scale;
  uint64_t G;
  FastDiv gpr;
  uint32_t K;
};

// The pass over g of the selection and the dequantisation of all groups from the codes they have, side by side: the first
// n_keys blocks read g, the others write weights.  A step takes few groups of many, and only those get their weights again
// with their new codes, from the search.
// What bounds it: HBM, both ways at once (11008x4096 2x8: 361 MB), or the gathers where the codebook is large.  Whole steps in
// us, one after the other / side by side: 4096x4096 1x16 118 / 113, 11008x4096 2x8 fp32 148 / 138, 3x8 fp16 223 / 214, groups
// of 16 88 / 82, seven layers of a block 1820 / 1740.
// Four blocks per SM, two of them at g with two groups in flight per thread, shares of a sixteenth of an SM's weights so that
// both kinds end together; three codebooks or more need the registers: two blocks, one of them at g with four groups, shares
// of an eighth.  (Three blocks, two / one at g: 1x16 114 / 113, 2x8 140 / 144, 3x8 216 / 218.  One share per SM in place of
// many: 1x16 144, 2x8 209.  Both in every thread, weights formed while g is on its way: 1x16 118, 2x8 144, 3x8 222.)
template <int M, bool CB_F16>
struct Both {
  static constexpr bool kMany = M < 3;
  static constexpr int kBlocks = kMany ? (M == 2 && !CB_F16 ? 3 : 4) : 2, kAtG = kMany ? 2 : 1, kGroups = kMany ? 2 : 4,
                       kShares = kMany ? 16 : 8;
};
template <int M, bool CB_F16, bool CODE_U16, bool OUT_F16, bool SMEM_BOOK, int DG>
__global__ void __launch_bounds__(kNormThreads, Both<M, CB_F16>::kBlocks)
    keys_dequant_kernel(void* __restrict__ W_hat, const select::SelParams p, const DequantIn in, uint32_t n_keys) {
  constexpr int kBook = SMEM_BOOK ? staged_bytes(M, (CB_F16 ? 2 : 4) * DG) : 16, kHist = 4 * kSelBins0;
  __shared__ __align__(16) unsigned char sh[kBook > kHist ? kBook : kHist];
  uint32_t* hist = reinterpret_cast<uint32_t*>(sh);
  pdl_trigger();
  constexpr int U = Both<M, CB_F16>::kGroups * 8 / DG;
  const uint64_t first = (uint64_t)blockIdx.x * (U * kNormThreads);
  if (blockIdx.x < n_keys) {
    for (uint32_t i = threadIdx.x; i < kSelBins0; i += kNormThreads) hist[i] = 0;
    if (threadIdx.x == 0 && first < p.G)  // what the block reads first comes to the L2 while it waits
      prefetch_l2(p.g + first * DG,
                  (uint32_t)((p.G - first < U * kNormThreads ? p.G - first : U * kNormThreads) * DG * sizeof(float)));
  }
  __syncthreads();
  pdl_wait();
  if (blockIdx.x < n_keys)
    select::keys_pass<DG, select::kKeyNorm, U>(p, hist, n_keys);
  else
    dequant_share<M, CB_F16, CODE_U16, OUT_F16, SMEM_BOOK, DG, kNormThreads, kDqUnroll>(
        in.codebooks, in.codes, in.scale, in.G, in.gpr, in.K, W_hat, nullptr, sh, blockIdx.x - n_keys, gridDim.x - n_keys);
}

// Dequantisation of the groups of a list: four weights per thread.
template <bool CB_F16>
__global__ void __launch_bounds__(kDqThreads) dequant_list_kernel(const DequantIn in, const uint32_t* idx, uint64_t k, int M,
                                                                  int code_u16, int out_f16, uint32_t parts, void* W_hat) {
  pdl_trigger();
  pdl_wait();
  for (uint64_t h = (uint64_t)blockIdx.x * kDqThreads + threadIdx.x; h < k * parts; h += (uint64_t)gridDim.x * kDqThreads) {
    const uint32_t j = idx[h / parts], part = (uint32_t)(h % parts);
    if (j >= in.G) continue;
    const float s = in.scale[fast_div(j, in.gpr)];
    float v[4];
    for (int m = 0; m < M; ++m) {
      const size_t at = (size_t)j * M + m;
      uint32_t b = code_u16 ? reinterpret_cast<const uint16_t*>(in.codes)[at] : reinterpret_cast<const uint8_t*>(in.codes)[at];
      if (b >= in.K) b = 0;
      const size_t cw = ((size_t)m * in.K + b) * parts + part;
      float c[4];
      if (CB_F16) {
        const uint2 raw = reinterpret_cast<const uint2*>(in.codebooks)[cw];
        const float2 lo = __half22float2(*reinterpret_cast<const __half2*>(&raw.x));
        const float2 hi = __half22float2(*reinterpret_cast<const __half2*>(&raw.y));
        c[0] = lo.x, c[1] = lo.y, c[2] = hi.x, c[3] = hi.y;
      } else {
        const float4 raw = reinterpret_cast<const float4*>(in.codebooks)[cw];
        c[0] = raw.x, c[1] = raw.y, c[2] = raw.z, c[3] = raw.w;
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) v[i] = m == 0 ? c[i] : __fadd_rn(v[i], c[i]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = __fmul_rn(s, v[i]);
    const size_t to = (size_t)j * parts + part;
    if (out_f16) {
      const __half2 a = __floats2half2_rn(v[0], v[1]), b = __floats2half2_rn(v[2], v[3]);
      reinterpret_cast<uint2*>(W_hat)[to] =
          make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
    } else {
      reinterpret_cast<float4*>(W_hat)[to] = make_float4(v[0], v[1], v[2], v[3]);
    }
  }
}

// where a launch of dequantisation goes
struct Target {
  void* W_hat;
  uint32_t* status;
  const select::SelParams* keys;  // null: dequantisation by itself
  int sm_count;
  cudaStream_t stream;
};

DequantIn dequant_in(const pvt_layer& L, uint64_t G) {
  return DequantIn{L.codebooks, L.codes, L.scale, G, make_fast_div((uint32_t)(L.cols / L.group_dim)),
                   (uint32_t)L.codebook_size};
}

template <int M, bool CB_F16, bool CODE_U16, bool OUT_F16, bool SMEM_BOOK, int DG>
cudaError_t launch_s(const pvt_layer& L, uint64_t G, const Target& t) {
  if (t.keys) {
    constexpr auto kernel = keys_dequant_kernel<M, CB_F16, CODE_U16, OUT_F16, SMEM_BOOK, DG>;
    const uint64_t keys = (G + 2 * kNormThreads - 1) / (2 * kNormThreads), most = (uint64_t)t.sm_count * Both<M, CB_F16>::kAtG;
    const uint64_t per_block = (uint64_t)kNormThreads * kDqUnroll;
    const uint64_t pieces = (DG / (OUT_F16 ? 8 : 4) * G + per_block - 1) / per_block;
    const uint32_t n_keys = (uint32_t)(keys < most ? keys : most);
    const uint64_t shares = (uint64_t)t.sm_count * Both<M, CB_F16>::kShares, rest = pieces < shares ? pieces : shares;
    return launch_dependent(kernel, n_keys + (unsigned)rest, kNormThreads, 0, t.stream, t.W_hat, *t.keys, dequant_in(L, G),
                            n_keys);
  }
  constexpr auto kernel = dequant_kernel<M, CB_F16, CODE_U16, OUT_F16, SMEM_BOOK, DG>;
  uint64_t cap = 0;
  const cudaError_t e = resident_blocks<kernel>(kDqThreads, t.sm_count, &cap);
  if (e != cudaSuccess) return e;
  const uint64_t per_block = (uint64_t)kDqThreads * kDqUnroll;
  const uint64_t want = (DG / (OUT_F16 ? 8 : 4) * G + per_block - 1) / per_block;
  return launch_dependent(kernel, (unsigned)(want < cap ? want : cap), kDqThreads, 0, t.stream, L.codebooks, L.codes, L.scale,
                          G, make_fast_div((uint32_t)(L.cols / DG)), (uint32_t)L.codebook_size, t.W_hat, t.status);
}

template <int M, bool CB_F16, bool CODE_U16, bool OUT_F16, int DG = 8>
cudaError_t launch_t(const pvt_layer& L, uint64_t G, const Target& t) {
  if constexpr (M == 1) {
    constexpr int cw_bytes = (CB_F16 ? 2 : 4) * DG;
    if ((uint64_t)L.codebook_size * cw_bytes > (uint64_t)staged_bytes(1, cw_bytes))
      return launch_s<M, CB_F16, CODE_U16, OUT_F16, false, DG>(L, G, t);
  }
  return launch_s<M, CB_F16, CODE_U16, OUT_F16, true, DG>(L, G, t);
}

template <int M, bool CB_F16, int DG = 8>
cudaError_t launch_c(const pvt_layer& L, uint64_t G, int32_t out_dtype, const Target& t) {
  if (L.code_dtype == PVT_U16)
    return out_dtype == PVT_F16 ? launch_t<M, CB_F16, true, true, DG>(L, G, t) : launch_t<M, CB_F16, true, false, DG>(L, G, t);
  return out_dtype == PVT_F16 ? launch_t<M, CB_F16, false, true, DG>(L, G, t) : launch_t<M, CB_F16, false, false, DG>(L, G, t);
}

cudaError_t launch_any(const pvt_layer& L, uint64_t G, int32_t out_dtype, const Target& t) {
  const bool f16 = L.codebook_dtype == PVT_F16;
  if (L.group_dim == 16)  // groups of 16 weights: one codebook
    return f16 ? launch_c<1, true, 16>(L, G, out_dtype, t) : launch_c<1, false, 16>(L, G, out_dtype, t);
  switch (L.num_codebooks) {
    case 1: return f16 ? launch_c<1, true>(L, G, out_dtype, t) : launch_c<1, false>(L, G, out_dtype, t);
    case 2: return f16 ? launch_c<2, true>(L, G, out_dtype, t) : launch_c<2, false>(L, G, out_dtype, t);
    case 3: return f16 ? launch_c<3, true>(L, G, out_dtype, t) : launch_c<3, false>(L, G, out_dtype, t);
    default: return f16 ? launch_c<4, true>(L, G, out_dtype, t) : launch_c<4, false>(L, G, out_dtype, t);
  }
}

}  // namespace

cudaError_t launch_dequant(const pvt_layer& L, uint64_t G, void* W_hat, int32_t out_dtype, uint32_t* status,
                           int sm_count, cudaStream_t stream) {
  timing_begin(kKernDequant, stream);
  const cudaError_t err = launch_any(L, G, out_dtype, Target{W_hat, status, nullptr, sm_count, stream});
  count_launches(1);
  timing_end(kKernDequant, stream);
  return err;
}

cudaError_t launch_keys_dequant(const select::SelParams& p, const pvt_layer& L, void* W_hat, int32_t out_dtype, int sm_count,
                                cudaStream_t stream) {
  return launch_any(L, p.G, out_dtype, Target{W_hat, nullptr, &p, sm_count, stream});
}

cudaError_t launch_dequant_list(const pvt_layer& L, uint64_t G, const uint32_t* idx, uint64_t k, void* W_hat, int32_t out_dtype,
                                cudaStream_t stream) {
  timing_begin(kKernDequant, stream);
  const uint32_t parts = (uint32_t)L.group_dim / 4;
  const uint64_t want = (k * parts + kDqThreads - 1) / kDqThreads;
  const unsigned blocks = (unsigned)(want < 65536 ? want : 65536);
  const int u16 = L.code_dtype == PVT_U16, o16 = out_dtype == PVT_F16, M = L.num_codebooks;
  auto run = [&](auto kernel) {
    return launch_dependent(kernel, blocks, kDqThreads, 0, stream, dequant_in(L, G), idx, k, M, u16, o16, parts, W_hat);
  };
  const cudaError_t err = L.codebook_dtype == PVT_F16 ? run(dequant_list_kernel<true>) : run(dequant_list_kernel<false>);
  count_launches(1);
  timing_end(kKernDequant, stream);
  return err;
}

}  // namespace pvt
