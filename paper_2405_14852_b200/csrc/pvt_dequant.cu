// dequantize_weights (Algorithm 3, first line): W_hat = s_row * sum_m C_m[b_m] for
// every weight group.  Streaming kernel, persistent grid: one thread per 16 bytes of the
// result, two of them in flight per thread, codes read coalesced, codewords gathered from
// the L2-resident codebook (small ones are first copied to shared memory), and a
// warp's stores contiguous: 512 bytes per instruction.
//
// Arithmetic per element, binary32, each step rounded once: v = c1 (+ c2);
// w = s * v; fp16 output = round-to-nearest-even of w.
#include <cuda_fp16.h>

#include "pvt_internal.h"

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
template <int M, bool CB_F16, bool CODE_U16, bool OUT_F16, bool SMEM_BOOK, int DG>
__global__ void __launch_bounds__(kDqThreads) dequant_kernel(const void* codebooks, const void* codes,
                                                              const float* scale, uint64_t G, FastDiv gpr, uint32_t K,
                                                              void* __restrict__ W_hat, uint32_t* status) {
  constexpr int EL = OUT_F16 ? 8 : 4, PARTS = DG / EL;
  constexpr int kCwBytes = (CB_F16 ? 2 : 4) * DG;
  __shared__ __align__(16) unsigned char sh_book[SMEM_BOOK ? staged_bytes(M, kCwBytes) : 16];
  const void* book = codebooks;
  pdl_wait();
  if (SMEM_BOOK) {
    const uint4* src = reinterpret_cast<const uint4*>(codebooks);
    uint4* dst = reinterpret_cast<uint4*>(sh_book);
    const int n16 = M * K * kCwBytes / 16;
    for (int i = threadIdx.x; i < n16; i += kDqThreads) dst[i] = src[i];
    __syncthreads();
    book = sh_book;
  }
  // kDqUnroll parts per thread and iteration, a block apart, all their loads issued
  // before the first use: the code -> codeword -> store chain of one group is two
  // dependent memory round trips, so several must be in flight per thread; the codes
  // and scales of the next iteration are asked for ahead of this one's stores (with the
  // loads behind the stores 11008x4096 2x8 fp32 takes 9 us more)
  const uint64_t H = (uint64_t)PARTS * G;
  const uint64_t stride = (uint64_t)gridDim.x * (kDqThreads * kDqUnroll);
  uint32_t b[kDqUnroll][M];
  float s[kDqUnroll];
  auto fetch = [&](uint64_t base) {
#pragma unroll
    for (int u = 0; u < kDqUnroll; ++u) {
      const uint64_t h = base + (uint64_t)u * kDqThreads + threadIdx.x;
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
  uint64_t base = (uint64_t)blockIdx.x * (kDqThreads * kDqUnroll);
  fetch(base);
  for (; base < H; base += stride) {
    bool bad = false;
#pragma unroll
    for (int u = 0; u < kDqUnroll; ++u) {
#pragma unroll
      for (int m = 0; m < M; ++m) {
        if (b[u][m] >= K) {
          bad = true;
          b[u][m] = 0;
        }
      }
    }
    if (bad && status) atomicOr(status, PVT_DEV_BAD_CODE);
    float v[kDqUnroll][EL], row_scale[kDqUnroll];
#pragma unroll
    for (int u = 0; u < kDqUnroll; ++u)
      load_part<CB_F16, EL, PARTS>(book, b[u][0], threadIdx.x % PARTS, v[u]);
#pragma unroll
    for (int m = 1; m < M; ++m) {  // codebooks added left to right, each sum rounded once
#pragma unroll
      for (int u = 0; u < kDqUnroll; ++u) {
        float v2[EL];
        load_part<CB_F16, EL, PARTS>(book, m * K + b[u][m], threadIdx.x % PARTS, v2);
#pragma unroll
        for (int i = 0; i < EL; ++i) v[u][i] = __fadd_rn(v[u][i], v2[i]);
      }
    }
#pragma unroll
    for (int u = 0; u < kDqUnroll; ++u) row_scale[u] = s[u];
    fetch(base + stride);
#pragma unroll
    for (int u = 0; u < kDqUnroll; ++u) {
      const uint64_t h = base + (uint64_t)u * kDqThreads + threadIdx.x;
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
cudaError_t launch_s(const pvt_layer& L, uint64_t G, void* W_hat, uint32_t* status, int sm_count, cudaStream_t stream) {
  constexpr auto kernel = dequant_kernel<M, CB_F16, CODE_U16, OUT_F16, SMEM_BOOK, DG>;
  uint64_t cap = 0;
  const cudaError_t e = resident_blocks<kernel>(kDqThreads, sm_count, &cap);
  if (e != cudaSuccess) return e;
  const uint64_t per_block = (uint64_t)kDqThreads * kDqUnroll;
  const uint64_t want = (DG / (OUT_F16 ? 8 : 4) * G + per_block - 1) / per_block;
  return launch_dependent(kernel, (unsigned)(want < cap ? want : cap), kDqThreads, 0, stream, L.codebooks, L.codes, L.scale,
                          G, make_fast_div((uint32_t)(L.cols / DG)), (uint32_t)L.codebook_size, W_hat, status);
}

template <int M, bool CB_F16, bool CODE_U16, bool OUT_F16, int DG = 8>
cudaError_t launch_t(const pvt_layer& L, uint64_t G, void* W_hat, uint32_t* status, int sm_count,
                     cudaStream_t stream) {
  if constexpr (M == 1) {
    constexpr int cw_bytes = (CB_F16 ? 2 : 4) * DG;
    if ((uint64_t)L.codebook_size * cw_bytes > (uint64_t)staged_bytes(1, cw_bytes))
      return launch_s<M, CB_F16, CODE_U16, OUT_F16, false, DG>(L, G, W_hat, status, sm_count, stream);
  }
  return launch_s<M, CB_F16, CODE_U16, OUT_F16, true, DG>(L, G, W_hat, status, sm_count, stream);
}

template <int M, bool CB_F16, bool CODE_U16>
cudaError_t launch_o(const pvt_layer& L, uint64_t G, void* W_hat, int32_t out_dtype, uint32_t* status,
                     int sm_count, cudaStream_t stream) {
  return out_dtype == PVT_F16 ? launch_t<M, CB_F16, CODE_U16, true>(L, G, W_hat, status, sm_count, stream)
                              : launch_t<M, CB_F16, CODE_U16, false>(L, G, W_hat, status, sm_count, stream);
}

template <int M, bool CB_F16>
cudaError_t launch_c(const pvt_layer& L, uint64_t G, void* W_hat, int32_t out_dtype, uint32_t* status,
                     int sm_count, cudaStream_t stream) {
  return L.code_dtype == PVT_U16 ? launch_o<M, CB_F16, true>(L, G, W_hat, out_dtype, status, sm_count, stream)
                                 : launch_o<M, CB_F16, false>(L, G, W_hat, out_dtype, status, sm_count, stream);
}

}  // namespace

cudaError_t launch_dequant(const pvt_layer& L, uint64_t G, void* W_hat, int32_t out_dtype, uint32_t* status,
                           int sm_count, cudaStream_t stream) {
  timing_begin(kKernDequant, stream);
  cudaError_t err;
  const bool f16 = L.codebook_dtype == PVT_F16;
  if (L.group_dim == 16) {  // groups of 16 weights: one codebook
    const bool u16 = L.code_dtype == PVT_U16, o16 = out_dtype == PVT_F16;
#define PVT_DQ16(CB, CU, OF) launch_t<1, CB, CU, OF, 16>(L, G, W_hat, status, sm_count, stream)
    if (f16)
      err = u16 ? (o16 ? PVT_DQ16(true, true, true) : PVT_DQ16(true, true, false))
                : (o16 ? PVT_DQ16(true, false, true) : PVT_DQ16(true, false, false));
    else
      err = u16 ? (o16 ? PVT_DQ16(false, true, true) : PVT_DQ16(false, true, false))
                : (o16 ? PVT_DQ16(false, false, true) : PVT_DQ16(false, false, false));
#undef PVT_DQ16
    count_launches(1);
    timing_end(kKernDequant, stream);
    return err;
  }
  switch (L.num_codebooks) {
    case 1:
      err = f16 ? launch_c<1, true>(L, G, W_hat, out_dtype, status, sm_count, stream)
                : launch_c<1, false>(L, G, W_hat, out_dtype, status, sm_count, stream);
      break;
    case 2:
      err = f16 ? launch_c<2, true>(L, G, W_hat, out_dtype, status, sm_count, stream)
                : launch_c<2, false>(L, G, W_hat, out_dtype, status, sm_count, stream);
      break;
    case 3:
      err = f16 ? launch_c<3, true>(L, G, W_hat, out_dtype, status, sm_count, stream)
                : launch_c<3, false>(L, G, W_hat, out_dtype, status, sm_count, stream);
      break;
    default:
      err = f16 ? launch_c<4, true>(L, G, W_hat, out_dtype, status, sm_count, stream)
                : launch_c<4, false>(L, G, W_hat, out_dtype, status, sm_count, stream);
      break;
  }
  count_launches(1);
  timing_end(kKernDequant, stream);
  return err;
}

}  // namespace pvt
