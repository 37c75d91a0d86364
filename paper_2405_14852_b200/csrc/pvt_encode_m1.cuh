// Pieces shared by the two M = 1 search kernels (FP32 pipe and tensor cores) and
// the rescoring kernel that follows either: parameters, the binary32 target, the
// order-preserving float <-> u32 map, mbarrier / bulk-copy PTX wrappers.
#pragma once

#include <cuda_fp16.h>

#include "pvt_internal.h"

namespace pvt {
namespace m1 {

constexpr uint32_t kMaxSpins = 1u << 22;     // polls after which a wait on an on-chip barrier gives up
constexpr uint32_t kNoWithhold = 0xffffffffu;

// Test hook for the give-up path of the waits (host side, process-wide): the poll limit the search kernels
// run with, and the number of one codebook copy that the producer leaves out so that a wait really runs out.
struct WaitTestHook {
  uint32_t max_spins;      // kMaxSpins unless a test lowered it
  uint32_t withhold_copy;  // kNoWithhold, or the per-CTA sequence number of the copy that is never issued
};
WaitTestHook wait_test_hook();
void set_wait_test_hook(uint32_t max_spins, uint32_t withhold_copy);

struct StepLists {
  const uint16_t* steps;     // rows of step numbers
  const uint32_t* counts;    // steps of each row; null: `most`
  const uint16_t* rows;      // row of each tile; null: its own
  uint32_t stride, most;
};

struct EncM1Params {
  const float* W;
  const float* g;
  const float* scale;
  const uint32_t* idx;
  const uint32_t* place;  // position in the caller's list of each of them (null: its own)
  uint64_t k, G;
  uint32_t gpr;
  FastDiv gpr_div;  // the same as a divisor
  uint32_t dg;  // weights per group: 8, or 16 (tensor engine and rescoring only)
  float eta;
  const float* cbx;
  const uint32_t* n2max_bits;
  uint32_t K, n_tiles, n_slices, tile;
  uint32_t n_units, unit_cw;  // the codebook is cut into n_units units of unit_cw codewords; a slice is a run of whole units
  FastDiv slice_div;          // n_slices as a divisor
  // codewords the fast score cannot represent, always rescored: their number (may be null), and by block of codewords the
  // number and the places in the list
  const uint32_t *any_exc, *n_exc;
  uint32_t exc_blocks, exc_per_block;
  const uint32_t* exc_list;
  uint32_t* gbest;
  float* margin;      // rounding-error margin of each target's fast scores, to which
  float rel_margin;   // this share of the score is added
  CandRecord* rec;
  const void* book;  // the caller's codebook [K][dg]
  void* codes;
  int code_u16;
  WeightsOut out;
  float* err_out;
  uint32_t* status;
  // the search over codewords and targets in spatial order (null elsewhere): the codebook in the order of the image, the
  // codeword at each of its positions, the steps of a tile
  const void* sorted_book;
  const uint32_t* order;
  StepLists lists;       // of the sweep at hand, for the rescoring of the second
  StepLists near_lists;  // for the rescoring: of the first
  uint32_t record, records;  // the record that a launch writes, of so many per target
  uint32_t max_spins;      // poll limit of every wait on an on-chip barrier
  uint32_t withhold_copy;  // kNoWithhold; otherwise the producer skips its copy of this sequence number (test hook)
};

// order-preserving map binary32 -> u32 (and back)
__device__ __forceinline__ uint32_t ord(float f) {
  const uint32_t b = __float_as_uint(f);
  return b ^ ((b >> 31) ? 0xffffffffu : 0x80000000u);
}
__device__ __forceinline__ float unord(uint32_t o) {
  return __uint_as_float(o ^ ((o >> 31) ? 0x80000000u : 0xffffffffu));
}

// t = (W - eta g) / s of group j in binary32: one fma, one division per element
struct TargetIn {
  float4 w0, w1, g0, g1;
  float sc;
};
__device__ __forceinline__ TargetIn load_target(const EncM1Params& p, uint32_t j) {
  const float4* W4 = reinterpret_cast<const float4*>(p.W);
  const float4* g4 = reinterpret_cast<const float4*>(p.g);
  return TargetIn{W4[2 * (size_t)j], W4[2 * (size_t)j + 1], g4[2 * (size_t)j], g4[2 * (size_t)j + 1],
                  p.scale[fast_div(j, p.gpr_div)]};
}
__device__ __forceinline__ void form_target(const TargetIn& in, float eta, float* t) {
  const float neg_eta = -eta;
  t[0] = __fdiv_rn(__fmaf_rn(neg_eta, in.g0.x, in.w0.x), in.sc);
  t[1] = __fdiv_rn(__fmaf_rn(neg_eta, in.g0.y, in.w0.y), in.sc);
  t[2] = __fdiv_rn(__fmaf_rn(neg_eta, in.g0.z, in.w0.z), in.sc);
  t[3] = __fdiv_rn(__fmaf_rn(neg_eta, in.g0.w, in.w0.w), in.sc);
  t[4] = __fdiv_rn(__fmaf_rn(neg_eta, in.g1.x, in.w1.x), in.sc);
  t[5] = __fdiv_rn(__fmaf_rn(neg_eta, in.g1.y, in.w1.y), in.sc);
  t[6] = __fdiv_rn(__fmaf_rn(neg_eta, in.g1.z, in.w1.z), in.sc);
  t[7] = __fdiv_rn(__fmaf_rn(neg_eta, in.g1.w, in.w1.w), in.sc);
}
__device__ __forceinline__ void form_target(const EncM1Params& p, uint32_t j, float* t) {
  form_target(load_target(p, j), p.eta, t);
}

// the same for a group of 16 weights
__device__ __forceinline__ void form_target16(const EncM1Params& p, uint32_t j, float* t) {
  const float4* W4 = reinterpret_cast<const float4*>(p.W) + 4 * (size_t)j;
  const float4* g4 = reinterpret_cast<const float4*>(p.g) + 4 * (size_t)j;
  const float sc = p.scale[fast_div(j, p.gpr_div)];
  const float neg_eta = -p.eta;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const float4 w = W4[q], gg = g4[q];
    t[4 * q + 0] = __fdiv_rn(__fmaf_rn(neg_eta, gg.x, w.x), sc);
    t[4 * q + 1] = __fdiv_rn(__fmaf_rn(neg_eta, gg.y, w.y), sc);
    t[4 * q + 2] = __fdiv_rn(__fmaf_rn(neg_eta, gg.z, w.z), sc);
    t[4 * q + 3] = __fdiv_rn(__fmaf_rn(neg_eta, gg.w, w.w), sc);
  }
}

// one codeword of DG elements as it lies in memory, and widened to binary32
template <bool CB_F16, int DG>
struct RawCodeword {
  uint4 part[CB_F16 ? DG / 8 : DG / 4];
};
template <bool CB_F16, int DG>
__device__ __forceinline__ void fetch_codeword(const void* book, uint32_t kappa, RawCodeword<CB_F16, DG>* raw) {
  constexpr int kParts = CB_F16 ? DG / 8 : DG / 4;
#pragma unroll
  for (int part = 0; part < kParts; ++part)
    raw->part[part] = reinterpret_cast<const uint4*>(book)[(size_t)kappa * kParts + part];
}
template <bool CB_F16, int DG>
__device__ __forceinline__ void widen_codeword(const RawCodeword<CB_F16, DG>& raw, float* c) {
  if (CB_F16) {
#pragma unroll
    for (int part = 0; part < DG / 8; ++part) {
      const __half2* h = reinterpret_cast<const __half2*>(&raw.part[part]);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float2 f = __half22float2(h[i]);
        c[8 * part + 2 * i] = f.x;
        c[8 * part + 2 * i + 1] = f.y;
      }
    }
  } else {
#pragma unroll
    for (int part = 0; part < DG / 4; ++part) {
      c[4 * part] = __uint_as_float(raw.part[part].x);
      c[4 * part + 1] = __uint_as_float(raw.part[part].y);
      c[4 * part + 2] = __uint_as_float(raw.part[part].z);
      c[4 * part + 3] = __uint_as_float(raw.part[part].w);
    }
  }
}
template <bool CB_F16, int DG>
__device__ __forceinline__ void load_codeword(const void* book, uint32_t kappa, float* c) {
  RawCodeword<CB_F16, DG> raw;
  fetch_codeword<CB_F16, DG>(book, kappa, &raw);
  widen_codeword<CB_F16, DG>(raw, c);
}

// largest ||c||^2 / 2 that the operand image of the tensor engine represents
constexpr float kMaxHalfNorm = 60000.0f;

// The power of two that a target of largest element m and squared norm nt2 is scaled by for the tensor engine (zero if it
// is outside the range served); cnmin: the smallest norm of a codeword.
struct TargetScale {
  bool in_range;
  float scale;
};
__device__ __forceinline__ TargetScale target_scale(float m, float nt2, float cnmin) {
  bool in_range = (m < 256.0f) && (nt2 == nt2);  // also false for Inf / NaN
  int e = 0;
  if (in_range && m > 0.0f) {
    e = -ilogbf(m) - 1;
    e = e > 15 ? 15 : e;
  }
  // the best score, at least -2^e (||t|| + min ||c||)^2 / 2, has to be a half
  // (and above that of the padding rows, -327520 2^e)
  const float far = sqrtf(nt2) + cnmin, low = 0.5f * far * far;
  in_range = in_range && low < 150000.0f;
  if (in_range && low > 1.0f) e = min(e, 14 - ilogbf(low));
  return TargetScale{in_range, in_range ? scalbnf(1.0f, e) : 0.0f};
}

// ---- PTX helpers ---------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// 1-D bulk copy global -> shared through the tensor memory accelerator; completes
// `bytes` on the mbarrier.  Both addresses 16-byte aligned, bytes % 16 == 0.
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
// Bounded wait.  Gives up after max_spins polls (or as soon as another thread gave
// up), flags the CTA as aborted and reports through the status word.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile uint32_t* abort_flag,
                                          uint32_t* status, uint32_t max_spins) {
  for (uint32_t spin = 0; spin < max_spins; ++spin) {
    if (mbar_try_wait(bar, parity)) return true;
    if (*abort_flag) return false;
    if (spin > 4096) __nanosleep(64);  // try_wait itself suspends the thread for a short while
  }
  *abort_flag = 1;
  atomicOr(status, PVT_DEV_WAIT_EXPIRED);
  return false;
}


// candidate records: sub-chunks are added one by one, the count last
__device__ __forceinline__ void cand_add(CandRecord& r, uint32_t n, uint32_t sub) {
  const uint32_t bits = sub << (12 * (n & 1u));
#pragma unroll
  for (uint32_t q = 0; q < 3; ++q) r.w[q] |= (n >> 1) == q ? bits : 0u;
}
__device__ __forceinline__ void cand_write(CandRecord* to, const CandRecord& r) {
  *reinterpret_cast<uint4*>(to) = make_uint4(__float_as_uint(r.best), r.w[0], r.w[1], r.w[2]);
}

// units [lo, hi) of slice sl
__device__ __forceinline__ void slice_units(const EncM1Params& p, uint32_t sl, uint32_t* lo, uint32_t* hi) {
  *lo = fast_div(sl * p.n_units, p.slice_div);  // (at most 16 slices of 512 units)
  *hi = fast_div((sl + 1) * p.n_units, p.slice_div);
}

}  // namespace m1

// exact rescoring + code write after either search kernel (defined with the FP32 search)
cudaError_t launch_rescore_m1(const m1::EncM1Params& p, bool codebook_f16, bool tensor_engine, cudaStream_t stream);

}  // namespace pvt
