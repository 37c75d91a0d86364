// Exhaustive nearest-codeword search of the V step for one fp16 codebook on the
// tensor cores (Appendix C / Appendix J: all codewords of the codebook are tried;
// Appendix D: the score ||c||^2 - 2 <t, c>; Eq. 8 for the target).
//
// The score matrix S[n][kappa] = -2^e_n ||t_n - c_kappa||^2 / 2 is a dense contraction of depth 8 plus norm terms: it is
// evaluated tile by tile with tcgen05.mma (fp16 operands, sums in binary32 that are rounded to fp16 accumulators in tensor
// memory) and never leaves the SM -- the epilogue reads each accumulator row once and keeps only its running maximum and
// the 64-codeword sub-chunks that come within an error margin of it.  The exact decision (binary64 distances, argmin of
// (distance, code)) is taken afterwards by the rescoring kernel on those sub-chunks, so the rounding of the operands and
// of the scores only has to be bounded, not small.
//
// Operands (16-byte K chunks of 8 halves, no swizzle, K-major "interleaved" core-matrix layout: 8 rows x 16 bytes per core
// matrix, K chunks 128 bytes apart, 8-row groups 256 bytes apart; one MMA instruction consumes two K chunks):
//   A row n     = [ hi_0 .. hi_7 | 2^e x 3, b_hi, b_lo, b_lo2, 2^e x 2 ]   hi_i = fp16(2^e t_i)
//   B row kappa = [ c_0 .. c_7   | -h_hi, -h_lo, -h_lo2, 1 x 3, 0 x 2 ]    h = ||c||^2/2 = h_hi + h_lo + h_lo2
// The bias b = sum of -t_i (hi_i - 2^e t_i / 2) completes <t, c> - h to minus half the squared distance.  A score near
// the best is therefore small, and with it the rounding to fp16, which is relative; and what the rounding of t to one half
// costs is (2^e t - hi) . (c - t), a small vector times the distance.  So one instruction of fp16 accuracy serves where
// <t, c> - h needed t in two halves, two instructions and binary32 scores, and few sub-chunks come within the margin.
// The codebook image is written once per call by a small kernel in exactly the shared-memory byte order, so eight steps of
// 128 codewords arrive with one 1-D bulk copy (32 KB); the A rows are written by threads of the CTA.
// e_n is chosen per target so that max_i |2^e t_i| lies in [1/2, 1), smaller if the best score would not be a half.
//
// CTA = 256 targets (two 128-row A blocks) x a slice of the codebook, one CTA per SM, persistent over (tile, slice) units.
// Tensor memory: 2 buffers x 2 A blocks x 128 columns = 512 columns.  Each of these four accumulators has one warp that
// issues its MMAs (warps 16-19) and four that read it out (warps 0-15; warp w reads lanes 32 (w % 4) ..): even steps of the
// codebook go through buffer 0, odd ones through buffer 1.  Warp 20 copies the codebook (two stages of eight steps), warps
// 21-23 form the targets of the next unit.  That is six warps on each scheduler; the ones that wait long sleep.
//
// What bounds it: the ring each accumulator goes round - MMA issued, executed, completion seen, read out, release seen -,
// with all of tensor memory in flight (a fp16 accumulator takes a 32-bit column too), and on it the instructions of the
// warps that share a scheduler.  By the SM's own clock counter (1820 MHz under this load) 1048576 targets x 65536 codewords
// take 298 cycles per 256 x 128 scores, an accumulator coming round once in two of these steps; MMAs and tensor-memory
// loads together keep their pipe busy for 200 of them, the minima the ALU for 130.  20971 targets: 64 us.
// Before, in us for 1048576 / 20971 targets: 3228 / 90.6.  The issuing thread elected inside the statement (umma_step):
// 2990; one codebook copy per run of steps in place of one per step: 2510; the limit as a member of the minima: 2402 / 72.4;
// the next unit's targets formed beside the search, units counted without 64-bit divisions: 2367 / 63.6.  (A unit used to
// begin 7500 cycles after the end of the one before it.)
// Tried and slower: two issuing warps (2800), the events of a step handled while the next one's columns are on their way
// (2520: spills), limits exchanged between the two sets (2450), the read-out warps issuing their own MMAs (a bare ring of
// this kind: 411 cycles for 250), 64-column accumulators (344), mma.sync beside tcgen05 (they share a pipe), four or five
// codebook stages (no change).  Against binary32 accumulators, two instructions per step and eight read-out warps: 4556.
// Where the stored codes exclude nothing (random ones), events make it 2703 / 84.  With the slices of a tile one after the
// other, each beginning with the best score so far, 20971 / 88473 such targets take 77 / 253 in place of 86 / 302, but a
// step over the layers of a block whose codes are near 1823 in place of 1802, as the rows of all tiles are then gathered at
// the same time; slices that run together and exchange their best scores after a few steps 78 / 278, and 1820.
// In spatial order (pvt_encode_m1_sorted.cu: many targets) a unit is a tile and goes over a list of steps in place of a slice:
// a copy for each step, the list in shared memory with the rows; 29360128 targets from random codes 74.5 -> 29.5 ms in two
// launches.
//
// Codewords whose half squared norm exceeds the fp16 range get a sentinel row
// that can never win and are listed as "exceptions": the rescoring kernel always
// evaluates them exactly.  Targets outside the range the scaling can serve
// (non-finite, or max |t_i| >= 256) are rescored against the whole codebook.
//
// Groups of 16 weights (Appendix J): two such rows side by side, one for each half of the group, hence two instructions per
// step and A block, the second accumulating onto the first, and 8 KB per step.
#include <atomic>

#include "pvt_encode_m1.cuh"
#include "pvt_encode_m1_sorted.cuh"

namespace pvt {

using namespace m1;

namespace {

constexpr int kTcTile = 256;            // targets per CTA tile
constexpr int kTcStepCw = 128;          // codewords per MMA step (the N of one instruction)
// Operand geometry: eight weights fill one instruction (two K chunks); groups of 16 are two of them, one onto the other:
//   A row = [ hi | 2^e x 3, bias x 3, 2^e x 2 ],   B row = [ c | norm terms x 3, 1 x 3, 0 x 2 ]   per eight weights
template <int DG>
struct TcDim {
  static constexpr int kARowBytes = DG == 8 ? 32 : 64;
  static constexpr int kAGroupBytes = 8 * kARowBytes;          // one 8-row group of A
  static constexpr int kABlockBytes = 128 * kARowBytes;        // one A block of 128 targets
  static constexpr int kBRowBytes = kARowBytes;
  static constexpr int kBGroupBytes = 8 * kBRowBytes;
  static constexpr int kStepBytes = kTcStepCw * kBRowBytes;    // codebook image per step: 4096 or 8192
  static constexpr int kMmas = DG / 8;                         // instructions per step and A block
  static constexpr int kPart = DG / 8;                         // K chunks per codeword
};
constexpr int kTcStepBytes = TcDim<8>::kStepBytes;
constexpr int kTcListLen = 8;           // remembered near-maximum sub-chunks per target
constexpr int kTcGroupSteps = 8;        // steps per codebook stage: the MMA warps wait for the codebook once per eight steps
constexpr int kTcStages = 2;            // codebook stages (eight steps each: 32 KB, or 64 KB for groups of 16)
constexpr int kTcEpiThreads = 512;      // two sets of 256, one thread per target each: even and odd steps
constexpr int kTcEpiWarps = kTcEpiThreads / 32;
constexpr int kTcMmaWarp = kTcEpiWarps;     // the first of four: one per A block and accumulator buffer
constexpr int kTcCopyWarp = kTcMmaWarp + 4;
constexpr int kTcFormWarp = kTcCopyWarp + 1;  // the first of three that form the next unit's targets
constexpr int kTcFormers = 96;
constexpr int kTcThreads = 32 * kTcFormWarp + kTcFormers;  // 24 warps, six per scheduler
// What the search has to know of the codewords, by block of 256 of them: written by the kernel that prepares the image, so
// that nothing has to be cleared before it.
constexpr uint32_t kTcPrepCw = 256;
static_assert(65536 / kTcPrepCw <= kTcTile, "one thread of the search per block");
struct TcStats {
  uint32_t any_exc;  // exceptions of all blocks
  uint32_t n_exc[65536 / kTcPrepCw];  // exceptions of a block, listed from its first place in the list on
  uint2 norms[65536 / kTcPrepCw];     // bit pattern of the largest ||c||^2; 0x7f800000 - that of the smallest (zero: none)
};
constexpr uint32_t kTmemCols = 512;
constexpr float kNegInf = -__builtin_huge_valf();
// share of a score that its error may take, doubled: see the kernel
__host__ __device__ constexpr float rel_margin(int dg) {
  return 2.0f * 1.01f * (dg == 8 ? 2.0f : 3.0f) * 0.0009765625f /* 2^-10 */;
}

}  // namespace

namespace {
std::atomic<int> g_m1_search{PVT_M1_AUTO};
std::atomic<uint32_t> g_max_spins{m1::kMaxSpins};
std::atomic<uint32_t> g_withhold_copy{m1::kNoWithhold};
}

namespace m1 {
WaitTestHook wait_test_hook() {
  return WaitTestHook{g_max_spins.load(std::memory_order_relaxed), g_withhold_copy.load(std::memory_order_relaxed)};
}
void set_wait_test_hook(uint32_t max_spins, uint32_t withhold_copy) {
  g_max_spins.store(max_spins, std::memory_order_relaxed);
  g_withhold_copy.store(withhold_copy, std::memory_order_relaxed);
}
}  // namespace m1

void set_m1_search(int mode) { g_m1_search.store(mode, std::memory_order_relaxed); }

bool encode_m1_use_tc(const pvt_layer& L, uint64_t k) {
  (void)k;
  if (L.num_codebooks != 1 || L.codebook_dtype != PVT_F16) return false;  // the operand image is fp16
  const int mode = g_m1_search.load(std::memory_order_relaxed);
  if (mode == PVT_M1_FP32) return false;
  if (mode == PVT_M1_TENSOR) return true;
  return L.codebook_size >= kM1TensorCodebook;
}

namespace {
// the scratch of the search in spatial order, from `base` on; returns its size
size_t sorted_scratch(char* base, void* records, uint32_t K, uint64_t k, uint32_t n_tiles, uint32_t n_steps,
                      m1::SortedScratch* s) {
  size_t at = 0;
  auto take = [&](size_t bytes) {
    char* p = base ? base + at : nullptr;
    at += align_up(bytes, kWsAlign);
    return p;
  };
  m1::SortedScratch out;
  out.dims = reinterpret_cast<uint32_t*>(take(sizeof(uint32_t) * m1::kSortedLevels));
  out.tree = reinterpret_cast<float*>(take(sizeof(float) << m1::kSortedLevels));
  out.order = reinterpret_cast<uint32_t*>(take(sizeof(uint32_t) << m1::kSortedLevels));
  out.order2 = reinterpret_cast<uint32_t*>(take(sizeof(uint32_t) << m1::kSortedLevels));
  out.book = reinterpret_cast<uint4*>(take(sizeof(uint4) * (size_t)K));
  out.boxes = reinterpret_cast<float*>(take(sizeof(float) * 16 * m1::kSortedSteps));
  out.packed = reinterpret_cast<uint4*>(take(32 * (size_t)(m1::kSortedSteps + m1::kSortedSteps / 8)));
  out.near = reinterpret_cast<uint16_t*>(take(sizeof(uint16_t) * m1::kSortedSteps * m1::kSortedNear));
  out.cells = reinterpret_cast<uint32_t*>(take(sizeof(uint32_t) << m1::kSortedLevels));
  out.starts = reinterpret_cast<uint32_t*>(take(sizeof(uint32_t) << m1::kSortedLevels));
  out.sidx = reinterpret_cast<uint32_t*>(take(sizeof(uint32_t) * k));
  out.place = reinterpret_cast<uint32_t*>(take(sizeof(uint32_t) * k));
  out.tile_step = reinterpret_cast<uint16_t*>(take(sizeof(uint16_t) * n_tiles));
  out.lists = reinterpret_cast<uint16_t*>(take(sizeof(uint16_t) * n_tiles * (size_t)m1::list_stride(n_steps)));
  out.counts = reinterpret_cast<uint32_t*>(take(sizeof(uint32_t) * n_tiles));  // (the last: counts_off)
  out.keys = reinterpret_cast<uint2*>(records);  // (8 bytes per target, done with before the first record of 32)
  if (s) *s = out;
  return at;
}
}  // namespace

EncodeM1TcLayout encode_m1_tc_layout(uint32_t K, uint64_t k, int sm_count, int group_dim) {
  EncodeM1TcLayout e = {};
  e.n_steps = (K + kTcStepCw - 1) / kTcStepCw;
  e.n_tiles = (uint32_t)((k + kTcTile - 1) / kTcTile);
  uint32_t best_s = 1;
  double best_eff = 0.0;
  // a slice should keep at least 16 steps so that building A stays a small part of a unit
  uint32_t s_max = e.n_steps / 16;
  if (s_max < 1) s_max = 1;
  if (s_max > (uint32_t)kMaxSlices) s_max = (uint32_t)kMaxSlices;
  for (uint32_t s = 1; s <= s_max; ++s) {
    const uint64_t units = (uint64_t)e.n_tiles * s;
    const uint64_t rounds = (units + sm_count - 1) / sm_count;
    const double eff = (double)units / (double)(rounds * sm_count);
    if (eff > best_eff + 0.03) {
      best_eff = eff;
      best_s = s;
    }
  }
  e.n_slices = best_s;
  const uint64_t units = (uint64_t)e.n_tiles * e.n_slices;
  e.sorted = group_dim == kGroupDim && m1_sorted(K, k);
  if (e.sorted) e.n_slices = 2;  // two sweeps, a record each
  e.n_ctas = (uint32_t)(units < (uint64_t)sm_count ? units : (uint64_t)sm_count);
  e.bimg_off = kWsHeaderBytes;
  e.stats_off = align_up(e.bimg_off + (size_t)e.n_steps * (group_dim == 16 ? TcDim<16>::kStepBytes : kTcStepBytes),
                         kWsAlign);
  e.exc_off = align_up(e.stats_off + sizeof(TcStats), kWsAlign);
  e.gbest_off = align_up(e.exc_off + sizeof(uint32_t) * K, kWsAlign);
  e.margin_off = align_up(e.gbest_off + sizeof(uint32_t) * k, kWsAlign);
  e.rec_off = align_up(e.margin_off + sizeof(float) * k, kWsAlign);
  e.bytes = align_up(e.rec_off + (size_t)e.n_tiles * e.n_slices * kTcTile * sizeof(CandRecord), kWsAlign);
  if (e.sorted) {
    e.sorted_off = e.bytes;
    e.bytes = sorted_scratch(nullptr, nullptr, K, k, e.n_tiles, e.n_steps, nullptr) + e.bytes;
    e.counts_off = e.bytes - align_up(sizeof(uint32_t) * e.n_tiles, kWsAlign);
  }
  return e;
}

namespace {

// ---- codebook image ------------------------------------------------------------
// SORTED: codewords in the order of `order`, of which a copy is left as well.
template <int DG, bool SORTED>
__global__ void __launch_bounds__(kTcPrepCw) tc_prep_kernel(const uint4* book, uint32_t K, uint32_t n_steps,
                                                       unsigned char* bimg, TcStats* stats, uint32_t* exc_list,
                                                       uint32_t* gbest, uint64_t k, const uint32_t* order,
                                                       uint4* sorted_book) {
  using D = TcDim<DG>;
  __shared__ uint32_t sh_exc, sh_max, sh_inv;
  if (threadIdx.x == 0) sh_exc = sh_max = sh_inv = 0;
  pdl_trigger();
  pdl_wait();
  __syncthreads();
  for (uint64_t n = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; n < k; n += (uint64_t)gridDim.x * blockDim.x)
    gbest[n] = 0xffffffffu;
  const uint32_t pos = blockIdx.x * blockDim.x + threadIdx.x;
  uint32_t n2bits = 0, n2inv = 0;
  if (pos < n_steps * kTcStepCw) {
    const bool real = pos < K;
    const uint32_t kappa = SORTED && real ? order[pos] : pos;
    uint4 raw[D::kPart];
    float n2 = 0.0f, part2[D::kPart];
#pragma unroll
    for (int part = 0; part < D::kPart; ++part) {
      raw[part] = make_uint4(0, 0, 0, 0);
      part2[part] = 0.0f;
      if (real) {
        raw[part] = book[(size_t)kappa * D::kPart + part];
        if (SORTED) sorted_book[(size_t)pos * D::kPart + part] = raw[part];
        const __half2* h = reinterpret_cast<const __half2*>(&raw[part]);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float2 f = __half22float2(h[i]);
          part2[part] = __fmaf_rn(f.x, f.x, part2[part]);
          part2[part] = __fmaf_rn(f.y, f.y, part2[part]);
        }
      }
      n2 += part2[part];
    }
    const bool rep = real && (0.5f * n2 <= kMaxHalfNorm);  // false for NaN / Inf as well
    if (real && !rep) {
      exc_list[blockIdx.x * kTcPrepCw + atomicAdd(&sh_exc, 1u)] = kappa;
    }
    if (rep) {
      n2bits = __float_as_uint(n2);
      n2inv = 0x7f800000u - n2bits;
    }
    const uint32_t step = pos / kTcStepCw, r = pos % kTcStepCw;
    unsigned char* row = bimg + (size_t)step * D::kStepBytes + (r >> 3) * D::kBGroupBytes + (r & 7) * 16;
#pragma unroll
    for (int part = 0; part < D::kPart; ++part) {
      uint4 k1;
      if (rep) {
        const float hn = 0.5f * part2[part];
        const __half h_hi = __float2half_rn(hn);
        const float r1 = hn - __half2float(h_hi);
        const __half h_lo = __float2half_rn(r1);
        const float r2 = r1 - __half2float(h_lo);
        const __half h_lo2 = __float2half_rn(r2);
        const __half2 a = __halves2half2(__hneg(h_hi), __hneg(h_lo));
        const __half2 b = __halves2half2(__hneg(h_lo2), __float2half_rn(1.0f));
        k1 = make_uint4(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b), 0x3c003c00u, 0u);
      } else {
        // padding and exceptions: zero codeword with five of the most negative norm terms, never a maximum
        raw[part] = make_uint4(0, 0, 0, 0);
        k1 = make_uint4(0xfbfffbffu, 0x0000fbffu, 0u, 0xfbfffbffu);
      }
      *reinterpret_cast<uint4*>(row + 256 * part) = raw[part];
      *reinterpret_cast<uint4*>(row + 256 * part + 128) = k1;
    }
  }
  n2bits = __reduce_max_sync(0xffffffffu, n2bits);
  n2inv = __reduce_max_sync(0xffffffffu, n2inv);
  if ((threadIdx.x & 31) == 0) {
    atomicMax(&sh_max, n2bits);
    atomicMax(&sh_inv, n2inv);
  }
  __syncthreads();
  if (threadIdx.x == 0 && blockIdx.x * kTcPrepCw < n_steps * kTcStepCw) {
    stats->n_exc[blockIdx.x] = sh_exc;
    stats->norms[blockIdx.x] = make_uint2(sh_max, sh_inv);
  }
}

// ---- tcgen05 wrappers -----------------------------------------------------------
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_alloc(uint32_t dst_smem, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(cols) : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
}
// One step of an accumulator, D[tmem] = A[smem] * B[smem]^T (fp16 x fp16 -> fp16, M = 128, N = 128, K = 16 per instruction,
// the second, for groups of 16, onto the first), and the arrival on the mbarrier that follows its completion.  The whole
// warp calls; one thread, always the same, is elected inside the statement.  (A branch on the lane in its place leaves the
// compiler without the knowledge that one thread runs it, and the operands go through a loop over the active lanes: issue
// and commit took 107 cycles by themselves, 310 to 370 beside the other warps, where this takes 9.)
template <int MMAS>
__device__ __forceinline__ void umma_step(uint32_t d_tmem, const uint64_t* a_desc, uint64_t b_desc, uint32_t idesc,
                                          uint32_t bar) {
  if constexpr (MMAS == 1) {
    asm volatile(
        "{\n\t.reg .pred one, onto;\n\t"
        "elect.sync _|one, 0xffffffff;\n\t"
        "setp.ne.b32 onto, 0, 0;\n\t"
        "@one tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, onto;\n\t"
        "@one tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%4];\n\t}" ::"r"(d_tmem),
        "l"(a_desc[0]), "l"(b_desc), "r"(idesc), "r"(bar)
        : "memory");
  } else {
    asm volatile(
        "{\n\t.reg .pred one, onto;\n\t"
        "elect.sync _|one, 0xffffffff;\n\t"
        "setp.ne.b32 onto, 0, 0;\n\t"
        "@one tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, onto;\n\t"
        "setp.eq.b32 onto, 0, 0;\n\t"
        "@one tcgen05.mma.cta_group::1.kind::f16 [%0], %5, %6, %3, onto;\n\t"
        "@one tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%4];\n\t}" ::"r"(d_tmem),
        "l"(a_desc[0]), "l"(b_desc), "r"(idesc), "r"(bar), "l"(a_desc[1]), "l"(b_desc + (uint64_t)(2 * (128 >> 4)))
        : "memory");
  }
}
// arrive on the mbarrier once all MMAs issued so far by the warp's elected thread have completed; called by the whole warp
__device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile(
      "{\n\t.reg .pred one;\n\t"
      "elect.sync _|one, 0xffffffff;\n\t"
      "@one tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(bar)
      : "memory");
}
// shared-memory operand descriptor: K-major, no swizzle, K chunks 128 B apart, 8-row groups group_bytes apart
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t group_bytes) {
  return (uint64_t)((saddr & 0x3ffffu) >> 4) | ((uint64_t)(128u >> 4) << 16) |
         ((uint64_t)(group_bytes >> 4) << 32) | (1ull << 46);
}
// instruction descriptor: D, A and B fp16, both K-major, N = 128, M = 128
constexpr uint32_t kIdesc = ((uint32_t)(kTcStepCw >> 3) << 17) | ((128u >> 4) << 24);

// 32 lanes x 128 consecutive columns of 16-bit accumulators -> 64 registers per thread, two columns each
__device__ __forceinline__ void tmem_ld64(uint32_t taddr, uint32_t* v) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.pack::16b.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
        "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
        "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
        "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(taddr)
      : "memory");
}
// Wait for the outstanding tensor-memory loads.  The registers are passed through the
// statement so that no use of them can be scheduled ahead of the wait.
__device__ __forceinline__ void tmem_ld_wait(uint32_t* v, uint32_t* w) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]),
                 "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15]),
                 "+r"(v[16]), "+r"(v[17]), "+r"(v[18]), "+r"(v[19]), "+r"(v[20]), "+r"(v[21]), "+r"(v[22]), "+r"(v[23]),
                 "+r"(v[24]), "+r"(v[25]), "+r"(v[26]), "+r"(v[27]), "+r"(v[28]), "+r"(v[29]), "+r"(v[30]), "+r"(v[31]),
                 "+r"(w[0]), "+r"(w[1]), "+r"(w[2]), "+r"(w[3]), "+r"(w[4]), "+r"(w[5]), "+r"(w[6]), "+r"(w[7]),
                 "+r"(w[8]), "+r"(w[9]), "+r"(w[10]), "+r"(w[11]), "+r"(w[12]), "+r"(w[13]), "+r"(w[14]), "+r"(w[15]),
                 "+r"(w[16]), "+r"(w[17]), "+r"(w[18]), "+r"(w[19]), "+r"(w[20]), "+r"(w[21]), "+r"(w[22]), "+r"(w[23]),
                 "+r"(w[24]), "+r"(w[25]), "+r"(w[26]), "+r"(w[27]), "+r"(w[28]), "+r"(w[29]), "+r"(w[30]), "+r"(w[31])
               :
               : "memory");
}

// The scores are at most zero but for rounding, and among halves with the sign bit set the largest value is the smallest
// unsigned number; one without it, a rounding error above zero, counts as better than all of them, and which of several is
// taken does not matter (all are within the error bound of the best).  So the maxima are minima of unsigned 16-bit
// halves: the three-operand minimum takes two registers per instruction, the two-operand f16x2 maximum one at twice the
// rate - as fast, with half as many instructions.
// Which of 64 keys are below a cap, in 16 instructions: both halves of the result are the cap if none is, otherwise one of
// them is the smallest key.
__device__ __forceinline__ uint32_t key_min64(const uint32_t* v, uint32_t cap) {
  uint32_t m[4] = {__vimin3_u16x2(v[0], v[1], cap), __vimin3_u16x2(v[2], v[3], v[4]), __vimin3_u16x2(v[5], v[6], v[7]),
                   __vimin3_u16x2(v[8], v[9], v[10])};
#pragma unroll
  for (int i = 11; i < 27; i += 8)
#pragma unroll
    for (int q = 0; q < 4; ++q) m[q] = __vimin3_u16x2(m[q], v[i + 2 * q], v[i + 2 * q + 1]);
  m[0] = __vimin3_u16x2(m[0], v[27], v[28]);
  m[1] = __vimin3_u16x2(m[1], v[29], v[30]);
  m[2] = __vimin3_u16x2(m[2], v[31], m[3]);
  return __vimin3_u16x2(m[0], m[1], m[2]);
}
__device__ __forceinline__ uint32_t lower_half(uint32_t x) { return min(x & 0xffffu, x >> 16); }
__device__ __forceinline__ float key_score(uint32_t key) { return __half2float(__ushort_as_half((unsigned short)key)); }
// the key of the largest half not above a score, and of -0 from there on: every half that reaches the score passes
__device__ __forceinline__ uint32_t key_limit(float score) {
  return score < 0.0f ? (uint32_t)__half_as_ushort(__float2half_rd(score)) : 0x8000u;
}

// ---- shared memory -----------------------------------------------------------------
constexpr float kOutOfRange = -1.0f, kAbsent = -2.0f;  // in place of a margin
template <int DG, bool SORTED>
struct TcSmem {
  alignas(128) unsigned char a[2][2][TcDim<DG>::kABlockBytes];  // of this unit and the next: two A blocks of 128 targets
  alignas(128) unsigned char b[kTcStages][kTcGroupSteps][TcDim<DG>::kStepBytes];
  alignas(8) uint64_t full_bar[kTcStages];
  uint64_t empty_bar[kTcStages];
  uint64_t tmem_full[2][2];   // per buffer and A block
  uint64_t tmem_empty[2][2];
  uint64_t a_first;               // the first unit's rows
  uint64_t a_ready[2], a_free[2];  // per unit parity
  uint64_t drain_bar[4];
  // key of the maximum (upper half) and number of the sub-chunk: of the even set, and of the odd one by unit parity
  uint32_t list[3][kTcListLen][kTcTile];
  float margin[2][kTcTile];   // per unit parity and target; kOutOfRange, kAbsent
  float seed[2][kTcTile];     // score of the stored code
  float odd_best[2][kTcTile];  // what the odd set leaves for the even one
  uint32_t odd_cnt[2][kTcTile], odd_evicted[2][kTcTile];
  // in spatial order: the steps of the units being formed and searched, and those the copying warp is at or will be next
  alignas(16) uint16_t steps[SORTED ? 4 : 1][SORTED ? kSortedSteps : 1];
  alignas(16) uint16_t ahead[SORTED ? 2 : 1][SORTED ? kSortedSteps : 1];
  uint32_t n_steps[4];
  uint32_t tmem_base;
  uint32_t abort_flag;
  uint32_t n2max_bits, n2min_inv, n_exc;  // over all codewords
};

// SORTED: a unit is a tile, and its steps are those of a list (pvt_encode_m1_sorted.cu) in place of a slice of the codebook.
template <int DG, bool SORTED>
__global__ void __launch_bounds__(kTcThreads, 1) encode_m1_tc_kernel(const EncM1Params p,
                                                                      const unsigned char* bimg, TcStats* stats) {
  using D = TcDim<DG>;
  constexpr int kStepBytes = D::kStepBytes;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  TcSmem<DG, SORTED>& sm = *reinterpret_cast<TcSmem<DG, SORTED>*>(smem_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  volatile uint32_t* abort_flag = &sm.abort_flag;

  if (tid == 0) {
    sm.abort_flag = 0;
    sm.n2max_bits = sm.n2min_inv = sm.n_exc = 0;
    for (int s = 0; s < kTcStages; ++s) {
      mbar_init(smem_u32(&sm.full_bar[s]), 1);
      mbar_init(smem_u32(&sm.empty_bar[s]), 4);  // one commit per MMA warp, at the stage's last step
    }
    for (int b = 0; b < 2; ++b) {
      for (int q = 0; q < 2; ++q) {
        mbar_init(smem_u32(&sm.tmem_full[b][q]), 1);
        mbar_init(smem_u32(&sm.tmem_empty[b][q]), 128);  // every thread of the four warps
      }
    }
    mbar_init(smem_u32(&sm.a_first), kTcTile);
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&sm.a_ready[b]), kTcFormers);
      mbar_init(smem_u32(&sm.a_free[b]), 4 + kTcEpiWarps);  // one commit per MMA warp, one arrival per read-out warp
    }
    for (int i = 0; i < 4; ++i) mbar_init(smem_u32(&sm.drain_bar[i]), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kTcMmaWarp) {
    tmem_alloc(smem_u32(&sm.tmem_base), kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *reinterpret_cast<volatile uint32_t*>(&sm.tmem_base);

  pdl_wait();
  // unit u is slice u % n_slices of tile u / n_slices
  const uint32_t units = p.n_tiles * p.n_slices;
  // (in 32 bits: at most 2^24 tiles of one slice, fewer of more; a 64-bit division takes a warp a thousand cycles)
  auto unit_steps = [&](uint32_t u, uint32_t* lo, uint32_t* hi) {
    if (SORTED) {  // places in the tile's list
      *lo = 0;
      *hi = p.lists.counts ? p.lists.counts[u] : p.lists.most;
      return u;
    }
    const uint32_t tile = fast_div(u, p.slice_div);
    slice_units(p, u - tile * p.n_slices, lo, hi);
    return tile;
  };
  auto step_list = [&](uint32_t tile) {
    return p.lists.steps + (size_t)(p.lists.rows ? p.lists.rows[tile] : tile) * p.lists.stride;
  };
  auto total_steps = [&] {  // of this CTA
    uint32_t total = 0;
    if (SORTED) {  // (called by whole warps)
      for (uint32_t u = blockIdx.x + lane * gridDim.x; u < units; u += 32 * gridDim.x) {
        uint32_t lo, hi;
        unit_steps(u, &lo, &hi);
        total += hi;
      }
      total = __reduce_add_sync(0xffffffffu, total);
    } else if (p.n_slices == 1) {
      total = ((units - 1 - blockIdx.x) / gridDim.x + 1) * p.n_units;
    } else {
      for (uint32_t u = blockIdx.x; u < units; u += gridDim.x) {
        uint32_t s_lo, s_hi;
        unit_steps(u, &s_lo, &s_hi);
        total += s_hi - s_lo;
      }
    }
    return total;
  };
  // a wait whose answer is the same in every lane: one poll by all of them when the phase is already over, otherwise
  // lane 0 polls, a bounded number of times, and tells the others (all threads polling one barrier slow every barrier
  // operation of the CTA down)
  auto wait_all = [&](uint32_t bar, uint32_t parity) -> bool {
    if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
    bool ok = true;
    if (lane == 0) ok = mbar_wait(bar, parity, abort_flag, p.status, p.max_spins);
    return __shfl_sync(0xffffffffu, ok, 0);
  };
  // the same for waits that are long: the warp sleeps between its polls, so that it takes no issue slots from the others
  auto wait_asleep = [&](uint32_t bar, uint32_t parity, uint32_t ns) -> bool {
    for (uint32_t spin = 0; spin < p.max_spins; ++spin) {
      if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
      if (__any_sync(0xffffffffu, *abort_flag != 0)) return false;
      __nanosleep(ns);
    }
    if (lane == 0) {
      *abort_flag = 1;
      atomicOr(p.status, PVT_DEV_WAIT_EXPIRED);
    }
    return false;
  };

  // the index of a tile's target (an impossible one beyond the last)
  auto target_index = [&](uint32_t tile, uint32_t own) -> uint32_t {
    const uint64_t n = (uint64_t)tile * kTcTile + own;
    return n < p.k ? p.idx[n] : 0xffffffffu;
  };
  // brings a tile's list to shared memory, `threads` threads of number `first` (16 bytes each; the last ones may be padding);
  // no number goes beyond the last step, whatever the list holds, so that none of them leads past the image
  auto bring_list = [&](uint32_t tile, uint16_t* to, uint32_t n, uint32_t first, uint32_t threads) {
    const uint4* from = reinterpret_cast<const uint4*>(step_list(tile));
    const uint32_t last = (p.n_units - 1) * 0x10001u;
    for (uint32_t i = first; i < (n + 7) / 8; i += threads) {
      const uint4 eight = from[i];
      reinterpret_cast<uint4*>(to)[i] =
          make_uint4(__vminu2(eight.x, last), __vminu2(eight.y, last), __vminu2(eight.z, last), __vminu2(eight.w, last));
    }
  };
  // What a target is formed from (index j): in spatial order, where it is farther away, asked for ahead of its use.
  struct RowIn {
    TargetIn in;
    uint32_t code;
    uint32_t best;  // in the second sweep: of the first
  };
  auto load_row = [&](uint32_t j, uint32_t tile, uint32_t own) {
    RowIn row = {};
    if (SORTED && j < p.G) {
      row.code = p.code_u16 ? reinterpret_cast<const uint16_t*>(p.codes)[j] : reinterpret_cast<const uint8_t*>(p.codes)[j];
      row.in = load_target(p, j);
      if (p.record > 0) row.best = p.gbest[(uint64_t)tile * kTcTile + own];
    }
    return row;
  };
  // Forms target `own` of a unit: the group's index j -> its A row, margin and seed.
  auto form_row = [&](uint32_t j, const RowIn& row, uint32_t own, uint32_t par) {
    const uint32_t rb = own >> 7, r = own & 127u;
    unsigned char* a_row = &sm.a[par][rb][(r >> 3) * D::kAGroupBytes + (r & 7) * 16];
    const float n2max = __uint_as_float(sm.n2max_bits);
    const float cnmax = sqrtf(n2max), hmax = 0.5f * n2max;
    const float cnmin = sqrtf(__uint_as_float(0x7f800000u - sm.n2min_inv));  // (infinite if there is none)
    // the target of this thread, its scaling, its A row
    float t[DG];
#pragma unroll
    for (int i = 0; i < DG; ++i) t[i] = 0.0f;
    float prev = -kNegInf;
    const bool have = j < p.G;  // an index out of range is reported by the rescoring kernel
    if (have) {
      // the distance to the stored code: only what comes near it has to be remembered
      uint32_t code = row.code;
      float c[DG];
      if (SORTED) {
        RawCodeword<true, DG> stored;
        fetch_codeword<true, DG>(p.book, code < p.K ? code : 0u, &stored);
        form_target(row.in, p.eta, t);
        widen_codeword<true, DG>(stored, c);
      } else {
        code = p.code_u16 ? reinterpret_cast<const uint16_t*>(p.codes)[j] : reinterpret_cast<const uint8_t*>(p.codes)[j];
        if (DG == 8)
          form_target(p, j, t);
        else
          form_target16(p, j, t);
        if (code < p.K) load_codeword<true, DG>(p.book, code, c);
      }
      if (code < p.K) {
        float d = 0.0f;
#pragma unroll
        for (int i = 0; i < DG; ++i) d = fmaf(t[i] - c[i], t[i] - c[i], d);
        if (d < 1e30f) prev = d;
      }
    }
    float m = 0.0f, nt2 = 0.0f;
#pragma unroll
    for (int i = 0; i < DG; ++i) {
      m = fmaxf(m, fabsf(t[i]));
      nt2 = fmaf(t[i], t[i], nt2);
    }
    const float norm = sqrtf(nt2);
    const TargetScale ts = target_scale(m, nt2, cnmin);
    const bool in_range = ts.in_range;
    const float sc = ts.scale;
    float r2 = 0.0f;  // ||2^e t - hi||^2
    {
      const uint32_t sb = __half_as_ushort(__float2half_rn(sc));
#pragma unroll
      for (int part = 0; part < D::kPart; ++part) {
        __half2 hi[4];
        float bias = 0.0f;  // sum over i of (2^e t_i - hi_i) t_i - 2^e t_i^2 / 2 = -t_i (hi_i - 2^e t_i / 2)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float tx = in_range ? t[8 * part + 2 * i] : 0.0f, ty = in_range ? t[8 * part + 2 * i + 1] : 0.0f;
          const float x = tx * sc, y = ty * sc;  // exact products
          hi[i] = __floats2half2_rn(x, y);
          const float2 back = __half22float2(hi[i]);
          r2 = fmaf(x - back.x, x - back.x, r2);
          r2 = fmaf(y - back.y, y - back.y, r2);
          bias = fmaf(-tx, fmaf(-0.5f, x, back.x), bias);
          bias = fmaf(-ty, fmaf(-0.5f, y, back.y), bias);
        }
        const __half b_hi = __float2half_rn(bias);
        const float r1 = bias - __half2float(b_hi);
        const __half b_lo = __float2half_rn(r1);
        const __half b_lo2 = __float2half_rn(r1 - __half2float(b_lo));
        *reinterpret_cast<uint4*>(a_row + 256 * part) = reinterpret_cast<const uint4*>(hi)[0];
        *reinterpret_cast<uint4*>(a_row + 256 * part + 128) =
            make_uint4(sb | (sb << 16), sb | ((uint32_t)__half_as_ushort(b_hi) << 16),
                       (uint32_t)__half_as_ushort(b_lo) | ((uint32_t)__half_as_ushort(b_lo2) << 16), sb | (sb << 16));
      }
    }
    // A score is S = -2^e ||t - c||^2 / 2 but for rounding: the bias takes 2^e ||t||^2 / 2 off and adds what the rounding
    // of the target costs at c = t.  Error bound, in the score's units: 2^-10 of itself for the rounding to a half
    // (rounded or truncated; twice for two instructions, whose parts have one sign); for the rest of the rounding of the
    // target r ||t - c|| <= 2^-10 |S| + 2^9 r^2 2^-e with r = ||2^e t - hi||; 2^-19 of the sum of magnitudes
    // 2^e (||t|| ||c|| + h + ||t||^2) for the sum of products in binary32, rounded or truncated (twice the terms for
    // groups of 16); 2^-24 where a half is subnormal, and the split of h and of the bias.  Twice that is the margin, the
    // last terms with a factor 2 to spare: margin + kRelMargin |S|.
    // How the tensor cores add and round is not documented: that a sum is formed to binary32 accuracy and is off by at
    // most one unit of 2^-10 of itself per instruction as a half is an assumption.  What supports it are the tests, in
    // which the codes are the same as those of binary64 distances.
    const float margin = 2.0f * (517.0f * r2 / (in_range ? sc : 1.0f) +
                                 (DG == 8 ? 3.814697265625e-6f /* 2^-18 */ : 7.62939453125e-6f) * sc *
                                     (norm * cnmax + hmax + nt2) +
                                 4.76837158203125e-7f /* 2^-21 */);
    sm.margin[par][own] = !have ? kAbsent : in_range ? margin : kOutOfRange;
    float seed = in_range ? -0.5f * sc * prev * 1.0001f : kNegInf;  // (minus infinity without a stored code)
    // the second sweep goes on from what the first one found
    if (SORTED && have && in_range && p.record > 0) seed = fmaxf(seed, -unord(row.best));
    sm.seed[par][own] = seed;
  };

  if (warp == kTcCopyWarp) {
    // ------------------------------------------------------------ bulk-copy producer
    // (the whole warp runs the loop, lane 0 issues the copies: no lane waits at the final barrier meanwhile)
    {
      // total number of steps of this CTA (for the byte count of the last, partial stage)
      const uint32_t total = total_steps();
      uint32_t it = 0;
      bool alive = true;
      // in spatial order: steps of the next unit, whose list is brought near while this one's is gone through
      uint32_t next_n = 0, place = 0;
      if (SORTED && blockIdx.x < units) {
        uint32_t lo;
        unit_steps(blockIdx.x, &lo, &next_n);
        bring_list(blockIdx.x, sm.ahead[0], next_n, lane, 32);
      }
      for (uint32_t u = blockIdx.x; u < units && alive; u += gridDim.x, place ^= 1) {
        uint32_t s_lo = 0, s_hi = next_n;
        if (!SORTED) {
          unit_steps(u, &s_lo, &s_hi);
        } else {
          __syncwarp();  // (all lanes are done with the list before)
          if (u + gridDim.x < units) {
            uint32_t lo;
            unit_steps(u + gridDim.x, &lo, &next_n);
            bring_list(u + gridDim.x, sm.ahead[place ^ 1], next_n, lane, 32);
          }
        }
        for (uint32_t st = s_lo; st < s_hi && alive;) {
          const uint32_t grp = it / kTcGroupSteps, sub = it % kTcGroupSteps, s = grp % kTcStages;
          const uint32_t fb = smem_u32(&sm.full_bar[s]);
          if (sub == 0) {
            if (grp >= (uint32_t)kTcStages) {
              const uint32_t eb = smem_u32(&sm.empty_bar[s]), ep = ((grp / kTcStages) - 1) & 1;
              alive = wait_asleep(eb, ep, 200);
            }
            if (!alive) break;
            const uint32_t left = total - it;
            if (lane == 0)
              mbar_expect_tx(fb, (left < (uint32_t)kTcGroupSteps ? left : (uint32_t)kTcGroupSteps) * kStepBytes);
            __syncwarp();
          }
          // the steps up to the end of the stage or of the unit lie one after the other on both sides: one copy
          const uint32_t room = kTcGroupSteps - sub, n = s_hi - st < room ? s_hi - st : room;
          // test hook: a step that is never copied leaves its stage's barrier incomplete, so the MMA warps' wait
          // for that stage runs out
          if (SORTED) {  // the steps of a list: a copy each
            if ((uint32_t)lane < n && p.withhold_copy != it + lane)
              bulk_g2s(smem_u32(&sm.b[s][sub + lane][0]), bimg + (size_t)sm.ahead[place][st + lane] * kStepBytes, kStepBytes,
                       fb);
          } else if (lane == 0 && p.withhold_copy - it >= n)
            bulk_g2s(smem_u32(&sm.b[s][sub][0]), bimg + (size_t)st * kStepBytes, n * kStepBytes, fb);
          st += n;
          it += n;
        }
      }
      if (!alive && lane == 0) {
        // let every copy that was issued land before the CTA may exit
        const uint32_t groups = (it + kTcGroupSteps - 1) / kTcGroupSteps;
        for (uint32_t back = 1; back <= (uint32_t)kTcStages && back <= groups; ++back) {
          const uint32_t j = groups - back;
          if (p.withhold_copy / kTcGroupSteps == j) continue;  // incomplete on purpose; its other copies landed long ago
          const uint32_t fb = smem_u32(&sm.full_bar[j % kTcStages]);
          for (uint32_t spin = 0; spin < p.max_spins; ++spin) {
            if (mbar_try_wait(fb, (j / kTcStages) & 1)) break;
            __nanosleep(64);
          }
        }
      }
    }
  } else if (warp >= kTcMmaWarp && warp < kTcCopyWarp) {
    // ------------------------------------------------------------ MMA issuers: one warp per A block and accumulator buffer
    // The whole warp runs the loop, so that everything the instructions need (descriptors, addresses, parities) is
    // computed once per warp in converged code; one lane issues.  The loop is part of the ring of the accumulators, so it
    // is kept to the bare sequence: a codebook stage (eight steps, four of this warp's buffer) is one trip, its steps are
    // unrolled with constant parities and descriptor offsets, and a wait that is already over costs a single poll.
    {
      const uint32_t iss = (uint32_t)(warp - kTcMmaWarp), q = iss & 1u, buf = iss >> 1;
      uint64_t a_desc[D::kMmas];
#pragma unroll
      for (int m = 0; m < D::kMmas; ++m)
        a_desc[m] = smem_desc(smem_u32(&sm.a[1][q][0]), D::kAGroupBytes) + (uint64_t)(2 * m * (128 >> 4));
      const uint32_t total = total_steps();
      const uint64_t b_desc0 = smem_desc(smem_u32(&sm.b[0][0][0]), D::kBGroupBytes);
      const uint32_t full = smem_u32(&sm.tmem_full[buf][q]), empty = smem_u32(&sm.tmem_empty[buf][q]);
      const uint32_t d = tmem_base + q * 128 + buf * 256;
      constexpr uint64_t kAUnit = (2 * D::kABlockBytes) >> 4;  // from the rows of even units to those of odd ones
      bool alive = true;
      uint32_t u = blockIdx.x;
      uint32_t unit_i = 0, unit_end = 0;  // units begun and their steps
      uint32_t s = 0, stage_par = 0;      // codebook stage of the trip and the parity of its barrier
      for (uint32_t base = 0; base < total && alive; base += kTcGroupSteps) {
        alive = wait_all(smem_u32(&sm.full_bar[s]), stage_par);
        const uint64_t b_s = b_desc0 + (uint64_t)((s * kTcGroupSteps + buf) * (kStepBytes >> 4));
#pragma unroll
        for (int j = 0; j < kTcGroupSteps / 2; ++j) {
          const uint32_t it = base + 2 * j + buf;
          if (it < total && alive) {
            while (it >= unit_end && alive) {  // the next unit begins: its A rows must be in place
              if (!SORTED) {
                uint32_t s_lo, s_hi;
                unit_steps(u, &s_lo, &s_hi);
                unit_end += s_hi - s_lo;
                u += gridDim.x;
              }
              if (unit_i > 0) umma_commit(smem_u32(&sm.a_free[(unit_i - 1) & 1]));  // the unit before is behind this warp
              alive = wait_all(smem_u32(&sm.a_ready[unit_i & 1]), (unit_i >> 1) & 1);
              if (SORTED && alive) unit_end += *reinterpret_cast<volatile uint32_t*>(&sm.n_steps[unit_i & 3]);
#pragma unroll
              for (int m = 0; m < D::kMmas; ++m) a_desc[m] = (unit_i & 1) ? a_desc[m] + kAUnit : a_desc[m] - kAUnit;
              ++unit_i;
            }
            // the buffer's use number base / 2 + j (base / 2 is even)
            if (alive) alive = wait_all(empty, (j & 1) ? 0u : 1u);
            if (alive) {
              tc_fence_after();
              umma_step<D::kMmas>(d, a_desc, b_s + (uint64_t)(2 * j * (kStepBytes >> 4)), kIdesc, full);
            }
          }
        }
        // this warp has read the whole stage (the last stage is not reused)
        if (alive && base + kTcGroupSteps < total) umma_commit(smem_u32(&sm.empty_bar[s]));
        s = (s == (uint32_t)kTcStages - 1) ? 0 : s + 1;
        if (s == 0) stage_par ^= 1;
      }
      if (!alive) {
        // wait (bounded) for whatever was issued before tensor memory is released
        umma_commit(smem_u32(&sm.drain_bar[2 * buf + q]));
        for (uint32_t spin = 0; spin < kMaxSpins; ++spin) {  // always the full limit: these MMAs do complete
          if (__all_sync(0xffffffffu, mbar_try_wait(smem_u32(&sm.drain_bar[2 * buf + q]), 0))) break;
          __nanosleep(64);
        }
      }
    }
  } else if (warp >= kTcFormWarp) {
    // ------------------------------------------------------------ formers: the targets of the next unit
    // The rows of one unit are formed while the search is at the one before, so that a unit begins with its first
    // instruction and not with three dependent trips to memory.  (The first unit's are formed by the even set.)
    const uint32_t first = (uint32_t)tid - 32 * kTcFormWarp;
    bool alive = wait_all(smem_u32(&sm.a_first), 0);
    __syncwarp();
    mbar_arrive(smem_u32(&sm.a_ready[0]));
    uint32_t unit_i = 1;
    for (uint32_t u = blockIdx.x + gridDim.x; u < units && alive; u += gridDim.x, ++unit_i) {
      const uint32_t par = unit_i & 1, tile = fast_div(u, p.slice_div);
      constexpr int kRounds = (kTcTile + kTcFormers - 1) / kTcFormers;
      uint32_t j[kRounds];
#pragma unroll
      for (int q = 0; q < kRounds; ++q)
        j[q] = first + q * kTcFormers < kTcTile ? target_index(tile, first + q * kTcFormers) : 0xffffffffu;
      RowIn row = load_row(j[0], tile, first);
      uint32_t lo, n = 0;
      if (SORTED) unit_steps(u, &lo, &n);
      alive = wait_asleep(smem_u32(&sm.a_free[par]), ((unit_i >> 1) & 1) ^ 1, 500);
      if (!alive) break;
      if (SORTED) {  // (four places: whoever still reads the list of three units ago has not let this unit's rows be formed)
        bring_list(u, sm.steps[unit_i & 3], n, first, kTcFormers);
        if (first == 0) sm.n_steps[unit_i & 3] = n;
      }
#pragma unroll 1
      for (int q = 0; q < kRounds; ++q) {
        const uint32_t mine = j[0];
#pragma unroll
        for (int i = 0; i + 1 < kRounds; ++i) j[i] = j[i + 1];
        const RowIn next = load_row(q + 1 < kRounds ? j[0] : 0xffffffffu, tile, first + (q + 1) * kTcFormers);
        if (first + q * kTcFormers < kTcTile) form_row(mine, row, first + q * kTcFormers, par);
        row = next;
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // generic-proxy writes -> visible to the MMA
      mbar_arrive(smem_u32(&sm.a_ready[par]));
    }
  } else {
    // ------------------------------------------------------------ read-out
    const uint32_t set = (uint32_t)tid / kTcTile, own = (uint32_t)tid % kTcTile, rb = own >> 7;
    const uint32_t acc = tmem_base + (((uint32_t)(warp & 3) * 32u) << 16) + set * 256 + rb * 128;
    const uint32_t full = smem_u32(&sm.tmem_full[set][rb]), empty = smem_u32(&sm.tmem_empty[set][rb]);
    constexpr float kRelMargin = rel_margin(DG);
    // A warp of the odd set and the one of the even set with the same targets meet once per unit, when the odd one has left
    // what it found.  It goes on at once: its next unit writes to the other of two places.
    auto pair_sync = [&] { asm volatile("bar.sync %0, 64;" ::"r"(1 + (warp & 7)) : "memory"); };
    if (set == 0) {
      const uint32_t j = target_index(fast_div(blockIdx.x, p.slice_div), own);
      const uint2 part = own < p.exc_blocks ? __ldcg(&stats->norms[own]) : make_uint2(0, 0);
      const uint32_t n2bits = __reduce_max_sync(0xffffffffu, part.x), n2inv = __reduce_max_sync(0xffffffffu, part.y);
      if (lane == 0) {
        atomicMax(&sm.n2max_bits, n2bits);
        atomicMax(&sm.n2min_inv, n2inv);
      }
      if (blockIdx.x == 0) {  // for the rescoring kernel
        const uint32_t exc = __reduce_add_sync(0xffffffffu, own < p.exc_blocks ? __ldcg(&stats->n_exc[own]) : 0u);
        if (lane == 0) atomicAdd(&sm.n_exc, exc);
      }
      asm volatile("bar.sync 9, %0;" ::"n"(kTcTile) : "memory");
      if (blockIdx.x == 0 && own == 0) stats->any_exc = sm.n_exc;
      form_row(j, load_row(j, fast_div(blockIdx.x, p.slice_div), own), own, 0);
      if (SORTED) {
        uint32_t lo, n;
        unit_steps(blockIdx.x, &lo, &n);
        bring_list(blockIdx.x, sm.steps[0], n, own, kTcTile);
        if (own == 0) sm.n_steps[0] = n;
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // generic-proxy writes -> visible to the MMA
      mbar_arrive(smem_u32(&sm.a_first));
    }
    uint32_t it = 0;    // steps of the CTA before the unit
    uint32_t uses = 0;  // of this set's buffer
    uint32_t unit_i = 0;
    bool alive = true;  // after a wait that ran out the set only keeps its turn at the barrier of each unit

    for (uint32_t u = blockIdx.x; u < units; u += gridDim.x, ++unit_i) {
      uint32_t s_lo = 0, s_hi = 0, tile = u;
      if (!SORTED) tile = unit_steps(u, &s_lo, &s_hi);
      const uint32_t sl = u - tile * p.n_slices, par = unit_i & 1;
      const uint64_t n = (uint64_t)tile * kTcTile + own;
      if (alive) alive = wait_all(smem_u32(&sm.a_ready[par]), (unit_i >> 1) & 1);
      __syncwarp();
      if (SORTED && alive) s_hi = *reinterpret_cast<volatile uint32_t*>(&sm.n_steps[unit_i & 3]);
      const float margin = sm.margin[par][own], seed = sm.seed[par][own];
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&sm.a_free[par]));
      const bool in_range = margin >= 0.0f;
      uint32_t* const list = &sm.list[set ? 1 + par : 0][0][own];
      float best = kNegInf;

      // Each set takes the steps of one buffer.  The accumulators go to registers in one go, and the buffer back to its MMA
      // warp: what follows, the minima of the 128 columns and their comparison, runs beside the next MMA, and the warps of
      // the other set and block (four per scheduler) fill the waits.
      uint32_t v[32], w[32];
      // the list of remembered sub-chunks lives in shared memory, its fill count and the best evicted entry
      // in registers: the common case of an event is one store and no load
      uint32_t list_cnt = 0, evicted = 0xffffffffu;
      // keys up to this one are remembered: at first those that may reach the score of the stored code.  (With no bound
      // to begin with, every thread remembers its first steps one after the other: 4096x4096 1x16 95 us instead of 90.)
      uint32_t lim = key_limit(seed - fmaf(kRelMargin, fabsf(seed), margin));
      // (a key is a half with the sign bit: the limit is far below 0xffff; nothing is below zero)
      uint32_t cap = in_range ? (lim + 1) * 0x10001u : 0u;
      auto note = [&](uint32_t key, uint32_t sub) {
        if (key <= lim) {
          const uint32_t slot = list_cnt & (kTcListLen - 1);
          if (list_cnt >= kTcListLen) evicted = min(evicted, list[slot * kTcTile]);
          list[slot * kTcTile] = (key << 16) | sub;
          ++list_cnt;
          best = fmaxf(best, key_score(key));
          lim = min(lim, key_limit(best - fmaf(kRelMargin, fabsf(best), margin)));
          cap = (lim + 1) * 0x10001u;
        }
      };
      for (uint32_t st = s_lo + ((it ^ set) & 1); st < s_hi && alive; st += 2, ++uses) {
        alive = wait_all(full, uses & 1);
        if (!alive) break;
        tc_fence_after();
        tmem_ld64(acc, v);
        tmem_ld64(acc + 64, w);
        tmem_ld_wait(v, w);
        tc_fence_before();
        mbar_arrive(empty);
        const uint32_t xa = key_min64(v, cap), xb = key_min64(w, cap);
        if ((xa ^ cap) | (xb ^ cap)) {
          note(lower_half(xa), 2 * st);
          note(lower_half(xb), 2 * st + 1);
        }
      }
      it += s_hi - s_lo;
      if (set == 1) {
        sm.odd_best[par][own] = best;
        sm.odd_cnt[par][own] = list_cnt;
        sm.odd_evicted[par][own] = evicted;
      }
      pair_sync();

      // leave the candidates of this (tile, slice) for the rescoring kernel (minimum convention: -S)
      if (set == 0 && alive && margin != kAbsent) {
        CandRecord rec;
        rec.w[0] = rec.w[1] = rec.w[2] = 0;
        if (in_range) {
          const uint32_t other_cnt = sm.odd_cnt[par][own];
          best = fmaxf(best, sm.odd_best[par][own]);
          lim = min(lim, key_limit(best - fmaf(kRelMargin, fabsf(best), margin)));
          uint32_t cnt_out = 0;
          auto pick = [&](const uint32_t* from, uint32_t cnt) {  // (seldom more than two)
            for (uint32_t q = 0; q < cnt && q < (uint32_t)kTcListLen; ++q) {
              const uint32_t entry = from[q * kTcTile];
              if ((entry >> 16) <= lim) {
                uint32_t sub = entry & 0xffffu;
                if (SORTED) sub = 2u * sm.steps[unit_i & 3][sub >> 1] + (sub & 1u);
                if (cnt_out < (uint32_t)kCandMost) cand_add(rec, cnt_out, sub);
                ++cnt_out;
              }
            }
          };
          pick(list, list_cnt);
          pick(&sm.list[1 + par][0][own], other_cnt);
          rec.best = -best;
          // (an evicted entry stays above every key while nothing was evicted)
          const bool all = cnt_out > (uint32_t)kCandMost || (min(evicted, sm.odd_evicted[par][own]) >> 16) <= lim;
          rec.w[0] |= (all ? kCandOverflow : cnt_out) << 24;
        } else {
          // passes every limit: the whole slice (in spatial order the whole codebook, on account of the first record) is
          // rescored exactly
          rec.best = SORTED && p.record > 0 ? -kNegInf : kNegInf;
          rec.w[0] = kCandOverflow << 24;
        }
        if (SORTED)
          cand_write(&p.rec[((size_t)tile * p.records + p.record) * kTcTile + own], rec);
        else
          cand_write(&p.rec[((size_t)tile * p.n_slices + sl) * kTcTile + own], rec);
        atomicMin(&p.gbest[n], ord(rec.best));
        if (sl == 0 && !(SORTED && p.record > 0)) p.margin[n] = in_range ? margin : 0.0f;
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  pdl_trigger();
  if (warp == kTcMmaWarp) {
    tc_fence_after();
    tmem_dealloc(tmem_base, kTmemCols);
  }
}

}  // namespace

namespace {

template <int DG, bool SORTED>
cudaError_t launch_image(const pvt_layer& L, const EncM1Params& p, const EncodeM1TcLayout& lay, char* base, TcStats* stats,
                         const uint32_t* order, uint4* sorted_book, cudaStream_t stream) {
  const uint32_t n_cw = lay.n_steps * kTcStepCw;
  // enough threads for one codeword each, and for no more than four of the initial minima each until the chip is full
  const uint64_t fill = (p.k + 1023) / 1024 < 592 ? (p.k + 1023) / 1024 : 592;
  const uint32_t image = (n_cw + kTcPrepCw - 1) / kTcPrepCw;
  count_launches(1);
  return launch_dependent(tc_prep_kernel<DG, SORTED>, fill > image ? (unsigned)fill : image, kTcPrepCw, 0, stream,
                          reinterpret_cast<const uint4*>(L.codebooks), p.K, lay.n_steps,
                          reinterpret_cast<unsigned char*>(base + lay.bimg_off), stats,
                          reinterpret_cast<uint32_t*>(base + lay.exc_off), p.gbest, p.k, order, sorted_book);
}

template <int DG, bool SORTED>
cudaError_t launch_search(const EncM1Params& p, const EncodeM1TcLayout& lay, char* base, TcStats* stats,
                          cudaStream_t stream) {
  const cudaError_t err = allow_smem<encode_m1_tc_kernel<DG, SORTED>>();
  if (err != cudaSuccess) return err;
  count_launches(1);
  return launch_dependent(encode_m1_tc_kernel<DG, SORTED>, lay.n_ctas, kTcThreads, sizeof(TcSmem<DG, SORTED>), stream, p,
                          reinterpret_cast<const unsigned char*>(base + lay.bimg_off), stats);
}

template <int DG>
cudaError_t launch_tc(const pvt_layer& L, const EncM1Params& p, const EncodeM1TcLayout& lay, char* base, TcStats* stats,
                      cudaStream_t stream) {
  timing_begin(kKernEncodeAux, stream);
  cudaError_t err = launch_image<DG, false>(L, p, lay, base, stats, nullptr, nullptr, stream);
  timing_end(kKernEncodeAux, stream);
  if (err != cudaSuccess) return err;
  timing_begin(kKernEncodeMain, stream);
  err = launch_search<DG, false>(p, lay, base, stats, stream);
  timing_end(kKernEncodeMain, stream);
  return err;
}

// the same with codewords and targets in spatial order; leaves in p what the rescoring kernel needs
cudaError_t launch_tc_sorted(const pvt_layer& L, EncM1Params& p, const EncodeM1TcLayout& lay, char* base, TcStats* stats,
                             int sm_count, cudaStream_t stream) {
  SortedScratch s;
  sorted_scratch(base + lay.sorted_off, p.rec, p.K, p.k, lay.n_tiles, lay.n_steps, &s);
  const uint32_t* idx = p.idx;
  const TcNorms norms{stats->norms, p.exc_blocks};
  p.n_slices = 1;
  p.slice_div = make_fast_div(1);
  p.sorted_book = s.book;
  p.order = s.order;
  timing_begin(kKernEncodeAux, stream);
  cudaError_t err = launch_sorted_codebook(p.book, p.K, s, stream);
  if (err == cudaSuccess) err = launch_image<8, true>(L, p, lay, base, stats, s.order, s.book, stream);
  if (err == cudaSuccess) err = launch_sorted_targets(p, idx, norms, s, sm_count, stream);
  timing_end(kKernEncodeAux, stream);
  if (err != cudaSuccess) return err;
  p.idx = s.sidx;
  p.place = s.place;
  p.records = 2;
  p.record = 0;
  p.lists = p.near_lists = StepLists{s.near, nullptr, s.tile_step, kSortedNear, kSortedNear};
  timing_begin(kKernEncodeMain, stream);
  err = launch_search<8, true>(p, lay, base, stats, stream);
  timing_end(kKernEncodeMain, stream);
  if (err != cudaSuccess) return err;
  timing_begin(kKernEncodeAux, stream);
  err = launch_sorted_reach(p, norms, s, sm_count, stream);
  timing_end(kKernEncodeAux, stream);
  if (err != cudaSuccess) return err;
  p.record = 1;
  p.lists = StepLists{s.lists, s.counts, nullptr, list_stride(lay.n_steps), 0};
  timing_begin(kKernEncodeMain, stream);
  err = launch_search<8, true>(p, lay, base, stats, stream);
  timing_end(kKernEncodeMain, stream);
  p.n_slices = p.records;
  return err;
}

}  // namespace

cudaError_t launch_encode_m1_tc(const pvt_layer& L, uint64_t G, const uint32_t* idx, uint64_t k, float* err_out,
                             WeightsOut out, void* ws, int sm_count, cudaStream_t stream) {
  const EncodeM1TcLayout lay = encode_m1_tc_layout((uint32_t)L.codebook_size, k, sm_count, L.group_dim);
  char* base = static_cast<char*>(ws);
  TcStats* stats = reinterpret_cast<TcStats*>(base + lay.stats_off);
  EncM1Params p = {};
  p.W = L.W;
  p.g = L.g;
  p.scale = L.scale;
  p.idx = idx;
  p.k = k;
  p.G = G;
  p.gpr = (uint32_t)(L.cols / L.group_dim);
  p.gpr_div = make_fast_div(p.gpr);
  p.dg = (uint32_t)L.group_dim;
  p.eta = L.eta;
  p.cbx = nullptr;
  p.n2max_bits = nullptr;
  p.K = (uint32_t)L.codebook_size;
  p.n_tiles = lay.n_tiles;
  p.n_slices = lay.n_slices;
  p.slice_div = make_fast_div(lay.n_slices);
  p.tile = kTcTile;
  p.n_units = lay.n_steps;
  p.unit_cw = kTcStepCw;
  p.rel_margin = rel_margin(L.group_dim);
  p.any_exc = &stats->any_exc;
  p.n_exc = stats->n_exc;
  p.exc_blocks = (lay.n_steps * kTcStepCw + kTcPrepCw - 1) / kTcPrepCw;
  p.exc_per_block = kTcPrepCw;
  p.exc_list = reinterpret_cast<const uint32_t*>(base + lay.exc_off);
  p.gbest = reinterpret_cast<uint32_t*>(base + lay.gbest_off);
  p.margin = reinterpret_cast<float*>(base + lay.margin_off);
  p.rec = reinterpret_cast<CandRecord*>(base + lay.rec_off);
  p.book = L.codebooks;
  p.codes = L.codes;
  p.code_u16 = L.code_dtype == PVT_U16;
  p.out = out;
  p.err_out = err_out;
  p.status = reinterpret_cast<uint32_t*>(base);
  const WaitTestHook hook = wait_test_hook();
  p.max_spins = hook.max_spins;
  p.withhold_copy = hook.withhold_copy;

  const cudaError_t err = L.group_dim == 16 ? launch_tc<16>(L, p, lay, base, stats, stream)
                          : lay.sorted      ? launch_tc_sorted(L, p, lay, base, stats, sm_count, stream)
                                            : launch_tc<8>(L, p, lay, base, stats, stream);
  if (err != cudaSuccess) return err;
  return launch_rescore_m1(p, true, true, stream);
}

}  // namespace pvt
