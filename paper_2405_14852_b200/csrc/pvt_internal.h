// Internal declarations shared by the translation units of libpvt (host side
// launchers, workspace layout, small device helpers).  Not part of the ABI.
#pragma once

#include <atomic>

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "pvt.h"

namespace pvt {

constexpr int kGroupDim = 8;
constexpr int kSmCountFallback = 148;

// ---- workspace layout -------------------------------------------------------
// [0, 256)            header: status word (u32 at 0)
// [256, ...)          region shared by select and encode (they run one after the
//                     other on a stream and never need each other's scratch)
constexpr size_t kWsHeaderBytes = 256;
constexpr size_t kWsAlign = 256;

// selection -------------------------------------------------------------------
constexpr int kSelThreads = 1024;     // passes over the keys
constexpr int kNormThreads = 512;     // pass over g
constexpr int kNormCtas = 2;          // its CTAs per SM
constexpr int kSelBins0 = 8192;       // key bits [30:18]
constexpr int kSelBins1 = 512;        // key bits [17:9]
constexpr int kSelBins2 = 512;        // key bits [8:0]
constexpr uint32_t kSelMaxCtas = 1024;
// counts per CTA, state, the histograms
constexpr uint32_t kSelCountStride = 4;  // a count (u64) per 32 bytes: all later CTAs poll it
constexpr uint32_t kSelScratchWords = 2 * kSelCountStride * kSelMaxCtas + 16 + kSelBins0 + kSelBins1 + kSelBins1 * kSelBins2;

struct SelectLayout {
  size_t scratch_off;  // u32 [kSelScratchWords]
  size_t keys_off;     // u32 [G]
  size_t masks_off;    // u32 [G / 32][2]
  size_t bytes;        // end of the region (from the workspace base)
};
SelectLayout select_layout(uint64_t G);

// encode, M = 1 ---------------------------------------------------------------
// The search kernel leaves, per (target, codebook slice), the sub-chunks of the
// codebook that may hold the nearest codeword; the rescoring kernel evaluates the
// exact distances of those codewords and writes the code.
constexpr int kEncThreads = 256;     // compute threads per CTA (8 warps) + 1 producer warp
constexpr int kChunkCodewords = 256; // codewords per staged chunk (one bulk copy)
constexpr int kSubCodewords = 32;    // tracking granularity of the running minimum
constexpr int kTcSubCodewords = 64;  // the same on the tensor engine
constexpr int kChunkBytes = kChunkCodewords * (kGroupDim * 4 + 4);  // 9216: pairs interleaved + half norms
constexpr int kEncStages = 4;
constexpr int kListLen = 4;          // near-minimum sub-chunks per (target, slice) that the FP32 engine remembers
constexpr int kMaxSlices = 16;

struct CandRecord {        // 16 bytes, one per (target, codebook slice)
  float best;              // smallest fast score of the slice
  uint32_t w[3];           // up to six sub-chunk ids (12 bits each, two per word) whose minimum lies within the margin of
                           // `best`; their number in the upper byte of w[0], kCandOverflow: rescan the whole slice
};
constexpr int kCandMost = 6;
constexpr uint32_t kCandOverflow = 0xffu;

struct EncodeM1Layout {
  size_t cbx_off;      // expanded codebook: n_chunks * kChunkBytes
  size_t n2max_off;    // u32 bit pattern of max ||c||^2
  size_t gbest_off;    // u32 [k]: order-preserving image of the smallest fast score over all slices
  size_t margin_off;   // f32 [k]: rounding-error margin of the fast score of each target
  size_t rec_off;      // CandRecord [n_tiles][n_slices][tile]
  size_t bytes;
  uint32_t n_chunks;
  uint32_t tile;       // targets per tile (kEncThreads * TT)
  uint32_t n_tiles;
  uint32_t n_slices;   // codebook slices per tile (whole chunks each)
  uint32_t n_ctas;
};
EncodeM1Layout encode_m1_layout(uint32_t K, uint64_t k, int sm_count, int targets_per_thread);
int encode_m1_targets_per_thread(uint64_t k, int sm_count);  // 4 or 8
size_t encode_beam_workspace_bytes();

// encode, M = 1 on the tensor cores (fp16 codebooks of at least 1024 codewords)
struct EncodeM1TcLayout {
  size_t bimg_off;    // codebook image in operand order: n_steps * 4096 bytes
  size_t stats_off;   // TcStats: exceptions and extreme norms by block of codewords
  size_t exc_off;     // u32 [K]: codewords the image cannot represent, by block
  size_t gbest_off, margin_off, rec_off;
  size_t sorted_off;  // scratch of the search in spatial order
  size_t counts_off;  // its u32 [n_tiles]: steps of the second sweep
  size_t bytes;
  bool sorted;
  uint32_t n_steps;   // 128-codeword steps
  uint32_t n_tiles;   // tiles of 256 targets
  uint32_t n_slices;
  uint32_t n_ctas;
};
bool encode_m1_use_tc(const pvt_layer& L, uint64_t k);
// fp16 codebooks from here on: the tensor engine (the line that pvt.h states).  20971 / 500000 targets, 512 codewords:
// small-codebook kernel 17 / 173 us, tensor engine 18 / 210; 768: 27 / 237 and 19 / 218; 1024: 29 / 299 and 19 / 224.
constexpr int kM1TensorCodebook = 1024;
// The tensor engine takes codewords and targets in spatial order if both are many: what that leaves out grows with either,
// and its making costs 0.2 ms and some passes over the targets.  Step over 500000 / 700000 / 1000000 / 2000000 targets from
// near stored codes in ms, 65536 codewords: every codeword 1.47 / 1.97 / 2.71 / 5.15, in spatial order 1.51 / 1.84 / 2.36 /
// 3.94; 50000: 1.21 / 1.60 / 2.20 / 4.14 and 1.35 / 1.65 / 2.11 / 3.43; 40000: 1.05 / 1.37 / 1.87 / 3.49 and 1.24 / 1.50 /
// 1.94 / 3.17; 33000: 0.92 / 1.20 / 1.63 / 3.04 and 1.17 / 1.41 / 1.79 / 2.95.  The two meet where targets times the square of
// the codewords is 1.7e15 to 2.6e15 (normally distributed weights; where less can be left out they meet later: Laplace weights,
// 700000 / 800000 / 900000 / 1000000 targets 1.80 / 2.09 / 2.27 / 2.55 and 1.92 / 2.14 / 2.31 / 2.53).
inline bool m1_sorted(uint32_t K, uint64_t k) {
  return K > 32768 && k >= 3000000000000000ull / ((uint64_t)K * K);
}
// Without the tensor engine: codebooks up to here stay in shared memory (both sides measured at the kernel).
constexpr uint32_t kM1SmallCodebook = 1024;
constexpr size_t kM1SmallWorkspace = kWsHeaderBytes + kWsAlign;
void set_m1_search(int mode);
EncodeM1TcLayout encode_m1_tc_layout(uint32_t K, uint64_t k, int sm_count, int group_dim = 8);

// Whether a step dequantises all groups from their present codes beside the selection, and those chosen again from the search:
// while these are few.  It saves the latency of a kernel and, where one alone does not fill HBM, some of its time (2 to 15 us,
// more in the largest layers and from fp32 codebooks to fp16 results); it costs a second write of the chosen groups, in pieces.
// us one after the other less us side by side, at an 8th / 12th / 16th / 24th of the groups, fp16 results: 11008 x 4096 1x16
// 4 / 5 / 6 / 8, 1x12 -4 / -1 / 0 / 1, 2x8 -7 / -2 / 0 / 2; 8192 x 8192 2x8 -12 / -3 / 1 / 4; 28672 x 8192 1x16 -21 / 10 / 40 /
// 23.  512 codewords at a 16th / 32nd / 64th / 100th: 8192 x 8192 1 / 5 / 7 / 8, 28672 x 8192 -21 / -10 / -4 / -1 (of 440).
// Four codebooks at the same: 11008 x 4096 -15 / -2 / 4 / 5, 8192 x 8192 -24 / -9 / -3 / 2.  fp32 codebooks to fp16 results at
// an 8th: 8192 x 8192 1x8 3, 2x8 11.  Three codebooks or more: fp32 results need the whole SM (28672 x 8192 4x8 636 one after
// the other, 699 side by side), and layers with few groups lose (196608 groups, fp32 codebooks, a 100th: 3x8 60 and 82, 4x8 74
// and 85; 131072, fp16: 4x8 72 and 78; from 262144 on side by side is 0 to 6 us less).
inline bool step_dequant_first(const pvt_layer& L, uint64_t k, uint64_t G, int32_t out_dtype) {
  const int M = L.num_codebooks;
  if (M >= 3 && (out_dtype != PVT_F16 || G < 250000)) return false;
  if (M == 4) return k <= G / 64;
  if (M <= 2 && L.codebook_dtype == PVT_F32 && out_dtype == PVT_F16) return k <= G / 8;
  if (M == 1 && L.group_dim == kGroupDim && L.codebook_size <= (int32_t)kM1SmallCodebook && k > 300000) return false;
  return k <= G / 16;
}

// Whether a step over every group of a layer with one small codebook leaves the weights to a kernel after its search: in large
// layers, where eight lanes with an element each store more slowly than 16 bytes per lane.  From the search itself / after it in
// us: fp16 weights, 256 fp16 codewords, 262144 groups 71.7 / 71.8, 524288 129.6 / 129.0, 1048576 243.7 / 239.6, 5636096 1246 /
// 1216, 29360128 6437 / 6282; 1000 codewords 524288 332 / 333, 2097152 1201 / 1199, 29360128 16400 / 16362.  fp32 weights, 256
// codewords: 1048576 243.3 / 242.9, 2097152 473.1 / 470.1, 29360128 6403 / 6348; 512: 2097152 710 / 709; 700: 895 / 896.
inline bool step_weights_after(const pvt_layer& L, uint64_t G, int32_t out_dtype) {
  return out_dtype == PVT_F16 ? G >= 500000 : L.codebook_size <= 512 && G >= 1000000;
}

// where a search writes the weights of the groups it re-encodes as well (null: nowhere)
struct WeightsOut {
  void* W_hat;
  int f16;
};

// launchers (each returns a cudaError_t) --------------------------------------
// (W_hat, k < G: dequantises all groups from their present codes beside the pass over g)
cudaError_t launch_select(const pvt_layer& L, uint64_t G, uint64_t k, uint32_t* idx_out, void* ws, int sm_count,
                          cudaStream_t stream, void* W_hat = nullptr, int32_t out_dtype = 0);
// the same selection on other keys: 0 squared update norm, 1 the same while a straight-through buffer takes the
// step, 2 uniformly random keys, 3 keys of a draw in proportion to the squared update norm (seeded)
cudaError_t launch_select_keyed(const pvt_layer& L, uint64_t G, uint64_t k, uint32_t* idx_out, void* ws, int sm_count,
                                cudaStream_t stream, int key_mode, float* buffer, uint64_t seed);
cudaError_t launch_encode_m1(const pvt_layer& L, uint64_t G, const uint32_t* idx, uint64_t k, float* err_out,
                             WeightsOut out, void* ws, int sm_count, cudaStream_t stream);
cudaError_t launch_encode_m1_small(const pvt_layer& L, uint64_t G, const uint32_t* idx, uint64_t k, float* err_out,
                                   WeightsOut out, void* ws, int sm_count, cudaStream_t stream);
// selection of all groups, their search and dequantisation (if there is anywhere to write) in one kernel
cudaError_t launch_step_m1_small(const pvt_layer& L, uint64_t G, uint32_t* idx_out, WeightsOut out, void* ws, int sm_count,
                                 cudaStream_t stream);
cudaError_t launch_encode_m1_tc(const pvt_layer& L, uint64_t G, const uint32_t* idx, uint64_t k, float* err_out,
                             WeightsOut out, void* ws, int sm_count, cudaStream_t stream);
cudaError_t launch_encode_beam(const pvt_layer& L, uint64_t G, const uint32_t* idx, uint64_t k, float* err_out,
                             WeightsOut out, void* ws, int sm_count, cudaStream_t stream);
cudaError_t launch_encode_g16(const pvt_layer& L, uint64_t G, const uint32_t* idx, uint64_t k, float* err_out,
                              void* ws, cudaStream_t stream);
cudaError_t launch_dequant(const pvt_layer& L, uint64_t G, void* W_hat, int32_t out_dtype, uint32_t* status,
                           int sm_count, cudaStream_t stream);

// the same for the groups of a list
cudaError_t launch_dequant_list(const pvt_layer& L, uint64_t G, const uint32_t* idx, uint64_t k, void* W_hat, int32_t out_dtype,
                                cudaStream_t stream);

cudaError_t launch_pstep_grad(const pvt_layer& L, uint64_t G, double* grad_books, double* grad_scale, uint32_t* status,
                              int sm_count, cudaStream_t stream);
cudaError_t launch_adam(float* param, void* param_f16, const double* grad, float* exp_avg, float* exp_avg_sq,
                        uint64_t n, float lr, float beta1, float beta2, float eps, float bias1, float bias2,
                        int sm_count, cudaStream_t stream);

cudaError_t launch_adam_direction(const float* grad, float* exp_avg, float* exp_avg_sq, float* dir, uint64_t n,
                                  float beta1, float beta2, float eps, float bias1, float bias2, int sm_count,
                                  cudaStream_t stream);

// V step with the subspace size taken from a trust ratio: scratch behind the selection's region
struct TrustLayout {
  size_t idx_off;       // u32 [k]: the selection, ascending
  size_t pairs_a_off;   // u64 [k]: (inverted key, position) pairs; the sorted order ends here
  size_t pairs_b_off;   // u64 [k]: second sort buffer, afterwards f64 [k] squared changes by rank
  size_t counts_off;    // u32 [4 or 1][256][sort_stride], afterwards f64: the changes' sums by block
  size_t saved_off;     // u32 [k]: previous codes by position
  size_t partial_off;   // f64 [norm_blocks]
  size_t stats_off;     // f64 [2] + ticket
  size_t encode_off;    // workspace of the search kernels (own header)
  size_t bytes;
  uint32_t sort_blocks, sort_stride, sort_rounds, norm_blocks;
  bool sort_direct;     // few blocks: one kernel per digit, with counts of all four digits
};
TrustLayout trust_layout(uint64_t G, uint64_t k, size_t encode_bytes, int sm_count);
cudaError_t launch_trust_rank(const pvt_layer& L, uint64_t G, uint64_t k, void* ws, const TrustLayout& t,
                              cudaStream_t stream);
cudaError_t launch_trust_before_search(const pvt_layer& L, uint64_t G, uint64_t k, void* ws, const TrustLayout& t,
                                       cudaStream_t stream);
cudaError_t launch_trust_after_search(const pvt_layer& L, uint64_t G, uint64_t k, float ratio, uint32_t* idx_out,
                                      uint64_t* n_out, double* stats_out, void* ws, const TrustLayout& t,
                                      cudaStream_t stream);

cudaError_t launch_refine(const pvt_layer& L, uint64_t G, const uint32_t* idx, uint64_t k, int max_moves,
                          float* err_out, uint32_t* moves_out, uint32_t* status, cudaStream_t stream);

// ---- division by an invariant 32-bit divisor ---------------------------------------------------------------
// n / d for every 32-bit n as one multiply-high, a subtraction, an addition and two shifts (Granlund and
// Montgomery, "Division by invariant integers using multiplication", 1994, unsigned case): with l = ceil(log2 d),
// mul = floor(2^32 (2^l - d) / d) + 1, t = mulhi(mul, n):  n / d = (t + ((n - t) >> min(l, 1))) >> max(l - 1, 0).
struct FastDiv {
  uint32_t mul, s1, s2;
};
inline FastDiv make_fast_div(uint32_t d) {
  uint32_t l = 0;
  while (l < 32 && ((uint64_t)1 << l) < d) ++l;
  FastDiv f;
  f.mul = (uint32_t)((((uint64_t)1 << 32) * (((uint64_t)1 << l) - d)) / d + 1);
  f.s1 = l < 1 ? l : 1;
  f.s2 = l > 1 ? l - 1 : 0;
  return f;
}
#ifdef __CUDACC__
__device__ __forceinline__ uint32_t fast_div(uint32_t n, const FastDiv& f) {
  const uint32_t t = __umulhi(f.mul, n);
  return (t + ((n - t) >> f.s1)) >> f.s2;
}
#endif

// ---- 32 bytes per thread --------------------------------------------------------------------------------
#ifdef __CUDACC__
// 32 bytes that are not read again: one 256-bit load where the pointer allows it
__device__ __forceinline__ void load8(const float* p, bool wide, float* v) {
  if (wide) {
    asm volatile("ld.global.L1::no_allocate.L2::evict_first.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
                 : "l"(p));
  } else {
    const float4 a = __ldcs(reinterpret_cast<const float4*>(p)), b = __ldcs(reinterpret_cast<const float4*>(p) + 1);
    v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w, v[4] = b.x, v[5] = b.y, v[6] = b.z, v[7] = b.w;
  }
}
// Asks for `bytes` (a multiple of 16, from a 16-byte boundary) to be brought into the L2.  It reads nothing, so it may
// stand before pdl_wait(): whoever writes there meanwhile writes in the same L2.
__device__ __forceinline__ void prefetch_l2(const void* p, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}
__device__ __forceinline__ void store8(float* p, bool wide, const float* v) {
  if (wide) {
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]),
                 "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
                 : "memory");
  } else {
    __stcs(reinterpret_cast<float4*>(p), make_float4(v[0], v[1], v[2], v[3]));
    __stcs(reinterpret_cast<float4*>(p) + 1, make_float4(v[4], v[5], v[6], v[7]));
  }
}
#endif

// ---- programmatic dependent launch --------------------------------------------------------------------
// Consecutive kernels of a call depend on one another, so between two of them the GPU would idle for a launch
// latency.  A kernel launched with launch_dependent() may be scheduled while the kernel before it on the stream
// is still running; every thread of it must execute pdl_wait() before its first access to global memory, which
// returns once that kernel has completed and its writes are visible.  There is no exception for what an earlier
// kernel of the chain wrote, or the caller: the wait is what makes it visible to this grid.  (A prefetch into the L2
// is no access.)  Nor may such a kernel read through the read-only path (__ldg, const ... __restrict__): that promises
// memory nobody writes as long as the kernel lives, while kernels ahead of it are still writing when it starts, and
// lets the compiler move the load ahead of the wait.  Every kernel of a chain calls pdl_trigger() at its start to allow
// the one after it to be scheduled early.  Both are no-ops for a kernel launched the plain way.
#ifdef __CUDACC__
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <typename... KArgs, typename... Args>
cudaError_t launch_dependent(void (*kernel)(KArgs...), unsigned grid, unsigned block, size_t smem, cudaStream_t stream,
                             Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}
#endif

// optional per-kernel timing (benchmark instrumentation) ----------------------
enum KernelId {
  kKernSelect = 0, kKernEncodeMain = 1, kKernEncodeAux = 2, kKernDequant = 3, kKernEncodeRescore = 4,
  kKernPstepGrad = 5, kKernAdam = 6, kKernTrust = 7, kKernRefine = 8, kKernCount = 9
};
void timing_begin(KernelId id, cudaStream_t stream);
void timing_end(KernelId id, cudaStream_t stream);

// remembers the CUDA error behind a PVT_ECUDA return for pvt_last_cuda_error (per host thread)
void record_cuda_error(cudaError_t e);

// multiprocessors of the current device
int device_sm_count();

// ordinal of the current device below kMaxDevices, or -1: for what is set up once per device
constexpr int kMaxDevices = 64;
int device_slot();

// Lets a kernel take all the dynamic shared memory there is; the driver is asked once per kernel and device.
#ifdef __CUDACC__
template <auto kernel>
cudaError_t allow_smem() {
  static std::atomic<bool> done[kMaxDevices];  // of this kernel: the instantiation is its own
  const int dev = device_slot();
  if (dev >= 0 && done[dev].load(std::memory_order_relaxed)) return cudaSuccess;
  cudaFuncAttributes fa;
  cudaError_t e = cudaFuncGetAttributes(&fa, kernel);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(227 * 1024 - fa.sharedSizeBytes));
  if (e == cudaSuccess && dev >= 0) done[dev].store(true, std::memory_order_relaxed);
  return e;
}

// Blocks of a kernel without dynamic shared memory that are resident at once on the device, the grid of a persistent
// kernel; the driver is asked once per kernel and device.
template <auto kernel>
cudaError_t resident_blocks(int threads, int sm_count, uint64_t* blocks) {
  static std::atomic<int> known[kMaxDevices];  // per SM
  const int dev = device_slot();
  int per_sm = dev >= 0 ? known[dev].load(std::memory_order_relaxed) : 0;
  if (per_sm < 1) {
    const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, 0);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) per_sm = 1;
    if (dev >= 0) known[dev].store(per_sm, std::memory_order_relaxed);
  }
  *blocks = (uint64_t)sm_count * (uint64_t)per_sm;
  return cudaSuccess;
}
#endif

// number of kernels launched by this process through the library (a claim the benchmark reports)
void count_launches(int n);

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

}  // namespace pvt
