// V step whose subspace size follows from a trust ratio (Section 4.3; Appendix J, hyper-parameter paragraph):
// the groups are taken in the order of decreasing update norm and re-encoded, and the longest prefix of that
// order is kept whose total squared change of the dequantised weights stays below ratio^2 * ||W_hat||^2; the
// other groups get their previous codes back; one group always keeps its new code.
//
// The appendix reaches this prefix by re-encoding a hundredth of the weights at a time and undoing the tail of
// the last portion.  Here the k_max groups of largest norm are re-encoded in one go (the search kernels want
// many targets at once), their changes are summed in rank order, and the codes behind the cut are restored:
// the same result whenever the cut falls inside the first k_max groups.
//
// Steps on the stream, after the top-k_max selection (ascending indices):
//   rank_init      key of every selected group (the binary32 norm again, bit for bit) paired with its position; previous
//                  codes; counts of the first digit
//   4 x radix pass stable LSD sort of the pairs by descending key: positions ascend, so equal norms keep the
//                  lowest index first
//   sq_norm        ||W_hat||^2 of the whole matrix in binary64 (fixed summation tree), beside the radix passes
//   search         the library's own encode kernels on the ascending list
//   change         squared change of each group's dequantised weights, summed along the rank order block by block
//   cut            running sum of the blocks, first position that breaks the bound
//   restore        previous codes for every position from the cut on
// Bound by the latency of these short dependent kernels: each is launched while the one before it runs, and up to
// kSortDirect blocks a radix pass is one kernel, with a quarter of the norm beside it.  (Three plain launches per pass: step
// of 4096x4096, k = 20971, 306 us; one kernel per pass 209; now, with a faster selection and search, 170.)
#include <cuda_fp16.h>

#include "pvt_internal.h"

namespace pvt {
namespace {

constexpr int kSortThreads = 256;
constexpr int kSortMaxRounds = 8;                       // pairs per thread
// Up to this many blocks the starts of a block's digits are summed by the block itself from all blocks' counts, and the
// scatter counts the next digit at the places that it writes to: one kernel per digit.  Beyond, the counts that every block
// would read (1 KB per block) and the scattered additions cost more than a counting and a scanning kernel.
constexpr uint32_t kSortDirect = 256;
constexpr int kSortBins = 256;                          // 8 bits per pass, 4 passes over the 32 key bits
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kScanThreads = 1024;
constexpr int kNormThreads = 256;
constexpr int kChangeThreads = 256;
constexpr int kCutThreads = 1024;

// ---- rank order ------------------------------------------------------------------------------------------------

// pair = (~key) << 32 | position in the ascending index list.  Sorting the pairs by their upper half in ascending
// order, stably, gives (norm descending, index ascending).
struct RankParams {
  const float* g;
  uint64_t G, k;
  float eta;
  const uint32_t* idx;
  uint64_t *pairs, *other;  // the two buffers of the sort
  uint32_t* counts;         // [4][256][stride] without a scan, else [256][stride]
  uint32_t n_blocks, stride, rounds;
  const void* codes;
  int M;
  bool code_u16;
  uint32_t* saved;
  uint32_t* status;
  uint32_t *clear_a, *clear_b;  // the statistics and the header of the search's workspace
  uint32_t n_clear_a, n_clear_b;
};

// codes of a group packed into one word: the two-byte code itself for two-byte codes (one codebook), otherwise
// byte m = code of codebook m
__device__ __forceinline__ uint32_t load_packed(const void* codes, uint32_t j, int M, bool code_u16) {
  if (code_u16 || M == 2) return reinterpret_cast<const uint16_t*>(codes)[j];  // (M = 2: first | second << 8)
  const uint8_t* c = reinterpret_cast<const uint8_t*>(codes) + (size_t)j * M;
  uint32_t packed = 0;
  for (int m = 0; m < M; ++m) packed |= (uint32_t)c[m] << (8 * m);
  return packed;
}

__device__ __forceinline__ uint32_t digit_of(uint64_t pair, int pass) { return (uint32_t)(pair >> (32 + 8 * pass)) & 255u; }

template <int DG>
__device__ __forceinline__ uint64_t rank_pair(const RankParams& p, uint64_t a) {
  const uint32_t j = p.idx[a];
  uint32_t key = 0, code = 0;
  if (j < p.G) {
    code = load_packed(p.codes, j, p.M, p.code_u16);
    const float eta = p.eta;
    const float4* src = reinterpret_cast<const float4*>(p.g) + (DG / 4) * (size_t)j;
    float acc = 0.0f;
#pragma unroll
    for (int q = 0; q < DG / 4; ++q) {  // one chain over the DG elements in index order
      const float4 x = src[q];
      float u;
      u = __fmul_rn(eta, x.x); acc = __fmaf_rn(u, u, acc);
      u = __fmul_rn(eta, x.y); acc = __fmaf_rn(u, u, acc);
      u = __fmul_rn(eta, x.z); acc = __fmaf_rn(u, u, acc);
      u = __fmul_rn(eta, x.w); acc = __fmaf_rn(u, u, acc);
    }
    key = __float_as_uint(acc);
  } else {
    atomicOr(p.status, PVT_DEV_BAD_INDEX);
  }
  p.saved[a] = code;
  return ((uint64_t)(~key) << 32) | (uint64_t)(uint32_t)a;
}

// Pairs, previous codes, and how many pairs of the block's tile carry each value of the first digit:
// counts[bin * stride + block].
template <int DG>
__global__ void __launch_bounds__(kSortThreads) rank_init_kernel(const RankParams p, bool direct) {
  __shared__ uint32_t h[kSortBins];
  h[threadIdx.x] = 0;
  pdl_trigger();
  __syncthreads();
  pdl_wait();
  if (blockIdx.x == 0) {
    for (uint32_t i = threadIdx.x; i < p.n_clear_a; i += kSortThreads) p.clear_a[i] = 0;
    for (uint32_t i = threadIdx.x; i < p.n_clear_b; i += kSortThreads) p.clear_b[i] = 0;
  }
  const uint64_t base = (uint64_t)blockIdx.x * p.rounds * kSortThreads;
  for (uint32_t r = 0; r < p.rounds; ++r) {
    const uint64_t a = base + (uint64_t)r * kSortThreads + threadIdx.x;
    if (a < p.k) {
      const uint64_t pair = rank_pair<DG>(p, a);
      p.pairs[a] = pair;
      atomicAdd(&h[digit_of(pair, 0)], 1u);
    }
  }
  __syncthreads();
  uint32_t* row = p.counts + (size_t)threadIdx.x * p.stride;
  row[blockIdx.x] = h[threadIdx.x];
  if (direct) {  // the later digits' counts begin at zero, and so do all counts beyond the last block
#pragma unroll
    for (int pass = 1; pass < 4; ++pass) row[(size_t)pass * kSortBins * p.stride + blockIdx.x] = 0;
    if (blockIdx.x == 0)
      for (uint32_t b = p.n_blocks; b < p.stride; ++b)
#pragma unroll
        for (int pass = 0; pass < 4; ++pass) row[(size_t)pass * kSortBins * p.stride + b] = 0;
  }
}

// the counts of a later digit (more than kSortDirect blocks)
__global__ void __launch_bounds__(kSortThreads) sort_count_kernel(const uint64_t* in, const RankParams p,
                                                                  int pass) {
  __shared__ uint32_t h[kSortBins];
  h[threadIdx.x] = 0;
  pdl_trigger();
  __syncthreads();
  pdl_wait();
  const uint64_t base = (uint64_t)blockIdx.x * p.rounds * kSortThreads;
  for (uint32_t r = 0; r < p.rounds; ++r) {
    const uint64_t a = base + (uint64_t)r * kSortThreads + threadIdx.x;
    if (a < p.k) atomicAdd(&h[digit_of(in[a], pass)], 1u);
  }
  __syncthreads();
  p.counts[(size_t)threadIdx.x * p.stride + blockIdx.x] = h[threadIdx.x];
}

// exclusive prefix sum of n counters in place, one block; every thread owns a contiguous run
__global__ void __launch_bounds__(kScanThreads) sort_scan_kernel(uint32_t* counts, uint32_t n) {
  __shared__ uint32_t part[kScanThreads];
  pdl_trigger();
  pdl_wait();
  const uint32_t per = (n + kScanThreads - 1) / kScanThreads;
  const uint32_t lo = threadIdx.x * per, hi = lo + per < n ? lo + per : n;
  uint32_t sum = 0;
  for (uint32_t i = lo; i < hi; ++i) sum += counts[i];
  part[threadIdx.x] = sum;
  __syncthreads();
  for (int off = 1; off < kScanThreads; off <<= 1) {  // inclusive scan of the run totals
    const uint32_t add = threadIdx.x >= (unsigned)off ? part[threadIdx.x - off] : 0u;
    __syncthreads();
    part[threadIdx.x] += add;
    __syncthreads();
  }
  uint32_t run = threadIdx.x ? part[threadIdx.x - 1] : 0u;
  for (uint32_t i = lo; i < hi; ++i) {
    const uint32_t c = counts[i];
    counts[i] = run;
    run += c;
  }
}

// stable scatter: within a block the pairs are visited in position order (round, then thread); a pair's slot is
// the block's start for its digit + the number of earlier pairs of the block with the same digit
struct ScatterSmem {
  uint32_t seen[kSortBins];             // pairs of earlier rounds, per digit, plus the block's start
  uint32_t cnt[kSortWarps][kSortBins];  // this round: per warp and digit
  uint32_t warp_total[kSortWarps];
};
template <bool DIRECT>
__device__ __forceinline__ void sort_scatter(const uint64_t* in, uint64_t* out, const RankParams& p, int pass,
                                             ScatterSmem& sm) {
  auto& seen = sm.seen;
  auto& cnt = sm.cnt;
  auto& warp_total = sm.warp_total;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint64_t k = p.k;
  if (DIRECT) {
    // thread = digit: pairs of the digit in earlier blocks and in all, then all pairs of smaller digits
    const uint4* row = reinterpret_cast<const uint4*>(p.counts + ((size_t)pass * kSortBins + threadIdx.x) * p.stride);
    uint32_t before = 0, all = 0;
#pragma unroll 8
    for (uint32_t b = 0; b < p.stride / 4; ++b) {
      const uint4 c = __ldcg(row + b);
      const uint32_t four[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        all += four[i];
        before += 4 * b + i < blockIdx.x ? four[i] : 0u;
      }
    }
    uint32_t sum = all;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t x = __shfl_up_sync(0xffffffffu, sum, off);
      if (lane >= off) sum += x;
    }
    if (lane == 31) warp_total[warp] = sum;
    __syncthreads();
    for (int w = 0; w < warp; ++w) before += warp_total[w];
    seen[threadIdx.x] = before + sum - all;
  } else {
    seen[threadIdx.x] = p.counts[(size_t)threadIdx.x * p.stride + blockIdx.x];
  }
  const uint64_t base = (uint64_t)blockIdx.x * p.rounds * kSortThreads;
  for (uint32_t r = 0; r < p.rounds; ++r) {
#pragma unroll
    for (int w = 0; w < kSortWarps; ++w) cnt[w][threadIdx.x] = 0;
    __syncthreads();
    const uint64_t a = base + (uint64_t)r * kSortThreads + threadIdx.x;
    const bool valid = a < k;
    const uint64_t pair = valid ? in[a] : 0;
    const uint32_t d = valid ? digit_of(pair, pass) : kSortBins;  // past the end: a digit of its own
    const uint32_t peers = __match_any_sync(0xffffffffu, d);
    const uint32_t before = __popc(peers & ((1u << lane) - 1u));
    if (valid && before == 0) cnt[warp][d] = __popc(peers);
    __syncthreads();
    {  // thread = digit: turn the per-warp counts into offsets, advance the running total
      uint32_t run = seen[threadIdx.x];
#pragma unroll
      for (int w = 0; w < kSortWarps; ++w) {
        const uint32_t c = cnt[w][threadIdx.x];
        cnt[w][threadIdx.x] = run;
        run += c;
      }
      seen[threadIdx.x] = run;
    }
    __syncthreads();
    if (valid) {
      const uint32_t slot = cnt[warp][d] + before;
      if (slot < k) {
        out[slot] = pair;
        if (DIRECT && pass < 3)
          atomicAdd(p.counts + ((size_t)(pass + 1) * kSortBins + digit_of(pair, pass + 1)) * p.stride +
                        slot / (p.rounds * kSortThreads), 1u);
      }
    }
    __syncthreads();
  }
}
__global__ void __launch_bounds__(kSortThreads) sort_scatter_kernel(const uint64_t* in, uint64_t* out, const RankParams p,
                                                                    int pass) {
  __shared__ ScatterSmem sm;
  pdl_trigger();
  pdl_wait();
  sort_scatter<false>(in, out, p, pass, sm);
}

// ---- codes and dequantised values ------------------------------------------------------------------------------

template <bool CODE_U16>
__device__ __forceinline__ uint32_t load_codes(const void* codes, uint32_t j, int M) {
  return load_packed(codes, j, M, CODE_U16);
}

template <bool CODE_U16>
__device__ __forceinline__ void store_codes(void* codes, uint32_t j, int M, uint32_t packed) {
  if (CODE_U16 || M == 2) {
    reinterpret_cast<uint16_t*>(codes)[j] = (uint16_t)packed;
  } else {
    uint8_t* c = reinterpret_cast<uint8_t*>(codes) + (size_t)j * M;
    for (int m = 0; m < M; ++m) c[m] = (uint8_t)(packed >> (8 * m));
  }
}

template <bool CB_F16, int DG>
__device__ __forceinline__ void codeword(const void* book, uint32_t code, float* c) {
  if (CB_F16) {
#pragma unroll
    for (int part = 0; part < DG / 8; ++part) {
      const uint4 raw = reinterpret_cast<const uint4*>(book)[(size_t)code * (DG / 8) + part];
      const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w[i]));
        c[8 * part + 2 * i] = f.x;
        c[8 * part + 2 * i + 1] = f.y;
      }
    }
  } else {
    const float4* src = reinterpret_cast<const float4*>(book) + (size_t)code * (DG / 4);
#pragma unroll
    for (int part = 0; part < DG / 4; ++part) {
      const float4 x = src[part];
      c[4 * part] = x.x, c[4 * part + 1] = x.y, c[4 * part + 2] = x.z, c[4 * part + 3] = x.w;
    }
  }
}

// the dequantised weights of a group, binary32 exactly as dequantisation forms them: v = c1 (+ c2 ...), w = s * v
template <bool CB_F16, int DG>
__device__ __forceinline__ bool group_weights(const void* books, uint32_t K, int M, uint32_t packed, bool code_u16,
                                              float s, float* w) {
  const uint32_t b0 = (M >= 2 && !code_u16) ? (packed & 0xffu) : packed;
  bool ok = b0 < K;
  for (int m = 1; m < M; ++m) ok = ok && ((packed >> (8 * m)) & 0xffu) < K;
  float v[DG];
  codeword<CB_F16, DG>(books, ok ? b0 : 0, v);
  for (int m = 1; m < M; ++m) {  // codebooks added left to right, each sum rounded once
    float v2[DG];
    codeword<CB_F16, DG>(books, (uint32_t)m * K + (ok ? ((packed >> (8 * m)) & 0xffu) : 0u), v2);
#pragma unroll
    for (int i = 0; i < DG; ++i) v[i] = __fadd_rn(v[i], v2[i]);
  }
#pragma unroll
  for (int i = 0; i < DG; ++i) w[i] = __fmul_rn(s, v[i]);
  return ok;
}

struct TrustParams {
  const void* books;
  void* codes;
  const float* scale;
  uint64_t G, k;
  FastDiv gpr;
  uint32_t K;
  int M;
  const uint32_t* idx;      // ascending list of the selection [k]
  const uint64_t* pairs;    // sorted pairs [k]: lower half = position in idx
  uint32_t* saved;          // previous codes by position [k]
  double* change;           // squared change by rank [k], summed up within blocks of kChangeThreads ranks
  double* block_sum;        // the blocks' sums, then the sums before each block
  uint32_t* rank_idx;       // group index by rank [k] (caller's output)
  double* partial;          // per-block sums of the norm kernel
  uint32_t* ticket;
  double* stats;            // [0] ||W_hat||^2, [1] total squared change of the kept groups
  double* stats_out;        // the caller's copy, or null
  uint64_t* n_out;
  float ratio;
  uint32_t* status;
  const uint32_t* enc_status;
};

// ||W_hat||^2: every thread adds its groups in index order, the block adds its threads in a fixed tree, the last
// block to finish adds the block sums in a fixed tree -- the same binary64 result on every run.
// Four groups are in flight per thread, since each is a chain code -> codeword.  (One at a time, and the last block's sums
// added by one thread: 32 us for 4096x4096 1x16.)
struct NormSmem {
  double sh[kNormThreads];
  bool last;
};
// share `part` of `parts`, one after the other: a share is a run of the trips that all blocks make side by side
template <bool CB_F16, bool CODE_U16, int DG>
__device__ __forceinline__ void sq_norm(const TrustParams& p, uint32_t block, uint32_t blocks, uint32_t part, uint32_t parts,
                                        NormSmem& sm) {
  constexpr int kFlight = DG == 8 ? 4 : 2;
  auto& sh = sm.sh;
  double acc = 0.0;
  bool bad = false;
  const uint64_t stride = (uint64_t)blocks * kNormThreads, trip = kFlight * stride, trips = (p.G + trip - 1) / trip;
  for (uint64_t t = trips * part / parts; t < trips * (part + 1) / parts; ++t) {
    const uint64_t j0 = t * trip + (uint64_t)block * kNormThreads + threadIdx.x;
    uint32_t packed[kFlight];
    float s[kFlight], w[kFlight][DG];
#pragma unroll
    for (int u = 0; u < kFlight; ++u) {
      const uint64_t j = j0 + u * stride;
      packed[u] = j < p.G ? load_codes<CODE_U16>(p.codes, (uint32_t)j, p.M) : 0u;
      s[u] = j < p.G ? p.scale[fast_div((uint32_t)j, p.gpr)] : 0.0f;
    }
#pragma unroll
    for (int u = 0; u < kFlight; ++u)
      bad |= !group_weights<CB_F16, DG>(p.books, p.K, p.M, packed[u], CODE_U16, s[u], w[u]);
#pragma unroll
    for (int u = 0; u < kFlight; ++u) {
      if (j0 + u * stride < p.G) {
#pragma unroll
        for (int i = 0; i < DG; ++i) acc = __fma_rn((double)w[u][i], (double)w[u][i], acc);
      }
    }
  }
  if (bad) atomicOr(p.status, PVT_DEV_BAD_CODE);
  auto block_sum = [&](double x) {
    sh[threadIdx.x] = x;
    __syncthreads();
    for (int off = kNormThreads / 2; off > 0; off >>= 1) {
      if (threadIdx.x < off) sh[threadIdx.x] += sh[threadIdx.x + off];
      __syncthreads();
    }
    return sh[0];
  };
  const double mine = block_sum(acc);
  if (threadIdx.x == 0) {
    p.partial[block] = part ? p.partial[block] + mine : mine;
    __threadfence();
    sm.last = part == parts - 1 && atomicAdd(p.ticket, 1u) == blocks - 1;
  }
  __syncthreads();
  if (sm.last) {
    __threadfence();
    double some = 0.0;
    for (unsigned b = threadIdx.x; b < blocks; b += kNormThreads) some += __ldcg(p.partial + b);
    const double total = block_sum(some);
    if (threadIdx.x == 0) {
      p.stats[0] = total;
      *p.ticket = 0;
    }
  }
}
template <bool CB_F16, bool CODE_U16, int DG>
__global__ void __launch_bounds__(kNormThreads) sq_norm_kernel(const TrustParams p) {
  __shared__ NormSmem sm;
  pdl_trigger();
  pdl_wait();
  sq_norm<CB_F16, CODE_U16, DG>(p, blockIdx.x, gridDim.x, 0, 1, sm);
}

// One pass of the sort, and beside it a quarter of the norm, which needs nothing of it: the few blocks of the sort leave
// the chip to a chain of dependent trips to memory.  (One after the other: 4096x4096 1x16, k = 20971, 175.8 us for 169.7.)
static_assert(kSortThreads == kNormThreads, "blocks of both kinds in one launch");
template <bool CB_F16, bool CODE_U16, int DG>
__global__ void __launch_bounds__(kSortThreads) sort_norm_kernel(const uint64_t* in, uint64_t* out, const RankParams p, int pass,
                                                                 const TrustParams norm, uint32_t norm_blocks) {
  __shared__ union {
    ScatterSmem sort;
    NormSmem norm;
  } sm;
  pdl_trigger();
  pdl_wait();
  if (blockIdx.x < p.n_blocks)
    sort_scatter<true>(in, out, p, pass, sm.sort);
  else
    sq_norm<CB_F16, CODE_U16, DG>(norm, blockIdx.x - p.n_blocks, norm_blocks, pass, 4, sm.norm);
}

// inclusive sums of a block's values in thread order (a fixed tree), by all of its threads; BLOCK / 32 warps
template <int BLOCK>
__device__ __forceinline__ double block_prefix(double x, double* warp_sums) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const double y = __shfl_up_sync(0xffffffffu, x, off);
    if (lane >= off) x += y;
  }
  if (lane == 31) warp_sums[warp] = x;
  __syncthreads();
  if (warp == 0) {
    double w = lane < BLOCK / 32 ? warp_sums[lane] : 0.0;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const double y = __shfl_up_sync(0xffffffffu, w, off);
      if (lane >= off) w += y;
    }
    if (lane < BLOCK / 32) warp_sums[lane] = w;
  }
  __syncthreads();
  return warp ? warp_sums[warp - 1] + x : x;
}

// squared change of the dequantised weights of the group at every rank, summed along the block's ranks; the group index in
// rank order
template <bool CB_F16, bool CODE_U16, int DG>
__global__ void __launch_bounds__(kChangeThreads) change_kernel(const TrustParams p) {
  __shared__ double warp_sums[kChangeThreads / 32];
  const uint64_t r = (uint64_t)blockIdx.x * kChangeThreads + threadIdx.x;
  pdl_trigger();
  pdl_wait();
  const uint32_t a = r < p.k ? (uint32_t)p.pairs[r] : 0xffffffffu;
  uint32_t j = a < p.k ? p.idx[a] : 0xffffffffu;
  double acc = 0.0;
  if (j < p.G) {
    const float s = p.scale[fast_div(j, p.gpr)];
    float wo[DG], wn[DG];
    bool ok = group_weights<CB_F16, DG>(p.books, p.K, p.M, p.saved[a], CODE_U16, s, wo);
    ok &= group_weights<CB_F16, DG>(p.books, p.K, p.M, load_codes<CODE_U16>(p.codes, j, p.M), CODE_U16, s, wn);
    if (!ok) atomicOr(p.status, PVT_DEV_BAD_CODE);
#pragma unroll
    for (int i = 0; i < DG; ++i) {
      const double diff = __dsub_rn((double)wn[i], (double)wo[i]);
      acc = __dadd_rn(acc, __dmul_rn(diff, diff));
    }
  } else {
    j = 0;
  }
  const double run = block_prefix<kChangeThreads>(acc, warp_sums);
  if (r < p.k) {
    p.change[r] = run;
    p.rank_idx[r] = j;
  }
  if (threadIdx.x == kChangeThreads - 1) p.block_sum[blockIdx.x] = run;
}

// One block.  Running sum of the changes in rank order; n = first rank whose running sum is not below
// ratio^2 * ||W_hat||^2, at least 1.  First the sums before each block of the change kernel (each thread owns a contiguous
// run of blocks), then the first block whose end breaks the bound, then the rank in it.
// (All ranks summed by one block's threads, their run totals by one of them: 14.5 us at k = 20971.)
__global__ void __launch_bounds__(kCutThreads) cut_kernel(const TrustParams p) {
  __shared__ double warp_sums[kCutThreads / 32];
  __shared__ unsigned long long first_block, first_bad;
  pdl_trigger();
  pdl_wait();
  const uint64_t n_blocks = (p.k + kChangeThreads - 1) / kChangeThreads;
  const uint64_t per = (n_blocks + kCutThreads - 1) / kCutThreads;
  const uint64_t lo = threadIdx.x * per, hi = lo + per < n_blocks ? lo + per : n_blocks;
  if (threadIdx.x == 0) first_block = first_bad = ~0ull;
  double sum = 0.0;
  for (uint64_t b = lo; b < hi; ++b) sum += __ldcg(p.block_sum + b);
  const double upto = block_prefix<kCutThreads>(sum, warp_sums);
  // (what lies before a thread's run is what its left neighbour has: the same number, taken from the same sum)
  double before = __shfl_up_sync(0xffffffffu, upto, 1);
  if ((threadIdx.x & 31) == 0) before = threadIdx.x ? warp_sums[(threadIdx.x >> 5) - 1] : 0.0;
  const double limit = ((double)p.ratio * (double)p.ratio) * p.stats[0];
  double run = before;
  bool found = false;
  for (uint64_t b = lo; b < hi; ++b) {
    const double mine = __ldcg(p.block_sum + b);
    p.block_sum[b] = run;  // now the sum before the block
    run += mine;
    if (!found && !(run < limit)) {
      found = true;
      atomicMin(&first_block, (unsigned long long)b);
    }
  }
  __syncthreads();
  uint64_t n = p.k;
  if (first_block != ~0ull) {
    const uint64_t r = first_block * kChangeThreads + threadIdx.x;
    if (threadIdx.x < kChangeThreads && r < p.k && !(p.block_sum[first_block] + p.change[r] < limit))
      atomicMin(&first_bad, (unsigned long long)r);
    __syncthreads();
    // (the block's end broke the bound, so some rank of it does: its last one if no other, which differs from the end in
    // the order of the sums if the block is not full)
    const uint64_t end = (first_block + 1) * kChangeThreads < p.k ? (first_block + 1) * kChangeThreads : p.k;
    n = first_bad < end ? first_bad : end - 1;
  }
  if (n < 1) n = 1;  // one change always goes through
  if (threadIdx.x == 0) {
    const double kept = p.block_sum[(n - 1) / kChangeThreads] + p.change[n - 1];
    p.stats[1] = kept;
    if (p.stats_out) {
      p.stats_out[0] = p.stats[0];
      p.stats_out[1] = kept;
    }
    *p.n_out = n;
    const uint32_t e = *p.enc_status;
    if (e) atomicOr(p.status, e);
  }
}

template <bool CODE_U16>
__global__ void __launch_bounds__(256) restore_kernel(const TrustParams p) {
  const uint64_t r = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  pdl_trigger();
  pdl_wait();
  if (r >= p.k || r < *p.n_out) return;
  const uint32_t a = (uint32_t)p.pairs[r];
  const uint32_t j = p.rank_idx[r];
  if (a < p.k && j < p.G) store_codes<CODE_U16>(p.codes, j, p.M, p.saved[a]);
}

size_t host_align(size_t x) { return (x + kWsAlign - 1) & ~(kWsAlign - 1); }

}  // namespace

TrustLayout trust_layout(uint64_t G, uint64_t k, size_t encode_bytes, int sm_count) {
  TrustLayout t;
  // one more round of pairs per thread for every 64 blocks: a block reads all blocks' counts
  const uint64_t rounds = (k + 64 * kSortThreads - 1) / (64 * kSortThreads);
  t.sort_rounds = (uint32_t)(rounds < (uint64_t)kSortMaxRounds ? rounds : (uint64_t)kSortMaxRounds);
  const uint64_t tile = (uint64_t)t.sort_rounds * kSortThreads;
  t.sort_blocks = (uint32_t)((k + tile - 1) / tile);
  t.sort_direct = t.sort_blocks <= kSortDirect;
  t.sort_stride = t.sort_direct ? (t.sort_blocks + 3) / 4 * 4 : t.sort_blocks;
  t.norm_blocks = (uint32_t)(4 * sm_count);
  t.idx_off = host_align(select_layout(G).bytes);
  t.pairs_a_off = host_align(t.idx_off + sizeof(uint32_t) * k);
  t.pairs_b_off = host_align(t.pairs_a_off + sizeof(uint64_t) * k);   // second sort buffer, later the changes
  t.counts_off = host_align(t.pairs_b_off + sizeof(uint64_t) * k);
  const size_t counts = sizeof(uint32_t) * kSortBins * (size_t)t.sort_stride * (t.sort_direct ? 4 : 1);
  const size_t sums = sizeof(double) * ((k + kChangeThreads - 1) / kChangeThreads);  // afterwards, of the changes
  t.saved_off = host_align(t.counts_off + (counts > sums ? counts : sums));
  t.partial_off = host_align(t.saved_off + sizeof(uint32_t) * k);
  t.stats_off = host_align(t.partial_off + sizeof(double) * t.norm_blocks);  // stats[2], ticket
  t.encode_off = host_align(t.stats_off + 64);
  t.bytes = t.encode_off + host_align(encode_bytes);
  return t;
}

namespace {

TrustParams make_params(const pvt_layer& L, uint64_t G, uint64_t k, float ratio, uint32_t* idx_out, uint64_t* n_out,
                        void* ws, const TrustLayout& t) {
  char* base = static_cast<char*>(ws);
  TrustParams p;
  p.books = L.codebooks;
  p.codes = L.codes;
  p.scale = L.scale;
  p.G = G;
  p.k = k;
  p.gpr = make_fast_div((uint32_t)(L.cols / L.group_dim));
  p.K = (uint32_t)L.codebook_size;
  p.M = L.num_codebooks;
  p.idx = reinterpret_cast<const uint32_t*>(base + t.idx_off);
  p.pairs = reinterpret_cast<const uint64_t*>(base + t.pairs_a_off);  // four passes end in the first buffer
  p.saved = reinterpret_cast<uint32_t*>(base + t.saved_off);
  p.change = reinterpret_cast<double*>(base + t.pairs_b_off);
  p.block_sum = reinterpret_cast<double*>(base + t.counts_off);
  p.stats_out = nullptr;
  p.rank_idx = idx_out;
  p.partial = reinterpret_cast<double*>(base + t.partial_off);
  p.stats = reinterpret_cast<double*>(base + t.stats_off);
  p.ticket = reinterpret_cast<uint32_t*>(base + t.stats_off + 2 * sizeof(double));
  p.n_out = n_out;
  p.ratio = ratio;
  p.status = reinterpret_cast<uint32_t*>(base);
  p.enc_status = reinterpret_cast<const uint32_t*>(base + t.encode_off);
  return p;
}

// a pass of the sort with a quarter of the norm
template <bool CB_F16, bool CODE_U16>
cudaError_t launch_sort_norm(const uint64_t* in, uint64_t* out, const RankParams& p, int pass, const TrustParams& norm, int dg,
                             uint32_t norm_blocks, cudaStream_t stream) {
  return launch_dependent(dg == 16 ? sort_norm_kernel<CB_F16, CODE_U16, 16> : sort_norm_kernel<CB_F16, CODE_U16, 8>,
                          p.n_blocks + norm_blocks, kSortThreads, 0, stream, in, out, p, pass, norm, norm_blocks);
}

}  // namespace

cudaError_t launch_trust_rank(const pvt_layer& L, uint64_t G, uint64_t k, void* ws, const TrustLayout& t,
                              cudaStream_t stream) {
  char* base = static_cast<char*>(ws);
  uint32_t* status = reinterpret_cast<uint32_t*>(base);
  const uint32_t* idx = reinterpret_cast<const uint32_t*>(base + t.idx_off);
  RankParams p;
  p.g = L.g;
  p.G = G;
  p.k = k;
  p.eta = L.eta;
  p.idx = idx;
  p.pairs = reinterpret_cast<uint64_t*>(base + t.pairs_a_off);
  p.other = reinterpret_cast<uint64_t*>(base + t.pairs_b_off);
  p.counts = reinterpret_cast<uint32_t*>(base + t.counts_off);
  p.n_blocks = t.sort_blocks;
  p.stride = t.sort_stride;
  p.rounds = t.sort_rounds;
  p.codes = L.codes;
  p.M = L.num_codebooks;
  p.code_u16 = L.code_dtype == PVT_U16;
  p.saved = reinterpret_cast<uint32_t*>(base + t.saved_off);
  p.status = status;
  p.clear_a = reinterpret_cast<uint32_t*>(base + t.stats_off);
  p.n_clear_a = 64 / 4;
  p.clear_b = reinterpret_cast<uint32_t*>(base + t.encode_off);
  p.n_clear_b = kWsHeaderBytes / 4;
  cudaError_t e = launch_dependent(L.group_dim == 16 ? rank_init_kernel<16> : rank_init_kernel<8>, t.sort_blocks,
                                   kSortThreads, 0, stream, p, t.sort_direct);
  count_launches(1);
  const TrustParams norm = make_params(L, G, k, 0.0f, nullptr, nullptr, ws, t);
  uint64_t *a = p.pairs, *b = p.other;
  for (int pass = 0; pass < 4 && e == cudaSuccess; ++pass) {
    if (t.sort_direct) {
      const bool f16 = L.codebook_dtype == PVT_F16, u16 = L.code_dtype == PVT_U16;
      const auto launch = f16 ? (u16 ? launch_sort_norm<true, true> : launch_sort_norm<true, false>)
                              : (u16 ? launch_sort_norm<false, true> : launch_sort_norm<false, false>);
      e = launch(a, b, p, pass, norm, L.group_dim, t.norm_blocks, stream);
      count_launches(1);
    } else {
      if (pass > 0) e = launch_dependent(sort_count_kernel, t.sort_blocks, kSortThreads, 0, stream, a, p, pass);
      if (e == cudaSuccess)
        e = launch_dependent(sort_scan_kernel, 1, kScanThreads, 0, stream, p.counts, kSortBins * t.sort_blocks);
      if (e == cudaSuccess)
        e = launch_dependent(sort_scatter_kernel, t.sort_blocks, kSortThreads, 0, stream, a, b, p, pass);
      count_launches(pass > 0 ? 3 : 2);
    }
    uint64_t* tmp = a;
    a = b;
    b = tmp;
  }
  return e;
}

namespace {

template <bool CB_F16, bool CODE_U16>
cudaError_t before_search(const TrustParams& p, int dg, unsigned norm_blocks, cudaStream_t stream) {
  count_launches(1);
  return launch_dependent(dg == 16 ? sq_norm_kernel<CB_F16, CODE_U16, 16> : sq_norm_kernel<CB_F16, CODE_U16, 8>, norm_blocks,
                          kNormThreads, 0, stream, p);
}

template <bool CB_F16, bool CODE_U16>
cudaError_t after_search(const TrustParams& p, int dg, cudaStream_t stream) {
  const unsigned blocks = (unsigned)((p.k + kChangeThreads - 1) / kChangeThreads);
  cudaError_t e = launch_dependent(dg == 16 ? change_kernel<CB_F16, CODE_U16, 16> : change_kernel<CB_F16, CODE_U16, 8>,
                                   blocks, kChangeThreads, 0, stream, p);
  if (e == cudaSuccess) e = launch_dependent(cut_kernel, 1, kCutThreads, 0, stream, p);
  if (e == cudaSuccess) e = launch_dependent(restore_kernel<CODE_U16>, (unsigned)((p.k + 255) / 256), 256, 0, stream, p);
  count_launches(3);
  return e;
}

}  // namespace

cudaError_t launch_trust_before_search(const pvt_layer& L, uint64_t G, uint64_t k, void* ws, const TrustLayout& t,
                                       cudaStream_t stream) {
  if (t.sort_direct) return cudaSuccess;  // the norm went along with the sort
  const TrustParams p = make_params(L, G, k, 0.0f, nullptr, nullptr, ws, t);
  const bool f16 = L.codebook_dtype == PVT_F16, u16 = L.code_dtype == PVT_U16;
  const int dg = L.group_dim;
  if (f16)
    return u16 ? before_search<true, true>(p, dg, t.norm_blocks, stream)
               : before_search<true, false>(p, dg, t.norm_blocks, stream);
  return u16 ? before_search<false, true>(p, dg, t.norm_blocks, stream)
             : before_search<false, false>(p, dg, t.norm_blocks, stream);
}

cudaError_t launch_trust_after_search(const pvt_layer& L, uint64_t G, uint64_t k, float ratio, uint32_t* idx_out,
                                      uint64_t* n_out, double* stats_out, void* ws, const TrustLayout& t,
                                      cudaStream_t stream) {
  TrustParams p = make_params(L, G, k, ratio, idx_out, n_out, ws, t);
  p.stats_out = stats_out;
  const bool f16 = L.codebook_dtype == PVT_F16, u16 = L.code_dtype == PVT_U16;
  cudaError_t e;
  if (f16)
    e = u16 ? after_search<true, true>(p, L.group_dim, stream) : after_search<true, false>(p, L.group_dim, stream);
  else
    e = u16 ? after_search<false, true>(p, L.group_dim, stream) : after_search<false, false>(p, L.group_dim, stream);
  return e;
}

}  // namespace pvt
