// Subspace choice of the V step (the top-tau selection of Algorithm 2; Section 3.4 ranks by
// update size, separately for every weight matrix): squared update norm per weight group,
// then an exact top-k by radix select on the binary32 bit patterns, ties at the
// threshold resolved towards the lowest group index, result in ascending order.
//
// Four kernels, each launched before the one ahead of it has finished.  What bounds them is the one pass over g (32 B
// per group); the others read keys that are in the L2 and cost little more than their launches:
//   0. clear:  zeroes the histograms; meanwhile the first 64 KB of g per block of pass 1 come to the L2
//   1. keys:   32 bytes per thread and load, four groups in flight per thread; writes the key of every group and sums
//              up key bits [30:18] -- 32 bins per octave, so that the threshold bin of ordinary updates holds a
//              fraction of a per cent of the groups
//   2. bin:    every CTA finds the threshold bin and writes two bits per group, above it and inside it; the members of
//              the bin are counted by their lower 18 bits, in a table of all 2^18 of them (few members: few atomics) and
//              in one of the upper nine of these bits
//   3. write:  the last warp of every CTA reads the threshold from those two tables, while the others ask for the masks and
//              the keys of the first members of the bin; then it counts what it takes, waits for the counts of the CTAs
//              before it and writes its part of the list by ballots:
//              position = (#greater before) + min(#equal before, ties to take)
// Measured as calls one after the other, 4096 x 4096 / 11008 x 4096: 27.7 / 52.2 us (29.7 / 54.5 with nothing asked for
// ahead, one CTA per SM and polls without a pause).  By counters of the kernels by themselves pass 1 takes 16 us of the
// first (4.2 TB/s of g from cold; 5.4 for the second), the others 4.5, 10 and 12; 28672 x 8192: 245 us.  Five passes with
// one bin per eighth of an octave took 45 / 74 / 344 us.  One cooperative kernel with the keys in shared memory takes
// 33 us, and about 10 us more to launch.  Clearing the large tables in pass 1, and contiguous shares there: no gain.  The
// counts that pass 3 waits for side by side, sixteen to a line: 27.1 / 49.0 us; each in a sector of its own: 24.8 / 48.0 (the
// pass 7.5 us after the one before it, 10.5 where its line was slow to reach: those that poll kept the counts from arriving).
#include "pvt_select.cuh"

namespace pvt {

using namespace select;

SelectLayout select_layout(uint64_t G) {
  SelectLayout s;
  s.scratch_off = kWsHeaderBytes;
  s.keys_off = align_up(s.scratch_off + sizeof(uint32_t) * kSelScratchWords, kWsAlign);
  s.masks_off = align_up(s.keys_off + sizeof(uint32_t) * G, kWsAlign);
  s.bytes = align_up(s.masks_off + 8 * ((G + 31) / 32), kWsAlign);
  return s;
}

namespace {

// inclusive scan over a block of 1024 threads; `sh` has one word per warp
__device__ __forceinline__ uint32_t block_scan(uint32_t v, uint32_t* sh) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t n = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += n;
  }
  __syncthreads();
  if (lane == 31) sh[warp] = v;
  __syncthreads();
  const uint32_t before = __reduce_add_sync(0xffffffffu, lane < warp ? sh[lane] : 0u);
  return v + before;
}

// Walk a histogram from its top bin downwards to the bin that holds the k_left-th largest key; found[0] = that bin,
// found[1] = how many keys are still to be taken from inside it.  A block of 1024 threads.
template <int NBINS>
__device__ __forceinline__ void find_digit(const uint32_t* hist, uint32_t k_left, uint32_t* sh, uint32_t* found) {
  constexpr int PER = NBINS >= kSelThreads ? NBINS / kSelThreads : 1;
  const bool own = threadIdx.x < NBINS / PER;
  const int hi = NBINS - 1 - (int)threadIdx.x * PER;
  uint32_t c[PER], mine = 0;
  if (PER >= 4 && own) {
#pragma unroll
    for (int i = 0; i < PER; i += 4) {
      const uint4 q = __ldcg(reinterpret_cast<const uint4*>(hist + hi + 1 - PER) + (PER - 4 - i) / 4);
      c[i] = q.w, c[i + 1] = q.z, c[i + 2] = q.y, c[i + 3] = q.x;
    }
  } else {
#pragma unroll
    for (int i = 0; i < PER; ++i) c[i] = own ? __ldcg(hist + hi - i) : 0u;
  }
#pragma unroll
  for (int i = 0; i < PER; ++i) mine += c[i];
  if (threadIdx.x == 0) found[0] = found[1] = 0;  // (nothing found: an inconsistent histogram, reported at the end)
  uint32_t above = block_scan(mine, sh) - mine;
#pragma unroll
  for (int i = 0; i < PER; ++i) {
    if (above < k_left && k_left - above <= c[i]) {
      found[0] = (uint32_t)(hi - i);
      found[1] = k_left - above;
    }
    above += c[i];
  }
  __syncthreads();
}

// The same for 512 bins by one warp (16 bins per lane); every lane gets the answer.
__device__ __forceinline__ void find_digit_warp(const uint32_t* hist, uint32_t k_left, uint32_t* digit, uint32_t* left) {
  const int lane = threadIdx.x & 31;
  const uint4* q = reinterpret_cast<const uint4*>(hist + 512 - 16 * (lane + 1));  // this lane's bins, ascending
  uint4 v[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) v[i] = __ldcg(q + i);
  const uint32_t c[16] = {v[3].w, v[3].z, v[3].y, v[3].x, v[2].w, v[2].z, v[2].y, v[2].x,
                          v[1].w, v[1].z, v[1].y, v[1].x, v[0].w, v[0].z, v[0].y, v[0].x};  // descending
  uint32_t mine = 0;
#pragma unroll
  for (int i = 0; i < 16; ++i) mine += c[i];
  uint32_t above = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t n = __shfl_up_sync(0xffffffffu, above, o);
    if (lane >= o) above += n;
  }
  above -= mine;
  uint32_t d = 0, l = 0;
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    if (above < k_left && k_left - above <= c[i]) {
      d = (uint32_t)(511 - 16 * lane - i);
      l = k_left - above;
    }
    above += c[i];
  }
  const uint32_t owner = __ballot_sync(0xffffffffu, l != 0);
  const int src = owner ? __ffs(owner) - 1 : 0;  // (no owner: an inconsistent histogram, reported at the end)
  *digit = __shfl_sync(0xffffffffu, d, src);
  *left = __shfl_sync(0xffffffffu, l, src);
}

// ---- 0. everything the passes count in starts at zero
__global__ void __launch_bounds__(kSelThreads) select_clear_kernel(uint4* scratch, uint32_t n16) {
  pdl_trigger();
  pdl_wait();
  for (uint32_t i = blockIdx.x * kSelThreads + threadIdx.x; i < n16; i += gridDim.x * kSelThreads)
    scratch[i] = make_uint4(0, 0, 0, 0);
}

// ---- 1. keys and the histogram of their upper bits: the one pass over g
template <int DG, int MODE>
__global__ void __launch_bounds__(kNormThreads, kNormCtas) select_keys_kernel(const SelParams p) {
  __shared__ uint32_t hist[kSelBins0];
  pdl_trigger();
  for (uint32_t i = threadIdx.x; i < kSelBins0; i += kNormThreads) hist[i] = 0;
  constexpr int U = kKeyGroups<DG, MODE>;
  const uint64_t first = (uint64_t)blockIdx.x * (U * kNormThreads);
  if (threadIdx.x == 0 && MODE != kKeyUniform && first < p.G) {  // what the block reads first comes to the L2 while it waits
    const uint64_t n = p.G - first < U * kNormThreads ? p.G - first : U * kNormThreads;
    prefetch_l2(p.g + first * DG, (uint32_t)(n * DG * sizeof(float)));
    if (MODE == kKeyNormBuffer) prefetch_l2(p.buffer + first * DG, (uint32_t)(n * DG * sizeof(float)));
  }
  __syncthreads();
  pdl_wait();
  keys_pass<DG, MODE>(p, hist, gridDim.x);
}

// ---- 2. the threshold bin: two bits per group (above it, inside it), and its members by their lower bits
__global__ void __launch_bounds__(kSelThreads) select_bin_kernel(const SelParams p) {
  __shared__ uint32_t hist[kSelBins1], sh[32], found[2];
  const uint32_t tid = threadIdx.x, lane = tid & 31;
  pdl_trigger();
  if (tid < kSelBins1) hist[tid] = 0;
  const uint64_t w_lo = (uint64_t)blockIdx.x * p.words, n_words = (p.G + 31) / 32;
  const uint64_t w_hi = w_lo + p.words < n_words ? w_lo + p.words : n_words;
  pdl_wait();
  find_digit<kSelBins0>(p.hist0, (uint32_t)p.k, sh, found);
  const uint32_t bin = found[0];
  constexpr uint32_t U = 16;  // words of 32 groups per warp and trip, all their keys in flight
  for (uint64_t w0 = w_lo + U * (tid >> 5); w0 < w_hi; w0 += U * (kSelThreads / 32)) {
    uint32_t key[U];
#pragma unroll
    for (uint32_t u = 0; u < U; ++u) {
      const uint64_t j = (w0 + u) * 32 + lane;
      key[u] = w0 + u < w_hi && j < p.G ? __ldcg(p.keys + j) : 0u;
    }
    uint32_t above = 0, inside = 0;
#pragma unroll
    for (uint32_t u = 0; u < U; ++u) {
      const bool real = w0 + u < w_hi && (w0 + u) * 32 + lane < p.G;
      const uint32_t m_gt = __ballot_sync(0xffffffffu, real && (key[u] >> 18) > bin);
      const uint32_t m_in = __ballot_sync(0xffffffffu, real && (key[u] >> 18) == bin);
      if (lane == u) {
        above = m_gt;
        inside = m_in;
      }
      if (m_in) {
        // equal keys of a warp add up first: many equal norms must not queue at one address
        const bool in = (m_in >> lane) & 1u;
        const uint32_t same = __match_any_sync(0xffffffffu, in ? key[u] : 0xffffffffu);
        if (in && lane == (uint32_t)__ffs(same) - 1) {
          atomicAdd(&hist[(key[u] >> 9) & 511u], (uint32_t)__popc(same));
          atomicAdd(&p.fine[key[u] & 0x3ffffu], (uint32_t)__popc(same));
        }
      }
    }
    if (lane < U && w0 + lane < w_hi) p.masks[w0 + lane] = make_uint2(above, inside);
  }
  __syncthreads();
  if (tid < kSelBins1 && hist[tid]) atomicAdd(&p.hist1[tid], hist[tid]);
  if (blockIdx.x == 0 && tid == 0) {
    p.state[0] = bin;
    p.state[1] = found[1];
  }
}

// ---- 3. threshold, and the ordered list of what is taken
// A CTA needs to know what the CTAs before it take.  It waits for their counts, and only for theirs: numbers are drawn
// at the start, so whoever is waited for is already running (and waits for nobody after it).  The wait is bounded.
constexpr uint32_t kSelMaxPolls = 1u << 21;

__global__ void __launch_bounds__(kSelThreads) select_write_kernel(const SelParams p) {
  __shared__ uint32_t sh[32], ticket, sh_threshold, sh_need, sum_gt, sum_eq, all_gt, all_eq;
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  pdl_trigger();
  pdl_wait();
  constexpr uint32_t kReaders = kSelThreads - 32;  // the last warp finds the threshold
  const uint64_t n_words = (p.G + 31) / 32;
  uint2 early = make_uint2(0, 0);  // of the first trip: this thread's masks, the key of its first member of the bin
  uint32_t early_key = 0;
  if (tid < kReaders) {
    if (tid == 0) {
      ticket = atomicAdd(&p.state[2], 1u);
      sum_gt = sum_eq = all_gt = all_eq = 0;
    }
    asm volatile("bar.sync 1, %0;" ::"n"(kReaders) : "memory");
    const uint64_t w = (uint64_t)ticket * p.words + tid;
    if (tid < p.words && w < n_words) {
      early = __ldcg(p.masks + w);
      if (early.y) early_key = __ldcg(p.keys + w * 32 + (uint32_t)__ffs(early.y) - 1);
    }
  } else {
    const uint32_t bin = __ldcg(p.state), in_bin = __ldcg(p.state + 1);
    uint32_t d1, d2, left;
    find_digit_warp(p.hist1, in_bin, &d1, &left);
    find_digit_warp(p.fine + 512 * d1, left, &d2, &left);
    if (lane == 0) {
      sh_threshold = (bin << 18) | (d1 << 9) | d2;
      sh_need = left;
    }
  }
  __syncthreads();
  const uint32_t cta = ticket, threshold = sh_threshold, need_eq = sh_need;
  const uint64_t w_lo = (uint64_t)cta * p.words;
  const uint64_t w_hi = w_lo + p.words < n_words ? w_lo + p.words : n_words;

  // one word of 32 groups per thread and trip; the members of the threshold bin (few) are looked up
  auto resolve = [&](uint64_t w) {
    const bool known = w == w_lo + tid && tid < kReaders;
    const uint2 m = known ? early : __ldcg(p.masks + w);
    uint32_t gt = m.x, eq = 0;
    for (uint32_t in = m.y; in; in &= in - 1) {
      const uint32_t b = (uint32_t)__ffs(in) - 1;
      const uint32_t key = known && in == m.y ? early_key : __ldcg(p.keys + w * 32 + b);
      gt |= key > threshold ? 1u << b : 0u;
      eq |= key == threshold ? 1u << b : 0u;
    }
    return make_uint2(gt, eq);
  };
  uint2 first = make_uint2(0, 0);  // the first trip's answer stays in registers, those of further trips go back
  uint32_t n_gt = 0, n_eq = 0;
  for (uint64_t w = w_lo + tid; w < w_hi; w += kSelThreads) {
    const uint2 m = resolve(w);
    if (w == w_lo + tid)
      first = m;
    else
      p.masks[w] = m;
    n_gt += __popc(m.x);
    n_eq += __popc(m.y);
  }
  n_gt = __reduce_add_sync(0xffffffffu, n_gt);
  n_eq = __reduce_add_sync(0xffffffffu, n_eq);
  if (lane == 0 && n_gt) atomicAdd(&all_gt, n_gt);
  if (lane == 0 && n_eq) atomicAdd(&all_eq, n_eq);
  __syncthreads();
  if (tid == 0) {
    const uint64_t mine = (1ull << 63) | ((uint64_t)all_eq << 31) | all_gt;  // a CTA has fewer than 2^31 groups
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p.counts + kSelCountStride * cta), "l"(mine) : "memory");
  }
  bool ok = true;
  uint32_t prev_gt = 0, prev_eq = 0;
  for (uint32_t b = tid; b < cta; b += kSelThreads) {
    uint64_t c = 0;
    for (uint32_t i = 0; i < kSelMaxPolls && !(c >> 63); ++i) {
      if (i) __nanosleep(40);
      asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(c) : "l"(p.counts + kSelCountStride * b) : "memory");
    }
    ok &= (c >> 63) != 0;
    prev_gt += (uint32_t)c & 0x7fffffffu;
    prev_eq += (uint32_t)(c >> 31) & 0x7fffffffu;
  }
  prev_gt = __reduce_add_sync(0xffffffffu, prev_gt);
  prev_eq = __reduce_add_sync(0xffffffffu, prev_eq);
  if (lane == 0 && prev_gt) atomicAdd(&sum_gt, prev_gt);
  if (lane == 0 && prev_eq) atomicAdd(&sum_eq, prev_eq);
  if (!__syncthreads_and(ok)) {
    if (tid == 0) atomicOr(p.status, PVT_DEV_WAIT_EXPIRED);
    return;
  }
  uint32_t at_gt = sum_gt, at_eq = sum_eq;  // what comes before the trip
  // all greater keys plus the ties taken must be exactly k
  if (cta == gridDim.x - 1 && tid == 0 && (uint64_t)at_gt + all_gt + min(at_eq + all_eq, need_eq) != p.k)
    atomicOr(p.status, PVT_DEV_INTERNAL);
  for (uint64_t w0 = w_lo; w0 < w_hi; w0 += kSelThreads) {
    const uint64_t w = w0 + tid;
    uint2 m = make_uint2(0, 0);
    if (w < w_hi) m = w0 == w_lo ? first : __ldcg(p.masks + w);
    // both counts in one scan: a trip has 2^15 groups
    const uint32_t mine = (uint32_t)__popc(m.x) | ((uint32_t)__popc(m.y) << 16);
    const uint32_t incl = block_scan(mine, sh);
    uint32_t my_gt = at_gt + ((incl - mine) & 0xffffu), my_eq = at_eq + ((incl - mine) >> 16);
    if (tid == kSelThreads - 1) {
      sum_gt = at_gt + (incl & 0xffffu);
      sum_eq = at_eq + (incl >> 16);
    }
    const uint32_t most = __reduce_max_sync(0xffffffffu, (uint32_t)__popc(m.x | m.y));
    if (most <= 6) {  // few bits: every lane writes its own word's
      for (uint32_t both = m.x | m.y; both; both &= both - 1) {
        const uint32_t b = (uint32_t)__ffs(both) - 1;
        const bool is_gt = (m.x >> b) & 1u;
        const uint32_t pos = my_gt + min(my_eq, need_eq);
        if ((is_gt || my_eq < need_eq) && pos < p.k) p.idx_out[pos] = (uint32_t)(w * 32) + b;
        my_gt += is_gt;
        my_eq += !is_gt;
      }
    } else {          // the warp writes one word after the other, a lane per group
      for (uint32_t left = __ballot_sync(0xffffffffu, (m.x | m.y) != 0); left; left &= left - 1) {
        const int src = __ffs(left) - 1;
        const uint32_t gt = __shfl_sync(0xffffffffu, m.x, src), eq = __shfl_sync(0xffffffffu, m.y, src);
        const uint32_t b_gt = __shfl_sync(0xffffffffu, my_gt, src), b_eq = __shfl_sync(0xffffffffu, my_eq, src);
        const uint32_t below = (1u << lane) - 1u;
        const uint32_t e = b_eq + __popc(eq & below), pos = b_gt + __popc(gt & below) + min(e, need_eq);
        const bool take = ((gt >> lane) & 1u) || (((eq >> lane) & 1u) && e < need_eq);
        if (take && pos < p.k) p.idx_out[pos] = (uint32_t)((w0 + 32 * warp + src) * 32) + lane;
      }
    }
    __syncthreads();
    at_gt = sum_gt;
    at_eq = sum_eq;
  }
}

__global__ void iota_kernel(uint32_t* idx_out, uint64_t k) {
  pdl_trigger();
  pdl_wait();
  const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < k) idx_out[i] = (uint32_t)i;
}

}  // namespace

namespace {

template <int DG, int MODE>
cudaError_t launch_keys(const SelParams& p, int sm_count, cudaStream_t stream) {
  const uint64_t blocks = (p.G + 2 * kNormThreads - 1) / (2 * kNormThreads), resident = (uint64_t)sm_count * kNormCtas;
  return launch_dependent(select_keys_kernel<DG, MODE>, (unsigned)(blocks < resident ? blocks : resident), kNormThreads, 0,
                          stream, p);
}

template <int DG>
cudaError_t launch_group(int mode, const SelParams& p, int sm_count, cudaStream_t stream) {
  switch (mode) {
    case kKeyNormBuffer: return launch_keys<DG, kKeyNormBuffer>(p, sm_count, stream);
    case kKeyUniform: return launch_keys<DG, kKeyUniform>(p, sm_count, stream);
    case kKeyProportional: return launch_keys<DG, kKeyProportional>(p, sm_count, stream);
    default: return launch_keys<DG, kKeyNorm>(p, sm_count, stream);
  }
}

}  // namespace

namespace {
// (W_hat: with the plain norms only)
cudaError_t launch_passes(const pvt_layer& L, uint64_t G, uint64_t k, uint32_t* idx_out, void* ws, int sm_count,
                          cudaStream_t stream, int key_mode, float* buffer, uint64_t seed, void* W_hat, int32_t out_dtype) {
  timing_begin(kKernSelect, stream);
  cudaError_t err;
  if (k == G && key_mode != kKeyNormBuffer) {  // every group is taken: the ascending index list itself
    err = launch_dependent(iota_kernel, (unsigned)((k + 255) / 256), 256, 0, stream, idx_out, k);
  } else {
    const SelectLayout lay = select_layout(G);
    char* base = static_cast<char*>(ws);
    SelParams p;
    p.g = L.g;
    p.buffer = buffer;
    p.G = G;
    p.k = k;
    p.seed = seed;
    p.eta = L.eta;
    p.idx_out = idx_out;
    p.status = reinterpret_cast<uint32_t*>(base);
    p.keys = reinterpret_cast<uint32_t*>(base + lay.keys_off);
    p.masks = reinterpret_cast<uint2*>(base + lay.masks_off);
    uint32_t* scratch = reinterpret_cast<uint32_t*>(base + lay.scratch_off);
    p.counts = reinterpret_cast<uint64_t*>(scratch);
    p.state = scratch + 2 * kSelCountStride * kSelMaxCtas;
    p.hist0 = p.state + 16;
    p.hist1 = p.hist0 + kSelBins0;
    p.fine = p.hist1 + kSelBins1;
    // the passes over the keys: a CTA per SM, fewer for small layers (at least two groups per thread)
    uint64_t n_cta = (G + 2 * kSelThreads - 1) / (2 * kSelThreads);
    const uint64_t most = sm_count < (int)kSelMaxCtas ? (uint64_t)sm_count : kSelMaxCtas;
    if (n_cta > most) n_cta = most;
    p.words = (uint32_t)(((G + n_cta - 1) / n_cta + 31) / 32);
    constexpr uint32_t n16 = kSelScratchWords / 4;
    err = launch_dependent(select_clear_kernel, (n16 + kSelThreads - 1) / kSelThreads, kSelThreads, 0, stream,
                           reinterpret_cast<uint4*>(scratch), n16);
    if (err == cudaSuccess)
      err = W_hat               ? launch_keys_dequant(p, L, W_hat, out_dtype, sm_count, stream)
            : L.group_dim == 16 ? launch_group<16>(key_mode, p, sm_count, stream)
                                : launch_group<8>(key_mode, p, sm_count, stream);
    if (err == cudaSuccess) err = launch_dependent(select_bin_kernel, (unsigned)n_cta, kSelThreads, 0, stream, p);
    // the last pass: one trip of words per CTA (of those that ask early), for which two CTAs of an SM may be needed
    // (11008 x 4096: 1 us less than two trips of one CTA)
    const uint64_t words = (G + 31) / 32, trip = kSelThreads - 32;
    uint64_t w_cta = n_cta;
    if (p.words > trip) w_cta = (words + trip - 1) / trip;
    if (w_cta > 2 * most) w_cta = 2 * most;
    if (w_cta > kSelMaxCtas) w_cta = kSelMaxCtas;
    p.words = (uint32_t)((words + w_cta - 1) / w_cta);
    if (err == cudaSuccess) err = launch_dependent(select_write_kernel, (unsigned)w_cta, kSelThreads, 0, stream, p);
    count_launches(3);
  }
  count_launches(1);
  timing_end(kKernSelect, stream);
  return err;
}
}  // namespace

cudaError_t launch_select(const pvt_layer& L, uint64_t G, uint64_t k, uint32_t* idx_out, void* ws, int sm_count,
                          cudaStream_t stream, void* W_hat, int32_t out_dtype) {
  return launch_passes(L, G, k, idx_out, ws, sm_count, stream, kKeyNorm, nullptr, 0, W_hat, out_dtype);
}

cudaError_t launch_select_keyed(const pvt_layer& L, uint64_t G, uint64_t k, uint32_t* idx_out, void* ws, int sm_count,
                                cudaStream_t stream, int key_mode, float* buffer, uint64_t seed) {
  return launch_passes(L, G, k, idx_out, ws, sm_count, stream, key_mode, buffer, seed, nullptr, 0);
}

}  // namespace pvt
