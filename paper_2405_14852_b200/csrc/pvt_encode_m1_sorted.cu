// Preparation of the tensor search over codewords and targets in spatial order (one fp16 codebook, groups of 8, many
// targets; Appendix C / Appendix J: the nearest of all codewords).
//
// The exhaustive search evaluates every codeword for every target.  Most of that cannot matter: with 65536 codewords in
// eight dimensions a target is nearer to some known codeword than to all but a twentieth of the codebook.  A tensor tile
// works on 256 targets and 128 codewords at once, so a tile of codewords may be left out only if that holds for each of
// the 256 targets - which takes targets that lie close together, and codewords as well:
//   1. A k-d tree of depth 16 over the codewords.  All nodes of a level split along the same dimension (the one whose
//      spread is largest when the splits above it are taken off), at the median.  Its leaves, in order, are the order of
//      the codebook image: a step of the search (128 codewords) is a cell of the tree.
//   2. The targets are sorted by the cell of the tree that they fall into (counting sort).
//   3. The search goes over the thirty-two steps nearest to a tile's cell.
//   4. From the best distance found, or that of the stored code, every target names the steps whose bounding box it can
//      reach; a tile's list is the union.
//   5. The search goes over the tiles' lists.
// What is left out is farther away than a codeword that is known, so codes are those of the exhaustive search, bit for bit.
//
// Normally distributed weights and 65536 codewords: with 1 / 8 / 29 million targets a tile keeps 0.53 / 0.42 / 0.38 of the
// steps (a target by itself 0.06: what is lost is the union over 256).  Whole step of 28672 x 8192, every group: 73.5 -> 43.0
// ms from near stored codes, 82.0 -> 45.4 from random ones; 8192 x 8192 20.8 -> 13.1, 8192 x 1024 2.65 -> 2.2.  Of 13.1 ms the
// second sweep takes 7.0, the first 1.6 (finds: each of its steps is near its targets), the boxes 2.0, rescoring 1.8, the
// codebook 0.2, the targets 0.4.  What it gives depends on the weights.  Search of 8388608 targets in ms, every codeword / in
// spatial order: normal 20.7 / 12.9, uniform 20.7 / 8.8, correlated elements 22.1 / 6.4, Laplace 20.8 / 16.4, groups of unlike
// size 20.8 / 15.2, a codebook ten times smaller than the targets 22.8 / 20.5, half of the targets zero 20.9 / 15.2; where more
// codewords are near than a record holds, log-normal sizes of groups 363 / 81, equal codewords 2143 / 1914.
// The tree is built by a block per node with the keys in shared memory (seven launches, 150 us) and by sorting nodes of 512
// positions; with nodes of 4096 sorted and the keys read again for every pass the codebook took 0.49 ms.  Tried for the boxes:
// bounds from the tree's planes alone (keeps 0.03 more steps), the box of 32 targets in place of the targets (0.82 of the
// steps).  Tried for the search: each half of a tile over the steps of its own (0.32 in place of 0.38 of them, but the issuing
// warps then look every step up: 7.1 -> 8.1).
#include "pvt_encode_m1.cuh"
#include "pvt_encode_m1_sorted.cuh"

namespace pvt {

using namespace m1;

namespace {

constexpr uint32_t kPositions = 1u << kSortedLevels;
constexpr int kSplitThreads = 1024;
constexpr int kTailThreads = 256;
constexpr uint32_t kTailPositions = 512;   // nodes up to this size are split in shared memory
constexpr uint32_t kPadKey = 0xffffu;     // positions without a codeword come after every codeword

// order-preserving image of a half (infinities and NaN at the ends, below kPadKey), and what it stands for
__device__ __forceinline__ uint32_t half_key(uint32_t b) {
  return (b & 0x8000u) ? (~b & 0xffffu) : min(b | 0x8000u, kPadKey - 1);
}
__device__ __forceinline__ float key_value(uint32_t key) {
  if (key >= kPadKey) return __uint_as_float(0x7f800000u);
  const uint32_t b = (key & 0x8000u) ? (key & 0x7fffu) : (~key & 0xffffu);
  return __half2float(__ushort_as_half((unsigned short)b));
}
__device__ __forceinline__ uint32_t element_bits(const uint4& raw, uint32_t dim) {
  const uint32_t w = dim < 4 ? (dim < 2 ? raw.x : raw.y) : (dim < 6 ? raw.z : raw.w);
  return (dim & 1u) ? w >> 16 : w & 0xffffu;
}

// Block 0 chooses the dimension of each level: that of the largest variance, which a split at the median of a normal
// distribution leaves 0.36 of.  A sample of the codewords tells.  The other blocks clear the counts of targets by cell.
__global__ void __launch_bounds__(kSplitThreads) sorted_dims_kernel(const uint4* book, uint32_t K, uint32_t* dims,
                                                                    uint32_t* cells) {
  pdl_trigger();
  pdl_wait();
  const uint32_t tid = threadIdx.x;
  if (blockIdx.x > 0) {
    for (uint32_t i = (blockIdx.x - 1) * kSplitThreads + tid; i < kPositions; i += (gridDim.x - 1) * kSplitThreads)
      cells[i] = 0;
    return;
  }
  __shared__ float part[kSplitThreads / 32][16];
  float sum[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) sum[i] = 0.0f;
  constexpr uint32_t kSample = 8 * kSplitThreads;
#pragma unroll
  for (uint32_t q = 0; q < kSample / kSplitThreads; ++q) {
    const uint4 raw = book[(uint64_t)(tid + q * kSplitThreads) * K / kSample];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      float f = __half2float(__ushort_as_half((unsigned short)element_bits(raw, i)));
      if (!(fabsf(f) < 1e4f)) f = 0.0f;
      sum[i] += f;
      sum[8 + i] = fmaf(f, f, sum[8 + i]);
    }
  }
#pragma unroll
  for (int i = 0; i < 16; ++i) {
#pragma unroll
    for (int o = 16; o; o >>= 1) sum[i] += __shfl_xor_sync(0xffffffffu, sum[i], o);
    if ((tid & 31) == 0) part[tid >> 5][i] = sum[i];
  }
  __syncthreads();
  if (tid == 0) {
    float spread[8];
    for (int i = 0; i < 8; ++i) {
      float s = 0.0f, q = 0.0f;
      for (int w = 0; w < kSplitThreads / 32; ++w) {
        s += part[w][i];
        q += part[w][8 + i];
      }
      s /= (float)kSample;
      spread[i] = fmaxf(q / (float)kSample - s * s, 0.0f);
    }
    for (int l = 0; l < kSortedLevels; ++l) {
      int best = 0;
      for (int i = 1; i < 8; ++i)
        if (spread[i] > spread[best]) best = i;
      spread[best] *= 0.36f;
      dims[l] = (uint32_t)best;
    }
  }
}

// One level of the tree for nodes of more than 512 positions: a block per node finds the median (the keys, in shared memory
// for all but the first pass, are counted by their first eleven bits and by the other five) and moves what is below it to the
// left half.  Which of several equal elements goes where does not matter.  (Halves of like size share their first bits: with
// eight bits at first all threads count in few bins.)
__global__ void __launch_bounds__(kSplitThreads) sorted_split_kernel(const uint4* book, uint32_t K, const uint32_t* dims,
                                                                     int level, const uint32_t* from, uint32_t* to,
                                                                     float* tree) {
  extern __shared__ __align__(16) unsigned char split_smem[];
  uint16_t* keys = reinterpret_cast<uint16_t*>(split_smem);  // [n]
  __shared__ uint32_t hist[2 * kSplitThreads];
  __shared__ uint32_t found[2], sums[3][32];
  pdl_trigger();
  pdl_wait();
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t n = kPositions >> level, first = blockIdx.x * n, half = n / 2, dim = dims[level];  // (n >= kSplitThreads)
  auto id_at = [&](uint32_t i) { return from ? from[first + i] : first + i; };
  const uint16_t* elements = reinterpret_cast<const uint16_t*>(book) + dim;
  auto inclusive = [&](uint32_t x) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t up = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= (uint32_t)o) x += up;
    }
    return x;
  };
  hist[tid] = hist[tid + kSplitThreads] = 0;
  __syncthreads();
  for (uint32_t i = tid; i < n; i += 8 * kSplitThreads) {
    uint32_t id[8], key[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) id[q] = i + q * kSplitThreads < n ? id_at(i + q * kSplitThreads) : K;
#pragma unroll
    for (int q = 0; q < 8; ++q) key[q] = id[q] < K ? half_key(elements[8 * (size_t)id[q]]) : kPadKey;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      if (i + q * kSplitThreads < n) {
        keys[i + q * kSplitThreads] = (uint16_t)key[q];
        atomicAdd(&hist[key[q] >> 5], 1u);
      }
    }
  }
  uint32_t below = 0, median = 0;
  for (int pass = 0; pass < 2; ++pass) {  // the bin that holds the element with `half` elements below it
    __syncthreads();
    const uint32_t h0 = hist[2 * tid], h = h0 + hist[2 * tid + 1], incl = inclusive(h);
    if (lane == 31) sums[0][warp] = incl;
    __syncthreads();
    const uint32_t before = below + __reduce_add_sync(0xffffffffu, lane < warp ? sums[0][lane] : 0u) + incl - h;
    if (before <= half && half < before + h) {
      const bool second = half >= before + h0;
      found[0] = 2 * tid + second;
      found[1] = before + (second ? h0 : 0u);
    }
    hist[2 * tid] = hist[2 * tid + 1] = 0;
    __syncthreads();
    median = (median << 5) + found[0];
    below = found[1];
    if (pass == 0) {
      for (uint32_t i = tid; i < n; i += kSplitThreads)
        if ((uint32_t)(keys[i] >> 5) == median) atomicAdd(&hist[keys[i] & 31u], 1u);
    }
  }
  if (tid == 0) tree[(1u << level) + blockIdx.x] = key_value(median);
  // a warp takes adjacent positions, so that what it moves lands side by side
  const uint32_t chunk = n / (kSplitThreads / 32), mine = warp * chunk;
  uint32_t less = 0, equal = 0;
  for (uint32_t i = lane; i < chunk; i += 32) {
    less += __popc(__ballot_sync(0xffffffffu, keys[mine + i] < median));
    equal += __popc(__ballot_sync(0xffffffffu, keys[mine + i] == median));
  }
  if (lane == 0) {
    sums[1][warp] = less;
    sums[2][warp] = equal;
  }
  __syncthreads();
  // elements ahead of this warp's: `less` and `equal` of them; of the equal ones half - below go to the left
  less = __reduce_add_sync(0xffffffffu, lane < warp ? sums[1][lane] : 0u);
  equal = __reduce_add_sync(0xffffffffu, lane < warp ? sums[2][lane] : 0u);
  const uint32_t equal_left = half - below, equal_all = __reduce_add_sync(0xffffffffu, sums[2][lane]);
  uint32_t more = mine - less - equal;
  const uint32_t ahead = (1u << lane) - 1u;
#pragma unroll 4
  for (uint32_t i = lane; i < chunk; i += 32) {
    const uint32_t key = keys[mine + i], id = id_at(mine + i);
    const uint32_t in_less = __ballot_sync(0xffffffffu, key < median), in_equal = __ballot_sync(0xffffffffu, key == median);
    const uint32_t in_more = ~(in_less | in_equal);
    const uint32_t e = equal + __popc(in_equal & ahead);
    const uint32_t pos = key < median    ? less + __popc(in_less & ahead)
                         : key > median ? below + equal_all + more + __popc(in_more & ahead)
                                        : (e < equal_left ? below + e : half + e - equal_left);
    to[first + pos] = id;
    less += __popc(in_less);
    equal += __popc(in_equal);
    more += __popc(in_more);
  }
}

// The rest of the tree, a block per node of 512 positions: on each level every node is sorted in shared memory.
__global__ void __launch_bounds__(kTailThreads) sorted_tail_kernel(const uint4* book, uint32_t K, const uint32_t* dims,
                                                                    const uint32_t* from, uint32_t* order, float* tree) {
  __shared__ uint4 pts[kTailPositions];
  __shared__ uint32_t word[kTailPositions], ids[kTailPositions];  // key and place in `pts`
  pdl_trigger();
  pdl_wait();
  const uint32_t tid = threadIdx.x, first = blockIdx.x * kTailPositions;
  for (uint32_t i = tid; i < kTailPositions; i += kTailThreads) {
    const uint32_t id = from[first + i];
    ids[i] = id;
    word[i] = i;
    pts[i] = id < K ? book[id] : make_uint4(0, 0, 0, 0);
  }
  __syncthreads();
  constexpr int kTop = kSortedLevels - 9;  // the level of this block's node
  for (int level = kTop; level < kSortedLevels; ++level) {
    const uint32_t n = kPositions >> level, dim = dims[level];
    for (uint32_t i = tid; i < kTailPositions; i += kTailThreads) {
      const uint32_t at = word[i] & (kTailPositions - 1);
      word[i] = ((ids[at] < K ? half_key(element_bits(pts[at], dim)) : kPadKey) << 12) | at;
    }
    __syncthreads();
    for (uint32_t size = 2; size <= n; size <<= 1) {
      for (uint32_t stride = size >> 1; stride; stride >>= 1) {
        for (uint32_t q = tid; q < kTailPositions / 2; q += kTailThreads) {
          const uint32_t i = ((q & ~(stride - 1)) << 1) | (q & (stride - 1));
          const uint32_t a = word[i], b = word[i + stride];
          const bool up = size == n || !(i & size);
          if ((a > b) == up) {
            word[i] = b;
            word[i + stride] = a;
          }
        }
        __syncthreads();
      }
    }
    for (uint32_t node = tid; node < kTailPositions / n; node += kTailThreads)
      tree[(1u << level) + blockIdx.x * (kTailPositions / n) + node] = key_value(word[node * n + n / 2] >> 12);
    __syncthreads();
  }
  for (uint32_t i = tid; i < kTailPositions; i += kTailThreads) order[first + i] = ids[word[i] & (kTailPositions - 1)];
}

// Bounding box of each step, over the codewords that the operand image holds.
__global__ void __launch_bounds__(128) sorted_box_kernel(const uint4* book, uint32_t K, float* boxes) {
  __shared__ uint32_t part[4][16];
  pdl_trigger();
  pdl_wait();
  const uint32_t tid = threadIdx.x, pos = blockIdx.x * 128 + tid;
  const uint4 raw = pos < K ? book[pos] : make_uint4(0, 0, 0, 0);
  float c[8], n2 = 0.0f;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    c[i] = __half2float(__ushort_as_half((unsigned short)element_bits(raw, i)));
    n2 = fmaf(c[i], c[i], n2);
  }
  const bool use = pos < K && 0.5f * n2 <= kMaxHalfNorm;  // (the same sum as for the image; false for NaN and infinities)
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const uint32_t lo = __reduce_min_sync(0xffffffffu, use ? ord(c[i]) : 0xffffffffu);
    const uint32_t hi = __reduce_max_sync(0xffffffffu, use ? ord(c[i]) : 0u);
    if ((tid & 31) == 0) {
      part[tid >> 5][i] = lo;
      part[tid >> 5][8 + i] = hi;
    }
  }
  __syncthreads();
  if (tid < 16) {
    uint32_t x = part[0][tid];
    for (int w = 1; w < 4; ++w) x = tid < 8 ? min(x, part[w][tid]) : max(x, part[w][tid]);
    // no codeword: an empty box
    boxes[blockIdx.x * 16 + tid] = tid < 8 ? (x == 0xffffffffu ? 1e30f : unord(x)) : (x == 0u ? -1e30f : unord(x));
  }
}

// ---- boxes in half precision ------------------------------------------------------
// Scaled by a power of two so that no element of a codeword exceeds 8, rounded outwards; two boxes side by side.
__device__ __forceinline__ float box_scale(uint32_t n2max_bits) {
  const float c = sqrtf(__uint_as_float(n2max_bits));
  return c > 1e-15f ? scalbnf(1.0f, 2 - ilogbf(c)) : 1.0f;
}
__device__ void put_box(__half* to, uint32_t which, const float* lo, const float* hi, float scale) {
  const uint32_t pair = which >> 1, side = which & 1u;
  for (int i = 0; i < 8; ++i) {
    // (empty: out of reach of everything)
    const bool some = lo[i] <= hi[i];
    to[pair * 32 + 4 * i + side] = __float2half_rd(some ? lo[i] * scale : 65504.0f);
    to[pair * 32 + 4 * i + 2 + side] = __float2half_ru(some ? hi[i] * scale : -65504.0f);
  }
}

// A block per step: the steps nearest to it, by their boxes' centres, and its box (the first of eight: theirs as well) in
// half precision.
__global__ void __launch_bounds__(kSortedSteps) sorted_near_kernel(const float* boxes, uint32_t n_steps, const uint2* norms,
                                                                   uint32_t norm_blocks, uint16_t* near, __half* packed) {
  __shared__ __align__(16) uint32_t dist[kSortedSteps];
  __shared__ float group[8 * 16];  // (the boxes of eight steps, this one among them)
  __shared__ uint32_t n2max;
  const uint32_t tid = threadIdx.x, s = blockIdx.x;
  if (tid == 0) n2max = 0;
  pdl_trigger();
  pdl_wait();
  __syncthreads();
  if (tid < 128) group[tid] = s / 8 * 8 + tid / 16 < n_steps ? boxes[s / 8 * 128 + tid] : tid % 16 < 8 ? 1e30f : -1e30f;
  const uint32_t most = __reduce_max_sync(0xffffffffu, tid < norm_blocks ? norms[tid].x : 0u);
  if ((tid & 31) == 0) atomicMax(&n2max, most);
  float d = __uint_as_float(0x7f800000u);
  if (tid < n_steps && s < n_steps) {
    const float *a = boxes + 16 * s, *b = boxes + 16 * tid;
    if (b[0] <= b[8] && a[0] <= a[8]) {
      d = 0.0f;
      for (int i = 0; i < 8; ++i) {
        const float e = (a[i] + a[8 + i]) - (b[i] + b[8 + i]);
        d = fmaf(e, e, d);
      }
    }
  }
  const uint32_t key = near_key(__float_as_uint(d), tid, s);
  dist[tid] = key;
  __syncthreads();
  if (s < n_steps && tid < n_steps) {
    uint32_t rank = 0;
#pragma unroll 4
    for (uint32_t i = 0; i < kSortedSteps / 4; ++i) {  // (steps that are not there are farthest)
      const uint4 four = reinterpret_cast<const uint4*>(dist)[i];
      rank += (four.x < key) + (four.y < key) + (four.z < key) + (four.w < key);
    }
    if (rank < kSortedNear) near[s * kSortedNear + rank] = (uint16_t)tid;
  }
  const float scale = box_scale(n2max);
  if (tid == 0) {
    put_box(packed, s, group + 16 * (s % 8), group + 16 * (s % 8) + 8, scale);
  } else if (tid == 32 && s % 8 == 0) {
    float lo[8], hi[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      lo[i] = group[i];
      hi[i] = group[8 + i];
#pragma unroll
      for (int q = 1; q < 8; ++q) {
        lo[i] = fminf(lo[i], group[16 * q + i]);
        hi[i] = fmaxf(hi[i], group[16 * q + 8 + i]);
      }
    }
    put_box(packed + kSortedSteps * 16, s / 8, lo, hi, scale);
  }
}

// ---- targets in the order of the cells ---------------------------------------------
constexpr uint32_t kKeyTree = 4096;  // nodes of the tree in shared memory

__global__ void __launch_bounds__(256) sorted_key_kernel(const EncM1Params p, const uint32_t* idx, const uint32_t* dims,
                                                         const float* tree, uint32_t* cells, uint2* keys) {
  __shared__ float top[kKeyTree];
  __shared__ uint32_t dim[kSortedLevels];
  pdl_trigger();
  pdl_wait();
  for (uint32_t i = threadIdx.x; i < kKeyTree; i += 256) top[i] = i ? tree[i] : 0.0f;
  if (threadIdx.x < kSortedLevels) dim[threadIdx.x] = dims[threadIdx.x];
  __syncthreads();
  // (whole warps; no target: a number that is no cell's)
  const uint32_t lane = threadIdx.x & 31;
  for (uint64_t n = (uint64_t)blockIdx.x * 256 + threadIdx.x; n - lane < p.k; n += (uint64_t)gridDim.x * 256) {
    const uint32_t j = n < p.k ? idx[n] : 0xffffffffu;
    uint32_t node = 1;
    if (j < p.G) {  // (the rescoring kernel reports an index out of range)
      float t[8];
      form_target(p, j, t);
#pragma unroll 1
      for (int l = 0; l < kSortedLevels; ++l) {
        const float v = node < kKeyTree ? top[node] : tree[node];
        const uint32_t d = dim[l];
        const float lo = d < 2 ? (d ? t[1] : t[0]) : (d & 1u ? t[3] : t[2]);
        const float hi = d < 6 ? (d & 1u ? t[5] : t[4]) : (d & 1u ? t[7] : t[6]);
        node = 2 * node + ((d < 4 ? lo : hi) >= v ? 1u : 0u);
      }
      node -= kPositions;
    } else {
      node = n < p.k ? 0 : 0xffffffffu;
    }
    // Targets of a warp in the same cell are counted at once: equal ones (the zero groups of a pruned matrix) would all queue
    // at one address (8388608 targets, half of them zero: 17.8 ms with an atomic each, 15.2 so).
    const uint32_t same = __match_any_sync(0xffffffffu, node), first = __ffs(same) - 1;
    uint32_t at = 0;
    if (lane == first && n < p.k) at = atomicAdd(&cells[node], (uint32_t)__popc(same));
    at = __shfl_sync(0xffffffffu, at, first) + __popc(same & ((1u << lane) - 1u));
    if (n < p.k) keys[n] = make_uint2(node, at);
  }
}

// Counts by cell -> first places: a block per 1024 cells, which adds up all cells before them as well.
__global__ void __launch_bounds__(1024) sorted_scan_kernel(const uint32_t* cells, uint32_t* starts) {
  __shared__ uint32_t part[32], ahead[32];
  pdl_trigger();
  pdl_wait();
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint32_t before = 0;
#pragma unroll 4
  for (uint32_t i = tid; i < blockIdx.x * 256; i += 1024) {
    const uint4 c = reinterpret_cast<const uint4*>(cells)[i];
    before += c.x + c.y + c.z + c.w;
  }
  const uint32_t own = cells[blockIdx.x * 1024 + tid];
  uint32_t incl = own;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t up = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= (uint32_t)o) incl += up;
  }
  before = __reduce_add_sync(0xffffffffu, before);
  if (lane == 0) ahead[warp] = before;
  if (lane == 31) part[warp] = incl;
  __syncthreads();
  starts[blockIdx.x * 1024 + tid] =
      __reduce_add_sync(0xffffffffu, ahead[lane] + (lane < warp ? part[lane] : 0u)) + incl - own;
}

__global__ void __launch_bounds__(256) sorted_place_kernel(const uint32_t* idx, uint64_t k, const uint32_t* starts,
                                                           const uint2* keys, uint32_t n_steps, uint32_t* sidx,
                                                           uint32_t* place, uint16_t* tile_step) {
  pdl_trigger();
  pdl_wait();
  for (uint64_t n = (uint64_t)blockIdx.x * 256 + threadIdx.x; n < k; n += (uint64_t)gridDim.x * 256) {
    const uint2 key = keys[n];
    const uint32_t at = starts[key.x] + key.y;
    sidx[at] = idx[n];
    place[at] = (uint32_t)n;
    if (at % 256 == 0) tile_step[at / 256] = (uint16_t)min(key.x >> 7, n_steps - 1);
  }
}

// ---- which steps a tile has to go over ----------------------------------------------
// A warp takes tiles of 256 sorted targets, a lane one of them at a time.  r is at least the distance to a codeword that is
// known: the stored one, or the best of the first sweep (its score and the margin of that).  A step is left out for a target if
// the distance to its box exceeds r for certain.  The distances are formed in half precision, two boxes per instruction,
// first to the boxes of eight steps, whose steps are looked at if any target of the warp comes that near.
// The target is rounded to half (2^-11 |t_i|), the boxes outwards, and the nearest point of a box is a half, so that a gap is
// at least b (1 - 2^-11) - 2^-11 |t_i| with b its value in half precision; the sum of the eight squares is off by less than
// ten units of 2^-11 of itself, and by 2^-20 where halves are subnormal.  Hence the limit
// (r + 1.01 2^-11 ||t||)^2 (1 + 2^-7) + 2^-14.  (Elements of codewords are scaled to at most 8.)
// What bounds it: the pipes of half-precision arithmetic, about evenly: 44 instructions for two boxes.  A block with a tile,
// every warp for itself: 2.34 ms for 8388608 targets; a warp with a tile, which leaves out what its earlier targets need,
// 2.13; the nearest point by minimum and maximum in place of centre and width 2.02.
constexpr int kReachThreads = 128, kReachBlocks = 10;
__global__ void __launch_bounds__(kReachThreads, kReachBlocks) sorted_reach_kernel(
    const EncM1Params p, const TcNorms norms, const uint4* packed, const uint16_t* near, const uint16_t* tile_step,
    uint16_t* lists, uint32_t* counts) {
  __shared__ __align__(16) uint4 box[(kSortedSteps + kSortedSteps / 8) * 2];  // pairs of boxes, 64 bytes
  __shared__ uint32_t n2max, n2min_inv;
  constexpr uint32_t kFull = 0xffffffffu;
  const uint32_t tid = threadIdx.x, lane = tid & 31;
  if (tid == 0) n2max = n2min_inv = 0;
  pdl_trigger();
  pdl_wait();
  __syncthreads();
  for (uint32_t i = tid; i - lane < norms.blocks; i += kReachThreads) {
    const uint2 part = i < norms.blocks ? norms.norms[i] : make_uint2(0, 0);
    const uint32_t a = __reduce_max_sync(kFull, part.x), b = __reduce_max_sync(kFull, part.y);
    if (lane == 0) {
      atomicMax(&n2max, a);
      atomicMax(&n2min_inv, b);
    }
  }
  for (uint32_t i = tid; i < (kSortedSteps + kSortedSteps / 8) * 2; i += kReachThreads) box[i] = packed[i];
  __syncthreads();
  const float scale = box_scale(n2max), cnmin = sqrtf(__uint_as_float(0x7f800000u - n2min_inv));
  const uint32_t n_steps = p.n_units, n_words = (n_steps + 31) / 32;
  const uint4* groups = box + kSortedSteps * 2;
  const uint32_t warps = gridDim.x * (kReachThreads / 32);
  for (uint32_t tile = blockIdx.x * (kReachThreads / 32) + (tid >> 5); tile < p.n_tiles; tile += warps) {
    // Lane w has word w of the steps that are needed; bit i: its step 2 i, bit 16 + i: step 2 i + 1.  What the first sweep has
    // seen, and what earlier targets of the tile need, is not looked at again.
    static_assert(kSortedNear == 32 && kSortedSteps == 512, "a step per lane, a word per lane of sixteen");
    uint32_t seen = 0, marked = 0;
    {
      const uint32_t s = near[(uint32_t)tile_step[tile] * kSortedNear + lane];
      const uint32_t bit = 1u << ((s >> 1 & 15) + 16 * (s & 1));
#pragma unroll 1
      for (uint32_t w = 0; w < n_words; ++w) {
        const uint32_t word = __reduce_or_sync(kFull, (s >> 5) == w ? bit : 0u);
        if (lane == w) seen = word;
      }
      marked = seen;
    }
    const uint64_t n0 = (uint64_t)tile * 256 + lane;
    uint32_t j_next = n0 < p.k ? p.idx[n0] : kFull;
#pragma unroll 1
    for (uint32_t turn = 0; turn < 8; ++turn) {
      const uint64_t n = n0 + 32 * turn;
      const uint32_t j = j_next;
      if (turn < 7) j_next = n + 32 < p.k ? p.idx[n + 32] : kFull;
      __half2 x[8], lim;
      {
        float t[8], r2 = -1.0f, nt2 = 0.0f;  // (nothing to look for)
#pragma unroll
        for (int i = 0; i < 8; ++i) t[i] = 0.0f;
        if (j < p.G) {
          const uint32_t code = p.code_u16 ? reinterpret_cast<const uint16_t*>(p.codes)[j]
                                           : reinterpret_cast<const uint8_t*>(p.codes)[j];
          form_target(p, j, t);
          float m = 0.0f;
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            m = fmaxf(m, fabsf(t[i]));
            nt2 = fmaf(t[i], t[i], nt2);
          }
          const TargetScale ts = target_scale(m, nt2, cnmin);
          if (ts.in_range) {  // (the others are rescored against the whole codebook)
            const float score = unord(p.gbest[n]);  // 2^e d^2 / 2 of the best so far, but for rounding
            r2 = 2.0f * (score + fmaf(p.rel_margin, fabsf(score), p.margin[n])) / ts.scale;
            if (code < p.K) {
              float c[8];
              load_codeword<true, 8>(p.book, code, c);
              float d = 0.0f;
#pragma unroll
              for (int i = 0; i < 8; ++i) d = fmaf(t[i] - c[i], t[i] - c[i], d);
              if (d < r2) r2 = d;
            }
            r2 = fmaxf(r2, 0.0f);
          }
        }
        float limit = -1.0f;
        if (r2 >= 0.0f) {
          const float r = scale * fmaf(4.94e-4f, sqrtf(nt2), sqrtf(r2) * 1.0001f);
          limit = fmaf(r * r, 1.0078125f, 6.103515625e-5f);
        }
        bool all = r2 != r2 || limit > 60000.0f;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float y = t[i] * scale;
          all = all || (r2 >= 0.0f && !(fabsf(y) < 1000.0f));
          x[i] = __float2half2_rn(y);
        }
        lim = __half2half2(__float2half_ru(limit));
        if (all) {  // beyond what halves can tell: every step
#pragma unroll
          for (int i = 0; i < 8; ++i) x[i] = __float2half2_rn(0.0f);
          lim = __half2half2(__ushort_as_half(0x7c00));
        }
      }
      // whether the target may reach each of the two boxes at `at`: all bits of the low and of the high half
      auto reached = [&](const uint4* at) -> uint32_t {
        __half2 sum = __float2half2_rn(0.0f);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const uint4 raw = at[q];
          const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const __half2 lo = *reinterpret_cast<const __half2*>(&w[2 * i]);
            const __half2 hi = *reinterpret_cast<const __half2*>(&w[2 * i + 1]);
            const __half2 gap = __hsub2(x[2 * q + i], __hmin2(__hmax2(x[2 * q + i], lo), hi));
            sum = __hfma2(gap, gap, sum);
          }
        }
        return __hle2_mask(sum, lim);
      };
#pragma unroll 1
      for (uint32_t w = 0; w < n_words; ++w) {
        const uint32_t open = ~__shfl_sync(kFull, marked, w);
        uint32_t in = 0;
#pragma unroll 1
        for (uint32_t q = 0; q < 2; ++q) {
          if (!(open & (0x00ff00ffu << (8 * q)))) continue;
          const uint32_t near8 = __reduce_or_sync(kFull, reached(groups + (2 * w + q) * 4));
#pragma unroll
          for (uint32_t side = 0; side < 2; ++side) {
            const uint32_t at = 8 * q + 4 * side;  // four pairs of steps
            if (near8 >> (16 * side) & 1u) {
#pragma unroll
              for (uint32_t i = 0; i < 4; ++i)
                if (open & (0x00010001u << (at + i))) in |= reached(box + (16 * w + at + i) * 4) & (0x00010001u << (at + i));
            }
          }
        }
        in = __reduce_or_sync(kFull, in);
        if (lane == w) marked |= in;
      }
    }
    // the list, without what the first sweep has seen
    auto in_order = [](uint32_t word) {  // of the steps: the halves of the word interleaved
      uint32_t x = word & 0xffffu, y = word >> 16;
      x = (x | (x << 8)) & 0x00ff00ffu, y = (y | (y << 8)) & 0x00ff00ffu;
      x = (x | (x << 4)) & 0x0f0f0f0fu, y = (y | (y << 4)) & 0x0f0f0f0fu;
      x = (x | (x << 2)) & 0x33333333u, y = (y | (y << 2)) & 0x33333333u;
      x = (x | (x << 1)) & 0x55555555u, y = (y | (y << 1)) & 0x55555555u;
      return x | (y << 1);
    };
    uint32_t b = in_order(marked & ~seen);
    if (32 * lane + 32 > n_steps) b &= 32 * lane < n_steps ? (1u << (n_steps & 31)) - 1u : 0u;  // (steps that are there)
    // A search needs a step.  One more than needed does no harm, if the first sweep has not gone over it either: the first such
    // (there are far more steps than that sweep takes).
    if (!__any_sync(kFull, b != 0)) {
      const uint32_t open = ~in_order(seen);
      if ((int)lane == __ffs(__ballot_sync(kFull, open != 0)) - 1) b = open & (0u - open);
    }
    const uint32_t c = __popc(b);
    uint32_t incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t up = __shfl_up_sync(kFull, incl, o);
      if (lane >= (uint32_t)o) incl += up;
    }
    uint16_t* to = lists + (size_t)tile * list_stride(n_steps) + incl - c;
    while (b) {
      *to++ = (uint16_t)(32 * lane + __ffs(b) - 1);
      b &= b - 1;
    }
    if (lane == 31) counts[tile] = incl;
  }
}

}  // namespace

namespace m1 {

cudaError_t launch_sorted_codebook(const void* book, uint32_t K, const SortedScratch& s, cudaStream_t stream) {
  const uint4* raw = reinterpret_cast<const uint4*>(book);
  cudaError_t e = launch_dependent(sorted_dims_kernel, 17, kSplitThreads, 0, stream, raw, K, s.dims, s.cells);
  if (e != cudaSuccess) return e;
  const uint32_t* from = nullptr;
  int launches = 1;
  if ((e = allow_smem<sorted_split_kernel>()) != cudaSuccess) return e;
  for (int level = 0; (kPositions >> level) > kTailPositions; ++level, ++launches) {
    uint32_t* to = (level & 1) ? s.order : s.order2;  // (seven levels)
    const size_t keys = sizeof(uint16_t) * (kPositions >> level);
    if ((e = launch_dependent(sorted_split_kernel, 1u << level, kSplitThreads, keys, stream, raw, K, (const uint32_t*)s.dims,
                              level, from, to, s.tree)) != cudaSuccess)
      return e;
    from = to;
  }
  e = launch_dependent(sorted_tail_kernel, kPositions / kTailPositions, kTailThreads, 0, stream, raw, K,
                       (const uint32_t*)s.dims, from, s.order, s.tree);
  count_launches(launches + 1);
  return e;
}

cudaError_t launch_sorted_targets(const EncM1Params& p, const uint32_t* idx, const TcNorms& norms, const SortedScratch& s,
                                  int sm_count, cudaStream_t stream) {
  cudaError_t e = launch_dependent(sorted_box_kernel, p.n_units, 128, 0, stream, (const uint4*)s.book, p.K, s.boxes);
  if (e != cudaSuccess) return e;
  if ((e = launch_dependent(sorted_near_kernel, kSortedSteps, kSortedSteps, 0, stream, (const float*)s.boxes, p.n_units,
                            norms.norms, norms.blocks, s.near, reinterpret_cast<__half*>(s.packed))) != cudaSuccess)
    return e;
  if ((e = launch_dependent(sorted_key_kernel, (unsigned)sm_count * 8, 256, 0, stream, p, idx, (const uint32_t*)s.dims,
                            (const float*)s.tree, s.cells, s.keys)) != cudaSuccess)
    return e;
  if ((e = launch_dependent(sorted_scan_kernel, kPositions / 1024, 1024, 0, stream, (const uint32_t*)s.cells, s.starts)) !=
      cudaSuccess)
    return e;
  e = launch_dependent(sorted_place_kernel, (unsigned)sm_count * 8, 256, 0, stream, idx, p.k, (const uint32_t*)s.starts,
                       (const uint2*)s.keys, p.n_units, s.sidx, s.place, s.tile_step);
  count_launches(5);
  return e;
}

cudaError_t launch_sorted_reach(const EncM1Params& p, const TcNorms& norms, const SortedScratch& s, int sm_count,
                                cudaStream_t stream) {
  uint64_t blocks;
  cudaError_t e = resident_blocks<sorted_reach_kernel>(kReachThreads, sm_count, &blocks);
  if (e != cudaSuccess) return e;
  const uint64_t want = (p.n_tiles + kReachThreads / 32 - 1) / (kReachThreads / 32);
  if (blocks > want) blocks = want;
  count_launches(1);
  return launch_dependent(sorted_reach_kernel, (unsigned)blocks, kReachThreads, 0, stream, p, norms, (const uint4*)s.packed,
                          (const uint16_t*)s.near, (const uint16_t*)s.tile_step, s.lists, s.counts);
}

}  // namespace m1
}  // namespace pvt
