// The tensor search over codewords and targets in spatial order: its scratch, and what prepares it.
#pragma once

#include "pvt_encode_m1.cuh"

namespace pvt {
namespace m1 {

constexpr int kSortedLevels = 16;            // of the tree: 65536 positions, those behind the last codeword empty
constexpr uint32_t kSortedSteps = 512;       // of 128 positions
constexpr uint32_t kSortedNear = 32;         // steps of the first sweep

// rows of the tiles' lists begin at 16-byte boundaries
__host__ __device__ constexpr uint32_t list_stride(uint32_t n_steps) { return (n_steps + 7) / 8 * 8; }

// What orders the steps by their distance from step `own` (its bit pattern; infinite where there is no step).  The keys of all
// kSortedSteps steps differ, so that they have the ranks 0, 1, 2, ...: the own one is zero, every other at least kSortedSteps
// with the step's number in its last bits.  (Without that least one step 0 would tie with `own` where the centres of their
// boxes are the same, as in a codebook of equal codewords, and a rank would have no step.)
__host__ __device__ constexpr uint32_t near_key(uint32_t distance_bits, uint32_t step, uint32_t own) {
  const uint32_t rounded = distance_bits & ~(kSortedSteps - 1);
  return step == own ? 0u : (rounded < kSortedSteps ? kSortedSteps : rounded) | step;
}

struct SortedScratch {
  uint32_t* dims;       // [16]: the dimension that a level splits
  float* tree;          // [65536]: values, node i of level l at 2^l + i
  uint32_t *order, *order2;  // [65536]: codeword by position
  uint4* book;          // [K]: the codebook by position
  float* boxes;         // [512][16]: smallest and largest elements by step
  uint4* packed;        // [288][4]: pairs of boxes of steps, of eight steps, in half precision
  uint16_t* near;       // [512][32]: the nearest steps
  uint32_t *cells, *starts;  // [65536]: targets by cell, their first place
  uint2* keys;          // [k]: cell and place in it, in the records' memory
  uint32_t *sidx, *place;  // [k]: group and place in the caller's list by sorted place
  uint16_t* tile_step;  // [tiles]
  uint16_t* lists;      // [tiles][steps]
  uint32_t* counts;     // [tiles]
};
// what the kernel that prepares the operand image leaves of the codewords' norms
struct TcNorms {
  const uint2* norms;
  uint32_t blocks;
};

cudaError_t launch_sorted_codebook(const void* book, uint32_t K, const SortedScratch& s, cudaStream_t stream);
cudaError_t launch_sorted_targets(const EncM1Params& p, const uint32_t* idx, const TcNorms& norms, const SortedScratch& s,
                                  int sm_count, cudaStream_t stream);
cudaError_t launch_sorted_reach(const EncM1Params& p, const TcNorms& norms, const SortedScratch& s, int sm_count,
                                cudaStream_t stream);

}  // namespace m1
}  // namespace pvt
