// rlb_quad.cuh -- the four-lanes-per-node arrangement of one D3Q19 distribution that the
// small-lattice steps and the quasi-1D reverse step share: which links a lane holds, and the
// sums over a node's lanes.
#pragma once
#include <cuda_runtime.h>

namespace {

constexpr int kTubeWarps = 4;                // warps of 8 nodes that a quasi-1D block holds
constexpr int kTubeTile = 8 * kTubeWarps;    // its nodes

__device__ __forceinline__ long long quad_sum64(long long v) {
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  v += __shfl_xor_sync(0xffffffffu, v, 2);
  return v;
}
__device__ __forceinline__ long long sel3(int j, long long v0, long long v1, long long v2) {
  return j == 0 ? v0 : (j == 1 ? v1 : v2);
}
// slot sl of lane j: link and direction (slots 0-1 the axis pair, 2-3 the first diagonal
// pair of the lane's plane, 4-5 the second); lane 3 reads the rest link in every slot
__device__ __forceinline__ int quad_link(int j, int sl) {
  const int pd = j == 0 ? 3 : (j == 1 ? 7 : 5);   // first diagonal pair of the plane
  return j == 3 ? 0 : sl < 2 ? 2 * j + 1 + sl : 2 * pd + 1 + (sl - 2);
}
__device__ __forceinline__ void quad_dir(int j, int sl, int& cx, int& cy, int& cz) {
  const int da = j == 1 ? 1 : 0, db = j == 0 ? 1 : 2;
  if (sl < 2) {
    const int c = sl == 0 ? 1 : -1;
    cx = j == 0 ? c : 0;
    cy = j == 1 ? c : 0;
    cz = j == 2 ? c : 0;
  } else {
    const int sa = (sl & 1) ? -1 : 1;              // +(e_a + e_b), -(e_a + e_b), +(e_a - e_b), -(e_a - e_b)
    const int sb = sl < 4 ? sa : -sa;
    cx = da == 0 ? sa : 0;                          // db is never x
    cy = (da == 1 ? sa : 0) + (db == 1 ? sb : 0);
    cz = db == 2 ? sb : 0;                          // da is never z
  }
  if (j == 3) cx = cy = cz = 0;
}
}  // namespace
