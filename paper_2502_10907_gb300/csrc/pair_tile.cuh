// Tiles of unordered index pairs: a block of n indices (triangles, or matrix
// rows) is cut into tiles of `size`; CTA t of the block takes the tile pair
// (I, J), I <= J, t = J (J + 1) / 2 + I.  prefix: first CTA of every block.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace mtf {

constexpr int kPairTile = 16;  // triangles per side of an assembly tile

struct PairTile {
  int blk, t0, s0;  // block, first index of either side (t0 <= s0)
};

__device__ __forceinline__ PairTile pair_tile(int64_t cta, const int64_t* __restrict__ prefix, int nblk,
                                              int size = kPairTile) {
  int lo = 0, hi = nblk - 1;
  while (lo < hi) {  // largest block with prefix <= cta
    const int mid = (lo + hi + 1) >> 1;
    if (prefix[mid] <= cta) lo = mid; else hi = mid - 1;
  }
  const int t = int(cta - prefix[lo]);
  int J = int((sqrtf(8.f * float(t) + 1.f) - 1.f) * 0.5f);
  while (int64_t(J) * (J + 1) / 2 > t) --J;  // the root is rounded
  while (int64_t(J + 1) * (J + 2) / 2 <= t) ++J;
  return {lo, (t - J * (J + 1) / 2) * size, J * size};
}

}  // namespace mtf
