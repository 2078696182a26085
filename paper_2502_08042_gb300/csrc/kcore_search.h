// Index arithmetic shared by device code and the host tests.
#pragma once

#ifdef __CUDACC__
#define KC_HD __host__ __device__ __forceinline__
#else
#define KC_HD inline
#endif

namespace kc {

// The middle of [lo, hi), 0 <= lo < hi < 2^31. Not (lo + hi) / 2: the sum
// leaves 32 bits in the upper half of a list of more than 2^30 entries.
KC_HD int middle(int lo, int hi) { return lo + ((hi - lo) >> 1); }

// Frontier vertices the batched peel lays out at a time: at most `block`, and
// so few that their arcs (at most dmax each) are counted in 32 bits.
KC_HD int chunk_vertices(int block, int dmax) {
  const int all = 0x7fffffff;
  if (dmax <= all / block) return block;
  return all / dmax;
}

}  // namespace kc
