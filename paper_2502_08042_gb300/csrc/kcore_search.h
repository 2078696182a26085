// Binary search steps shared by device code and the host tests.
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

}  // namespace kc
