// Index rules of the gathers that the CPU can check too (plain C++ outside nvcc).
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define XKV_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define XKV_HOST_DEVICE inline
#endif

namespace xkv {

// Quantised bases: the group of 32 columns, counted in the row, that lane `lane` (0..3) of a row's quad fetches for the pair
// of 64-column slabs (ks, ks + 1), ks even; `rank` is a multiple of 32.  Beyond the rank it is the row's first group, inside
// the row also where that has fewer than four: no key step reaches those columns, and the value side keeps none of theirs.
XKV_HOST_DEVICE uint32_t quant_group(int ks, uint32_t lane, int rank) {
  return ks * 64 + (int)lane * 32 < rank ? 2u * (uint32_t)ks + lane : 0u;
}

}  // namespace xkv
