// reduce_final.cuh -- the last stage of the scalar reductions: one warp per
// quantity sums the blocks' partials in a fixed order.  (One thread per
// quantity had added 608 partials one after another, 114 us of dependent
// FP64 additions and loads; a warp's lanes take every 32nd partial.)
#pragma once

#include "flame_internal.h"

namespace flame {

// Quantity v of `nblocks` blocks' partials (kRedVals each; 14 is a maximum,
// the others sums), by the calling warp; the result is lane 0's.
__device__ __forceinline__ double reduce_partials_warp(const double* __restrict__ partials, int nblocks, int v) {
  const int lane = threadIdx.x & 31;
  double a = 0.0;
  for (int b = lane; b < nblocks; b += 32) {
    const double t = partials[(long long)b * kRedVals + v];
    a = v == 14 ? fmax(a, t) : a + t;
  }
  for (int o = 16; o > 0; o >>= 1) {
    const double t = __shfl_down_sync(0xffffffffu, a, o);
    a = v == 14 ? fmax(a, t) : a + t;
  }
  return a;
}

}  // namespace flame
