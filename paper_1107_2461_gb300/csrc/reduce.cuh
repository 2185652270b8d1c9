// Fixed-order sums of FP64 values over a warp and a block.  GB300 adds FP64 at 2
// lanes per clock and SM, so one warp-wide add occupies an SM quarter's FP64
// pipe for 64 clocks whatever the number of lanes that matter: the components
// are packed into disjoint lanes before the butterfly (two components cost 5
// adds instead of 10, four cost 6 instead of 20), and the warps' sums are added
// by a butterfly as well instead of one thread's chain.
#pragma once
#include <cuda_runtime.h>

namespace fdi {
namespace red {

// sum over the warp of the component that belongs to the lane: with two
// components lanes 0-15 carry a and 16-31 carry b (every one of them the total)
__device__ __forceinline__ double warp_sum2(double a, double b) {
  const int lane = threadIdx.x & 31;
  const bool hi = lane & 16;
  double v = (hi ? b : a) + __shfl_xor_sync(0xffffffffu, hi ? a : b, 16);
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// four components: lanes 0-7 a, 8-15 c, 16-23 b, 24-31 d
__device__ __forceinline__ double warp_sum4(double a, double b, double c, double d) {
  const int lane = threadIdx.x & 31;
  const bool hi = lane & 16, hq = lane & 8;
  const double ab = (hi ? b : a) + __shfl_xor_sync(0xffffffffu, hi ? a : b, 16);
  const double cd = (hi ? d : c) + __shfl_xor_sync(0xffffffffu, hi ? c : d, 16);
  double v = (hq ? cd : ab) + __shfl_xor_sync(0xffffffffu, hq ? ab : cd, 8);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// sums of a and b over the first `warps` (<= 16) warps of a one-dimensional
// block, returned to warp 0 (sh: 32 doubles); every thread of the block calls it
__device__ __forceinline__ void block_sum2(double& a, double& b, int warps, double* sh) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (w < warps) {
    const double v = warp_sum2(a, b);
    if ((lane & 15) == 0) sh[lane + w] = v;  // a of warp w at w, b at 16 + w
  }
  __syncthreads();
  if (w == 0) {
    double v = (lane & 15) < warps ? sh[lane] : 0.0;
    if (warps > 1) {
      for (int o = warps > 8 ? 8 : (warps > 4 ? 4 : (warps > 2 ? 2 : 1)); o > 0; o >>= 1)
        v += __shfl_xor_sync(0xffffffffu, v, o);
    }
    a = __shfl_sync(0xffffffffu, v, 0);
    b = __shfl_sync(0xffffffffu, v, 16);
  }
}

}  // namespace red
}  // namespace fdi
