// Pointwise pieces of the lateral kernels: the soft threshold and the block sums
// of the norm partials.
#pragma once

#include "common.cuh"

namespace isam {

// T_tau(u) = u max(|u| - tau, 0) / (max(|u| - tau, 0) + tau)  (Eq. 14),
// evaluated as u max(1 - tau / |u|, 0); 0 where |u| = 0.
__device__ __forceinline__ float2 soft_threshold(float2 u, float tau) {
  const float m2 = fmaf(u.x, u.x, u.y * u.y);
  const float f = m2 > 0.0f ? fmaxf(1.0f - tau * rsqrtf(m2), 0.0f) : 0.0f;
  return cscale(u, f);
}
__device__ __forceinline__ double2 soft_threshold(double2 u, double tau) {
  const double m2 = fma(u.x, u.x, u.y * u.y);
  const double f = m2 > 0.0 ? fmax(1.0 - tau / sqrt(m2), 0.0) : 0.0;
  return cscale(u, f);
}

// Sum of v over the threads of one warp that exist: a block of nt threads
// (any count, e.g. 8, 24 or 48 for short or 3 * 2^p lateral lengths) has a
// last warp of n = nt - 32 w lanes, and a shuffle may only name lanes that
// exist, so the mask holds lanes [0, n) and a lane adds a partner's value only
// when that partner exists.  The sum lands in lane 0.
__device__ __forceinline__ double warp_sum_lanes(double v, int n) {
  const unsigned mask = n >= 32 ? 0xffffffffu : ((1u << n) - 1u);
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double t = __shfl_down_sync(mask, v, o);
    if (lane + o < n) v += t;
  }
  return v;
}

}  // namespace isam
