// Shared device/host helpers of the CASPT2 library (not part of the C ABI).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include "../../include/caspt2.h"

#define CASPT2_CUDA_TRY(expr)                                  \
  do {                                                         \
    cudaError_t _e = (expr);                                   \
    if (_e != cudaSuccess) return CASPT2_ECUDA;                \
  } while (0)

namespace caspt2 {

constexpr int kMaxStates = 16;   // n <= 16 reference states

// Number of kernels this thread has launched through the library (read by the
// C ABI around a solve to report launches per solve).
inline long& launch_counter() {
  static thread_local long count = 0;
  return count;
}

// Block-wide FP64 sum in a fixed order (warp shuffle tree, then warp 0 over the
// per-warp partials).  Every thread must call it; the result is valid in thread 0.
__device__ __forceinline__ double block_sum(double v, double* smem32) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nwarp = (blockDim.x + 31) >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  __syncthreads();
  if (lane == 0) smem32[warp] = v;
  __syncthreads();
  v = (threadIdx.x < nwarp) ? smem32[threadIdx.x] : 0.0;
  if (warp == 0) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  }
  return v;
}

// 1/d for the energy denominators: one third-order step x <- x + x (e + e^2), e = 1 - d x (the
// first terms of the geometric series for 1 / (1 - e)), from the hardware's approximate double
// reciprocal (rcp.approx.ftz.f64, |e| < 2^-20), in three FP64 operations where two Newton steps
// take four.  Error: e^3 (2^-60) beside the last rounding, at most 0.51 units in the last place
// (0.505 measured over 2^22 arguments).  d must be a normal number, not zero.
__device__ __forceinline__ double recip(double d) {
  double x;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(x) : "d"(d));
  const double e = fma(-d, x, 1.0);
  return fma(x, fma(e, e, e), x);
}

// r = sqrt(s) and ir = 1 / sqrt(s) from the hardware's approximate reciprocal root y by the
// binomial series (1 - z)^(-1/2) = 1 + z/2 + 3 z^2/8, z = 1 - s y^2 (|z| < 2^-19).  Relative error:
// 5 z^3/16 (2^-58), half the rounding of s y and the last rounding, 1.6 2^-53 together.
__device__ __forceinline__ void root_and_recip(double s, double& r, double& ir) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(s));
  const double s0 = s * y, z = fma(-s0, y, 1.0), c = z * fma(0.375, z, 0.5);
  r = fma(s0, c, s0);
  ir = fma(y, c, y);
}

__device__ __forceinline__ double block_min(double v, double* smem32) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nwarp = (blockDim.x + 31) >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmin(v, __shfl_down_sync(0xffffffffu, v, o));
  __syncthreads();
  if (lane == 0) smem32[warp] = v;
  __syncthreads();
  v = (threadIdx.x < nwarp) ? smem32[threadIdx.x] : 1e300;
  if (warp == 0) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmin(v, __shfl_down_sync(0xffffffffu, v, o));
  }
  return v;
}

}  // namespace caspt2
