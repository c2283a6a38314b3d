// FP64 reciprocal and reciprocal square root in a few FP64 instructions.  One
// warp issues an FP64 instruction every 64 cycles on this part, and the IEEE
// divide and square root are long sequences of them (1400 cycles together);
// these start from the FP32 approximation (relative error e of about 1e-7) and
// make one third-order step of Householder's method, 1 + e + e^2 and
// 1 + e / 2 + 3 e^2 / 8, whose error is of the order of e^3.  What is left are
// the roundings of the last operations: at most 0.6 ulp for the reciprocal, 1.1 for
// the root.  Arguments whose exponent the FP32 range does not hold (zero, infinity
// and NaN among them) take the library's divide and reciprocal square root.
#pragma once

#include <cuda_runtime.h>

namespace ofm {

__device__ __forceinline__ bool fp32_range(double x) {
  const int e = (__double2hiint(x) >> 20) & 0x7ff;
  return e > 1023 - 100 && e < 1023 + 100;
}

__device__ __forceinline__ double rcp64(double x) {
  if (!fp32_range(x)) return 1.0 / x;
  const double y = (double)__fdividef(1.0f, (float)x);
  const double e = fma(-x, y, 1.0);
  return fma(y * e, 1.0 + e, y);
}

__device__ __forceinline__ double rsqrt64(double x) {
  if (!fp32_range(x)) return rsqrt(x);
  const double y = (double)rsqrtf((float)x);
  const double e = fma(-(x * y), y, 1.0);
  return fma(y * e, fma(e, 0.375, 0.5), y);
}

}  // namespace ofm
