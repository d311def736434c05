// FP64 values through integer operations and the FP32 pipe (the FP64 pipe has two lanes a clock and SM).
#pragma once
#include <cuda_runtime.h>

namespace fthms {

__device__ __forceinline__ double f2d_bits(float f) {       // exact for normal f (zero gives 2^-127-ish)
  const unsigned u = __float_as_uint(f);
  return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7FFFFFFFu) >> 3) + 0x38000000u)), (int)(u << 29));
}

// Distance from its square R2 without the library's square root: R2 = m 4^k with m in [1, 4), the FP32 reciprocal root of
// m and two Newton steps on R2 (relative error 2^-22 -> 2^-45 -> below 2^-53).  Zero and every normal R2, so
// whatever the unit of length (an FP32 reciprocal root of R2 itself holds for distances of 1e-19 to 1e19 alone).
__device__ __forceinline__ double dist_f64(double R2) {
  const int h = __double2hiint(R2), l = __double2loint(R2);
  const int k = ((h >> 20) - 1023) >> 1, mh = h - k * 0x200000;
  const float y = rsqrtf(__uint_as_float((unsigned)((mh - 0x38000000) << 3) | ((unsigned)l >> 29)));   // m truncated
  const unsigned u = __float_as_uint(y);
  const int yh = (int)((u >> 3) + 0x38000000u) - k * 0x100000, yl = (int)(u << 29);
  const double yd = __hiloint2double(yh, yl), hy = __hiloint2double(yh - 0x100000, yl);             // 1/R, 1/(2 R)
  double r = R2 * yd;
  r = fma(fma(-r, r, R2), hy, r);
  return fma(fma(-r, r, R2), hy, r);
}

}  // namespace fthms
