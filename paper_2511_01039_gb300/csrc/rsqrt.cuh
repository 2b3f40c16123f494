#pragma once

#include <cuda_runtime.h>

namespace fpeps {

// 1 / sqrt(x) from the FP32 value by one step of Householder's third-order iteration (the Taylor
// series of (1 - r)^(-1/2), r = 1 - x y^2 ~ 2^-22): about 320 cycles of dependent FP64 operations, half
// of what rsqrt() takes here, on the critical path of every column.
__device__ __forceinline__ double rsqrt_fast(double x) {
  const int hi = __double2hiint(x);
  if (hi < 0x00100000) return rsqrt(x);   // below the normal range
  const int e = ((hi >> 20) - 1023) & ~1;
  const double m = __hiloint2double(hi - (e << 20), __double2loint(x));   // [1, 4)
  const double y = (double)rsqrtf((float)m);
  const double r = fma(-m, y * y, 1.0);   // y has 24 bits: y y is exact, and r rounded once
  const double p = fma(fma(r, 0.3125, 0.375), r, 0.5);
  const double z = fma(p, y * r, y);
  return __hiloint2double(__double2hiint(z) - ((e / 2) << 20), __double2loint(z));
}

}  // namespace fpeps
