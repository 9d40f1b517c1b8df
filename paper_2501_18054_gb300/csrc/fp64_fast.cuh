// Reciprocals for short FP64 chains: a division occupies the FP64 pipe of this
// part for ten instructions (640 cycles of a warp), a Newton step for two.
#pragma once

#include "sweep_common.cuh"

namespace pngf {
namespace {

// biased exponent
__device__ __forceinline__ int oz_exp(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// 1 / x for x > 0: FP32 seed and two Newton steps (2^-22, 2^-44, 2^-88), no
// FP64 division (ten instructions' time on the FP64 pipe)
__device__ __forceinline__ double rcp_pos(double x) {
  const int ex = oz_exp(x);
  if (ex < 1023 - 120 || ex > 1023 + 120) return 1.0 / x;
  double r = (double)(1.0f / (float)x);
  r = fma(r, fma(-x, r, 1.0), r);
  return fma(r, fma(-x, r, 1.0), r);
}

// 1 / z: z is scaled by a power of two to [1, 2), |z|^-2 by an FP32
// seed and two Newton steps
__device__ __forceinline__ c128 crecip(c128 z) {
  const int ex = max(oz_exp(z.x), oz_exp(z.y));
  if (ex < 64 || ex > 1980) return cdiv(mk(1.0, 0.0), z);  // zero, tiny, huge, infinite, NaN
  const double sc = __longlong_as_double((long long)(2046 - ex) << 52);  // 2^(1023 - ex)
  const double x = z.x * sc, y = z.y * sc;
  const double d = fma(x, x, y * y);  // in [1, 8)
  double r = (double)(1.0f / (float)d);
  r = fma(r, fma(-d, r, 1.0), r);
  r = fma(r, fma(-d, r, 1.0), r);
  r *= sc;
  return mk(x * r, -y * r);
}

}  // namespace
}  // namespace pngf
