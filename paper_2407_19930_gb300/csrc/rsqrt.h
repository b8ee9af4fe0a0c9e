// Reciprocal square root of the pivots of the diagonal blocks (k_ec.cu).
#pragma once

#include <cuda_runtime.h>

namespace librpa {

// 1 / sqrt(d) for a normal d > 0 in five FP64 instructions: FP32 seed r0 of the mantissa and one step of Householder's
// method of third order for the zero of 1 / r^2 - d, i.e. the binomial series of (1 - e)^(-1/2) in e = 1 - d r0^2 cut after
// e^2: r0 (1 + e / 2 + 3 e^2 / 8), error 5 e^3 / 16 < 2^-60.  Conversions and scaling by integer instructions.  The
// rounding of d r0 adds half a unit in the last place to that of the result.
__device__ __forceinline__ double fast_rsqrt(double d) {
  const int hi = __double2hiint(d), ex = hi >> 20;
  if (ex < 1 || ex > 2046) return rsqrt(d);
  const int q = (ex - 1023) & ~1;   // d 2^-q in [1, 4)
  const double x = __hiloint2double(hi - (q << 20), __double2loint(d));
  const float f = __int_as_float(((ex - q - 896) << 23) | ((hi & 0xFFFFF) << 3));
  const int rb = __float_as_int(rsqrtf(f));
  const double r0 = __hiloint2double((rb >> 3) + (896 << 20), rb << 29);
  const double e = fma(-(x * r0), r0, 1.0);
  const double r = fma(r0 * e, fma(0.375, e, 0.5), r0);
  return __hiloint2double(__double2hiint(r) - ((q / 2) << 20), __double2loint(r));
}

// sqrt(d) from ri = fast_rsqrt(d): d ri and one Newton step
__device__ __forceinline__ double sqrt_from(double d, double ri) {
  const double s = d * ri;
  return fma(0.5 * ri, fma(-s, s, d), s);
}

}  // namespace librpa
