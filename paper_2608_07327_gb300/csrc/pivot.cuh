// 1/d and 1/sqrt(d) of the pivots of the k x k steps.
#pragma once
#include <cuda_runtime.h>

namespace mbpcg {

// 1/d for a positive normal d below 2^1000, within about an ulp: the hardware approximation
// (rcp.approx.f32) of d's leading 23 significand bits, rescaled by d's exponent with integer
// operations, then one third-order Newton step y = y0 (1 + e + e^2), e = 1 - d y0 (the truncated
// series of 1 / (1 - e)); the seed's relative error is below 2^-22, so e^3 is below 2^-66.
__device__ __forceinline__ double rcp_pos(double d) {
  const long long bits = __double_as_longlong(d);
  const int e = (int)(bits >> 52) & 0x7FF;
  const float f = __int_as_float(0x3F800000 | (int)((bits >> 29) & 0x7FFFFF));  // in [1, 2)
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(f));  // in (0.5, 1]
  const int rb = __float_as_int(r);
  const long long ex = (long long)(((rb >> 23) & 0xFF) - 127 + 2046 - e);
  const double y0 = __longlong_as_double((ex << 52) | ((long long)(rb & 0x7FFFFF) << 29));
  const double eps = fma(-d, y0, 1.0);
  const double e2 = fma(eps, eps, eps);
  return fma(y0, e2, y0);
}

// 1/sqrt(d) for a positive normal d, within about an ulp: rsqrt.approx.f32 of the leading
// significand bits with the exponent's parity folded in (argument in [1, 4)), then one third-order
// Newton step y = y0 (1 + e/2 + 3 e^2/8), e = 1 - d y0^2 (the series of (1 - e)^{-1/2}).
__device__ __forceinline__ double rsqrt_pos(double d) {
  const long long bits = __double_as_longlong(d);
  const int E = ((int)(bits >> 52) & 0x7FF) - 1023;
  const int odd = E & 1;
  const float f = __int_as_float(((127 + odd) << 23) | (int)((bits >> 29) & 0x7FFFFF));  // in [1, 4)
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(f));  // in (0.5, 1]
  const int rb = __float_as_int(r);
  const int half = (E - odd) / 2;
  const long long ex = (long long)(((rb >> 23) & 0xFF) - 127 - half + 1023);
  const double y0 = __longlong_as_double((ex << 52) | ((long long)(rb & 0x7FFFFF) << 29));
  const double t = d * y0;
  const double eps = fma(-t, y0, 1.0);
  const double q = eps * fma(eps, 0.375, 0.5);
  return fma(y0, q, y0);
}

}  // namespace mbpcg
