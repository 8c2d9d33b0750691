// Reciprocal square root and reciprocal of the FP64 factorisations.
#pragma once

namespace gcx {

// Both take the hardware's approximation y, of relative error delta (measured on GB300: at most 2^-20.1 for the root,
// 2^-19.9 for the reciprocal), and one step of the binomial series of (1 - e)^p (p = -1/2, -1), e = 1 - a y^2 or
// 1 - a y, cut after e^2.  A warp's FP64 instruction holds its sub-partition's pipe for 64 cycles whatever its lanes
// do: these take five and four.
//
// 1 / sqrt(a) for a in the normal range: y (1 + e/2 + 3 e^2/8).  e is about 2 delta, so the cut 5 e^3/16 is 2.5 delta^3,
// 2^-59; e is rounded at 2^-53 and enters halved, the last operation rounds once: 1.52 x 2^-53 in all (measured 1.23;
// 80,072 values of 2^-963 to 2^900).
__device__ __forceinline__ double rsqrt_fast(double a) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(a));
  const double e = fma(-(a * y), y, 1.0);
  return fma(y * e, fma(0.375, e, 0.5), y);
}
// 1 / a for a in the normal range, by y (1 + e + e^2): the cut is delta^3, the last operation rounds once (measured
// 1.00 x 2^-53).
__device__ __forceinline__ double rcp_fast(double a) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(a));
  const double e = fma(-a, y, 1.0);
  return fma(y * e, 1.0 + e, y);
}

}  // namespace gcx
