// fp64_math.cuh -- FP64 functions in few operations for arguments of known
// range (the FP64 pipe issues one warp instruction per 16 cycles and SM).
//
// cos(2 pi x) for finite |x| < 2^51: with r = x - rint(x) and b = 1/4 - |r| in [-1/4, 1/4], cos(2 pi x) =
// sin(2 pi b) = b P(b^2), P of degree 8 (interpolation of sin(2 pi b) / b at the
// Chebyshev nodes of [0, 1/16] in b^2; with the coefficients rounded to FP64
// within 4e-17).
#pragma once

namespace sde {

// P(s) = sin(2 pi b) / b, s = b^2 <= 1/16.
__device__ __forceinline__ double sin2pi64_poly(double s) {
  double p = 0.10089695501646812;
  p = fma(p, s, -0.7177337921413454);
  p = fma(p, s, 3.8199280942271643);
  p = fma(p, s, -15.0946416761179);
  p = fma(p, s, 42.058693925428685);
  p = fma(p, s, -76.70585975282492);
  p = fma(p, s, 81.60524927607362);
  p = fma(p, s, -41.341702240399755);
  return fma(p, s, 6.283185307179586);
}

__device__ __forceinline__ double cos2pi64(double x) {
  const double b = 0.25 - fabs(x - rint(x));
  return b * sin2pi64_poly(b * b);
}

// sqrt(L), L >= 0, by Goldschmidt's iteration from the hardware's approximate
// reciprocal square root and a final correction by the residual L - g^2.
__device__ __forceinline__ double sqrt_goldschmidt(double L) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(L));
  y = L > 0.0 ? y : 0.0;
  double g = L * y, h = 0.5 * y;
  const double r = fma(-g, h, 0.5);
  g = fma(g, r, g);
  h = fma(h, r, h);
  return fma(fma(-g, g, L), h, g);
}

}  // namespace sde
