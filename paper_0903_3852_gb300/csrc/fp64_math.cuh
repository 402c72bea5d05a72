// fp64_math.cuh -- FP64 functions in few operations for arguments of known
// range (the FP64 pipe issues one warp instruction per 16 cycles and SM).
#pragma once

namespace sde {

// sin(2 pi b) / b, s = b^2 <= 1/16: degree 8, interpolation at the Chebyshev nodes
// of [0, 1/16] (with the coefficients rounded to FP64 within 4e-17).
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

// cos(2 pi k / P), k in [0, P], inv4P = 1 / (4 P): sin(2 pi b) with b = 1/4 - min(k, P -
// k) / P, whose numerator is an exact integer.  Within 2.7e-16 for P up to 4096 (a
// correctly rounded cosine of the rounded quotient k / P: 3.6e-16).
__device__ __forceinline__ double cos_ratio64(int k, int P, double inv4P) {
  const int m = k <= P - k ? k : P - k;
  const double b = (double)(P - 4 * m) * inv4P;
  return b * sin2pi64_poly(b * b);
}

// sqrt(L), L >= 0 (0 below 2^-1022), by Goldschmidt's iteration from the hardware's
// approximate reciprocal square root and a final correction by the residual L -
// g^2.  The test for zero and the halving are done on the high word, off the FP64
// pipe.
__device__ __forceinline__ double sqrt_goldschmidt(double L) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(L));
  const bool zero = __double2hiint(L) < 0x00100000;
  const int yh = __double2hiint(y), yl = __double2loint(y);
  double g = L * (zero ? 0.0 : y), h = zero ? 0.0 : __hiloint2double(yh - 0x00100000, yl);
  const double r = fma(-g, h, 0.5);
  g = fma(g, r, g);
  h = fma(h, r, h);
  return fma(fma(-g, g, L), h, g);
}

}  // namespace sde
