// FP64 reciprocal, square root and exponential in few FP64 instructions (the
// FP64 pipe issues one warp instruction per 64 cycles and SM partition;
// integer and FP32 work beside it is free).
#pragma once

#include "qmc_internal.cuh"

namespace qmc {

// FP32 value of a (|a| in 2^[-120, 120]) by integer operations on its bits
__device__ __forceinline__ bool fp32_seed(double a, float& f) {
  const int hi = __double2hiint(a);
  const int e = (hi >> 20) & 0x7ff;
  f = __uint_as_float(((unsigned)hi & 0x80000000u) | ((unsigned)(e - 896) << 23) |
                      (((unsigned)hi & 0xfffffu) << 3) | ((unsigned)__double2loint(a) >> 29));
  return e >= 1023 - 120 && e <= 1023 + 120;
}

// 1 / a: Householder's cubic step r (1 + e + e^2), e = 1 - a r, from the FP32
// reciprocal (relative error < 2^-21, cubed below 2^-63); 3 FP64 instructions
__device__ __forceinline__ double recip3(double a) {
  float f;
  if (!fp32_seed(a, f)) return 1.0 / a;
  const double r = widen(__frcp_rn(f));
  const double e = fma(-a, r, 1.0);
  return fma(r, fma(e, e, e), r);
}

// 1 / sqrt(a): the cubic step y (1 + e/2 + 3 e^2/8), e = 1 - a y^2; 5 instructions
__device__ __forceinline__ double rsqrt3(double a) {
  float f;
  if (!fp32_seed(a, f) || !(f > 0.f)) return 1.0 / sqrt(a);
  const double y = widen(rsqrtf(f));
  const double e = fma(-(a * y), y, 1.0);
  return fma(y * e, fma(e, 0.375, 0.5), y);
}

// sqrt(a) from its reciprocal iy (0 for a = 0): a iy corrected by the residual
// a - s^2, to within half an ulp and a little (3 instructions; distances enter
// exponentials, where an ulp of rho is zeta rho ulps of the orbital)
__device__ __forceinline__ double sqrt_from(double a, double iy) {
  const double s = a * iy;
  return __double_as_longlong(a) == 0 ? 0.0 : fma(0.5 * iy, fma(-s, s, a), s);
}

// 2^((nak x) / 2048): e^(-alpha x) with nak = -2048 alpha / ln 2.  Table-driven
// reduction in the manner of Tang (ACM TOMS 15, 1989) in base 2^(1/2048): the
// nearest integer n of nak x comes from one FMA with 1.5 x 2^52, the
// remainder |r| <= 1/2 from a second FMA (one rounding: the product is never
// rounded on its own), 2^(r/2048) from its Taylor polynomial to the third
// order (the next term is below 2^-54).  7 FP64 instructions.  Results below
// 2^-1022 are flushed to zero; NaN propagates.
__device__ __forceinline__ double exp_scaled(double nak, double x, const double* __restrict__ tab) {
  constexpr double kMagic = 6755399441055744.0;       // 1.5 x 2^52
  constexpr double kC1 = 3.3845077175778578e-04;       // ln 2 / 2048
  constexpr double kC2 = 5.7274462451720406e-08;       // kC1^2 / 2
  constexpr double kC3 = 6.4615286729323654e-12;       // kC1^3 / 6
  const double t = fma(nak, x, kMagic);
  const double n = t - kMagic;
  const double r = fma(nak, x, -n);
  const int ni = __double2loint(t);
  const double T = __ldg(tab + (ni & 2047));
  const int m = ni >> 11;
  const unsigned th = (unsigned)__double2hiint(t);
  const double Ts = __hiloint2double(__double2hiint(T) + (m << 20), __double2loint(T));
  const double q = r * fma(r, fma(r, kC3, kC2), kC1);
  const double v = fma(Ts, q, Ts);
  if (th - 0x4337ffffu <= 1u && m >= -1022 && m <= 1022) return v;  // n fits 32 bits
  const unsigned ta = th & 0x7fffffffu;
  if (ta > 0x7ff00000u || (ta == 0x7ff00000u && __double2loint(t) != 0)) return t;  // NaN
  const bool up = (th & 0x80000000u) == 0u && (th >= 0x43380000u) && !(th == 0x43380000u && m < 0);
  return up ? __longlong_as_double(0x7ff0000000000000ll) : 0.0;
}

}  // namespace qmc
