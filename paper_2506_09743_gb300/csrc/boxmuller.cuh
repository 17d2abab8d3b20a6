// Random numbers of the Metropolis chain: Philox4x32-10 (Salmon, Moraes, Dror,
// Shaw, SC'11) and Box-Muller Gaussians from table-driven logarithms and sines.
#pragma once

#include <cstdint>

#include "fp64_math.cuh"
#include "qmc_internal.cuh"

namespace qmc {

struct u4 { uint32_t x, y, z, w; };

// ---- Box-Muller in FP64 by table-driven argument reduction (in the manner
// of Tang, ACM TOMS 15 (1989) and 16 (1990)): the uniforms are 32-bit
// integers x with u = (x + 1/2) 2^-32, so
//   2 pi u = A + B,  A = 2 pi (x >> 16) 2^-16 (table: sin A, cos A),
//                    B = 2 pi ((x & 0xffff) + 1/2) 2^-32 < 1e-4 (short Taylor series),
//   sin(A + B) = sin A cos B + cos A sin B, cos(A + B) = cos A cos B - sin A sin B;
//   log u = (e - 32) ln 2 + log(1 + j 2^-16) + log1p(r),
//           x + 1/2 = 2^e m, j = the top 16 fraction bits of m,
//           r = (m - (1 + j 2^-16)) / (1 + j 2^-16) < 2^-16 (three Taylor terms),
// with ln 2 split so that (e - 32) ln2_hi is exact; for u within 2^-7 of 1
// the series of log1p(-(1 - u)) instead, which keeps a tiny log u accurate.  About a third of the FP64
// work of the library functions, to within a few ulp of them; the tables
// (2 x 65,536 pairs of doubles, 2 MB, L2-resident) are built on the host in
// extended precision, once per device.
constexpr int kBmBits = 16;
constexpr int kBmN = 1 << kBmBits;

// the tables of the current device (pointers to device memory)
struct BmTables {
  const double2* sincos;  // [j] = sin, cos of 2 pi j 2^-16
  const double2* log;     // [j] = log(1 + j 2^-16), 1 / (1 + j 2^-16)
};

// x + 1/2, exact, with one FP64 instruction: 2^52 + x is a bit pattern, and
// 2^52 - 1/2 is subtracted from it
__device__ __forceinline__ double half_up(uint32_t x) {
  return __hiloint2double(0x43300000, (int)x) - 4503599627370495.5;
}

__device__ __forceinline__ void sincos_2pi_u(const BmTables& tb, uint32_t x, double* s, double* c) {
  const double2 sc = __ldg(tb.sincos + (x >> kBmBits));
  const double sa = sc.x, ca = sc.y;
  const double b = half_up(x & (kBmN - 1)) * (6.283185307179586 * 0x1p-32);
  const double b2 = b * b;
  const double sb = b - b * b2 * (1.0 / 6.0);                  // next term < 1e-18 relative
  const double cb = 1.0 - b2 * 0.5;                             // next term < 5e-18
  *s = sa * cb + ca * sb;
  *c = ca * cb - sa * sb;
}

__device__ __forceinline__ double log_u(const BmTables& tb, uint32_t x) {
  if (x >= 0xFE000000u) {
    // u within 2^-7 of 1: log u = log1p(-w) = -(w + w^2/2 + ... + w^9/9), with
    // w = 1 - u exact (the table form would lose the digits of a tiny log u
    // to the cancellation of e ln2 against the table entry)
    const double w = half_up(0xFFFFFFFFu - x) * 0x1p-32;
    double q = 1.0 / 9.0;
    q = 1.0 / 8.0 + w * q;
    q = 1.0 / 7.0 + w * q;
    q = 1.0 / 6.0 + w * q;
    q = 1.0 / 5.0 + w * q;
    q = 1.0 / 4.0 + w * q;
    q = 1.0 / 3.0 + w * q;
    q = 0.5 + w * q;
    return -(w + w * w * q);
  }
  const double v = half_up(x);
  const unsigned long long bits = (unsigned long long)__double_as_longlong(v);
  const int e = (int)(bits >> 52) - 1023;
  const unsigned j = (unsigned)(bits >> (52 - kBmBits)) & (kBmN - 1);
  const double m = __longlong_as_double((long long)((bits & 0xFFFFFFFFFFFFFull) | 0x3FF0000000000000ull));
  const double mh =
      __longlong_as_double((long long)((bits & (((1ull << kBmBits) - 1) << (52 - kBmBits))) | 0x3FF0000000000000ull));
  const double2 lg = __ldg(tb.log + j);
  const double r = (m - mh) * lg.y;  // m - mh exact
  const double p = r - r * r * (0.5 - r * (1.0 / 3.0));  // next term < 2e-20, |log u| > 2^-7
  // e - 32 in [-33, 0) as a double: one FP64 add on a bit pattern
  const double k = __hiloint2double(0x43300000, e) - 4503599627370528.0;
  const double ln2_hi = 6.93147180369123816490e-01, ln2_lo = 1.90821492927058770002e-10;
  return (k * ln2_hi + lg.x) + (k * ln2_lo + p);
}

// sqrt(-2 log u), to about an ulp
__device__ __forceinline__ double bm_radius(const BmTables& tb, uint32_t x) {
  const double a = -2.0 * log_u(tb, x);
  return a * rsqrt3(a);
}

// four Gaussians from one Philox block: (x0, x1) and (x2, x3) -> z[0..3]
__device__ __forceinline__ void box_muller4(const BmTables& tb, const u4& x, double z[4]) {
  const double r1 = bm_radius(tb, x.x), r2 = bm_radius(tb, x.z);
  double s1, c1, s2, c2;
  sincos_2pi_u(tb, x.y, &s1, &c1);
  sincos_2pi_u(tb, x.w, &s2, &c2);
  z[0] = r1 * c1; z[1] = r1 * s1; z[2] = r2 * c2; z[3] = r2 * s2;
}

__device__ __forceinline__ u4 philox4x32_10(u4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r) { k0 += 0x9E3779B9u; k1 += 0xBB67AE85u; }
    const uint32_t lo0 = 0xD2511F53u * c.x, hi0 = __umulhi(0xD2511F53u, c.x);
    const uint32_t lo1 = 0xCD9E8D57u * c.z, hi1 = __umulhi(0xCD9E8D57u, c.z);
    c = u4{hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0};
  }
  return c;
}

__device__ __forceinline__ double u01(uint32_t x) { return half_up(x) * 0x1p-32; }

}  // namespace qmc
