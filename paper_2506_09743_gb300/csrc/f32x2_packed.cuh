// Pairs of FP32 (f32x2.cuh) for two independent numbers at once: every word is a
// packed f32x2 register pair, every operation one add / mul / fma.rn.f32x2
// instruction.  Each lane is rounded as its scalar instruction rounds, so the
// functions below give f32x2.cuh's results bit for bit; where they take fewer
// instructions (a product that is exact joined with its sum, a power of two
// folded into a factor, a negated constant), the result is the same number.
// A packed instruction takes the FMA pipe as long as its two scalar ones but one
// issue slot: on kernels bound by issue that is what it saves.
#pragma once

#include "f32x2.cuh"
#include "oz_digits.cuh"

namespace qmc {

struct v2f {
  unsigned long long u;
};

__device__ __forceinline__ v2f v2_make(float a, float b) {
  v2f r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.u) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ v2f v2_all(float a) { return v2_make(a, a); }
__device__ __forceinline__ void v2_get(v2f v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v.u));
}
__device__ __forceinline__ v2f v2_add(v2f a, v2f b) {
  v2f r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.u) : "l"(a.u), "l"(b.u));
  return r;
}
__device__ __forceinline__ v2f v2_fma(v2f a, v2f b, v2f c) {
  v2f r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.u) : "l"(a.u), "l"(b.u), "l"(c.u));
  return r;
}
__device__ __forceinline__ v2f v2_mul(v2f a, v2f b) {
  v2f r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.u) : "l"(a.u), "l"(b.u));
  return r;
}
// a b as an FMA with a -0 that the assembler cannot see through, for a product
// whose only use is a sum: measured, a packed product followed by a packed
// addition comes out as one FMA, without the product's rounding
__device__ __forceinline__ v2f v2_mul_rounded(v2f a, v2f b, v2f neg_zero) { return v2_fma(a, b, neg_zero); }
// a - b (the product with -1 is exact: one rounding)
__device__ __forceinline__ v2f v2_sub(v2f a, v2f b) { return v2_fma(b, v2_all(-1.0f), a); }

// -0 in both lanes, handed to the kernel as a parameter for v2_mul_rounded
constexpr unsigned long long kNegZero2 = 0x8000000080000000ull;
__device__ __forceinline__ v2f v2_neg(v2f a) { return v2f{a.u ^ kNegZero2}; }

struct p2 {
  v2f hi, lo;
};

__device__ __forceinline__ p2 p2_zero() { return p2{v2f{0ull}, v2f{0ull}}; }
__device__ __forceinline__ p2 p2_make(f32x2 a, f32x2 b) { return p2{v2_make(a.hi, b.hi), v2_make(a.lo, b.lo)}; }

__device__ __forceinline__ p2 p2_two_sum(v2f a, v2f b) {
  const v2f s = v2_add(a, b), bb = v2_sub(s, a);
  return p2{s, v2_add(v2_sub(a, v2_sub(s, bb)), v2_sub(b, bb))};
}
__device__ __forceinline__ p2 p2_fast_two_sum(v2f a, v2f b) {
  const v2f s = v2_add(a, b);
  return p2{s, v2_sub(b, v2_sub(s, a))};
}
__device__ __forceinline__ p2 operator-(p2 a) { return p2{v2_neg(a.hi), v2_neg(a.lo)}; }
__device__ __forceinline__ p2 operator+(p2 a, p2 b) {
  const p2 s = p2_two_sum(a.hi, b.hi);
  return p2_fast_two_sum(s.hi, v2_add(s.lo, v2_add(a.lo, b.lo)));
}
__device__ __forceinline__ p2 operator-(p2 a, p2 b) {
  const p2 s = p2_two_sum(a.hi, v2_neg(b.hi));
  return p2_fast_two_sum(s.hi, v2_add(s.lo, v2_sub(a.lo, b.lo)));
}
__device__ __forceinline__ p2 operator*(p2 a, p2 b) {
  const v2f p = v2_mul(a.hi, b.hi), pe = v2_fma(a.hi, b.hi, v2_neg(p));
  return p2_fast_two_sum(p, v2_fma(a.hi, b.lo, v2_fma(a.lo, b.hi, pe)));
}
__device__ __forceinline__ p2 operator*(p2 a, v2f b) {
  const v2f p = v2_mul(a.hi, b), pe = v2_fma(a.hi, b, v2_neg(p));
  return p2_fast_two_sum(p, v2_fma(a.lo, b, pe));
}
// times a power of two (exact on a normalised pair)
__device__ __forceinline__ p2 p2_scale(p2 a, float s) { return p2{v2_mul(a.hi, v2_all(s)), v2_mul(a.lo, v2_all(s))}; }

// mac_x2: acc += a b, with neg_bh = -b.hi (the negated product feeds the FMA of its
// rounding error and, subtracted, the sum), and the normalisation
__device__ __forceinline__ void p2_mac(p2& acc, p2 a, p2 b, v2f neg_bh) {
  const v2f np = v2_mul(a.hi, neg_bh), pe = v2_fma(a.hi, b.hi, np);
  const v2f cross = v2_fma(a.hi, b.lo, v2_fma(a.lo, b.hi, pe));
  const v2f s = v2_sub(acc.hi, np), bb = v2_sub(s, acc.hi);
  const v2f e = v2_sub(v2_sub(acc.hi, v2_sub(s, bb)), v2_add(np, bb));
  acc.hi = s;
  acc.lo = v2_add(acc.lo, v2_add(e, cross));
}
__device__ __forceinline__ p2 p2_normalize(p2 a) { return p2_fast_two_sum(a.hi, a.lo); }

// exp_x2 of both lanes (x <= about 0); tab holds 2^(j/64) as (hi, lo) in shared memory
__device__ __forceinline__ p2 p2_exp(p2 x, const float2* tab, v2f neg_zero) {
  // arguments below -87 give zero: they are replaced here and 2^m at the end
  float x0, x1;
  v2_get(x.hi, x0, x1);
  const bool z0 = x0 < -87.0f, z1 = x1 < -87.0f;
  x.hi = v2_make(z0 ? -87.0f : x0, z1 ? -87.0f : x1);
  const v2f t = v2_add(v2_mul_rounded(x.hi, v2_all(k64ByLn2), neg_zero), v2_all(12582912.0f));
  const v2f nf = v2_sub(t, v2_all(12582912.0f));
  // x.hi - n A: the product is exact for |n| < 2^13
  const v2f r0 = v2_fma(nf, v2_all(-kLn2By64A), x.hi);
  const v2f nb = v2_mul(nf, v2_all(-kLn2By64B)), nbl = v2_fma(nf, v2_all(kLn2By64B), nb);
  const p2 r1 = p2_two_sum(r0, nb);
  const p2 r2 = p2_two_sum(r1.hi, x.lo);
  const p2 r = p2_fast_two_sum(r2.hi, v2_sub(v2_add(r1.lo, r2.lo), v2_fma(nf, v2_all(kLn2By64C), nbl)));
  // r^2 / 2, r^3 (1/6 + r (1/24 + r/120)) with the factors of two folded
  const v2f hr = v2_mul(v2_all(0.5f), r.hi), qh = v2_mul(hr, r.hi);
  const p2 q{qh, v2_fma(r.hi, r.lo, v2_fma(hr, r.hi, v2_neg(qh)))};
  const v2f poly = v2_fma(r.hi, v2_fma(r.hi, v2_all(2.0f * (1.0f / 120.0f)), v2_all(2.0f * (1.0f / 24.0f))), v2_all(2.0f * (1.0f / 6.0f)));
  const v2f tail = v2_mul_rounded(v2_mul(r.hi, qh), poly, neg_zero);
  p2 em1 = r + q;
  em1 = p2_fast_two_sum(em1.hi, v2_add(em1.lo, tail));
  const p2 one_p = p2_fast_two_sum(v2_all(1.0f), em1.hi);
  const p2 er = p2_fast_two_sum(one_p.hi, v2_add(one_p.lo, em1.lo));
  // n from the bits of t, the table entries and 2^m per lane
  float t0, t1;
  v2_get(t, t0, t1);
  const int n0 = (int)(__float_as_uint(t0) - 0x4b400000u), n1 = (int)(__float_as_uint(t1) - 0x4b400000u);
  const float2 e0 = tab[n0 & 63], e1 = tab[n1 & 63];
  const p2 v = er * p2{v2_make(e0.x, e1.x), v2_make(e0.y, e1.y)};
  // 2^m, or zero
  const unsigned u0 = (unsigned)((n0 >> 6) + 127) << 23, u1 = (unsigned)((n1 >> 6) + 127) << 23;
  const v2f sc = v2_make(__uint_as_float(z0 ? 0u : u0), __uint_as_float(z1 ? 0u : u1));
  return p2{v2_mul(v.hi, sc), v2_mul(v.lo, sc)};
}

// The digits of oz_digits, negated: x = v s, s256 = 2^8 s, s24 = 2^24 s with s a
// power of two (s up to 2^100: the scales stay finite)
__device__ __forceinline__ void p2_digits_neg(p2 v, v2f s256, v2f s24, v2f d[kOzDigits]) {
  const v2f magic = v2_all(12582912.0f), k256 = v2_all(256.0f);
  d[0] = v2_sub(magic, v2_fma(v.hi, s256, magic));
  v2f h = v2_fma(v.hi, s256, d[0]);
  d[1] = v2_sub(magic, v2_fma(h, k256, magic));
  h = v2_fma(h, k256, d[1]);
  d[2] = v2_sub(magic, v2_fma(h, k256, magic));
  h = v2_fma(h, k256, d[2]);  // units of 2^-24
  const p2 s = p2_two_sum(h, v2_mul(v.lo, s24));
  d[3] = v2_sub(magic, v2_fma(s.hi, k256, magic));
  v2f r = v2_fma(s.lo, k256, v2_fma(s.hi, k256, d[3]));
  d[4] = v2_sub(magic, v2_fma(r, k256, magic));
  r = v2_fma(r, k256, d[4]);
  d[5] = v2_sub(magic, v2_fma(r, k256, magic));
}

}  // namespace qmc
