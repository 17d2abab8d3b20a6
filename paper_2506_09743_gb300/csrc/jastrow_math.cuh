// Compensated sums and pair distances of the Jastrow and Coulomb terms.
#pragma once

#include "ao_eval.cuh"
#include "qmc_internal.cuh"

namespace qmc {

// compensated FP32 accumulator
struct KahanF {
  float s = 0.f, c = 0.f;
  __device__ __forceinline__ void add(float x) {
    const float y = x - c;
    const float t = s + y;
    c = (t - s) - y;
    s = t;
  }
  // add(a b) with the product unrounded
  __device__ __forceinline__ void add_product(float a, float b) {
    const float y = __fmaf_rn(a, b, -c);
    const float t = s + y;
    c = (t - s) - y;
    s = t;
  }
  __device__ __forceinline__ double value() const { return (double)s - (double)c; }
};

// r_i - r_j (d) of two positions held as float pairs, as a pair
// (the low words' difference is formed exactly too: near a nucleus, where
// |a - b| is far below |a|, rounding it would cost 2^-48 |a| absolute, a
// relative error of 2^-48 |a| / |a - b| in 1 / |a - b|)
__device__ __forceinline__ f32x2 pair_diff_x2(float ah, float al, float bh, float bl) {
  const f32x2 s = two_sum(ah, -bh);
  const f32x2 t = two_sum(al, -bl);
  const f32x2 u = two_sum(s.hi, t.hi);
  return fast_two_sum(u.hi, x2_add_rn(u.lo, x2_add_rn(s.lo, t.lo)));
}
// 1 / |v| of a difference vector given as pairs
__device__ __forceinline__ f32x2 inv_dist_x2(f32x2 x, f32x2 y, f32x2 z) { return rsqrt_x2(x * x + y * y + z * z); }

}  // namespace qmc
