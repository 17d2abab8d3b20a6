// Shared pieces of the tensor-core FP32X2 AO stage (k_ao_mo_oz.cu, the general
// kernel, and k_ao_mo_oz_pk.cu, two rows per thread): tcgen05 descriptors and
// issue, bounded waits, group barriers, row scales and the epilogue.
#pragma once

#include "ao_eval.cuh"
#include "oz_digits.cuh"

namespace qmc {

namespace {

constexpr int kRows = 128;
constexpr int kThreads = 512;
constexpr int kNPad = 16;
constexpr int kPass = kTcPass;
constexpr uint32_t kTmemCols = 256;              // per group: 2 x 6 x 16 = 192 used
constexpr int kStackBlocks = kOzDigits + 1;       // zero block + digit slices of the B stack
constexpr int kChCols = kOzClasses * kNPad;       // accumulator columns of one channel
constexpr int kTileBytes = kRows * kPass * 2;     // one digit slice of one channel (BF16)

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// SM100 shared-memory matrix descriptor, no swizzle
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((addr >> 4) & 0x3FFFu);
  d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1 << 46;
  return d;
}

// Instruction descriptor: D = F32, A = B = BF16, both K-major, M = 128, N = n
// (a multiple of 16 up to 96 here).
__device__ __forceinline__ uint32_t idesc_bf16(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(kRows >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc,
                                         uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d_tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate));
}

// Barrier of one thread group: the whole CTA for one group, named barrier
// 1 + group (n threads) for two
template <int G>
__device__ __forceinline__ void group_sync(int grp, int n) {
  if (G == 1) {
    __syncthreads();
  } else {
    asm volatile("bar.sync %0, %1;" ::"r"(1 + grp), "r"(n) : "memory");
  }
}

template <int G>
__device__ __forceinline__ bool group_and(int grp, int n, bool v) {
  if (G == 1) return __syncthreads_and(v) != 0;
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.b32 q, %1, 0;\n\t"
      "bar.red.and.pred p, %2, %3, q;\n\t"
      "selp.b32 %0, 1, 0, p;\n\t}\n"
      : "=r"(r)
      : "r"((uint32_t)v), "r"(1 + grp), "r"(n)
      : "memory");
  return r != 0;
}

__device__ __forceinline__ bool mbar_wait_bounded(uint32_t mbar, uint32_t phase, long long budget) {
  const long long t0 = clock64();
  for (int it = 0; it < (1 << 24); ++it) {
    if (clock64() - t0 >= budget) break;
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.b32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok)
        : "r"(mbar), "r"(phase)
        : "memory");
    if (ok) return true;
  }
  return false;
}

constexpr long long kDrainCycles = 1ll << 31;

// byte offset of element (row, k) of a [128][32] BF16 K-major core-matrix
// tile: 8-row x 16-byte core matrices, LBO = 128 B along K, SBO = 512 B
__device__ __forceinline__ uint32_t a_off(int row, int k) {
  return (uint32_t)((row >> 3) * 512 + (k >> 3) * 128 + (row & 7) * 16 + (k & 7) * 2);
}

// power-of-two exponent e of a row scale: bound <= 2^(e - 1), clamped so that
// 2^-e stays a normal float
__device__ __forceinline__ int scale_exponent(uint32_t bound_bits) {
  const int E = (int)((bound_bits >> 23) & 0xffu) - 127;
  return max(-100, min(E + 2, 126));
}

// FP64 value of f * 2^k (f widened exactly, k added to the exponent field)
__device__ __forceinline__ double widen_scaled(float f, int k) {
  const double d = widen(f);
  if (d == 0.0) return d;
  return __longlong_as_double(__double_as_longlong(d) + ((long long)k << 52));
}

// The same for a normal float f when f 2^k is a normal double (always so in
// the epilogue: f is zero or a multiple of 2^-40 below 2^25, |k| < 300): the
// FP64 bit pattern is assembled by integer operations, so the epilogue
// spends one FP64 instruction (the final add) per output instead of five.
__device__ __forceinline__ double widen_scaled_int(float f, int k) {
  const uint32_t u = __float_as_uint(f);
  const uint32_t e32 = (u >> 23) & 0xffu;
  if (e32 == 0u || e32 == 0xffu) return widen_scaled(f, k);  // zero, subnormal, inf, NaN
  const uint32_t hi = (u & 0x80000000u) | ((e32 + 896u + (uint32_t)k) << 20) | ((u >> 3) & 0xfffffu);
  return __hiloint2double((int)hi, (int)(u << 29));
}

// FP32 upper bounds of |AO value| and |kinetic value| over the AOs of a shell
// at distance rho (r2 = rho^2) with |grad J| = gn
__device__ __forceinline__ void shell_bounds(const ShellDev& sh, float r2, float rho, float irho, float gn,
                                             float& bv, float& bk) {
  float rb0 = 0.f, rb1 = 0.f, rb2 = 0.f;
  if (sh.kind == 0) {
    float rk = 1.f;
    for (int k = 0; k < sh.kn; ++k) rk *= rho;
    const float f = fabsf(sh.coef_f[0]) * rk * __expf(-sh.expo_f[0] * rho);
    const float q = (float)sh.kn * irho + sh.expo_f[0];
    rb0 = f;
    rb1 = q * f * irho;
    rb2 = (q * q + (float)sh.kn * irho * irho) * f;
  } else {
    for (int p = 0; p < sh.n_prim; ++p) {
      const float al = sh.expo_f[p];
      const float ce = fabsf(sh.coef_f[p]) * __expf(-al * r2);
      rb0 += ce;
      rb1 += 2.f * al * ce;
      rb2 += (4.f * al * al * r2 + 2.f * al) * ce;
    }
  }
  const int l = sh.l;
  float rl = 1.f, rl1 = 0.f, rl2 = 0.f;  // rho^l, rho^(l-1), rho^(l-2) (0 for negative powers)
  for (int k = 0; k < l; ++k) {
    rl2 = rl1;
    rl1 = rl;
    rl *= rho;
  }
  bv = rb0 * rl;
  bk = rb0 * (float)(l * (l - 1)) * rl2 + rl * (rb2 + (float)(2 * (l + 1)) * rb1 + 2.f * rb1 * gn * rho) +
       2.f * rb0 * gn * (float)l * rl1;
}

// The epilogue of a tile: the six classes of 8 MO columns per thread,
// recombined.  A warp reads the tensor-memory lanes of its rank mod 4 (`quad`);
// the jobs (channel, half of the 16 MO columns) go round the `roles` warps of
// the group that read the same lanes.
template <int NCH>
__device__ __forceinline__ void oz_epilogue(uint32_t tmem, int quad, int role, int roles, const int* rowe,
                                            const int* colf, int i, int64_t wb, int64_t W,
                                            double* __restrict__ mo_out, int nmp, int64_t ldm) {
  for (int job = role; job < 2 * NCH; job += roles) {
    const int ch = job >> 1, half = job & 1;
    uint32_t v[kOzClasses][8];
#pragma unroll
    for (int g = 0; g < kOzClasses; ++g) {
      const uint32_t taddr =
          tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)((ch * kOzClasses + g) * kNPad + half * 8);
      asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                   : "=r"(v[g][0]), "=r"(v[g][1]), "=r"(v[g][2]), "=r"(v[g][3]), "=r"(v[g][4]), "=r"(v[g][5]),
                     "=r"(v[g][6]), "=r"(v[g][7])
                   : "r"(taddr));
    }
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
    const int rr = quad * 32 + (threadIdx.x & 31);
    const int64_t wr = wb * kRows + rr;
    if (wr < W) {
      const int er = rowe[ch * kRows + rr];
      double* dst = mo_out + (size_t)(i * NCH + ch) * nmp * ldm + wr;
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const int m = half * 8 + c;
        if (m < nmp) {
          float acc[kOzClasses];
#pragma unroll
          for (int g = 0; g < kOzClasses; ++g) acc[g] = __uint_as_float(v[g][c]);
          const f32x2 s = oz_combine(acc);
          const int k = er + colf[m] - 16;
          dst[(size_t)m * ldm] = widen_scaled_int(s.hi, k) + widen_scaled_int(s.lo, k);
        }
      }
    }
  }
}

// the MMAs of one pass (issued by one thread): even digits k take the window
// B_0 .. B_{5-k} (stack block 1 on) onto classes k .. 5, odd ones the zero block
// first, onto classes k - 1 .. 5.  k = 0 comes first and writes all six classes
// of the channel.
template <int NCH>
__device__ __forceinline__ void oz_issue_pass(uint32_t a0, uint32_t b0, uint32_t tmem, int kp, int pass,
                                              uint32_t& written, uint32_t mbar) {
  const uint32_t lbo = 128, sbo_a = 512, sbo_b = (uint32_t)(kp / 8) * 128;
  for (int ch = 0; ch < NCH; ++ch)
    for (int ks = 0; ks < kPass / 16; ++ks)
      for (int k = 0; k < kOzDigits; ++k) {
        const uint32_t a = a0 + (uint32_t)(ch * kOzDigits + k) * kTileBytes + (uint32_t)ks * 256;
        const int odd = k & 1;
        const int n = kNPad * (kOzDigits - k + odd);
        const uint32_t b =
            b0 + (uint32_t)(1 - odd) * (kNPad * kp * 2) + (uint32_t)(pass * (kPass / 8) + 2 * ks) * 128;
        const uint32_t d = tmem + (uint32_t)(ch * kChCols + kNPad * (k - odd));
        mma_bf16(d, smem_desc(a, lbo, sbo_a), smem_desc(b, lbo, sbo_b), idesc_bf16(n), (written >> ch) & 1u);
        written |= 1u << ch;
      }
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar) : "memory");
}

// NaN outputs of a group's tiles from `tile` on (a bounded wait gave up)
template <int NCH>
__device__ __forceinline__ void oz_poison(int64_t tile, int64_t tile_step, int64_t n_tiles, int n_elec, int row,
                                          int part, int parts, int64_t W, double* __restrict__ mo_out, int nmp,
                                          int64_t ldm) {
  for (int64_t t = tile; t < n_tiles; t += tile_step) {
    const int ti = (int)(t % n_elec);
    const int64_t tw = (t / n_elec) * kRows + row;
    if (tw < W)
      for (int ch = part; ch < NCH; ch += parts)
        for (int m = 0; m < nmp; ++m)
          mo_out[((size_t)(ti * NCH + ch) * nmp + m) * ldm + tw] = __longlong_as_double(0x7ff8000000000000ll);
  }
}

}  // namespace

}  // namespace qmc
