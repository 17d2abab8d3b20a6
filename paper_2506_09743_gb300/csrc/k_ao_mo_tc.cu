// AO evaluation fused with the AO->MO contraction on the 5th-generation
// tensor cores (tcgen05, sm_103a).  Mixed forms only.
//
// Persistent CTAs walk over tiles of 128 walkers x one electron (MMA M = 128
// rows) with the tables staged once.  The AO columns are packed on the host into
// K-passes of 32 columns (a shell never straddles two passes; unused columns are
// zero).  For each pass the four thread parts of a pair of rows (r and r + 64 of
// the tile) evaluate the pass's shells (dealt to the parts by cost) and write the
// FP32 AO channels into shared memory as the MMA A operand,
// split into TF32 high and low parts
//     a = a_hi + a_lo,  a_hi = rna_tf32(a),  a_lo = rna_tf32(a - a_hi),
// and one thread issues, per channel c (value / kinetic operator) and K step,
//     D_c += A_c,hi B_hi + A_c,hi B_lo + A_c,lo B_hi        (kind::tf32)
// with N = 16 (MOs, padded), K = 8 per instruction, accumulating in FP32 in
// tensor memory (two 16-column accumulators) across all passes.  The
// dropped a_lo b_lo term and the TF32 rounding of the low parts leave an
// error of order 2^-21 relative to |a||b|, i.e. FP32-level accuracy.
// B = MO^T (scaled by the AO angular factors) is prepared on the host in the
// same core-matrix layout, for all passes, and copied into shared memory.
// The A buffer holds one pass (64 KB with the kinetic channel, 32 KB without), so
// two CTAs of 256 threads fit on an SM (three without); a pass's buffer is reused
// once its MMAs have completed (mbarrier).
//
// The kernel is bound by issue slots.  With one row per thread and each part
// splitting the FP64 positions for itself it issued 7,400 instructions per row
// (273 us on 65,536 CO walkers with derivatives, 50 us on 16,384 without).  Two
// rows per thread share table loads, addresses and control; the displacements are
// formed once per tile, one coordinate per part, and shared; primitives are
// 16-byte records; the walk over the tiles takes no division: 4,300 instructions,
// 205 and 32 us.  What is left waits on dependent FMAs, on the tile's barriers and
// on the issue slots (half of them taken).
//
// Shared-memory operand layout (K-major, no swizzle): 8-row x 16-byte core
// matrices; element (row, k) at byte (row / 8) * SBO + (k / 4) * 128 +
// (row % 8) * 16 + (k % 4) * 4, LBO = 128 B (next core matrix along K) and
// SBO = (K extent / 4) * 128 B (next 8-row group).
//
// Every wait on an mbarrier is bounded (WfDev::wait_cycles, about one second
// by default), after which the CTA raises the error flags, waits (bounded
// again) for the MMAs it has issued, writes NaN for its remaining outputs,
// frees its tensor memory and stops instead of hanging; the host reports
// QMC_ERR_TIMEOUT (qmc_check_status, and the calls that synchronise).
#include <algorithm>

#include "ao_eval.cuh"

namespace qmc {

namespace {

constexpr int kRows = 128;
constexpr int kThreads = 256;
constexpr int kPairs = kRows / 2;              // a thread takes rows rp and rp + 64
constexpr int kParts = kThreads / kPairs;      // thread parts of a row pair
constexpr int kNPad = 16;
constexpr int kPass = kTcPass;
constexpr uint32_t kTmemCols = 32;

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// round to TF32 (10 stored mantissa bits), to nearest with ties away from
// zero, on the bit pattern: adding half a TF32 unit to the magnitude and
// clearing the 13 dropped bits (a carry moves into the exponent as it
// should; infinities and NaNs keep their class).  Two integer operations,
// measured slightly faster here than the conversion instruction.
__device__ __forceinline__ uint32_t tf32_rna(float x) { return (__float_as_uint(x) + 0x1000u) & 0xffffe000u; }

// SM100 shared-memory matrix descriptor, no swizzle.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((addr >> 4) & 0x3FFFu);
  d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1 << 46;  // descriptor version for tcgen05
  return d;                // base offset 0, layout type 0 (no swizzle)
}

// Instruction descriptor: D = F32, A = B = TF32, both K-major, N = 16, M = 128.
constexpr uint32_t kIdescTf32 = (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(kNPad >> 3) << 17) |
                                ((uint32_t)(kRows >> 4) << 24);

__device__ __forceinline__ void mma_tf32(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d_tmem),
      "l"(a), "l"(b), "r"(kIdescTf32), "r"(accumulate));
}

// Wait for the mbarrier phase of the given parity for at most `budget` SM
// clock cycles (and 2^24 tries); false if it did not complete in time.  A
// budget of 0 gives up before the first try (the timeout path's test).
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

// budget of the drain after a failed wait: the MMAs a CTA issued must have
// completed before its shared and tensor memory are released (~1 s)
constexpr long long kDrainCycles = 1ll << 31;

// Shell record: two 16-byte loads
struct TcShell {
  int atom, kind, n_prim, first;  // first: its primitives in the table below
  int kn, l, ao_first, n_ao;
};

// int words of the AO power, column and shell-list tables, rounded up so that
// the mbarrier behind them is 16-byte aligned
__host__ __device__ inline int tc_int_words(const WfDev& wf) { return (2 * wf.n_ao + wf.n_shell + 3) & ~3; }

// The roundings below are written out (products with __fmul_rn, fused products
// with fmaf): the energy of an expansion amplifies a change of the last bit of an
// AO by the square of the reference matrix's condition number, so the channels
// must not depend on which products a compiler joins with their sums.
__device__ __forceinline__ float tc_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float tc_mul(float a, float b, float c) { return __fmul_rn(__fmul_rn(a, b), c); }
// x . y
__device__ __forceinline__ float tc_dot(const float* x, float y0, float y1, float y2) {
  return fmaf(x[2], y2, fmaf(x[0], y0, tc_mul(x[1], y1)));
}
// a b + c d
__device__ __forceinline__ float tc_sum2(float a, float b, float c, float d) { return fmaf(c, d, tc_mul(a, b)); }

// radial factor, f'/rho and f'' - f'/rho of a Slater shell
__device__ __forceinline__ void tc_slater(float zeta, float c, int kn, float rho, float irho, float& f, float& g1,
                                          float& f2, bool deriv) {
  float rk = 1.f;
  for (int k = 0; k < kn; ++k) rk = tc_mul(rk, rho);
  f = tc_mul(c, rk, expf(tc_mul(-zeta, rho)));
  if (deriv) {
    const float q = fmaf(float(kn), irho, -zeta);
    g1 = tc_mul(q, f, irho);
    f2 = tc_mul(fmaf(q, q, -tc_mul(float(kn), irho, irho)), f);
  }
}

// Angular monomial x^a y^b z^c, its gradient and its Laplacian
__device__ __forceinline__ void tc_angular(int pw, const float* px, const float* py, const float* pz, float& P,
                                           float* dP, float& lapP, bool deriv) {
  const int a = pw & 15, b = (pw >> 4) & 15, c = (pw >> 8) & 15;
  const float xa = pick(px, a), yb = pick(py, b), zc = pick(pz, c);
  P = tc_mul(xa, yb, zc);
  if (deriv) {
    dP[0] = a ? tc_mul(tc_mul(float(a), pick(px, a - 1)), yb, zc) : 0.f;
    dP[1] = b ? tc_mul(tc_mul(float(b), xa), pick(py, b - 1), zc) : 0.f;
    dP[2] = c ? tc_mul(tc_mul(float(c), xa), yb, pick(pz, c - 1)) : 0.f;
    lapP = 0.f;
    if (a >= 2) lapP = fmaf(tc_mul(float(a * (a - 1)), pick(px, a - 2), yb), zc, lapP);
    if (b >= 2) lapP = fmaf(tc_mul(float(b * (b - 1)), xa, pick(py, b - 2)), zc, lapP);
    if (c >= 2) lapP = fmaf(tc_mul(float(c * (c - 1)), xa, yb), pick(pz, c - 2), lapP);
  }
}

}  // namespace

template <int NCH>
__global__ void __launch_bounds__(kThreads, NCH == 2 ? 2 : 3)
    k_ao_mo_tc(const __grid_constant__ WfDev wf, const double* __restrict__ walkers, int64_t W, int64_t ldw,
               const float* __restrict__ gradJ, double* __restrict__ mo_out, int64_t ldm, int* __restrict__ err_flag,
               int* __restrict__ err_wf) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  const int kp = wf.k_pad;
  constexpr size_t tile_words = (size_t)kRows * kPass;
  uint32_t* A = reinterpret_cast<uint32_t*>(smem_raw);                // [NCH][2][128][kPass]
  uint32_t* B = A + (size_t)NCH * 2 * tile_words;                     // [2][16][kp]
  float4* prim_s = reinterpret_cast<float4*>(B + 2 * kNPad * kp);    // [n_shell][8] alpha, c, 2 alpha, 4 alpha^2
  TcShell* sh_s = reinterpret_cast<TcShell*>(prim_s + wf.n_shell * QMC_MAX_PRIM);  // [n_shell]
  float* disp = reinterpret_cast<float*>(sh_s + wf.n_shell);            // [n_atom][3][128] electron - nucleus
  float2* atom_s = reinterpret_cast<float2*>(disp + wf.n_atom * 3 * kRows);  // [n_atom][3] positions as float pairs
  int* pow_s = reinterpret_cast<int*>(atom_s + ((wf.n_atom * 3 + 1) & ~1));  // [n_ao]
  int* col_s = pow_s + wf.n_ao;                                         // [n_ao]
  int* list_s = col_s + wf.n_ao;                                        // [n_shell]
  uint64_t* mbar = reinterpret_cast<uint64_t*>(pow_s + tc_int_words(wf));
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(mbar + 1);

  const int tid = threadIdx.x, warp = tid >> 5;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(kTmemCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  }
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(mbar)));
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  for (int k = tid; k < 2 * kNPad * kp; k += kThreads)
    B[k] = k < kNPad * kp ? wf.mo_tc_hi[k] : wf.mo_tc_lo[k - kNPad * kp];
  for (int k = tid; k < wf.n_shell * QMC_MAX_PRIM; k += kThreads) {
    const ShellDev& sh = wf.shells[k / QMC_MAX_PRIM];
    const float al = sh.expo_f[k % QMC_MAX_PRIM];
    prim_s[k] = make_float4(al, sh.coef_f[k % QMC_MAX_PRIM], 2.f * al, 4.f * al * al);
    if (k % QMC_MAX_PRIM == 0)
      sh_s[k / QMC_MAX_PRIM] = TcShell{sh.atom, sh.kind, sh.n_prim, k, sh.kn, sh.l, sh.ao_first, sh.n_ao};
  }
  for (int k = tid; k < 3 * wf.n_atom; k += kThreads) {
    float ah, al;
    split_f64(wf.atom_xyz[k / 3][k % 3], ah, al);
    atom_s[k] = make_float2(ah, al);
  }
  for (int k = tid; k < wf.n_ao; k += kThreads) {
    pow_s[k] = wf.ao_pow[k];
    col_s[k] = wf.ao_col[k];
  }
  for (int k = tid; k < wf.n_shell; k += kThreads) list_s[k] = wf.tc_shells[k];
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  const int rp = tid & (kPairs - 1), part = tid / kPairs;
  const uint32_t lbo = 128, sbo_a = (uint32_t)(kPass / 4) * 128, sbo_b = (uint32_t)(kp / 4) * 128;
  const int64_t n_wblk = (W + kRows - 1) / kRows;
  const int64_t n_tiles = n_wblk * wf.n_elec;
  uint32_t commits = 0;  // mbarrier phases completed so far (each pass commits once)
  // persistent CTA: the tables stay in shared memory and the tensor memory
  // stays allocated while the CTA walks over (walker block, electron) tiles
  double nr[2] = {0.0, 0.0};  // coordinate `part` of both rows of the next tile (parts 0 .. 2)
  float ng[2][3];
  // (walker block, electron) of the next tile, advanced without divisions
  const unsigned n_el = (unsigned)wf.n_elec;
  int64_t next_wb = blockIdx.x / n_el;
  unsigned next_i = blockIdx.x % n_el;
  const unsigned step_wb = gridDim.x / n_el, step_i = gridDim.x % n_el;
  auto advance = [&]() {
    next_wb += step_wb;
    next_i += step_i;
    if (next_i >= n_el) {
      next_i -= n_el;
      ++next_wb;
    }
  };
  auto fetch = [&]() {
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      nr[q] = 0.0;
      ng[q][0] = ng[q][1] = ng[q][2] = 0.f;
    }
    const int64_t tw = next_wb * kRows + rp;
    const int ti = (int)next_i;
#pragma unroll
    for (int q = 0; q < 2; ++q)
      if (tw + q * kPairs < W) {  // false past the last tile
        if (part < 3) nr[q] = walkers[(int64_t)(3 * ti + part) * ldw + tw + q * kPairs];
        if (NCH == 2)
#pragma unroll
          for (int d = 0; d < 3; ++d) ng[q][d] = gradJ[(int64_t)(3 * ti + d) * ldm + tw + q * kPairs];
      }
  };
  // displacements of the fetched positions (as `displacement` of ao_eval.cuh)
  auto place = [&]() {
    if (part >= 3) return;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      float xh, xl;
      split_f64(nr[q], xh, xl);
      for (int a = 0; a < wf.n_atom; ++a) {
        const float2 at = atom_s[3 * a + part];
        disp[(3 * a + part) * kRows + rp + q * kPairs] = (xh - at.x) + (xl - at.y);
      }
    }
  };
  fetch();
  place();
  __syncthreads();
  unsigned char* const a_row = reinterpret_cast<unsigned char*>(A) + (rp >> 3) * (kPass / 4) * 128 + (rp & 7) * 16;
  constexpr int kRow2 = (kPairs / 8) * (kPass / 4) * 128;  // from row rp to row rp + 64
  constexpr int kTile = (int)(tile_words * 4);
  for (int64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
    const int i = (int)next_i;
    const int64_t wb = next_wb;
    float gj[2][3];
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int d = 0; d < 3; ++d) gj[q][d] = ng[q][d];
    advance();
    fetch();
    // one, two (k even) or four (k = 0 mod 4) consecutive columns from k of row
    // rp + 64 q: one 4-, 8- or 16-byte store per buffer
    auto at = [&](int ch, int q, int k) { return a_row + ch * 2 * kTile + q * kRow2 + (k >> 2) * 128 + (k & 3) * 4; };
    auto put = [&](int ch, int q, int k, float v) {
      unsigned char* o = at(ch, q, k);
      const uint32_t hi = tf32_rna(v);
      *reinterpret_cast<uint32_t*>(o) = hi;
      *reinterpret_cast<uint32_t*>(o + kTile) = tf32_rna(v - __uint_as_float(hi));
    };
    auto put2 = [&](int ch, int q, int k, float v0, float v1) {
      unsigned char* o = at(ch, q, k);
      const uint32_t h0 = tf32_rna(v0), h1 = tf32_rna(v1);
      *reinterpret_cast<uint2*>(o) = make_uint2(h0, h1);
      *reinterpret_cast<uint2*>(o + kTile) =
          make_uint2(tf32_rna(v0 - __uint_as_float(h0)), tf32_rna(v1 - __uint_as_float(h1)));
    };
    auto put4 = [&](int ch, int q, int k, float v0, float v1, float v2, float v3) {
      unsigned char* o = at(ch, q, k);
      const uint32_t h0 = tf32_rna(v0), h1 = tf32_rna(v1), h2 = tf32_rna(v2), h3 = tf32_rna(v3);
      *reinterpret_cast<uint4*>(o) = make_uint4(h0, h1, h2, h3);
      *reinterpret_cast<uint4*>(o + kTile) =
          make_uint4(tf32_rna(v0 - __uint_as_float(h0)), tf32_rna(v1 - __uint_as_float(h1)),
                     tf32_rna(v2 - __uint_as_float(h2)), tf32_rna(v3 - __uint_as_float(h3)));
    };
    bool ok = true;
    for (int pass = 0; pass < wf.n_pass; ++pass) {
      if (pass > 0) {
        // the previous pass's MMAs must have read the A buffer before it is overwritten
        ok = mbar_wait_bounded(smem_u32(mbar), (commits - 1) & 1, wf.wait_cycles) && ok;
      }
      // unused columns of the pass are zero (disjoint from the shells' columns)
      const unsigned zero_cols = wf.pass_zero[pass];
      for (int k = part; k < kPass; k += kParts)
        if ((zero_cols >> k) & 1u)
#pragma unroll
          for (int q = 0; q < 2 * NCH; ++q) put(q >> 1, q & 1, k, 0.f);
      const int s_begin = wf.part_off[pass][part], s_end = wf.part_off[pass][part + 1];
      int cur_atom = -1, pow_atom = -1;
      float dx[2], dy[2], dz[2], r2[2], G[2];
      float px[2][5], py[2][5], pz[2][5];
      // value channel P f and kinetic channel
      //   (lap + 2 grad J . grad)(P f) = f lap P + P (f2 + 2 (l+1) g1 + 2 g1 gJ.d) + 2 f gJ.grad P
      // (rows past the last walker keep whatever their (zero) positions give:
      // an MMA row depends on its own A row only, and those rows are never stored)
      for (int e = s_begin; e < s_end; ++e) {
        const int ent = list_s[e];
        const TcShell sh = sh_s[ent & 0xff];
        const int c0 = (ent >> 8) & 0xff, type = ent >> 16;
        if (sh.atom != cur_atom) {
          cur_atom = sh.atom;
          const float* dp = disp + cur_atom * 3 * kRows + rp;
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            dx[q] = dp[q * kPairs], dy[q] = dp[kRows + q * kPairs], dz[q] = dp[2 * kRows + q * kPairs];
            r2[q] = dx[q] * dx[q] + dy[q] * dy[q] + dz[q] * dz[q];
            G[q] = tc_dot(gj[q], dx[q], dy[q], dz[q]);
          }
        }
        float f[2], g1[2], f2[2];
        const float4* pr = prim_s + sh.first;
        if (sh.kind == 0) {
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            const float irho = rsqrtf(r2[q]), rho = r2[q] * irho;
            tc_slater(pr[0].x, pr[0].y, sh.kn, rho, irho, f[q], g1[q], f2[q], NCH == 2);
          }
        } else {
#pragma unroll
          for (int q = 0; q < 2; ++q) f[q] = g1[q] = f2[q] = 0.f;
          for (int p = 0; p < sh.n_prim; ++p) {
            const float4 c = pr[p];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
              const float ex = expf(tc_mul(-c.x, r2[q])), t = tc_mul(c.y, ex);
              f[q] = NCH == 2 ? __fadd_rn(f[q], t) : fmaf(c.y, ex, f[q]);
              if (NCH == 2) {
                g1[q] = fmaf(-c.z, t, g1[q]);
                f2[q] = fmaf(fmaf(c.w, r2[q], -c.z), t, f2[q]);
              }
            }
          }
        }
        float RL[2], tf[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          RL[q] = fmaf(2.f * g1[q], G[q], fmaf(float(2 * (sh.l + 1)), g1[q], f2[q]));
          tf[q] = 2.f * f[q];
        }
        if (type == 1) {
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            put(0, q, c0, f[q]);
            if (NCH == 2) put(1, q, c0, RL[q]);
          }
        } else if (type == 2) {  // c0 even
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            put2(0, q, c0, dx[q] * f[q], dy[q] * f[q]);
            put(0, q, c0 + 2, dz[q] * f[q]);
            if (NCH == 2) {
              put2(1, q, c0, tc_sum2(dx[q], RL[q], tf[q], gj[q][0]), tc_sum2(dy[q], RL[q], tf[q], gj[q][1]));
              put(1, q, c0 + 2, tc_sum2(dz[q], RL[q], tf[q], gj[q][2]));
            }
          }
        } else if (type == 3) {  // c0 a multiple of four
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            const float x = dx[q], y = dy[q], z = dz[q];
            const float fx = f[q] * x, fy = f[q] * y, fz = f[q] * z;
            put4(0, q, c0, fx * x, fx * y, fx * z, fy * y);
            put2(0, q, c0 + 4, fy * z, fz * z);
            if (NCH == 2) {
              const float gx = gj[q][0], gy = gj[q][1], gz = gj[q][2], t = tf[q];
              const float Rx = RL[q] * x, Ry = RL[q] * y, Rz = RL[q] * z;
              const float t2 = 2.f * t;
              const float k0 = fmaf(tc_mul(t2, gx), x, fmaf(Rx, x, t)),
                          k1 = tc_sum2(Rx, y, t, fmaf(gx, y, tc_mul(gy, x))),
                          k2 = tc_sum2(Rx, z, t, fmaf(gx, z, tc_mul(gz, x))),
                          k3 = fmaf(tc_mul(t2, gy), y, fmaf(Ry, y, t)),
                          k4 = tc_sum2(Ry, z, t, fmaf(gy, z, tc_mul(gz, y))),
                          k5 = fmaf(tc_mul(t2, gz), z, fmaf(Rz, z, t));
              put4(1, q, c0, k0, k1, k2, k3);
              put2(1, q, c0 + 4, k4, k5);
            }
          }
        } else {
          if (pow_atom != cur_atom) {
            pow_atom = cur_atom;
#pragma unroll
            for (int q = 0; q < 2; ++q) {
              pow_table(dx[q], px[q]);
              pow_table(dy[q], py[q]);
              pow_table(dz[q], pz[q]);
            }
          }
          for (int k = 0; k < sh.n_ao; ++k) {
            const int b = sh.ao_first + k;
            const int col = col_s[b] - pass * kPass;
#pragma unroll
            for (int q = 0; q < 2; ++q) {
              float P, dP[3], lapP;
              tc_angular(pow_s[b], px[q], py[q], pz[q], P, dP, lapP, NCH == 2);
              put(0, q, col, P * f[q]);
              if (NCH == 2)
                put(1, q, col, fmaf(tf[q], tc_dot(gj[q], dP[0], dP[1], dP[2]), tc_sum2(f[q], lapP, P, RL[q])));
            }
          }
        }
      }
      // generic-proxy shared stores -> visible to the tensor core (async proxy);
      // every thread learns whether all the waits of this CTA succeeded
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      ok = __syncthreads_and(ok) != 0;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (!ok) break;
      if (tid == 0) {
        const uint32_t b_hi = smem_u32(B), b_lo = smem_u32(B + kNPad * kp);
        for (int ch = 0; ch < NCH; ++ch) {
          const uint32_t a_hi = smem_u32(A + (size_t)(ch * 2) * tile_words);
          const uint32_t a_lo = smem_u32(A + (size_t)(ch * 2 + 1) * tile_words);
          const uint32_t d = tmem + (uint32_t)(ch * kNPad);
          for (int ks = 0; ks < kPass / 8; ++ks) {
            const uint32_t aoff = (uint32_t)ks * 256;                            // two core matrices along K
            const uint32_t boff = (uint32_t)(pass * (kPass / 4) + 2 * ks) * 128;  // same columns of B
            const uint32_t acc = (pass > 0 || ks > 0) ? 1u : 0u;
            mma_tf32(d, smem_desc(a_hi + aoff, lbo, sbo_a), smem_desc(b_hi + boff, lbo, sbo_b), acc);
            mma_tf32(d, smem_desc(a_hi + aoff, lbo, sbo_a), smem_desc(b_lo + boff, lbo, sbo_b), 1u);
            mma_tf32(d, smem_desc(a_lo + aoff, lbo, sbo_a), smem_desc(b_hi + boff, lbo, sbo_b), 1u);
          }
        }
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                         smem_u32(mbar))
                     : "memory");
      }
      ++commits;
    }
    if (ok) {  // every thread has read this tile's displacements
      place();
      ok = mbar_wait_bounded(smem_u32(mbar), (commits - 1) & 1, wf.wait_cycles);
    }
    ok = __syncthreads_and(ok) != 0;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (!ok) {
      // an MMA did not complete in time: record it (per call and per
      // wavefunction), let the MMAs already issued finish (at most one commit
      // is outstanding: every pass waits for the previous one before it
      // commits), poison this CTA's remaining outputs (this tile and the
      // tiles it would have taken) and stop
      if (tid == 0) {
        atomicExch(err_flag, 1);
        atomicExch(err_wf, 1);
      }
      if (commits > 0) mbar_wait_bounded(smem_u32(mbar), (commits - 1) & 1, kDrainCycles);
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const int ch = tid >> 7, row = tid & (kRows - 1);
      for (int64_t t = tile; t < n_tiles; t += gridDim.x) {
        const int ti = (int)(t % wf.n_elec);
        const int64_t tw = (t / wf.n_elec) * kRows + row;
        if (ch < NCH && tw < W)
          for (int m = 0; m < kNPad; ++m)
            mo_out[((size_t)(ti * NCH + ch) * kNPad + m) * ldm + tw] = __longlong_as_double(0x7ff8000000000000ll);
      }
      break;
    }
    // ---- epilogue: TMEM -> registers -> MO channels in HBM
    // (two warps per quarter of the rows: one channel each, or half the orbitals)
    {
      constexpr int kCols = kNPad * NCH / 2;
      const int quad = warp & 3, ch = NCH == 2 ? warp >> 2 : 0, m0 = NCH == 2 ? 0 : (warp >> 2) * kCols;
      uint32_t v[kCols];
      const uint32_t taddr = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(ch * kNPad + m0);
#pragma unroll
      for (int h = 0; h < kCols; h += 8)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                     : "=r"(v[h]), "=r"(v[h + 1]), "=r"(v[h + 2]), "=r"(v[h + 3]), "=r"(v[h + 4]), "=r"(v[h + 5]),
                       "=r"(v[h + 6]), "=r"(v[h + 7])
                     : "r"(taddr + h));
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
      const int64_t wr = wb * kRows + quad * 32 + (tid & 31);
      if (wr < W) {  // walker-fastest MO layout: a warp stores 32 consecutive walkers per orbital
        double* dst = mo_out + (size_t)((i * NCH + ch) * kNPad + m0) * ldm + wr;
#pragma unroll
        for (int m = 0; m < kCols; ++m) dst[(size_t)m * ldm] = widen(__uint_as_float(v[m]));
      }
    }
    // the next tile's first MMA overwrites the accumulators: the loads above
    // are complete (wait::ld) before the barrier that precedes it
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  }
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols));
}

size_t tc_smem_bytes(const WfDev& wf, int nch) {
  size_t b = (size_t)nch * 2 * kRows * kPass * 4 + 2 * kNPad * (size_t)wf.k_pad * 4;
  b += (sizeof(float4) * QMC_MAX_PRIM + sizeof(TcShell)) * (size_t)wf.n_shell;
  b += (size_t)wf.n_atom * 3 * kRows * 4 + sizeof(float2) * ((wf.n_atom * 3 + 1) & ~1);
  b += 4 * (size_t)tc_int_words(wf) + 16;
  return b;
}

cudaError_t launch_ao_mo_tc(const WfDev& wf, int prec, const double* walkers, int64_t W, int64_t ldw,
                            const Workspace& ws, int nch, int* err_flag, int* err_wf, cudaStream_t st) {
  if (W == 0) return cudaSuccess;
  if (prec != QMC_MIXED_TF32) return cudaErrorInvalidValue;
  // persistent grid: as many CTAs per SM as the kernel is built for and shared
  // memory holds, never more CTAs than tiles
  int dev = 0, n_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
  const int64_t n_tiles = ((W + kRows - 1) / kRows) * wf.n_elec;
  const size_t smem = tc_smem_bytes(wf, nch);
  const int per_sm = std::min(nch == 2 ? 2 : 3, std::max(1, (int)((227 * 1024 + 1024) / (smem + 1024))));
  const dim3 grid((unsigned)std::min<int64_t>(n_tiles, per_sm * (int64_t)std::max(n_sm, 1)));
  const float* gj = static_cast<const float*>(ws.gradJ);
  double* mo = ws.mo;
  if (nch == 2) {
    cudaFuncSetAttribute(k_ao_mo_tc<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    k_ao_mo_tc<2><<<grid, kThreads, smem, st>>>(wf, walkers, W, ldw, gj, mo, ws.ldm, err_flag, err_wf);
  } else {
    cudaFuncSetAttribute(k_ao_mo_tc<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    k_ao_mo_tc<1><<<grid, kThreads, smem, st>>>(wf, walkers, W, ldw, gj, mo, ws.ldm, err_flag, err_wf);
  }
  return cudaGetLastError();
}

}  // namespace qmc
