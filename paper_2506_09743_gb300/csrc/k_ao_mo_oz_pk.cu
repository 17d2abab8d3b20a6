// The tensor-core FP32X2 AO stage (k_ao_mo_oz.cu) with two rows per thread.
//
// The AO evaluation of k_ao_mo_oz is bound by the issue slots: 72% busy, 70% of
// its instructions FP32 additions, products and FMAs (25,000 per row; 3.39 ms on
// 262,144 CO walkers).  Here a thread takes rows r and r + 64 of the tile of 128
// walkers and evaluates them in packed FP32 instructions (f32x2_packed.cuh), one
// issue slot for both; integer work, table look-ups and stores stay per row.
// Digits, row scales and sums are those of k_ao_mo_oz bit for bit.
//
// Served: Gaussian bases of complete s, p and d shells with bound tables, where
// two groups' digit tiles fit in shared memory (CO's 58 AOs); everything else
// runs k_ao_mo_oz.  Two groups of six warps on alternate tiles, 64 row pairs x 3
// parts of the shell lists each, one CTA of 384 threads (168 registers) per SM.
// The kernel has 36% fewer instructions than k_ao_mo_oz, and what is left waits on
// dependent FMAs and the FMA pipe: 2, 3 and 4 parts, that is as many warps per
// scheduler, issue 38%, 49% and 53% of the time and took 3.59, 3.11 and 3.14 ms
// (k_ao_mo_oz 3.39 ms).  A primitive's constants are kept in shared memory in
// both lanes of a packed word (64 bytes, four broadcast loads).
// The digits are stored negated (their remainders then come from one FMA), and
// so are the MO digits of the B stack: the products are the same.
#include <algorithm>

#include "f32x2_packed.cuh"
#include "oz_tc.cuh"

namespace qmc {

namespace {

constexpr int kPkThreads = 384;
constexpr int kPkParts = 3;                    // thread parts per row pair
constexpr int kPkGroups = 2;
constexpr int kPkGT = kPkThreads / kPkGroups;  // threads of a group
constexpr int kPkPairs = kRows / 2;            // row pairs of a tile

struct PkPrim {  // each constant twice (both lanes)
  float4 al, c, c2a, c4a;  // (hi, hi, lo, lo) of -alpha, c, 2 alpha c, 4 alpha^2 c
};

__device__ __forceinline__ p2 pk_const(const float4& v) {
  return p2{v2_make(v.x, v.y), v2_make(v.z, v.w)};
}

}  // namespace

template <int NCH>
__global__ void __launch_bounds__(kPkThreads, 1)
    k_ao_mo_oz_pk(const __grid_constant__ WfDev wf, unsigned long long neg_zero, int n_prim,
                  const double* __restrict__ walkers, int64_t W, int64_t ldw, const float* __restrict__ gradJ,
                  double* __restrict__ mo_out, int nmp, int64_t ldm, int* __restrict__ err_flag,
                  int* __restrict__ err_wf) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  const int kp = wf.k_pad;
  const int tid = threadIdx.x, warp = tid >> 5;
  const int grp = tid / kPkGT, gtid = tid % kPkGT;
  unsigned char* A = smem_raw + (size_t)grp * NCH * kOzDigits * kTileBytes;     // [NCH][6][128 x 32] BF16
  unsigned char* B = smem_raw + (size_t)kPkGroups * NCH * kOzDigits * kTileBytes;  // [7 x 16][kp] BF16 stack
  PkPrim* prim_s = reinterpret_cast<PkPrim*>(B + (size_t)kStackBlocks * kNPad * kp * 2);  // [n_prim]
  int4* sh_s = reinterpret_cast<int4*>(prim_s + n_prim);                 // [n_shell] atom, l, n_prim, first primitive
  float2* xtab = reinterpret_cast<float2*>(sh_s + wf.n_shell);           // [64]
  int* list_s = reinterpret_cast<int*>(xtab + 64);                       // [n_shell] three-part lists
  int* rowe_buf = list_s + ((wf.n_shell + 3) & ~3) + grp * 4 * kRows;    // [groups][2 tiles][2][128] exponents
  int* colf = list_s + ((wf.n_shell + 3) & ~3) + kPkGroups * 4 * kRows;  // [16]
  uint64_t* mbar_all = reinterpret_cast<uint64_t*>(colf + kNPad);        // [groups]
  uint64_t* mbar = mbar_all + grp;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(mbar_all + kPkGroups);

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(kTmemCols * kPkGroups));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  }
  if (gtid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(mbar)));
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  {  // the stack: one zero block, then the six digit slices of the MO table, negated
    const uint32_t* src = reinterpret_cast<const uint32_t*>(wf.mo_oz);
    uint32_t* dst = reinterpret_cast<uint32_t*>(B);
    const int zero_words = (kStackBlocks - kOzDigits) * kNPad * kp / 2;
    for (int k = tid; k < kStackBlocks * kNPad * kp / 2; k += kPkThreads)
      dst[k] = k < zero_words ? 0u : src[k - zero_words] ^ 0x80008000u;
  }
  if (tid == 0) {
    int first = 0;
    for (int s = 0; s < wf.n_shell; ++s) {
      const ShellDev& sh = wf.shells[s];
      sh_s[s] = make_int4(sh.atom, sh.l, sh.n_prim, first);
      first += sh.n_prim;
    }
  }
  for (int k = tid; k < 64; k += kPkThreads) xtab[k] = make_float2(wf.exp_tab[2 * k], wf.exp_tab[2 * k + 1]);
  for (int k = tid; k < wf.n_shell; k += kPkThreads) list_s[k] = wf.tc_shells[2 * wf.n_shell + k];
  for (int k = tid; k < kNPad; k += kPkThreads) colf[k] = wf.oz_colexp[k];
  __syncthreads();
  for (int k = tid; k < wf.n_shell * QMC_MAX_PRIM; k += kPkThreads) {
    const int s = k / QMC_MAX_PRIM, p = k % QMC_MAX_PRIM;
    const ShellDev& sh = wf.shells[s];
    if (p < sh.n_prim) {
      PkPrim& q = prim_s[sh_s[s].w + p];
      q.al = make_float4(-sh.expo_f[p], -sh.expo_f[p], -sh.expo_lo[p], -sh.expo_lo[p]);
      q.c = make_float4(sh.coef_f[p], sh.coef_f[p], sh.coef_lo[p], sh.coef_lo[p]);
      q.c2a = make_float4(sh.c2a_f[p], sh.c2a_f[p], sh.c2a_lo[p], sh.c2a_lo[p]);
      q.c4a = make_float4(sh.c4a_f[p], sh.c4a_f[p], sh.c4a_lo[p], sh.c4a_lo[p]);
    }
  }
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot + (uint32_t)(grp * kTmemCols);

  const int rp = gtid & (kPkPairs - 1), part = gtid / kPkPairs;  // rows rp and rp + 64
  const int64_t n_wblk = (W + kRows - 1) / kRows;
  const int64_t n_tiles = n_wblk * wf.n_elec;
  uint32_t commits = 0, iter = 0;
  double nr[2][3];
  float ng[2][3];
  // (walker block, electron) of the next tile, advanced without divisions
  const unsigned n_el = (unsigned)wf.n_elec, first = blockIdx.x + grp * gridDim.x;
  int64_t next_wb = first / n_el;
  unsigned next_i = first % n_el;
  const unsigned step_wb = kPkGroups * gridDim.x / n_el, step_i = kPkGroups * gridDim.x % n_el;
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
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        nr[q][d] = 0.0;
        ng[q][d] = 0.f;
      }
    const int64_t tw = next_wb * kRows + rp;  // past W past the last tile
    const int ti = (int)next_i;
#pragma unroll
    for (int q = 0; q < 2; ++q)
      if (tw + q * kPkPairs < W)
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          nr[q][d] = walkers[(int64_t)(3 * ti + d) * ldw + tw + q * kPkPairs];
          if (NCH == 2) ng[q][d] = gradJ[(int64_t)(3 * ti + d) * ldm + tw + q * kPkPairs];
        }
  };
  const int64_t tile_step = (int64_t)kPkGroups * gridDim.x;
  fetch();
  for (int64_t tile = blockIdx.x + (int64_t)grp * gridDim.x; tile < n_tiles; tile += tile_step, ++iter) {
    int* rowe = rowe_buf + (iter & 1u) * 2 * kRows;
    const int i = (int)next_i;
    const int64_t wb = next_wb;
    double r[2][3];
    float gq[2][3];
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        r[q][d] = nr[q][d];
        gq[q][d] = ng[q][d];
      }
    // ---- 1. row scales (as in k_ao_mo_oz, per row)
    float sc[2][2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const float gn = NCH == 2 ? sqrtf(gq[q][0] * gq[q][0] + gq[q][1] * gq[q][1] + gq[q][2] * gq[q][2]) : 0.f;
      float bv = 0.f, bk = 0.f;
      bool direct = false;
      for (int a = 0; a < wf.n_atom; ++a) {
        float dx, dy, dz;
        displacement(r[q][0], r[q][1], r[q][2], wf.atom_xyz[a], dx, dy, dz);
        const float r2 = dx * dx + dy * dy + dz * dz;
        const int idx = oz_bound_bin(r2);
        if (idx == 0) {
          direct = true;
          continue;
        }
        const float4 t = __ldg(wf.oz_bound + (size_t)a * kOzBoundBins + idx);
        bv = fmaxf(bv, t.x);
        bk = fmaxf(bk, fmaf(gn, t.z, t.y));
      }
      if (direct) {  // within 2^-12 bohr of a nucleus: bound every shell
        int cur_atom = -1;
        float r2 = 0.f, rho = 0.f, irho = 0.f;
        for (int s = 0; s < wf.n_shell; ++s) {
          const ShellDev& sh = wf.shells[s];
          if (sh.atom != cur_atom) {
            cur_atom = sh.atom;
            float dx, dy, dz;
            displacement(r[q][0], r[q][1], r[q][2], wf.atom_xyz[cur_atom], dx, dy, dz);
            r2 = dx * dx + dy * dy + dz * dz;
            irho = rsqrtf(r2);
            rho = r2 * irho;
          }
          float sv, sk;
          shell_bounds(sh, r2, rho, irho, gn, sv, sk);
          bv = fmaxf(bv, sv);
          bk = fmaxf(bk, sk);
        }
      }
      const int e0 = scale_exponent(__float_as_uint(bv)), e1 = scale_exponent(__float_as_uint(bk));
      if (part == 0) {
        rowe[rp + q * kPkPairs] = e0;
        rowe[kRows + rp + q * kPkPairs] = e1;
      }
      sc[0][q] = __uint_as_float((unsigned)(127 - e0) << 23);
      sc[1][q] = __uint_as_float((unsigned)(127 - e1) << 23);
    }
    // 2^8 s and 2^24 s of both channels
    v2f s256[2], s24[2];
#pragma unroll
    for (int ch = 0; ch < NCH; ++ch) {
      s256[ch] = v2_make(sc[ch][0] * 256.0f, sc[ch][1] * 256.0f);
      s24[ch] = v2_make(sc[ch][0] * 16777216.0f, sc[ch][1] * 16777216.0f);
    }
    const v2f gjx = v2_make(gq[0][0], gq[1][0]), gjy = v2_make(gq[0][1], gq[1][1]), gjz = v2_make(gq[0][2], gq[1][2]);

    // digits of one column or of two (k even: complete p and d shells start at
    // even columns) of a channel in both rows (row rp + 64 is 8 core-matrix
    // groups further)
    constexpr uint32_t kRow2 = (kPkPairs / 8) * 512;
    auto words = [](const v2f& a, uint32_t& w0, uint32_t& w1) {
      w0 = (uint32_t)a.u;
      w1 = (uint32_t)(a.u >> 32);
    };
    auto put1 = [&](int ch, int k, p2 v) {
      v2f d[kOzDigits];
      p2_digits_neg(v, s256[ch], s24[ch], d);
      unsigned char* base = A + (size_t)ch * kOzDigits * kTileBytes + a_off(rp, k);
#pragma unroll
      for (int j = 0; j < kOzDigits; ++j) {
        uint32_t w0, w1;
        words(d[j], w0, w1);
        *reinterpret_cast<uint16_t*>(base + (size_t)j * kTileBytes) = (uint16_t)(w0 >> 16);
        *reinterpret_cast<uint16_t*>(base + (size_t)j * kTileBytes + kRow2) = (uint16_t)(w1 >> 16);
      }
    };
    auto put2 = [&](int ch, int k, p2 v0, p2 v1) {
      v2f d0[kOzDigits], d1[kOzDigits];
      p2_digits_neg(v0, s256[ch], s24[ch], d0);
      p2_digits_neg(v1, s256[ch], s24[ch], d1);
      unsigned char* base = A + (size_t)ch * kOzDigits * kTileBytes + a_off(rp, k);
#pragma unroll
      for (int j = 0; j < kOzDigits; ++j) {
        uint32_t a0, a1, b0, b1;
        words(d0[j], a0, a1);
        words(d1[j], b0, b1);
        *reinterpret_cast<uint32_t*>(base + (size_t)j * kTileBytes) = __byte_perm(a0, b0, 0x7632);
        *reinterpret_cast<uint32_t*>(base + (size_t)j * kTileBytes + kRow2) = __byte_perm(a1, b1, 0x7632);
      }
    };

    // ---- 2. passes
    bool ok = true;
    uint32_t written = 0u;
    for (int pass = 0; pass < wf.n_pass; ++pass) {
      if (pass > 0) ok = mbar_wait_bounded(smem_u32(mbar), (commits - 1) & 1, wf.wait_cycles) && ok;
      const unsigned zero_cols = wf.pass_zero[pass];
      for (int k = part; k < kPass; k += kPkParts)
        if ((zero_cols >> k) & 1u)
#pragma unroll
          for (int q = 0; q < NCH * kOzDigits; ++q) {
            *reinterpret_cast<uint16_t*>(A + (size_t)q * kTileBytes + a_off(rp, k)) = 0;
            *reinterpret_cast<uint16_t*>(A + (size_t)q * kTileBytes + a_off(rp, k) + kRow2) = 0;
          }
      int cur_atom = -1;
      p2 dx = p2_zero(), dy = p2_zero(), dz = p2_zero(), r2 = p2_zero(), G = p2_zero();
      const int q1 = wf.part3_off[pass][part + 1];
      for (int q = wf.part3_off[pass][part]; q < q1; ++q) {
        const int ent = list_s[q];
        const int4 sh = sh_s[ent & 0xff];
        const int c0 = (ent >> 8) & 0xff, l = sh.y;
        if (sh.x != cur_atom) {
          cur_atom = sh.x;
          dx = p2_make(diff_x2(r[0][0], wf.atom_xyz[cur_atom][0]), diff_x2(r[1][0], wf.atom_xyz[cur_atom][0]));
          dy = p2_make(diff_x2(r[0][1], wf.atom_xyz[cur_atom][1]), diff_x2(r[1][1], wf.atom_xyz[cur_atom][1]));
          dz = p2_make(diff_x2(r[0][2], wf.atom_xyz[cur_atom][2]), diff_x2(r[1][2], wf.atom_xyz[cur_atom][2]));
          r2 = dx * dx + dy * dy + dz * dz;
          if (NCH == 2) G = dx * gjx + dy * gjy + dz * gjz;
        }
        p2 f = p2_zero(), t1 = p2_zero(), t2 = p2_zero();
        const PkPrim* pr = prim_s + sh.w;
        for (int p = 0; p < sh.z; ++p) {
          const p2 e = p2_exp(pk_const(pr[p].al) * r2, xtab, v2f{neg_zero});
          const v2f neg_eh = v2_neg(e.hi);
          p2_mac(f, pk_const(pr[p].c), e, neg_eh);
          if (NCH == 2) {
            p2_mac(t1, pk_const(pr[p].c2a), e, neg_eh);
            p2_mac(t2, pk_const(pr[p].c4a), e, neg_eh);
          }
        }
        f = p2_normalize(f);
        p2 RL = p2_zero(), tf = p2_zero();
        if (NCH == 2) {
          t1 = p2_normalize(t1);
          t2 = p2_normalize(t2);
          const p2 g1 = -t1, f2 = r2 * t2 - t1;
          // 2 (l + 1) g1: a power of two for s and p
          const p2 lg = l == 2 ? g1 * v2_all(6.0f) : p2_scale(g1, (float)(2 * (l + 1)));
          RL = f2 + lg + p2_scale(g1 * G, 2.0f);
          tf = p2_scale(f, 2.0f);
        }
        if (l == 0) {
          put1(0, c0, f);
          if (NCH == 2) put1(1, c0, RL);
        } else if (l == 1) {
          put2(0, c0, dx * f, dy * f);
          if (NCH == 2) put2(1, c0, dx * RL + tf * gjx, dy * RL + tf * gjy);
          put1(0, c0 + 2, dz * f);
          if (NCH == 2) put1(1, c0 + 2, dz * RL + tf * gjz);
        } else {
          const p2 fx = f * dx, fy = f * dy, fz = f * dz;
          put2(0, c0, fx * dx, fx * dy);
          put2(0, c0 + 2, fx * dz, fy * dy);
          put2(0, c0 + 4, fy * dz, fz * dz);
          if (NCH == 2) {
            const p2 Rx = RL * dx, Ry = RL * dy, Rz = RL * dz;
            const p2 tx = tf * gjx, ty = tf * gjy, tz = tf * gjz;
            const p2 k0 = tf + (Rx + p2_scale(tx, 2.0f)) * dx, k1 = Rx * dy + tx * dy + ty * dx;
            put2(1, c0, k0, k1);
            const p2 k2 = Rx * dz + tx * dz + tz * dx, k3 = tf + (Ry + p2_scale(ty, 2.0f)) * dy;
            put2(1, c0 + 2, k2, k3);
            const p2 k4 = Ry * dz + ty * dz + tz * dy, k5 = tf + (Rz + p2_scale(tz, 2.0f)) * dz;
            put2(1, c0 + 4, k4, k5);
          }
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      ok = group_and<2>(grp, kPkGT, ok);
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (!ok) break;
      if (gtid == 0)
        oz_issue_pass<NCH>(smem_u32(A), smem_u32(B), tmem, kp, pass, written, smem_u32(mbar));
      ++commits;
    }
    if (ok) ok = mbar_wait_bounded(smem_u32(mbar), (commits - 1) & 1, wf.wait_cycles);
    ok = group_and<2>(grp, kPkGT, ok);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (!ok) {  // as in k_ao_mo_oz: record, drain, poison this group's remaining outputs, stop
      if (gtid == 0) {
        atomicExch(err_flag, 1);
        atomicExch(err_wf, 1);
      }
      if (commits > 0) mbar_wait_bounded(smem_u32(mbar), (commits - 1) & 1, kDrainCycles);
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      oz_poison<NCH>(tile, tile_step, n_tiles, wf.n_elec, rp, part, kPkParts, W, mo_out, nmp, ldm);
      oz_poison<NCH>(tile, tile_step, n_tiles, wf.n_elec, rp + kPkPairs, part, kPkParts, W, mo_out, nmp, ldm);
      break;
    }
    advance();
    fetch();
    // ---- 3. epilogue
    // (six warps: two quarters of the rows have two warps, two have one)
    const int lw = warp % (kPkGT / 32);
    oz_epilogue<NCH>(tmem, warp & 3, lw >> 2, (lw & 3) < 2 ? 2 : 1, rowe, colf, i, wb, W, mo_out, nmp, ldm);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  }
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(*tmem_slot),
                 "r"(kTmemCols * kPkGroups));
}

namespace {

size_t oz_pk_smem_bytes(const WfDev& wf, int nch, int n_prim) {
  size_t b = (size_t)kPkGroups * nch * kOzDigits * kTileBytes + (size_t)kStackBlocks * kNPad * wf.k_pad * 2;
  b += sizeof(PkPrim) * (size_t)n_prim + sizeof(int4) * (size_t)wf.n_shell + sizeof(float2) * 64;
  b += sizeof(int) * (((wf.n_shell + 3) & ~3) + kPkGroups * 4 * kRows + kNPad) + 8 * kPkGroups + 8;
  return b;
}

}  // namespace

bool oz_pk_supported(const WfDev& wf, int nch) {
  return wf.oz_pk_prims > 0 && wf.oz_bound != nullptr && oz_pk_smem_bytes(wf, nch, wf.oz_pk_prims) <= 227 * 1024;
}

cudaError_t launch_ao_mo_oz_pk(const WfDev& wf, const double* walkers, int64_t W, int64_t ldw, const Workspace& ws,
                               int nch, int* err_flag, int* err_wf, cudaStream_t st) {
  int dev = 0, n_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
  const int64_t n_tiles = ((W + kRows - 1) / kRows) * wf.n_elec;
  const unsigned grid = (unsigned)std::min<int64_t>(n_tiles, std::max(n_sm, 1));
  const size_t smem = oz_pk_smem_bytes(wf, nch, wf.oz_pk_prims);
  const float* gj = static_cast<const float*>(ws.gradJ);
  if (nch == 2) {
    cudaFuncSetAttribute(k_ao_mo_oz_pk<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    k_ao_mo_oz_pk<2><<<grid, kPkThreads, smem, st>>>(wf, kNegZero2, wf.oz_pk_prims, walkers, W, ldw, gj, ws.mo,
                                                     ws.nmp, ws.ldm, err_flag, err_wf);
  } else {
    cudaFuncSetAttribute(k_ao_mo_oz_pk<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    k_ao_mo_oz_pk<1><<<grid, kPkThreads, smem, st>>>(wf, kNegZero2, wf.oz_pk_prims, walkers, W, ldw, gj, ws.mo,
                                                     ws.nmp, ws.ldm, err_flag, err_wf);
  }
  return cudaGetLastError();
}

}  // namespace qmc
