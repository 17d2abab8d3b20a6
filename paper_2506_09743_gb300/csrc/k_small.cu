// Small-molecule path: local energy and Metropolis chains of one-determinant
// wavefunctions with at most 8 electrons (H2, LiH, Li2 with backflow), one
// lane per electron (small_eval.cuh).  FP64; with PAIRS (FP32X2 form with
// backflow) the orbitals are evaluated in pairs of FP32.
#include "boxmuller.cuh"
#include "small_eval.cuh"

namespace qmc {

using namespace small;

cudaError_t box_muller_tables(BmTables* t);

namespace {

// Warps are the unit of work.  FP64: one-warp blocks spread a small batch over
// all SM partitions evenly, and the tables are read through L1 (their latency
// hides behind the FP64 pipe).  Pairs of FP32: the orbitals are bound by latency
// and issue, so four warps share tables staged in shared memory.
constexpr int kBlock = 32;
constexpr int kBlockPairs = 128;

// the orbital tables: in global memory, or (STAGE) copied to the block's
// dynamic shared memory
size_t table_bytes(const WfDev& wf) {
  return sizeof(ShellDev) * (size_t)wf.n_shell + sizeof(float2) * (size_t)wf.n_ao * wf.n_mo + sizeof(float) * 128;
}

template <bool STAGE>
__device__ __forceinline__ Tables tables(const WfDev& wf) {
  if constexpr (!STAGE) {
    return Tables{wf.shells, wf.mo_x2, wf.exp_tab};
  } else {
    extern __shared__ __align__(16) unsigned char tab_raw[];
    ShellDev* sh = reinterpret_cast<ShellDev*>(tab_raw);
    float2* C = reinterpret_cast<float2*>(sh + wf.n_shell);
    float* ex = reinterpret_cast<float*>(C + (size_t)wf.n_ao * wf.n_mo);
    for (int k = threadIdx.x; k < wf.n_shell * (int)(sizeof(ShellDev) / 4); k += blockDim.x)
      reinterpret_cast<int*>(sh)[k] = reinterpret_cast<const int*>(wf.shells)[k];
    for (int k = threadIdx.x; k < wf.n_ao * wf.n_mo; k += blockDim.x) C[k] = wf.mo_x2[k];
    for (int k = threadIdx.x; k < 128; k += blockDim.x) ex[k] = wf.exp_tab[k];
    __syncthreads();
    return Tables{sh, C, ex};
  }
}

}  // namespace

template <int NE, int NO, bool BF, bool PAIRS>
__global__ void __launch_bounds__(PAIRS ? kBlockPairs : kBlock, PAIRS ? 3 : 1) k_small_energy(const __grid_constant__ WfDev wf,
                                                         const double* __restrict__ walkers, int64_t W, int64_t ldw,
                                                         double* __restrict__ e_loc, double* __restrict__ log_psi) {
  constexpr int MODE = BF ? 2 : 1;
  using U = typename std::conditional<PAIRS, f32x2, double>::type;
  const Tables tb = tables<PAIRS>(wf);
  const Group g = make_group(wf.n_elec, blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), W);
  const int N = g.N, nu = wf.n_up;
  const int s = g.e >= nu ? 1 : 0, n = s ? wf.n_down : nu, i0 = s ? nu : 0, a = g.e - i0;
  double r[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) r[d] = walkers[(int64_t)(3 * g.e + d) * ldw + g.w];

  PairTerms<NE> pt;
  pair_terms<NE, false>(wf, g, r, pt);
  double rt[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) rt[d] = BF ? fma(wf.bf_w, pt.drt[d], r[d]) : r[d];

  // ---- orbitals, this electron's column of the inverse
  Mo<NO, MODE> mo;
  orbitals<U, NO, MODE>(wf, tb, rt, mo);
  double ai[NO];
  const double det = cofactors<NO>(g, mo.phi, a, n, i0, ai);
  const double idet = recip3(det);
#pragma unroll
  for (int m = 0; m < NO; ++m) ai[m] = m < n ? ai[m] * idet : 0.0;

  // ---- m_a and the traced second derivatives
  double ma[3] = {0.0, 0.0, 0.0}, hc[Mo<NO, MODE>::kH];
#pragma unroll
  for (int q = 0; q < Mo<NO, MODE>::kH; ++q) hc[q] = 0.0;
#pragma unroll
  for (int m = 0; m < NO; ++m) {
#pragma unroll
    for (int d = 0; d < 3; ++d) ma[d] = fma(ai[m], mo.d[m][d], ma[d]);
#pragma unroll
    for (int q = 0; q < Mo<NO, MODE>::kH; ++q) hc[q] = fma(ai[m], mo.h[m][q], hc[q]);
  }
  double kin;
  if constexpr (!BF) {
    // no backflow: J1 = I, and the squares of m_a cancel
    kin = pt.lap + hc[0];
#pragma unroll
    for (int d = 0; d < 3; ++d) kin = fma(pt.gj[d], fma(2.0, ma[d], pt.gj[d]), kin);
  } else {
    const double w = wf.bf_w;
    Blocks bl;
    backflow_blocks<NE>(g, pt, w, ma, bl);
    kin = pt.lap;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const double t = pt.gj[d] + bl.dS[d];  // |g + dS|^2 = |g|^2 + 2 g.dS + |dS|^2
      kin = fma(t, t, kin);
      kin = fma(-4.0 * w * bl.j2[d], ma[d], kin);
      kin = fma(bl.N[d], fma(-ma[d], ma[d], hc[d]), kin);
    }
    kin = fma(2.0 * bl.N[3], fma(-ma[0], ma[1], hc[3]), kin);
    kin = fma(2.0 * bl.N[4], fma(-ma[0], ma[2], hc[4]), kin);
    kin = fma(2.0 * bl.N[5], fma(-ma[1], ma[2], hc[5]), kin);
    // same-spin pairs (a, b), b = a + kk cyclic: each unordered pair once
    if constexpr (NO > 1) {
#pragma unroll
      for (int kk = 1; kk <= NO / 2; ++kk) {
        const bool pair = 2 * kk < n || (2 * kk == n && a < kk);
        const int b = a + kk >= n ? a + kk - n : a + kk;
        const int eb = pair ? i0 + b : g.e;
        const int src = g.base + eb;
        // x = M[a][b], y = M[b][a]; M[b][a] needs lane b's derivatives with
        // this lane's column of the inverse
        double x[3] = {0.0, 0.0, 0.0}, y[3] = {0.0, 0.0, 0.0};
#pragma unroll
        for (int m = 0; m < NO; ++m) {
          const double ab = shfl(ai[m], src);
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            x[d] = fma(ab, mo.d[m][d], x[d]);
            y[d] = fma(ai[m], shfl(mo.d[m][d], src), y[d]);
          }
        }
        double Sb[6], Sx[3], Sy[3], gx[3] = {0.0, 0.0, 0.0}, gy[3] = {0.0, 0.0, 0.0}, acc = 0.0;
#pragma unroll
        for (int q = 0; q < 6; ++q) Sb[q] = shfl(bl.S[q], src);
        symv(bl.S, x, Sx);
        symv(Sb, y, Sy);
#pragma unroll
        for (int k = 1; k < NE; ++k)
          if (k < N) {
            const int j = g.next(k);
            PairGeo pb;
            partner_geo<NE>(g, pt, src, eb, j, pb);
            double px[3], py[3];
            project(pt.pg[k - 1], x, px);
            const double ea = w * pt.pg[k - 1].iv;
            const bool at_b = j == eb;
            // j = b: px = P_ab x and P_ab y; otherwise P_bj y
            PairGeo pj;
#pragma unroll
            for (int d = 0; d < 3; ++d) pj.n[d] = dsel(at_b, pt.pg[k - 1].n[d], pb.n[d]);
            project(pj, y, py);
            const double c = ea * (w * pb.iv) * dot3(px, py);
            acc += at_b ? 0.0 : c;
#pragma unroll
            for (int d = 0; d < 3; ++d) {
              gx[d] = dsel(at_b, ea * px[d], gx[d]);
              gy[d] = dsel(at_b, ea * py[d], gy[d]);
            }
          }
        const double c = acc - dot3(Sx, gy) - dot3(gx, Sy);
        if (pair) kin = fma(-2.0, c, kin);
      }
    }
  }
  // ---- E_L = -1/2 kin + V, log|Psi| = J + log|D_up| + log|D_down| + log|d_0|
  double v = fma(-0.5, kin, 0.5 * pt.vee);
  for (int at = 0; at < wf.n_atom; ++at) {
    double x[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) x[d] = r[d] - wf.atom_xyz[at][d];
    v = fma(-wf.atom_z[at], rsqrt3(dot3(x, x)), v);
  }
  const double e = group_sum<NE>(g, v);
  const double lp = group_sum<NE>(g, a == 0 ? fma(0.5, pt.J, log(fabs(det))) : 0.5 * pt.J);
  if (g.first) {
    e_loc[g.w] = e + wf.vnn;
    if (log_psi) log_psi[g.w] = lp + wf.log_w0;
  }
}

// A chain of n_steps Metropolis steps per walker (App. B), kept in registers:
// chains of different walkers never meet, so the whole stretch is one launch
// (before, each step was five kernels and a counter update).  Step t draws the
// numbers of k_propose and k_accept: Philox block j of counter (j, walker,
// step) gives the Gaussians 4j .. 4j + 3, block ceil(3N/4) the acceptance
// uniform.  Box-Muller pair p (Gaussians 2p, 2p + 1) is formed by lane p of
// the walker (pairs beyond the N lanes in a second round) and handed to the
// coordinates by shuffles.  The acceptance test u < |Psi'/Psi|^2 is made on the
// ratio of the determinants and exp(2 (J' - J)), so a step takes no logarithm.
template <int NE, int NO, bool BF, bool PAIRS>
__global__ void __launch_bounds__(PAIRS ? kBlockPairs : kBlock) k_small_chain(const __grid_constant__ WfDev wf, double* __restrict__ walkers,
                                                        int64_t W, int64_t ldw, int n_steps, double step,
                                                        uint64_t seed, uint64_t first_walker, uint64_t step0,
                                                        BmTables bm, double* __restrict__ log_psi,
                                                        int64_t* __restrict__ n_accept) {
  using U = typename std::conditional<PAIRS, f32x2, double>::type;
  const Tables tb = tables<PAIRS>(wf);
  const Group g = make_group(wf.n_elec, blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), W);
  const int N = g.N, nu = wf.n_up;
  const int s = g.e >= nu ? 1 : 0, n = s ? wf.n_down : nu, i0 = s ? nu : 0, a = g.e - i0;
  const int n3 = 3 * N, n_pairs = (n3 + 1) / 2;
  const uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
  const uint32_t wi = (uint32_t)(first_walker + (uint64_t)g.w);
  const double two_over_ln2 = 2.0 * 2954.6394437405970;  // 2 (2048 / ln 2)
  double r[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) r[d] = walkers[(int64_t)(3 * g.e + d) * ldw + g.w];
  double J = 0.0, det = 1.0;
  int taken = 0;
  // t = -1 evaluates the starting positions (the same code as every step, so
  // that a chain cut into several calls is the same chain bit for bit)
  for (int t = -1; t < n_steps; ++t) {
    double q[3] = {r[0], r[1], r[2]};
    double u = 0.0;
    if (t >= 0) {
      const uint64_t gs = step0 + (uint64_t)t;
      const uint32_t c2 = (uint32_t)gs, c3 = (uint32_t)(gs >> 32);
      double z[2][2];
#pragma unroll
      for (int round = 0; round < 2; ++round) {
        const int p = g.e + round * N;
        z[round][0] = z[round][1] = 0.0;
        if (round == 0 || N < n_pairs) {
          const u4 x = philox4x32_10(u4{(uint32_t)(p >> 1), wi, c2, c3}, k0, k1);
          const uint32_t xa = (p & 1) ? x.z : x.x, xb = (p & 1) ? x.w : x.y;
          const double rad = bm_radius(bm, xa);
          double sn, cs;
          sincos_2pi_u(bm, xb, &sn, &cs);
          z[round][0] = rad * cs;
          z[round][1] = rad * sn;
        }
      }
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const int k = 3 * g.e + d, p = k >> 1;
        const bool second = p >= N;
        const int src = g.base + (second ? p - N : p);
        const double z00 = shfl(z[0][0], src), z01 = shfl(z[0][1], src), z10 = shfl(z[1][0], src),
                     z11 = shfl(z[1][1], src);
        const double zk = dsel(second, dsel(k & 1, z11, z10), dsel(k & 1, z01, z00));
        q[d] = fma(step, zk, r[d]);
      }
      const u4 x = philox4x32_10(u4{(uint32_t)((n3 + 3) / 4), wi, c2, c3}, k0, k1);
      u = u01(x.x);
    }
    // J' and the determinants at q
    double Jn = 0.0, drt[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int k = 1; k <= NE / 2; ++k) {
      // partner e + k; with N even the middle distance meets every pair twice
      if (2 * k <= N) {
        const int j = g.next(k), src = g.base + j;
        double v[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) v[d] = q[d] - shfl(q[d], src);
        const double d2 = dot3(v, v), iv = rsqrt3(d2), dist = d2 * iv;
        const double w0 = (j >= nu) == (g.e >= nu) ? wf.w0_par : wf.w0_anti;
        const double term = w0 * dist * recip3(fma(wf.jb, dist, 1.0));
        Jn += 2 * k == N ? 0.5 * term : term;
        if (BF) {
          const int e = g.e - k < 0 ? g.e - k + N : g.e - k;  // the lane whose partner this is
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            const double nd = v[d] * iv;
            const double back = shfl(nd, g.base + e);
            drt[d] += 2 * k == N ? nd : nd - back;
          }
        }
      }
    }
    double rt[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) rt[d] = BF ? fma(wf.bf_w, drt[d], q[d]) : q[d];
    Mo<NO, 0> mo;
    orbitals<U, NO, 0>(wf, tb, rt, mo);
    double cof[NO];
    const double dn = cofactors<NO>(g, mo.phi, a, n, i0, cof);
    Jn = shfl(group_sum<NE>(g, Jn), g.base);
    bool take = t < 0;
    if (t >= 0) {
      const double ratio = dn * recip3(det);
      // the two spins' ratios (an empty spin has no lane and ratio one)
      double f = shfl(ratio, g.base);
      if (nu > 0 && wf.n_down > 0) f *= shfl(ratio, g.base + nu);
      take = u < f * f * exp_scaled(two_over_ln2, Jn - J, wf.exp2_tab);
      taken += take ? 1 : 0;
    }
    if (take) {
#pragma unroll
      for (int d = 0; d < 3; ++d) r[d] = q[d];
      J = Jn;
      det = dn;
    }
  }
  if (g.live) {
#pragma unroll
    for (int d = 0; d < 3; ++d) walkers[(int64_t)(3 * g.e + d) * ldw + g.w] = r[d];
  }
  if (log_psi) {
    const double lp = group_sum<NE>(g, a == 0 ? log(fabs(det)) : 0.0);
    if (g.first) log_psi[g.w] = J + lp + wf.log_w0;
  }
  if (n_accept && g.first && n_steps > 0) n_accept[g.w] += taken;
}

namespace {

int64_t warps_of(const WfDev& wf, int64_t W) {
  const int per = 32 / wf.n_elec;
  return (W + per - 1) / per;
}

}  // namespace

cudaError_t launch_small_energy(const WfDev& wf, const double* walkers, int64_t W, int64_t ldw, double* e_loc,
                                double* log_psi, cudaStream_t st) {
  if (W == 0) return cudaSuccess;
  const unsigned grid = (unsigned)warps_of(wf, W);
  if (wf.bf_w == 0.0) {
    QMC_SMALL_DISPATCH((k_small_energy<NE, NO, false, false><<<grid, kBlock, 0, st>>>(wf, walkers, W, ldw, e_loc, log_psi)));
  } else if (wf.gen_x2) {
    const size_t tb = table_bytes(wf);
    QMC_SMALL_DISPATCH((cudaFuncSetAttribute(k_small_energy<NE, NO, true, true>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tb),
                        k_small_energy<NE, NO, true, true><<<(grid + 3) / 4, kBlockPairs, tb, st>>>(
                            wf, walkers, W, ldw, e_loc, log_psi)));
  } else {
    QMC_SMALL_DISPATCH((k_small_energy<NE, NO, true, false><<<grid, kBlock, 0, st>>>(wf, walkers, W, ldw, e_loc, log_psi)));
  }
  return cudaGetLastError();
}

// Steps per launch: long chains are cut so that a launch stays short next to
// other streams' work; every further launch re-evaluates its starting
// positions (one evaluation in kChainSteps).
constexpr int kChainSteps = 64;

cudaError_t launch_small_chain(const WfDev& wf, double* walkers, int64_t W, int64_t ldw, int32_t n_steps, double step,
                               uint64_t seed, uint64_t first_walker, uint64_t step_offset, double* log_psi,
                               int64_t* n_accept, cudaStream_t st) {
  if (W == 0) return cudaSuccess;
  BmTables bm;
  cudaError_t e = box_muller_tables(&bm);
  if (e != cudaSuccess) return e;
  const unsigned grid = (unsigned)warps_of(wf, W);
  for (int32_t t0 = 0; t0 == 0 || t0 < n_steps; t0 += kChainSteps) {
    const int nt = n_steps - t0 < kChainSteps ? n_steps - t0 : kChainSteps;
    double* lp = t0 + nt >= n_steps ? log_psi : nullptr;
    const uint64_t off = step_offset + (uint64_t)t0;
    if (wf.bf_w == 0.0) {
      QMC_SMALL_DISPATCH((k_small_chain<NE, NO, false, false><<<grid, kBlock, 0, st>>>(
          wf, walkers, W, ldw, nt, step, seed, first_walker, off, bm, lp, n_accept)));
    } else if (wf.gen_x2) {
      const size_t tb = table_bytes(wf);
      QMC_SMALL_DISPATCH((cudaFuncSetAttribute(k_small_chain<NE, NO, true, true>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tb),
                          k_small_chain<NE, NO, true, true><<<(grid + 3) / 4, kBlockPairs, tb, st>>>(
          wf, walkers, W, ldw, nt, step, seed, first_walker, off, bm, lp, n_accept)));
    } else {
      QMC_SMALL_DISPATCH((k_small_chain<NE, NO, true, false><<<grid, kBlock, 0, st>>>(
          wf, walkers, W, ldw, nt, step, seed, first_walker, off, bm, lp, n_accept)));
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace qmc
