// Parameter gradient of log|Psi| and nuclear forces of one-determinant
// wavefunctions (Eqs. nabla_loss, force), one lane per electron
// (small_eval.cuh), in one pass with the local energy.
//
// Forces.  At fixed walkers E_L depends on a nucleus through the orbital
// channels phi, d phi, H phi at r~ and through the potential, so the kernel
// forms the adjoints of the kinetic sum K = sum_k d_k^2 Psi/Psi with respect to
// the channels once, and contracts them with one derivative more of each
// nucleus's AOs (before, three forward tangents per nucleus went through the
// whole energy: 2.9 ms on 10,000 Li2 walkers).  With the notation of
// small_eval.cuh, g_a = grad_a J, s_a = g_a + dS_a, L(x)_a = x_a + sum_j G_aj (x_a - x_j):
//   adjoint of M[a][a]:  B_aa = 2 L(s)_a - 2 N_a m_a - 4 w sum_j n_aj / r_aj^2   (2 g_a without backflow)
//   adjoint of M[a][b]:  B_ab = -2 C_ab M[b][a]                     (same spin, a != b)
//   adjoint of Hc_a:     N_a                                        (I without backflow)
// and through M_d[a][b] = sum_m d_d phi_m(a) (A^-1)_{m b}, Hc_a = sum_m (A^-1)_{m a} H phi_m(a),
//   bar d phi_m(a) = sum_b B_ab (A^-1)_{m b},      bar H phi_m(a) = N_a (A^-1)_{m a},
//   bar (A^-1)_{m b} = sum_a B_ab . d phi_m(a) + N_b : H phi_m(b),
//   bar phi_m(a) = - sum_{m' b} bar (A^-1)_{m' b} (A^-1)_{m' a} (A^-1)_{m b}.
// The Hessian adjoint is N_a times the weight u = sum_m C_m (A^-1)_{m a} of each
// AO, so an AO takes five sums over the orbitals, not eleven, and its radial
// products are gathered per nucleus before they are expanded.
//
// Sums.  Every value v (parameter derivative, force term) of a lane goes to
// shared memory, and lane k of the warp then sums value k over the lanes in
// order, plain and weighted with E_L - E_c, E_c the warp's first energy.  Per
// warp sum v and sum (E_L - E_c) v are stored with E_c, and k_small_reduce
// forms sum (E_L - c) v = A + (E_c - c) B for any centre c without
// cancellation.  All orders are fixed: results are bitwise reproducible.
#include <algorithm>

#include "small_eval.cuh"

namespace qmc {

using namespace small;

namespace {

constexpr int kRow = 33;         // doubles per value in shared memory (32 lanes, odd stride)
constexpr int kRedWarps = 16;    // warps' sums per block of the first reduction

// third radial derivative factor t = q'/rho (q = (f'' - f'/rho)/rho^2)
__device__ __forceinline__ double radial_third(const WfDev& wf, const ShellDev& sh, int s, const Geo<double>& g,
                                               double f, double q) {
  if (sh.kind == 0) {
    const double z = sh.expo[0], kn = (double)sh.kn;
    const double kr = kn * g.ir2;          // -h'
    const double h = fma(kn, g.irho, -z);
    // F''' = (h^3 + 3 h h' + h'') F, h' = -kn/rho^2, h'' = 2 kn/rho^3
    const double f3 = f * fma(h, fma(h, h, -3.0 * kr), 2.0 * kr * g.irho);
    return g.ir2 * fma(f3, g.irho, -3.0 * q);
  }
  const double* nak = wf.nak + (size_t)s * QMC_MAX_PRIM;
  double t = 0.0;
  for (int p = 0; p < sh.n_prim; ++p) {
    const double a2 = 2.0 * sh.expo[p];
    t = fma(-(a2 * a2 * a2) * sh.coef[p], exp_scaled(nak[p], g.r2, wf.exp2_tab), t);
  }
  return t;
}

__device__ __forceinline__ double tr_sym(const double (&S)[6]) { return S[0] + S[1] + S[2]; }

}  // namespace

// Values per lane: [0, n_prim) exponents, then n_ao x NO MO coefficients
// (canonical AO rows), CI weight, Jastrow b, backflow w, and per nucleus
// d E_L / d R (3) and d ln rho / d R (3).
__host__ __device__ inline int small_n_val(int n_prim, int n_ao, int no, int n_atom) {
  return n_prim + n_ao * no + 3 + 6 * n_atom;
}

template <int NE, int NO, bool BF>
__global__ void __launch_bounds__(32) k_small_grad(const __grid_constant__ WfDev wf,
                                                   const double* __restrict__ walkers, int64_t W, int64_t ldw,
                                                   const int* __restrict__ prim_start, int n_prim,
                                                   double* __restrict__ e_loc, double* __restrict__ sums) {
  extern __shared__ double val[];  // [n_val][kRow]
  const Group g = make_group(wf.n_elec, blockIdx.x, W);
  const int lane = threadIdx.x;
  const int N = g.N, nu = wf.n_up;
  const int s = g.e >= nu ? 1 : 0, n = s ? wf.n_down : nu, i0 = s ? nu : 0, a = g.e - i0;
  const int off_c = n_prim, off_m = off_c + wf.n_ao * NO, off_f = off_m + 3;
  const int n_val = off_f + 6 * wf.n_atom;
  auto put = [&](int k, double v) { val[(size_t)k * kRow + lane] = v; };
  double r[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) r[d] = walkers[(int64_t)(3 * g.e + d) * ldw + g.w];
  PairTerms<NE> pt;
  pair_terms<NE, true>(wf, g, r, pt);
  double rt[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) rt[d] = BF ? fma(wf.bf_w, pt.drt[d], r[d]) : r[d];
  Mo<NO, 2> mo;
  const Tables tb{wf.shells, wf.mo_x2, wf.exp_tab};
  orbitals<double, NO, 2>(wf, tb, rt, mo);
  double ai[NO];
  const double det = cofactors<NO>(g, mo.phi, a, n, i0, ai);
  const double idet = recip3(det);
#pragma unroll
  for (int m = 0; m < NO; ++m) ai[m] = m < n ? ai[m] * idet : 0.0;
  double ma[3] = {0.0, 0.0, 0.0}, hc[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
#pragma unroll
  for (int m = 0; m < NO; ++m) {
#pragma unroll
    for (int d = 0; d < 3; ++d) ma[d] = fma(ai[m], mo.d[m][d], ma[d]);
#pragma unroll
    for (int q = 0; q < 6; ++q) hc[q] = fma(ai[m], mo.h[m][q], hc[q]);
  }
  put(off_m, g.e == 0 ? 1.0 / wf.det_w[0] : 0.0);
  put(off_m + 1, -0.5 * pt.gb);
  put(off_m + 2, dot3(ma, pt.drt));

  // ---- the kinetic sum and its adjoints: Bd[k] belongs to M[a][a + k]
  double kin = pt.lap, Nn[6], Bd[NO][3];
#pragma unroll
  for (int k = 0; k < NO; ++k)
#pragma unroll
    for (int d = 0; d < 3; ++d) Bd[k][d] = 0.0;
  if constexpr (!BF) {
#pragma unroll
    for (int q = 0; q < 6; ++q) Nn[q] = q < 3 ? 1.0 : 0.0;
    kin += tr_sym(hc);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      kin = fma(pt.gj[d], fma(2.0, ma[d], pt.gj[d]), kin);
      Bd[0][d] = 2.0 * pt.gj[d];
    }
  } else {
    const double w = wf.bf_w;
    Blocks bl;
    backflow_blocks<NE>(g, pt, w, ma, bl);
    double sv[3], Nm[3];
    symv(bl.N, ma, Nm);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      sv[d] = pt.gj[d] + bl.dS[d];
      kin = fma(sv[d], sv[d], kin);
      const double j2 = -4.0 * w * bl.j2[d];
      kin = fma(ma[d], j2 - Nm[d], kin);
      Bd[0][d] = fma(2.0, sv[d] - Nm[d], j2);
      kin = fma(bl.N[d], hc[d], kin);
    }
#pragma unroll
    for (int q = 3; q < 6; ++q) kin = fma(2.0 * bl.N[q], hc[q], kin);
#pragma unroll
    for (int q = 0; q < 6; ++q) Nn[q] = bl.N[q];
    // the G part of 2 L(s)
#pragma unroll
    for (int k = 1; k < NE; ++k)
      if (k < N) {
        const int src = g.base + g.next(k);
        double x[3], y[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) x[d] = sv[d] - shfl(sv[d], src);
        project(pt.pg[k - 1], x, y);
        const double e2 = 2.0 * w * pt.pg[k - 1].iv;
#pragma unroll
        for (int d = 0; d < 3; ++d) Bd[0][d] = fma(e2, y[d], Bd[0][d]);
      }
    // off-diagonal adjoints, every ordered same-spin pair (a, b = a + kk)
#pragma unroll
    for (int kk = 1; kk < NO; ++kk) {
      const bool pair = kk < n;
      const int b = a + kk >= n ? a + kk - n : a + kk;
      const int eb = pair ? i0 + b : g.e;
      const int src = g.base + eb;
      double x[3] = {0.0, 0.0, 0.0}, y[3] = {0.0, 0.0, 0.0};  // M[a][b], M[b][a]
#pragma unroll
      for (int m = 0; m < NO; ++m) {
        const double ab = shfl(ai[m], src);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          x[d] = fma(ab, mo.d[m][d], x[d]);
          y[d] = fma(ai[m], shfl(mo.d[m][d], src), y[d]);
        }
      }
      double Sb[6], Sy[3], Sg[3], gy[3] = {0.0, 0.0, 0.0}, gS[3] = {0.0, 0.0, 0.0}, v[3] = {0.0, 0.0, 0.0};
#pragma unroll
      for (int q = 0; q < 6; ++q) Sb[q] = shfl(bl.S[q], src);
      symv(Sb, y, Sy);
#pragma unroll
      for (int k = 1; k < NE; ++k)
        if (k < N) {
          const int j = g.next(k);
          PairGeo pb;
          partner_geo<NE>(g, pt, src, eb, j, pb);
          const bool at_b = j == eb;
          const double ea = w * pt.pg[k - 1].iv;
          // j = b: G_ab y and G_ab (I + S_b) y; otherwise G_aj G_jb y
          PairGeo pj;
#pragma unroll
          for (int d = 0; d < 3; ++d) pj.n[d] = dsel(at_b, pt.pg[k - 1].n[d], pb.n[d]);
          double t[3], in[3], out[3];
          project(pj, y, t);
          const double eb_j = w * pb.iv;
#pragma unroll
          for (int d = 0; d < 3; ++d) in[d] = dsel(at_b, Sy[d], eb_j * t[d]);
          project(pt.pg[k - 1], in, out);
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            const double o = ea * out[d];
            gy[d] = dsel(at_b, ea * t[d], gy[d]);
            gS[d] = dsel(at_b, o, gS[d]);
            v[d] += at_b ? 0.0 : o;
          }
        }
      symv(bl.S, gy, Sg);
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const double c = v[d] - Sg[d] - gS[d];  // (C_ab y)_d
        if (pair) {
          kin = fma(-x[d], c, kin);
          Bd[kk][d] = -2.0 * c;
        }
      }
    }
  }
  // ---- energy
  double ev = fma(-0.5, kin, 0.5 * pt.vee);
  for (int at = 0; at < wf.n_atom; ++at) {
    double x[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) x[d] = r[d] - wf.atom_xyz[at][d];
    ev = fma(-wf.atom_z[at], rsqrt3(dot3(x, x)), ev);
  }
  const double el = shfl(group_sum<NE>(g, ev), g.base) + wf.vnn;
  if (g.first) e_loc[g.w] = el;
  const double e_c = shfl(el, 0), de = el - e_c;

  // ---- adjoints of the channels (of the kinetic sum)
  double bphi[NO], bd[NO][3], binv[NO];  // bar phi, bar d phi, bar (A^-1)_{. a}
#pragma unroll
  for (int m = 0; m < NO; ++m) {
    bphi[m] = 0.0;
    double t = 0.0;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      bd[m][d] = Bd[0][d] * ai[m];
      t = fma(Bd[0][d], mo.d[m][d], t);
      t = fma(Nn[d], mo.h[m][d], t);
    }
    if (BF)
#pragma unroll
      for (int q = 3; q < 6; ++q) t = fma(2.0 * Nn[q], mo.h[m][q], t);
    binv[m] = t;
  }
  if constexpr (BF && NO > 1) {
#pragma unroll
    for (int kk = 1; kk < NO; ++kk) {
      const int b = a + kk >= n ? a + kk - n : a + kk, c = a - kk < 0 ? a - kk + n : a - kk;
      const bool pair = kk < n;
      const int src_b = g.base + (pair ? i0 + b : g.e), src_c = g.base + (pair ? i0 + c : g.e);
      // electron c = a - kk holds B_ca in its slot kk
      double Bc[3];
#pragma unroll
      for (int d = 0; d < 3; ++d) Bc[d] = shfl(Bd[kk][d], src_c);
#pragma unroll
      for (int m = 0; m < NO; ++m) {
        const double ab = shfl(ai[m], src_b);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          bd[m][d] = fma(Bd[kk][d], ab, bd[m][d]);
          binv[m] = fma(Bc[d], shfl(mo.d[m][d], src_c), binv[m]);
        }
      }
    }
  }
#pragma unroll
  for (int kk = 0; kk < NO; ++kk) {
    const int b = a + kk >= n ? a + kk - n : a + kk;
    const bool pair = kk < n;
    const int src = g.base + (pair ? i0 + b : g.e);
    double t = 0.0, ab[NO];
#pragma unroll
    for (int m = 0; m < NO; ++m) {
      ab[m] = shfl(ai[m], src);
      t = fma(ai[m], shfl(binv[m], src), t);
    }
    t = pair ? -t : 0.0;
#pragma unroll
    for (int m = 0; m < NO; ++m) bphi[m] = fma(t, ab[m], bphi[m]);
  }

  // ---- per run of a nucleus's shells: parameter values, weights, force
  for (int k = 0; k < 6 * wf.n_atom; ++k) put(off_f + k, 0.0);
  Geo<double> gg;
  const double trN = tr_sym(Nn);
  for (int sh0 = 0; sh0 < wf.n_shell;) {
    const int atom = wf.shells[sh0].atom;
    geometry<2>(rt, wf.atom_xyz[atom], wf.any_sto != 0, gg);
    // gathered radial products (names: radial factor, weight)
    double sg0 = 0.0, squ = 0.0, stu = 0.0, sgu = 0.0, sqw = 0.0;
    double g1w[3] = {0.0, 0.0, 0.0}, qw[3] = {0.0, 0.0, 0.0};
    double f0[3] = {0.0, 0.0, 0.0}, g0[3] = {0.0, 0.0, 0.0}, fu[3] = {0.0, 0.0, 0.0}, gu[3] = {0.0, 0.0, 0.0},
           qu[3] = {0.0, 0.0, 0.0}, gW[3][3] = {{0.0, 0.0, 0.0}, {0.0, 0.0, 0.0}, {0.0, 0.0, 0.0}}, tu = 0.0;
    for (; sh0 < wf.n_shell; ++sh0) {
      const ShellDev& sh = wf.shells[sh0];
      if (sh.atom != atom) break;
      double f, g1, f2, q;
      radial<2>(wf, tb, sh, sh0, gg, f, g1, f2, q);
      const double t3 = radial_third(wf, sh, sh0, gg, f, q);
      const int row = sh.ao_first, mask = sh.l == 0 ? 1 : sh.p_mask, p0 = prim_start[row];
      double uu[3] = {0.0, 0.0, 0.0};
#pragma unroll
      for (int e = 0; e < 3; ++e)
        if ((mask >> e) & 1) {
          const int k = e == 0 ? 0 : __popc(mask & ((1 << e) - 1));  // its AO within the shell
          double w0 = 0.0, w1[3] = {0.0, 0.0, 0.0}, u = 0.0;
          const double pf = sh.l == 0 ? f : gg.v[e] * f;
#pragma unroll
          for (int m = 0; m < NO; ++m) {
            const double c = mo_coef(wf, tb, row + k, m, 0.0);
            u = fma(c, ai[m], u);
            w0 = fma(c, bphi[m], w0);
#pragma unroll
            for (int d = 0; d < 3; ++d) w1[d] = fma(c, bd[m][d], w1[d]);
            put(off_c + (row + k) * NO + m, pf * ai[m]);
          }
          uu[e] = u;
          if (sh.kind == 0) {
            const double nq = (double)(sh.kn + sh.l + 1) + 0.5;
            put(p0 + k, u * pf * (nq * recip3(sh.expo[0]) - gg.rho));
          }
          if (sh.l == 0) {
            sg0 = fma(g1, w0, sg0);
            squ = fma(q, u, squ);
            stu = fma(t3, u, stu);
            sgu = fma(g1, u, sgu);
#pragma unroll
            for (int d = 0; d < 3; ++d) {
              g1w[d] = fma(g1, w1[d], g1w[d]);
              qw[d] = fma(q, w1[d], qw[d]);
            }
          } else {
            f0[e] = fma(f, w0, f0[e]);
            g0[e] = fma(g1, w0, g0[e]);
            fu[e] = fma(f, u, fu[e]);
            gu[e] = fma(g1, u, gu[e]);
            qu[e] = fma(q, u, qu[e]);
            tu = fma(t3 * u, gg.v[e], tu);
            double z = 0.0;
#pragma unroll
            for (int d = 0; d < 3; ++d) {
              gW[e][d] = fma(g1, w1[d], gW[e][d]);
              z = fma(w1[d], gg.v[d], z);
            }
            sqw = fma(q * gg.v[e], z, sqw);
          }
        }
      if (sh.kind == 1) {  // exponents: d(N_p e^(-alpha r^2))/d alpha = term ((3/4 + l/2)/alpha - r^2)
        const double* nak = wf.nak + (size_t)sh0 * QMC_MAX_PRIM;
        for (int p = 0; p < sh.n_prim; ++p) {
          const double term = sh.coef[p] * exp_scaled(nak[p], gg.r2, wf.exp2_tab) *
                              ((0.75 + 0.5 * sh.l) * recip3(sh.expo[p]) - gg.r2);
#pragma unroll
          for (int e = 0; e < 3; ++e)
            if ((mask >> e) & 1)
              put(p0 + __popc(mask & ((1 << e) - 1)) * sh.n_prim + p, uu[e] * (sh.l == 0 ? term : gg.v[e] * term));
        }
      }
    }
    // expansion: first derivatives with bar phi, second with bar d phi, third
    // with N u; the orbitals move with r~ - R, so a nucleus takes minus each
    double Nv[3], Ngu[3];
    symv(Nn, gg.v, Nv);
    symv(Nn, gu, Ngu);
    const double vNv = dot3(gg.v, Nv), quv = dot3(qu, gg.v), quN = dot3(qu, Nv);
    double along = sg0 + dot3(g0, gg.v);                   // times v_c
    along += dot3(qw, gg.v);                               // s, second
    along += gW[0][0] + gW[1][1] + gW[2][2] + sqw;         // p, second
    along = fma(squ + quv, trN, along);                    // third, trace
    along = fma(stu + tu, vNv, along);
    along = fma(2.0, quN, along);
    const double alongN = 2.0 * (squ + quv);               // times (N v)_c
    const double lr = sgu + dot3(gu, gg.v);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      double k1 = f0[c] + g1w[c];
      k1 = fma(along, gg.v[c], k1);
      k1 = fma(alongN, Nv[c], k1);
      k1 = fma(2.0, Ngu[c], k1);
      k1 = fma(gu[c], trN, k1);
      k1 = fma(qu[c], vNv, k1);
#pragma unroll
      for (int d = 0; d < 3; ++d) k1 = fma(gW[c][d] + gW[d][c], gg.v[d], k1);
      // dE/dR = -1/2 (-k1) + dV/dR; ln rho = 2 log|Psi|
      val[(size_t)(off_f + 6 * atom + c) * kRow + lane] += 0.5 * k1;
      val[(size_t)(off_f + 6 * atom + 3 + c) * kRow + lane] -= 2.0 * fma(lr, gg.v[c], fu[c]);
    }
  }
  // the potential's part: -Z / |r - R| and, once per walker, V_nn
  for (int at = 0; at < wf.n_atom; ++at) {
    double x[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) x[d] = r[d] - wf.atom_xyz[at][d];
    const double iv = rsqrt3(dot3(x, x)), c3 = wf.atom_z[at] * iv * iv * iv;
    double vn[3] = {0.0, 0.0, 0.0};
    if (g.e == 0)
      for (int b = 0; b < wf.n_atom; ++b) {
        if (b == at) continue;
        double y[3];
        for (int d = 0; d < 3; ++d) y[d] = wf.atom_xyz[at][d] - wf.atom_xyz[b][d];
        const double ib = rsqrt3(dot3(y, y)), zz = -wf.atom_z[at] * wf.atom_z[b] * ib * ib * ib;
        for (int d = 0; d < 3; ++d) vn[d] = fma(zz, y[d], vn[d]);
      }
#pragma unroll
    for (int d = 0; d < 3; ++d)
      val[(size_t)(off_f + 6 * at + d) * kRow + lane] += fma(-c3, x[d], vn[d]);
  }
  // ---- sums over the warp's lanes (those of walkers that exist), in lane order
  __syncwarp();
  const int per = 32 / N;
  const int64_t left = W - (int64_t)blockIdx.x * per;
  const int used = (int)(left < per ? left : per) * N;
  double* out = sums + (size_t)blockIdx.x * (2 * n_val + 1);
  for (int k0 = 0; k0 < n_val; k0 += 32) {
    const int k = k0 + lane;
    double A = 0.0, B = 0.0;
    const double* v = val + (size_t)(k < n_val ? k : 0) * kRow;
#pragma unroll 4
    for (int l = 0; l < used; ++l) {
      const double x = v[l];
      B += x;
      A = fma(x, shfl(de, l), A);
    }
    if (k < n_val) {
      out[k] = A;
      out[n_val + k] = B;
    }
  }
  if (lane == 0) out[2 * n_val] = e_c;
}

// First reduction: value k over the warps of a chunk, in order; rows
// [chunk][2][n_val]: sum (E_L - c) v and sum v, with c = stats[0] (centred) or 0
__global__ void __launch_bounds__(128) k_small_reduce(const double* __restrict__ sums, int64_t n_warps, int n_val,
                                                      const double* __restrict__ stats, bool centred,
                                                      double* __restrict__ part) {
  const int k = blockIdx.x * 128 + threadIdx.x;
  if (k >= n_val) return;
  const double c = centred ? stats[0] : 0.0;
  const int64_t w0 = (int64_t)blockIdx.y * kRedWarps;
  const int64_t w1 = w0 + kRedWarps < n_warps ? w0 + kRedWarps : n_warps;
  const size_t stride = 2 * (size_t)n_val + 1;
  double A = 0.0, B = 0.0;
#pragma unroll 4
  for (int64_t w = w0; w < w1; ++w) {
    const double* p = sums + (size_t)w * stride;
    const double b = p[n_val + k];
    B += b;
    A += fma(p[2 * n_val] - c, b, p[k]);
  }
  part[((size_t)blockIdx.y * 2) * n_val + k] = A;
  part[((size_t)blockIdx.y * 2 + 1) * n_val + k] = B;
}

// Second reduction and assembly.  One warp per output: its lanes take every
// 32nd chunk in order, then a fixed shuffle tree.  Outputs [0, n_param) are
// parameters, then 3 n_atom force components.  mode 0: gradient 2 A / M and
// forces -(sum dE + A') / M; mode 1: raw sums (sum v, sum E v of the parameters,
// and the three force sums) in the layout of qmc_energy_grad_sums.
__global__ void __launch_bounds__(128) k_small_assemble(WfDev wf, const double* __restrict__ part, int64_t n_chunks,
                                                        int n_val, int n_prim, int no, int n_param, double M, int mode,
                                                        double* __restrict__ grad, double* __restrict__ forces) {
  const int o = (blockIdx.x * 128 + threadIdx.x) / 32, lane = threadIdx.x & 31;
  const int nf = 3 * wf.n_atom;
  if (o >= n_param + nf) return;
  int va = -1, vb = -1;  // value indices: the parameter's, or d ln rho / dR and dE / dR
  double fac = 1.0;
  const int off_c = n_prim, off_m = off_c + wf.n_ao * no;
  if (o < n_param) {
    const int q = o - n_prim;
    if (q < 0) {
      va = wf.prim_val[o];
    } else if (q < wf.n_ao * wf.n_mo) {
      const int b = q / wf.n_mo, m = q % wf.n_mo;
      if (m < no) va = off_c + wf.ao_row[b] * no + m;
      fac = wf.ao_ang[b];
    } else {
      va = off_m + (q - wf.n_ao * wf.n_mo);
    }
  } else {
    const int c = o - n_param;
    vb = off_m + 3 + 6 * (c / 3) + c % 3;
    va = vb + 3;
  }
  double A = 0.0, B = 0.0, E = 0.0;
  if (va >= 0)
    for (int64_t c = lane; c < n_chunks; c += 32) {
      A += part[(size_t)c * 2 * n_val + va];
      B += part[((size_t)c * 2 + 1) * n_val + va];
      if (vb >= 0) E += part[((size_t)c * 2 + 1) * n_val + vb];
    }
#pragma unroll
  for (int s = 16; s >= 1; s >>= 1) {
    A += __shfl_xor_sync(0xffffffffu, A, s);
    B += __shfl_xor_sync(0xffffffffu, B, s);
    E += __shfl_xor_sync(0xffffffffu, E, s);
  }
  if (lane != 0) return;
  if (o < n_param) {
    if (!grad) return;
    if (mode == 0) {
      grad[o] = 2.0 * fac * A / M;
    } else {
      grad[o] = fac * B;
      grad[n_param + o] = fac * A;
    }
  } else if (forces) {
    const int c = o - n_param;
    if (mode == 0) {
      forces[c] = -(E + A) / M;
    } else {
      forces[c] = E;
      forces[nf + c] = B;
      forces[2 * nf + c] = A;
    }
  }
}

// ----------------------------------------------------------------------------

namespace {

int small_no(const WfDev& wf) {
  const int ns = wf.n_up > wf.n_down ? wf.n_up : wf.n_down;
  const int by_n = wf.n_elec <= 2 ? 1 : wf.n_elec <= 4 ? 2 : wf.n_elec <= 6 ? 3 : 4;
  return ns > by_n ? ns : by_n;
}

int64_t small_warps(const WfDev& wf, int64_t W) {
  const int per = 32 / wf.n_elec;
  return (W + per - 1) / per;
}

size_t small_smem(const WfDev& wf, int n_prim) {
  return sizeof(double) * kRow * (size_t)small_n_val(n_prim, wf.n_ao, small_no(wf), wf.n_atom);
}

}  // namespace

bool small_grad_supported(const WfDev& wf, int n_prim) { return wf.small && small_smem(wf, n_prim) <= 227 * 1024; }

size_t small_grad_scratch_bytes(const WfDev& wf, int64_t W, int n_prim) {
  const int64_t nw = small_warps(wf, W), nc = (nw + kRedWarps - 1) / kRedWarps;
  const size_t nv = small_n_val(n_prim, wf.n_ao, small_no(wf), wf.n_atom);
  return sizeof(double) * ((size_t)nw * (2 * nv + 1) + (size_t)nc * 2 * nv);
}

cudaError_t launch_small_grad(const WfDev& wf, const double* walkers, int64_t W, int64_t ldw, const int* prim_start,
                              int n_prim, double* e_loc, double* scratch, cudaStream_t st) {
  const unsigned grid = (unsigned)small_warps(wf, W);
  const size_t smem = small_smem(wf, n_prim);
#define QMC_SMALL_GRAD(BF)                                                                                        \
  QMC_SMALL_DISPATCH((cudaFuncSetAttribute(k_small_grad<NE, NO, BF>, cudaFuncAttributeMaxDynamicSharedMemorySize, \
                                           (int)smem),                                                            \
                      k_small_grad<NE, NO, BF><<<grid, 32, smem, st>>>(wf, walkers, W, ldw, prim_start, n_prim,   \
                                                                       e_loc, scratch)))
  if (wf.bf_w != 0.0) QMC_SMALL_GRAD(true) else QMC_SMALL_GRAD(false)
#undef QMC_SMALL_GRAD
  return cudaGetLastError();
}

cudaError_t launch_small_assemble(const WfDev& wf, int64_t W, int n_prim, int n_param, const double* stats, int mode,
                                  double* scratch, double* grad, double* forces, cudaStream_t st) {
  const int no = small_no(wf), nv = small_n_val(n_prim, wf.n_ao, no, wf.n_atom);
  const int64_t nw = small_warps(wf, W), nc = (nw + kRedWarps - 1) / kRedWarps;
  double* part = scratch + (size_t)nw * (2 * (size_t)nv + 1);
  k_small_reduce<<<dim3((unsigned)((nv + 127) / 128), (unsigned)nc), 128, 0, st>>>(scratch, nw, nv, stats, mode == 0,
                                                                                  part);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const int outs = n_param + 3 * wf.n_atom;
  k_small_assemble<<<(outs + 3) / 4, 128, 0, st>>>(wf, part, nc, nv, n_prim, no, n_param, (double)W, mode, grad,
                                                   forces);
  return cudaGetLastError();
}

}  // namespace qmc
