// Device code of the small-molecule path: one determinant, at most 8
// electrons (4 per spin), s and p shells, with or without backflow.
// One lane per electron, 32 / N walkers per warp.
//
// What bounds these kernels is the FP64 pipe: a warp-wide FP64 instruction
// occupies an SM partition's pipe for 64 cycles whatever its active lanes, and a
// dependent one can follow after the same 64 cycles (both measured), so one
// warp per partition keeps the pipe busy and the run time is the FP64
// instructions per lane times the warps per partition.  The decomposition
// therefore (a) spreads a walker's electrons over lanes, so that a batch of
// 10,000 walkers reaches every partition (one thread per walker left half of
// them idle), (b) exchanges pair data and matrix rows by shuffles, which cost
// no FP64 issue, and (c) keeps the FP64 instruction count of each lane low:
// table-driven exponentials, reciprocals and square roots from FP32 seeds with
// one cubic step, radial sums contracted with the MO coefficients before they
// are expanded into derivative channels, and the backflow Laplacian through
// the projector form of its Jacobian blocks (below).
//
// Backflow algebra.  With n_ij = (r_i - r_j) / r_ij and eta = w / r, the
// Jacobian blocks of g(v) = w v / |v| are
//   d g_d / d v_e = G = eta (I - n n^T),   sum_e d^2 g_d / d v_e^2 = -2 w n_d / r^2.
// J1_a(k) = d r~_a / d x_k is I + S_a (own coordinates, S_a = sum_j G_aj) or
// -G_ak, so that, over all 3N coordinates k,
//   N_a  = sum_k J1_a J1_a^T = (I + S_a)^2 + sum_j G_aj^2,  G_aj^2 = eta (G_aj),
//   C_ab = sum_k J1_a J1_b^T = -(I + S_a) G_ab - G_ab (I + S_b) + sum_{j != a,b} G_aj G_jb,
//   sum_k J2_a(k) = -4 w sum_j n_aj / r_aj^2,
//   sum_a J1_a(k)^T m_a = m_k + sum_j G_kj (m_k - m_j)            (per electron k).
// Per spin, M_d[a][b] = sum_m d_d phi_m(r~_a) (A^-1)_{m b}, m_a = M[a][a] and
// Hc_a = sum_m (A^-1)_{m a} Hess phi_m(r~_a), and Eqs. nabla_d, nabla_sigma,
// delta_sigma summed over the coordinates give
//   sum_k d_k^2 Sigma/Sigma = sum_a [ N_a : (Hc_a - m_a m_a^T) + J2_a . m_a + dS_a . dS_a ]
//                             - 2 sum_{a < b, same spin} M[a][b]^T C_ab M[b][a],
//   dS_a = m_a + sum_j G_aj (m_a - m_j),
// to which the Jastrow adds lap J + sum_a (|g_a|^2 + 2 g_a . dS_a) (App. F).
#pragma once

#include <type_traits>

#include "ao_eval.cuh"
#include "fp64_math.cuh"
#include "qmc_internal.cuh"

namespace qmc {

namespace small {

constexpr unsigned kAll = 0xffffffffu;

__device__ __forceinline__ double shfl(double v, int src) { return __shfl_sync(kAll, v, src); }

// ---- lane geometry: N lanes per walker, 32 / N walkers per warp.  Lanes past
// the last whole group repeat its first lanes (their results are not stored).
struct Group {
  int N, e, base;    // electrons, this lane's electron, first lane of the group
  int64_t w;         // walker
  bool live, first;  // stores results; stores the walker's scalars
  __device__ __forceinline__ int next(int k) const {  // electron e + k (cyclic)
    const int q = e + k;
    return q >= N ? q - N : q;
  }
};

__device__ __forceinline__ Group make_group(int N, int64_t warp, int64_t W) {
  Group g;
  const int lane = threadIdx.x & 31, per = 32 / N;
  int slot = lane / N;
  const bool extra = slot >= per;
  if (extra) slot = per - 1;
  g.N = N;
  g.base = slot * N;
  g.e = extra ? lane - per * N : lane - g.base;
  const int64_t w = warp * per + slot;
  g.live = !extra && w < W;
  g.first = g.live && g.e == 0;
  g.w = w < W ? w : W - 1;
  return g;
}

// sum over the lanes of a group, valid on its first lane (electron order)
template <int NE>
__device__ __forceinline__ double group_sum(const Group& g, double v) {
  double s = v;
#pragma unroll
  for (int k = 1; k < NE; ++k)
    if (k < g.N) s += shfl(v, g.base + g.next(k));
  return s;
}

// ---- pair terms

struct PairGeo {
  double n[3], iv;  // unit vector from the partner, 1 / r
};

// P (x) = x - n (n . x)
__device__ __forceinline__ void project(const PairGeo& p, const double (&x)[3], double (&y)[3]) {
  const double c = fma(p.n[2], x[2], fma(p.n[1], x[1], p.n[0] * x[0]));
#pragma unroll
  for (int d = 0; d < 3; ++d) y[d] = fma(-c, p.n[d], x[d]);
}

__device__ __forceinline__ double dot3(const double (&x)[3], const double (&y)[3]) {
  return fma(x[2], y[2], fma(x[1], y[1], x[0] * y[0]));
}

// symmetric 3x3 (xx yy zz xy xz yz) times vector
__device__ __forceinline__ void symv(const double (&S)[6], const double (&x)[3], double (&y)[3]) {
  y[0] = fma(S[4], x[2], fma(S[3], x[1], S[0] * x[0]));
  y[1] = fma(S[5], x[2], fma(S[3], x[0], S[1] * x[1]));
  y[2] = fma(S[5], x[1], fma(S[4], x[0], S[2] * x[2]));
}

// Jastrow and Coulomb terms of one electron with every other (full sums over
// partners: a pair counts in both its electrons' J, vee and dJ/db), and the
// pair geometry.
template <int NE>
struct PairTerms {
  PairGeo pg[NE > 1 ? NE - 1 : 1];  // slot k - 1: partner e + k (cyclic)
  double J, lap, vee, gb;           // J, lap_e J, sum 1/r, -dJ/db
  double gj[3], drt[3];             // grad_e J, sum_j n_ej
};

template <int NE, bool DB>
__device__ __forceinline__ void pair_terms(const WfDev& wf, const Group& g, const double (&r)[3], PairTerms<NE>& t) {
  const int N = g.N, nu = wf.n_up;
  t.J = t.lap = t.vee = t.gb = 0.0;
#pragma unroll
  for (int d = 0; d < 3; ++d) t.gj[d] = t.drt[d] = 0.0;
#pragma unroll
  for (int k = 1; k < NE; ++k)
    if (k < N) {
      const int j = g.next(k), src = g.base + j;
      double v[3];
#pragma unroll
      for (int d = 0; d < 3; ++d) v[d] = r[d] - shfl(r[d], src);
      const double d2 = dot3(v, v), iv = rsqrt3(d2), dist = d2 * iv;
      const double w0 = (j >= nu) == (g.e >= nu) ? wf.w0_par : wf.w0_anti;
      const double rd = recip3(fma(wf.jb, dist, 1.0)), u = w0 * rd, u1 = u * rd;
      t.J = fma(u, dist, t.J);
      t.vee += iv;
      t.lap += fma(-2.0 * wf.jb * rd, u1, 2.0 * u1 * iv);
      if (DB) t.gb = fma(u1, dist * dist, t.gb);
      PairGeo& p = t.pg[k - 1];
      p.iv = iv;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        p.n[d] = v[d] * iv;
        t.gj[d] = fma(u1, p.n[d], t.gj[d]);
        t.drt[d] += p.n[d];
      }
    }
}

// G = eta (I - n n^T) (xx yy zz xy xz yz)
__device__ __forceinline__ void g_block(const PairGeo& p, double eta, double (&t)[6]) {
  double en[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) en[d] = eta * p.n[d];
  t[0] = fma(-en[0], p.n[0], eta);
  t[1] = fma(-en[1], p.n[1], eta);
  t[2] = fma(-en[2], p.n[2], eta);
  t[3] = -en[0] * p.n[1];
  t[4] = -en[0] * p.n[2];
  t[5] = -en[1] * p.n[2];
}

// The backflow blocks of electron a: I + S_a, N_a, sum_j n / r^2 and
// dS_a = m_a + sum_j G_aj (m_a - m_j)
struct Blocks {
  double S[6], N[6], j2[3], dS[3];
};

template <int NE>
__device__ __forceinline__ void backflow_blocks(const Group& g, const PairTerms<NE>& pt, double w,
                                                const double (&ma)[3], Blocks& b) {
#pragma unroll
  for (int q = 0; q < 6; ++q) b.S[q] = b.N[q] = 0.0;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    b.j2[d] = 0.0;
    b.dS[d] = ma[d];
  }
#pragma unroll
  for (int k = 1; k < NE; ++k)
    if (k < g.N) {
      const PairGeo& p = pt.pg[k - 1];
      const int src = g.base + g.next(k);
      const double eta = w * p.iv, iv2 = p.iv * p.iv;
      double t[6], x[3], y[3];
      g_block(p, eta, t);
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        x[d] = ma[d] - shfl(ma[d], src);
        b.j2[d] = fma(p.n[d], iv2, b.j2[d]);
      }
#pragma unroll
      for (int q = 0; q < 6; ++q) {
        b.S[q] += t[q];
        b.N[q] = fma(eta, t[q], b.N[q]);
      }
      symv(t, x, y);
#pragma unroll
      for (int d = 0; d < 3; ++d) b.dS[d] += y[d];
    }
#pragma unroll
  for (int d = 0; d < 3; ++d) b.S[d] += 1.0;
  const double* S = b.S;
  b.N[0] = fma(S[0], S[0], fma(S[3], S[3], fma(S[4], S[4], b.N[0])));
  b.N[1] = fma(S[3], S[3], fma(S[1], S[1], fma(S[5], S[5], b.N[1])));
  b.N[2] = fma(S[4], S[4], fma(S[5], S[5], fma(S[2], S[2], b.N[2])));
  b.N[3] = fma(S[0], S[3], fma(S[3], S[1], fma(S[4], S[5], b.N[3])));
  b.N[4] = fma(S[0], S[4], fma(S[3], S[5], fma(S[4], S[2], b.N[4])));
  b.N[5] = fma(S[3], S[4], fma(S[1], S[5], fma(S[5], S[2], b.N[5])));
}

// lane src's geometry with electron j, eb being src's own electron (zero for j = eb)
template <int NE>
__device__ __forceinline__ void partner_geo(const Group& g, const PairTerms<NE>& pt, int src, int eb, int j,
                                            PairGeo& pb) {
  const int kb = j >= eb ? j - eb : j - eb + g.N;
  pb.n[0] = pb.n[1] = pb.n[2] = pb.iv = 0.0;
#pragma unroll
  for (int q = 1; q < NE; ++q)
    if (q < g.N) {
      // every lane publishes slot q; the reader keeps the one it needs
      const double t0 = shfl(pt.pg[q - 1].n[0], src), t1 = shfl(pt.pg[q - 1].n[1], src),
                   t2 = shfl(pt.pg[q - 1].n[2], src), t3 = shfl(pt.pg[q - 1].iv, src);
      const bool hit = q == kb;
      pb.n[0] = dsel(hit, t0, pb.n[0]);
      pb.n[1] = dsel(hit, t1, pb.n[1]);
      pb.n[2] = dsel(hit, t2, pb.n[2]);
      pb.iv = dsel(hit, t3, pb.iv);
    }
}

// ---- orbitals of one electron at p: the occupied MO values, gradients and
// (MODE 1) Laplacians or (MODE 2) Hessians (xx yy zz xy xz yz); MODE 0 values
// only.  Radial sums are contracted with the MO coefficients per atom first:
// for an s function f (coefficient c_m) and a p shell (vector c_m)
//   phi = f c + f (c.v),  grad = f c + (g1 c + g1 c.v) v,
//   Hess = (U1) I + g1 (c v^T + v c^T) + U2 v v^T,  U1 = g1 c + g1 c.v, U2 = q c + q c.v,
//   lap = (f2 + 2 g1) c + (f2 + 4 g1) c.v,     g1 = f'/rho, f2 = f'', q = (f2 - g1)/rho^2,
// so a p shell costs 9 multiply-accumulates per orbital and the expansion is
// paid once per atom.  U is double, or f32x2 (FP32X2 form).
template <int NO, int MODE>
struct Mo {
  static constexpr int kH = MODE == 2 ? 6 : 1;
  double phi[NO];
  double d[MODE ? NO : 1][3];
  double h[MODE ? NO : 1][kH];
};

__device__ __forceinline__ void macc(double& acc, double a, double b) { acc = fma(a, b, acc); }
__device__ __forceinline__ void macc(f32x2& acc, f32x2 a, f32x2 b) { mac_x2(acc, a, b); }
__device__ __forceinline__ double settle(double a) { return a; }
__device__ __forceinline__ f32x2 settle(f32x2 a) { return normalize_x2(a); }

// where the orbital tables are read (global or shared memory)
struct Tables {
  const ShellDev* shells;
  const float2* mo_x2;     // pairs of FP32
  const float* exp_tab;
};

template <typename U>
struct Geo {  // an electron's displacement from a nucleus
  U v[3], r2, rho, irho, ir2;
};
template <int MODE>
__device__ __forceinline__ void geometry(const double p[3], const double* R, bool sto, Geo<double>& g) {
#pragma unroll
  for (int d = 0; d < 3; ++d) g.v[d] = p[d] - R[d];
  g.r2 = fma(g.v[2], g.v[2], fma(g.v[1], g.v[1], g.v[0] * g.v[0]));
  if (sto) {
    g.irho = rsqrt3(g.r2);
    g.rho = sqrt_from(g.r2, g.irho);
    if (MODE) g.ir2 = g.irho * g.irho;
  }
}
template <int MODE>
__device__ __forceinline__ void geometry(const double p[3], const double* R, bool sto, Geo<f32x2>& g) {
#pragma unroll
  for (int d = 0; d < 3; ++d) g.v[d] = diff_x2(p[d], R[d]);
  g.r2 = g.v[0] * g.v[0] + g.v[1] * g.v[1] + g.v[2] * g.v[2];
  if (sto) {
    g.rho = sqrt_x2(g.r2);
    g.irho = recip_x2(g.rho);
    if (MODE) g.ir2 = g.irho * g.irho;
  }
}

// f, g1 = f'/rho, f2 = f'' and q = (f2 - g1)/rho^2 of a shell
template <int MODE>
__device__ __forceinline__ void radial(const WfDev& wf, const Tables&, const ShellDev& sh, int s,
                                       const Geo<double>& g, double& f, double& g1, double& f2, double& q) {
  const double* nak = wf.nak + (size_t)s * QMC_MAX_PRIM;
  if (sh.kind == 0) {
    const double z = sh.expo[0];
    f = sh.coef[0] * exp_scaled(nak[0], g.rho, wf.exp2_tab);
    for (int k = 0; k < sh.kn; ++k) f *= g.rho;
    if (MODE) {
      const double kn = (double)sh.kn, h = fma(kn, g.irho, -z), hf = h * f;
      g1 = hf * g.irho;
      f2 = fma(h, hf, -(kn * g.ir2) * f);
      if (MODE == 2) q = (f2 - g1) * g.ir2;
    }
  } else {
    f = 0.0;
    double t1 = 0.0, t2 = 0.0;
    for (int p = 0; p < sh.n_prim; ++p) {
      const double al2 = 2.0 * sh.expo[p];
      const double ce = sh.coef[p] * exp_scaled(nak[p], g.r2, wf.exp2_tab);
      f += ce;
      if (MODE) {
        const double a = al2 * ce;
        t1 += a;
        t2 = fma(al2, a, t2);
      }
    }
    if (MODE) {
      g1 = -t1;
      f2 = fma(g.r2, t2, -t1);
      if (MODE == 2) q = t2;
    }
  }
}
template <int MODE>
__device__ __forceinline__ void radial(const WfDev&, const Tables& tb, const ShellDev& sh, int, const Geo<f32x2>& g,
                                       f32x2& f, f32x2& g1, f32x2& f2, f32x2& q) {
  if (sh.kind == 0) {
    const f32x2 z(sh.expo_f[0], sh.expo_lo[0]);
    f = f32x2(sh.coef_f[0], sh.coef_lo[0]) * exp_x2(-(z * g.rho), tb.exp_tab);
    for (int k = 0; k < sh.kn; ++k) f = f * g.rho;
    if (MODE) {
      const f32x2 h = g.irho * (float)sh.kn - z, hf = h * f;
      g1 = hf * g.irho;
      f2 = h * hf - (g.ir2 * (float)sh.kn) * f;
      if (MODE == 2) q = (f2 - g1) * g.ir2;
    }
  } else {
    f = f32x2(0.f);
    f32x2 t1(0.f), t2(0.f);
    for (int p = 0; p < sh.n_prim; ++p) {
      const f32x2 e = exp_x2(-(f32x2(sh.expo_f[p], sh.expo_lo[p]) * g.r2), tb.exp_tab);
      mac_x2(f, f32x2(sh.coef_f[p], sh.coef_lo[p]), e);
      if (MODE) {
        mac_x2(t1, f32x2(sh.c2a_f[p], sh.c2a_lo[p]), e);
        mac_x2(t2, f32x2(sh.c4a_f[p], sh.c4a_lo[p]), e);
      }
    }
    f = normalize_x2(f);
    if (MODE) {
      t1 = normalize_x2(t1);
      t2 = normalize_x2(t2);
      g1 = -t1;
      f2 = g.r2 * t2 - t1;
      if (MODE == 2) q = t2;
    }
  }
}

__device__ __forceinline__ double mo_coef(const WfDev& wf, const Tables&, int row, int m, double) {
  return __ldg(wf.mo64c + (size_t)row * wf.n_mo + m);
}
__device__ __forceinline__ f32x2 mo_coef(const WfDev& wf, const Tables& tb, int row, int m, f32x2) {
  const float2 c = tb.mo_x2[(size_t)row * wf.n_mo + m];
  return f32x2(c.x, c.y);
}

template <typename U, int NO, int MODE>
__device__ __forceinline__ void orbitals(const WfDev& wf, const Tables& tb, const double p[3], Mo<NO, MODE>& out) {
  constexpr int ND = MODE ? NO : 1, NH = MODE == 2 ? 6 : 1;
  constexpr bool kPair = std::is_same<U, f32x2>::value;
  U phi[NO], dm[ND][3], hm[ND][NH];
  U s0[NO], s1[ND], s2[ND], p0[NO][3], p1[ND][3], p2[ND][3];
  const U zero(0.f);
#pragma unroll
  for (int m = 0; m < NO; ++m) phi[m] = zero;
#pragma unroll
  for (int m = 0; m < ND; ++m) {
#pragma unroll
    for (int d = 0; d < 3; ++d) dm[m][d] = zero;
#pragma unroll
    for (int q = 0; q < NH; ++q) hm[m][q] = zero;
  }
  Geo<U> g;
  for (int s = 0; s < wf.n_shell;) {
    const int atom = tb.shells[s].atom;
    geometry<MODE>(p, wf.atom_xyz[atom], wf.any_sto != 0, g);
#pragma unroll
    for (int m = 0; m < NO; ++m) {
      s0[m] = zero;
#pragma unroll
      for (int d = 0; d < 3; ++d) p0[m][d] = zero;
    }
#pragma unroll
    for (int m = 0; m < ND; ++m) {
      s1[m] = s2[m] = zero;
#pragma unroll
      for (int d = 0; d < 3; ++d) p1[m][d] = p2[m][d] = zero;
    }
    for (; s < wf.n_shell; ++s) {  // the shells of this run of the atom
      const ShellDev& sh = tb.shells[s];
      if (sh.atom != atom) break;
      U f, g1 = zero, f2 = zero, q = zero;
      radial<MODE>(wf, tb, sh, s, g, f, g1, f2, q);
      const int row = sh.ao_first;
      if (sh.l == 0) {
        if (MODE == 1) q = f2 + g1 * U(2.0f);
#pragma unroll
        for (int m = 0; m < NO; ++m) {
          const U c = mo_coef(wf, tb, row, m, zero);
          macc(s0[m], c, f);
          if (MODE) {
            macc(s1[m], c, g1);
            macc(s2[m], c, q);
          }
        }
      } else {
        if (MODE == 1) q = f2 + g1 * U(4.0f);
        // (the functions that the shell holds: all three, or fewer where the
        // exponents of x, y and z differ, as after an optimisation step)
        int r = row;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          if (!((sh.p_mask >> d) & 1)) continue;
#pragma unroll
          for (int m = 0; m < NO; ++m) {
            const U c = mo_coef(wf, tb, r, m, zero);
            macc(p0[m][d], c, f);
            if (MODE) {
              macc(p1[m][d], c, g1);
              macc(p2[m][d], c, q);
            }
          }
          ++r;
        }
      }
    }
    U dd[6];
    if (MODE == 2) {
      dd[0] = g.v[0] * g.v[0];
      dd[1] = g.v[1] * g.v[1];
      dd[2] = g.v[2] * g.v[2];
      dd[3] = g.v[0] * g.v[1];
      dd[4] = g.v[0] * g.v[2];
      dd[5] = g.v[1] * g.v[2];
    }
#pragma unroll
    for (int m = 0; m < NO; ++m) {
      if (kPair) {
        s0[m] = settle(s0[m]);
#pragma unroll
        for (int d = 0; d < 3; ++d) p0[m][d] = settle(p0[m][d]);
      }
      phi[m] = phi[m] + s0[m];
#pragma unroll
      for (int d = 0; d < 3; ++d) macc(phi[m], p0[m][d], g.v[d]);
      if (MODE) {
        U u1 = s1[m], u2 = s2[m];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          p1[m][d] = settle(p1[m][d]);
          p2[m][d] = settle(p2[m][d]);
          macc(u1, p1[m][d], g.v[d]);
          macc(u2, p2[m][d], g.v[d]);
        }
        u1 = settle(u1);
        u2 = settle(u2);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          dm[m][d] = dm[m][d] + p0[m][d];
          macc(dm[m][d], u1, g.v[d]);
        }
        if (MODE == 1) {
          hm[m][0] = hm[m][0] + u2;
        } else {
          const U two(2.0f);
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            hm[m][d] = hm[m][d] + u1;
            macc(hm[m][d], p1[m][d] * two, g.v[d]);
          }
          macc(hm[m][3], p1[m][0], g.v[1]);
          macc(hm[m][3], p1[m][1], g.v[0]);
          macc(hm[m][4], p1[m][0], g.v[2]);
          macc(hm[m][4], p1[m][2], g.v[0]);
          macc(hm[m][5], p1[m][1], g.v[2]);
          macc(hm[m][5], p1[m][2], g.v[1]);
#pragma unroll
          for (int q = 0; q < 6; ++q) macc(hm[m][q], u2, dd[q]);
        }
      }
    }
    if (kPair && s < wf.n_shell) {
#pragma unroll
      for (int m = 0; m < NO; ++m) phi[m] = settle(phi[m]);
#pragma unroll
      for (int m = 0; m < ND; ++m) {
#pragma unroll
        for (int d = 0; d < 3; ++d) dm[m][d] = settle(dm[m][d]);
#pragma unroll
        for (int q = 0; q < NH; ++q) hm[m][q] = settle(hm[m][q]);
      }
    }
  }
#pragma unroll
  for (int m = 0; m < NO; ++m) out.phi[m] = widen(settle(phi[m]));
  if (MODE) {
#pragma unroll
    for (int m = 0; m < NO; ++m) {
#pragma unroll
      for (int d = 0; d < 3; ++d) out.d[m][d] = widen(settle(dm[m][d]));
#pragma unroll
      for (int q = 0; q < NH; ++q) out.h[m][q] = widen(settle(hm[m][q]));
    }
  }
}

// ---- the reference determinant of the lane's spin: lane a holds row a of A
// (phi of its electron).  The generalised cross product of the other rows, in
// cyclic order, gives row a's cofactors, so the lane forms its own column of
// the inverse, (A^-1)_{m a} = cof_m / det, without the elimination's serial
// chain.  Spins with n < NO rows are padded with unit rows.
template <int NO>
__device__ __forceinline__ double cofactors(const Group& g, const double (&phi)[NO], int a, int n, int i0,
                                            double (&cof)[NO]) {
  double row[NO];
#pragma unroll
  for (int m = 0; m < NO; ++m) row[m] = m < n ? phi[m] : 0.0;
  double o[NO > 1 ? NO - 1 : 1][NO];  // rows a + 1, a + 2, ... (cyclic in NO)
#pragma unroll
  for (int k = 1; k < NO; ++k) {
    const int q = a + k >= NO ? a + k - NO : a + k;
    const int src = g.base + (q < n ? i0 + q : i0);
#pragma unroll
    for (int m = 0; m < NO; ++m) {
      const double v = shfl(row[m], src);
      o[k - 1][m] = q < n ? v : (m == q ? 1.0 : 0.0);
    }
  }
  if constexpr (NO == 1) {
    cof[0] = 1.0;
  } else if constexpr (NO == 2) {
    // the cyclic order of two rows is odd for a = 1
    const double sg = a == 0 ? 1.0 : -1.0;
    cof[0] = sg * o[0][1];
    cof[1] = -sg * o[0][0];
  } else if constexpr (NO == 3) {
    cof[0] = fma(o[0][1], o[1][2], -(o[0][2] * o[1][1]));
    cof[1] = fma(o[0][2], o[1][0], -(o[0][0] * o[1][2]));
    cof[2] = fma(o[0][0], o[1][1], -(o[0][1] * o[1][0]));
  } else {
    const double sg = (a & 1) ? -1.0 : 1.0;  // a cyclic shift of four rows is odd
    // 2x2 minors of the last two rows
    double M[4][4];
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
      for (int d = c + 1; d < 4; ++d) M[c][d] = fma(o[1][c], o[2][d], -(o[1][d] * o[2][c]));
    auto det3 = [&](int c0, int c1, int c2) {
      return fma(o[0][c0], M[c1][c2], fma(-o[0][c1], M[c0][c2], o[0][c2] * M[c0][c1]));
    };
    cof[0] = sg * det3(1, 2, 3);
    cof[1] = -sg * det3(0, 2, 3);
    cof[2] = sg * det3(0, 1, 3);
    cof[3] = -sg * det3(0, 1, 2);
  }
  double det = row[0] * cof[0];
#pragma unroll
  for (int m = 1; m < NO; ++m) det = fma(row[m], cof[m], det);
  // one value per spin: the expansion along its first row
  return shfl(det, g.base + i0);
}

}  // namespace small

}  // namespace qmc

#define QMC_SMALL_DISPATCH(CALL)                                                      \
  {                                                                                   \
    const int ns = wf.n_up > wf.n_down ? wf.n_up : wf.n_down;                         \
    if (wf.n_elec <= 2 && ns <= 1) { constexpr int NE = 2, NO = 1; CALL; }            \
    else if (wf.n_elec <= 4 && ns <= 2) { constexpr int NE = 4, NO = 2; CALL; }       \
    else if (wf.n_elec <= 6 && ns <= 3) { constexpr int NE = 6, NO = 3; CALL; }       \
    else if (wf.n_elec <= 8 && ns <= 4) { constexpr int NE = 8, NO = 4; CALL; }       \
    else return cudaErrorInvalidValue;                                                \
  }
