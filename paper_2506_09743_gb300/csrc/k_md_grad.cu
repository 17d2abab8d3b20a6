// Parameter gradient of log|Psi| for a multi-determinant expansion without
// backflow (FP64): the estimator of Eq. nabla_loss for Psi of Eq. psimol
// with the CI sum, through the tables of the reference inverse (Eq. table).
//
// Per spin (n electrons a, orbitals m, Phi_{a m} = phi_m(r_a), A = Phi[:, occ]
// the reference matrix, T = A^-1 Phi, so that an excitation X with holes h
// and particles p has D_X / D_0 = R_X = det T[h, p]):
//   log|Psi| = log|D_0^up| + log|D_0^dn| + log|S|,   S = sum_n d_n R_n^up R_n^dn.
// The derivative of log|Psi| with respect to Phi_{a m} is Gamma_{m a}:
//   d log|D_0| / d Phi_{a m} = (A^-1)_{m a}                 (m occupied)
//   d log S / d Phi_{a m}    = [(I - P T) Y A^-1]_{m a},
// where Y_{p h} = (dS / dT_{h p}) / S collects, per unique excitation e of
// the spin, c_e = sum_{n: e_n = e} d_n R_n^(other spin) / S times dR_e/dT_{hp}
// (rank 1: 1; rank 2: the 2x2 cofactors), and P selects the occupied rows
// (dT = A^-1 (dPhi - dPhi[:, occ] T)).  Y has rows for particles only, so
//   Gamma_{m a} = (A^-1)_{m a} - sum_p T_{m p} Z_{p a}   (m occupied),
//   Gamma_{p a} = Z_{p a}                                 (particles),
//   Z = Y A^-1.
// Then with AO values phi_b (angular normalisation ang_b), MO coefficients
// C_{b m} and u_b = sum_m C_{b m} ang_b Gamma_{m a} per electron row:
//   d log|Psi| / d C_{b m}  = sum_a ang_b phi_b(r_a) Gamma_{m a}
//   d log|Psi| / d alpha_p  = sum_a u_b d phi_b / d alpha_p      (as k_grad_logpsi)
//   d log|Psi| / d d_n      = R_n^up R_n^dn / S
//   d log|Psi| / d b        = -sum_{i<j} w0 r_ij^2 / (1 + b r_ij)^2
//   d log|Psi| / d w        = sum_a sum_b u_b grad phi_b(r_a) . sum_{j != a} (r_a - r_j) / r_ij
// (the last at w = 0: the derivative of turning the backflow on).
//
// Two kernels: k_md_gamma (one thread per walker: the reference inverses,
// tables, CI sum, Gamma, the CI-weight and Jastrow terms) writes Gamma to
// scratch; k_md_rows (one thread per electron row) evaluates the AOs and
// adds the coefficient, exponent and backflow terms.  Per-walker values are
// weighted (estimator 2 (E_L - E_v) / M, one, or E_L) and summed per warp in a
// fixed order, per block over the warps in order, and over the blocks by
// k_row_sums: the result is bitwise reproducible.
#include "fp64_math.cuh"
#include "general_eval.cuh"

namespace qmc {

namespace {

constexpr int kMdNS = 8;        // electrons per spin
constexpr int kMdNM = 16;       // orbitals
constexpr int kMdThreads = 128;
constexpr int kMdWarps = kMdThreads / 32;

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;  // lane 0 holds the sum
}

__device__ __forceinline__ double walker_weight(int weight, const double* e_loc, const double* stats, int64_t w,
                                                int64_t W) {
  if (weight == 1) return 1.0;
  if (weight == 2) return e_loc[w];
  return 2.0 * (e_loc[w] - stats[0]) / (double)W;
}

// per-warp accumulators [warps][n_param] -> partial[k][col] in a fixed order
__device__ void flush_acc(const double* acc, int n_param, double* partial, int64_t ld_partial, int col) {
  __syncthreads();
  for (int k = threadIdx.x; k < n_param; k += blockDim.x) {
    double s = 0.0;
    for (int q = 0; q < (int)(blockDim.x >> 5); ++q) s += acc[(size_t)q * n_param + k];
    partial[(size_t)k * ld_partial + col] = s;
  }
}

}  // namespace

__global__ void __launch_bounds__(kMdThreads) k_md_gamma(WfDev wf, const double* __restrict__ walkers, int64_t W,
                                                          int64_t ldw, const double* __restrict__ mo, int nmp,
                                                          int64_t ldm, const double* __restrict__ e_loc,
                                                          const double* __restrict__ stats, int weight, int n_param,
                                                          int off_d, double* __restrict__ gam,
                                                          double* __restrict__ partial, int64_t ld_partial) {
  extern __shared__ __align__(16) double acc[];  // [kMdWarps][n_param]
  for (int k = threadIdx.x; k < kMdWarps * n_param; k += blockDim.x) acc[k] = 0.0;
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nu = wf.n_up, N = wf.n_elec, nmo = wf.n_mo;
  const int off_b = off_d + wf.n_det;
  const int64_t n_iter = (W + (int64_t)gridDim.x * kMdThreads - 1) / ((int64_t)gridDim.x * kMdThreads);
  for (int64_t it = 0; it < n_iter; ++it) {
    const int64_t w = (it * gridDim.x + blockIdx.x) * kMdThreads + threadIdx.x;
    const bool live = w < W;
    const double wt = live ? walker_weight(weight, e_loc, stats, w, W) : 0.0;
    double R[2][kMaxExc > 128 ? 128 : kMaxExc];  // ratios of the unique excitations
    double ainv[2][kMdNS][kMdNS], T[2][kMdNS][kMdNM];
    for (int s = 0; s < 2; ++s) {
      const int n = s == 0 ? nu : wf.n_down, i0 = s == 0 ? 0 : nu;
      const int p_hi = wf.p_hi[s];
      for (int a = 0; a < n; ++a)
        for (int m = 0; m < n; ++m)
          ainv[s][a][m] = live ? mo[((size_t)((i0 + a) * 2) * nmp + m) * ldm + w] : (a == m ? 1.0 : 0.0);
      if (n > 0) small_inverse<double, kMdNS>(ainv[s], n);
      // T_{h p} = sum_a (A^-1)_{h a} Phi_{a p} for every occupied row h and particle p
      for (int h = 0; h < n; ++h)
        for (int p = n; p < p_hi; ++p) {
          double t = 0.0;
          for (int a = 0; a < n; ++a)
            t += ainv[s][h][a] * (live ? mo[((size_t)((i0 + a) * 2) * nmp + p) * ldm + w] : 0.0);
          T[s][h][p] = t;
        }
      for (int e = 0; e < wf.n_exc[s]; ++e) {
        const int* x = wf.exc + (s * kMaxExc + e) * 5;
        const int rank = x[0];
        R[s][e] = rank == 0 ? 1.0
                  : rank == 1 ? T[s][x[1]][x[3]]
                              : T[s][x[1]][x[3]] * T[s][x[2]][x[4]] - T[s][x[1]][x[4]] * T[s][x[2]][x[3]];
      }
    }
    double S = 0.0;
    for (int n = 0; n < wf.n_det; ++n) S += wf.det_w[n] * R[0][wf.det_idx[2 * n]] * R[1][wf.det_idx[2 * n + 1]];
    const double iS = live ? 1.0 / S : 0.0;
    // CI weights (stored sorted; the gradient goes to the original order)
    for (int n = 0; n < wf.n_det; ++n) {
      const double v = warp_sum(wt * R[0][wf.det_idx[2 * n]] * R[1][wf.det_idx[2 * n + 1]] * iS);
      if (lane == 0) acc[(size_t)warp * n_param + off_d + wf.det_orig[n]] += v;
    }
    // Jastrow b
    {
      double gb = 0.0;
      if (live)
        for (int i = 0; i < N; ++i)
          for (int j = i + 1; j < N; ++j) {
            double d2 = 0.0;
            for (int c = 0; c < 3; ++c) {
              const double dd = walkers[(int64_t)(3 * i + c) * ldw + w] - walkers[(int64_t)(3 * j + c) * ldw + w];
              d2 += dd * dd;
            }
            const double dist = sqrt(d2);
            const double w0 = ((i < nu) == (j < nu)) ? wf.w0_par : wf.w0_anti;
            const double den = 1.0 + wf.jb * dist;
            gb -= w0 * dist * dist / (den * den);
          }
      const double v = warp_sum(wt * gb);
      if (lane == 0) acc[(size_t)warp * n_param + off_b] += v;
    }
    // many-body Jastrow (App. D), after the backflow weight:
    //   K_en = (w0 r + w1 r^2) / (1 + w2 r) over atoms and electrons:
    //     d/dw0 = r / d, d/dw1 = r^2 / d, d/dw2 = -(w0 r + w1 r^2) r / d^2, d = 1 + w2 r;
    //   K_een = 1/2 sum over atoms, ordered pairs i != j and terms of
    //     c f(a1, b1; r_ai) f(a2, b2; r_aj) f(a3, b3; r_ij), f(a, b; r) = a r / (1 + b r):
    //     df/da = r / (1 + b r), df/db = -a r^2 / (1 + b r)^2
    if (wf.mb_en || wf.n_een) {
      int k = off_b + 2;
      if (wf.mb_en) {
        double g3[3] = {0.0, 0.0, 0.0};
        if (live)
          for (int a = 0; a < wf.n_atom; ++a)
            for (int i = 0; i < N; ++i) {
              double d2 = 0.0;
              for (int c = 0; c < 3; ++c) {
                const double dd = walkers[(int64_t)(3 * i + c) * ldw + w] - wf.atom_xyz[a][c];
                d2 += dd * dd;
              }
              const double r = sqrt(d2), d = 1.0 + wf.jen[2] * r;
              g3[0] += r / d;
              g3[1] += r * r / d;
              g3[2] -= (wf.jen[0] * r + wf.jen[1] * r * r) * r / (d * d);
            }
        for (int q = 0; q < 3; ++q) {
          const double v = warp_sum(wt * g3[q]);
          if (lane == 0) acc[(size_t)warp * n_param + k + q] += v;
        }
        k += 3;
      }
      for (int t = 0; t < wf.n_een; ++t) {
        const double c = wf.jeen[t][0], a1 = wf.jeen[t][1], b1 = wf.jeen[t][2], a2 = wf.jeen[t][3],
                     b2 = wf.jeen[t][4], a3 = wf.jeen[t][5], b3 = wf.jeen[t][6];
        double g7[7] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
        if (live)
          for (int a = 0; a < wf.n_atom; ++a)
            for (int i = 0; i < N; ++i)
              for (int j = 0; j < N; ++j) {
                if (i == j) continue;
                double x2 = 0.0, y2 = 0.0, z2 = 0.0;
                for (int q = 0; q < 3; ++q) {
                  const double ri = walkers[(int64_t)(3 * i + q) * ldw + w], rj = walkers[(int64_t)(3 * j + q) * ldw + w];
                  x2 += (ri - wf.atom_xyz[a][q]) * (ri - wf.atom_xyz[a][q]);
                  y2 += (rj - wf.atom_xyz[a][q]) * (rj - wf.atom_xyz[a][q]);
                  z2 += (ri - rj) * (ri - rj);
                }
                const double x = sqrt(x2), y = sqrt(y2), z = sqrt(z2);
                const double d1 = 1.0 + b1 * x, d2 = 1.0 + b2 * y, d3 = 1.0 + b3 * z;
                const double h1 = x / d1, h2 = y / d2, h3 = z / d3;  // df/da
                const double f1 = a1 * h1, f2 = a2 * h2, f3 = a3 * h3;
                g7[0] += 0.5 * f1 * f2 * f3;
                g7[1] += 0.5 * c * h1 * f2 * f3;
                g7[2] -= 0.5 * c * a1 * h1 * h1 * f2 * f3;
                g7[3] += 0.5 * c * f1 * h2 * f3;
                g7[4] -= 0.5 * c * f1 * a2 * h2 * h2 * f3;
                g7[5] += 0.5 * c * f1 * f2 * h3;
                g7[6] -= 0.5 * c * f1 * f2 * a3 * h3 * h3;
              }
        for (int q = 0; q < 7; ++q) {
          const double v = warp_sum(wt * g7[q]);
          if (lane == 0) acc[(size_t)warp * n_param + k + q] += v;
        }
        k += 7;
      }
    }
    if (!live) continue;
    // Gamma per spin
    for (int s = 0; s < 2; ++s) {
      const int n = s == 0 ? nu : wf.n_down, i0 = s == 0 ? 0 : nu;
      const int p_hi = wf.p_hi[s];
      // c_e and Y_{p h}
      double c[kMaxExc > 128 ? 128 : kMaxExc];
      for (int e = 0; e < wf.n_exc[s]; ++e) c[e] = 0.0;
      for (int k = 0; k < wf.n_det; ++k)
        c[wf.det_idx[2 * k + s]] += wf.det_w[k] * R[1 - s][wf.det_idx[2 * k + 1 - s]] * iS;
      double Y[kMdNM][kMdNS];
      for (int p = n; p < p_hi; ++p)
        for (int h = 0; h < n; ++h) Y[p][h] = 0.0;
      for (int e = 0; e < wf.n_exc[s]; ++e) {
        const int* x = wf.exc + (s * kMaxExc + e) * 5;
        if (x[0] == 1) {
          Y[x[3]][x[1]] += c[e];
        } else if (x[0] == 2) {
          Y[x[3]][x[1]] += c[e] * T[s][x[2]][x[4]];
          Y[x[4]][x[2]] += c[e] * T[s][x[1]][x[3]];
          Y[x[4]][x[1]] -= c[e] * T[s][x[2]][x[3]];
          Y[x[3]][x[2]] -= c[e] * T[s][x[1]][x[4]];
        }
      }
      // Z = Y A^-1 (particle rows), then Gamma
      double Z[kMdNM][kMdNS];
      for (int p = n; p < p_hi; ++p)
        for (int a = 0; a < n; ++a) {
          double z = 0.0;
          for (int h = 0; h < n; ++h) z += Y[p][h] * ainv[s][h][a];
          Z[p][a] = z;
        }
      for (int a = 0; a < n; ++a) {
        double* g = gam + (size_t)((i0 + a) * nmo) * ldm + w;
        for (int m = 0; m < nmo; ++m) {
          double v = 0.0;
          if (m < n) {
            v = ainv[s][m][a];
            for (int p = n; p < p_hi; ++p) v -= T[s][m][p] * Z[p][a];
          } else if (m < p_hi) {
            v = Z[m][a];
          }
          g[(size_t)m * ldm] = v;
        }
      }
    }
  }
  flush_acc(acc, n_param, partial, ld_partial, blockIdx.x);
}

// Row kernel.  It is bound by the FP64 pipe, so the split minimises FP64
// instructions: 65,536 CO walkers took 16.6 ms when every coefficient and
// exponent value was formed per row and summed over the warp by shuffles (about
// 95 instructions per AO and row).  A warp takes 32 rows of one electron, and
//   1. each lane evaluates its row's AOs, a chunk of up to kChunkAo at a time:
//      values phi_b, the weighted exponent factors q_b = w u_b P_b and the
//      shells' radial derivatives go to shared memory;
//   2. the chunk's outputs are then formed as sums over the 32 rows,
//        C: sum_r phi_b[r] (w Gamma_m)[r],   alpha: sum_r q_b[r] (d f/d alpha_p)[r],
//      one output per lane and round, one FMA per row (the reduction over the
//      rows is the FMA chain itself), added to the warp's sums in shared memory.
// Rows, chunks, warps and blocks are taken in a fixed order.
constexpr int kChunkAo = 16;
constexpr int kChunkRad = 24;   // radial derivatives (shells x primitives) of a chunk
constexpr int kRowPad = 33;

// doubles of a warp's chunk buffers: phi, q, w Gamma, radial derivatives
constexpr int kRowsBuf = (2 * kChunkAo + kMdNM + kChunkRad) * kRowPad;

__global__ void __launch_bounds__(kMdThreads) k_md_rows(const __grid_constant__ WfDev wf,
                                                         const double* __restrict__ walkers, int64_t W, int64_t ldw,
                                                         const double* __restrict__ gam, int64_t ldm,
                                                         const double* __restrict__ e_loc,
                                                         const double* __restrict__ stats, int weight,
                                                         const double* __restrict__ ang,
                                                         const int* __restrict__ prim_start, int n_param,
                                                         double* __restrict__ partial, int64_t ld_partial, int col0) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warp = blockDim.x >> 5;
  const int N = wf.n_elec, nmo = wf.n_mo, n_ao = wf.n_ao;
  const int n_prim = prim_start[n_ao];
  const int off_c = n_prim, off_w = off_c + n_ao * nmo + wf.n_det + 1;
  double* acc = reinterpret_cast<double*>(smem_raw);                      // [n_warp][n_param]
  double* buf = acc + (size_t)n_warp * n_param + (size_t)warp * kRowsBuf;
  // exponent parameter -> AO within its chunk << 8 | radial derivative within the chunk
  unsigned short* slot = reinterpret_cast<unsigned short*>(acc + (size_t)n_warp * (n_param + kRowsBuf));
  double* phi_s = buf;                           // [kChunkAo][33]
  double* q_s = phi_s + kChunkAo * kRowPad;      // [kChunkAo][33]
  double* wg_s = q_s + kChunkAo * kRowPad;       // [kMdNM][33]
  double* rd_s = wg_s + kMdNM * kRowPad;         // [kChunkRad][33]
  for (int k = threadIdx.x; k < n_warp * n_param; k += blockDim.x) acc[k] = 0.0;
  // chunk of shell s: consecutive shells while their AOs and radial
  // derivatives fit (the same rule in the loop below)
  auto fits = [&](int ao, int rad, const ShellDev& sh) {
    return ao == 0 || (ao + sh.n_ao <= kChunkAo && rad + sh.n_prim <= kChunkRad);
  };
  if (threadIdx.x == 0) {
    int ao = 0, rad = 0;
    for (int s = 0; s < wf.n_shell; ++s) {
      const ShellDev& sh = wf.shells[s];
      if (!fits(ao, rad, sh)) ao = rad = 0;
      for (int k = 0; k < sh.n_ao; ++k)
        for (int p = 0; p < sh.n_prim; ++p)
          slot[prim_start[sh.ao_first + k] + p] = (unsigned short)(((ao + k) << 8) | (rad + p));
      ao += sh.n_ao;
      rad += sh.n_prim;
    }
  }
  __syncthreads();
  double* my = acc + (size_t)warp * n_param;
  const int64_t n_tile = (W + 31) / 32;  // tiles of 32 walkers, per electron
  const int64_t n_work = n_tile * N;
  for (int64_t t = (int64_t)blockIdx.x * n_warp + warp; t < n_work; t += (int64_t)gridDim.x * n_warp) {
    const int i = (int)(t / n_tile);
    const int64_t w0 = (t - (int64_t)i * n_tile) * 32 + lane;
    const bool live = w0 < W;
    const int64_t w = live ? w0 : W - 1;
    const double wt = live ? walker_weight(weight, e_loc, stats, w, W) : 0.0;
    double r[3], drt[3] = {0.0, 0.0, 0.0};
    for (int c = 0; c < 3; ++c) r[c] = walkers[(int64_t)(3 * i + c) * ldw + w];
    for (int j = 0; j < N; ++j) {
      if (j == i) continue;
      double v[3];
      for (int c = 0; c < 3; ++c) v[c] = r[c] - walkers[(int64_t)(3 * j + c) * ldw + w];
      const double inv = rsqrt3(fma(v[2], v[2], fma(v[1], v[1], v[0] * v[0])));
      for (int c = 0; c < 3; ++c) drt[c] = fma(inv, v[c], drt[c]);
    }
    double G[kMdNM];
#pragma unroll
    for (int m = 0; m < kMdNM; ++m) {
      G[m] = m < nmo ? gam[((size_t)i * nmo + m) * ldm + w] : 0.0;
      wg_s[m * kRowPad + lane] = wt * G[m];
    }
    double gw = 0.0;
    int cur_atom = -1;
    double dv[3] = {0.0, 0.0, 0.0}, r2 = 0.0, rho = 0.0, irho = 0.0, D = 0.0;
    for (int s0 = 0; s0 < wf.n_shell;) {
      int ao = 0, rad = 0, s = s0;
      const int b0 = wf.shells[s0].ao_first;
      for (; s < wf.n_shell; ++s) {
        const ShellDev& sh = wf.shells[s];
        if (!fits(ao, rad, sh)) break;
        if (sh.atom != cur_atom) {
          cur_atom = sh.atom;
          for (int c = 0; c < 3; ++c) dv[c] = r[c] - wf.atom_xyz[cur_atom][c];
          r2 = fma(dv[2], dv[2], fma(dv[1], dv[1], dv[0] * dv[0]));
          D = fma(dv[2], drt[2], fma(dv[1], drt[1], dv[0] * drt[0]));
          if (wf.any_sto) {
            irho = rsqrt3(r2);
            rho = sqrt_from(r2, irho);
          }
        }
        // radial factor, f'/rho, and per primitive the exponent derivative of
        // its normalised term: d(N_p e^(-alpha r^2))/d alpha = term ((3/4 + l/2)/alpha - r^2)
        const double* nak = wf.nak + (size_t)s * QMC_MAX_PRIM;
        double f = 0.0, g1 = 0.0;
        if (sh.kind == 0) {
          f = sh.coef[0] * exp_scaled(nak[0], rho, wf.exp2_tab);
          for (int k = 0; k < sh.kn; ++k) f *= rho;
          g1 = fma((double)sh.kn, irho, -sh.expo[0]) * f * irho;
          rd_s[rad * kRowPad + lane] = f * (((double)(sh.kn + sh.l + 1) + 0.5) * recip3(sh.expo[0]) - rho);
        } else {
          for (int p = 0; p < sh.n_prim; ++p) {
            const double al = sh.expo[p];
            const double term = sh.coef[p] * exp_scaled(nak[p], r2, wf.exp2_tab);
            f += term;
            g1 = fma(nak[p], term, g1);  // -2048 alpha / ln 2, scaled below
            rd_s[(rad + p) * kRowPad + lane] = term * fma(0.75 + 0.5 * sh.l, recip3(al), -r2);
          }
          g1 *= 2.0 * (0.69314718055994530942 / 2048.0);
        }
        const double h = g1 * D;
        for (int k = 0; k < sh.n_ao; ++k) {
          const int b = sh.ao_first + k;
          const int pw = wf.ao_pow[b];
          const int pa[3] = {pw & 15, (pw >> 4) & 15, (pw >> 8) & 15};
          // P and grad(P f) . drt = f grad P . drt + P g1 (v . drt)
          double P, gd;
          if (sh.l == 0) {
            P = 1.0;
            gd = h;
          } else if (sh.l == 1) {
            const bool px = pa[0] != 0, py = pa[1] != 0;
            P = px ? dv[0] : py ? dv[1] : dv[2];
            gd = fma(P, h, f * (px ? drt[0] : py ? drt[1] : drt[2]));
          } else if (sh.l == 2) {
            const int c = pa[0] ? 0 : pa[1] ? 1 : 2;                  // first factor
            const int e = pa[c] == 2 ? c : (pa[2] ? 2 : 1);           // second
            const double vc = c == 0 ? dv[0] : c == 1 ? dv[1] : dv[2], ve = e == 0 ? dv[0] : e == 1 ? dv[1] : dv[2];
            const double tc = c == 0 ? drt[0] : c == 1 ? drt[1] : drt[2],
                         te = e == 0 ? drt[0] : e == 1 ? drt[1] : drt[2];
            P = vc * ve;
            gd = fma(P, h, f * fma(vc, te, ve * tc));
          } else {
            P = mono(dv[0], dv[1], dv[2], pa[0], pa[1], pa[2]);
            double dP = 0.0;
            for (int c = 0; c < 3; ++c)
              if (pa[c] > 0)
                dP += pa[c] * mono(dv[0], dv[1], dv[2], pa[0] - (c == 0), pa[1] - (c == 1), pa[2] - (c == 2)) * drt[c];
            gd = fma(P, h, f * dP);
          }
          const double* Cb = wf.mo64 + (size_t)b * nmo;  // angular factor folded in
          double u0 = 0.0, u1 = 0.0;
#pragma unroll
          for (int m = 0; m < kMdNM; m += 2) {
            if (m < nmo) u0 = fma(__ldg(Cb + m), G[m], u0);
            if (m + 1 < nmo) u1 = fma(__ldg(Cb + m + 1), G[m + 1], u1);
          }
          const double u = u0 + u1;
          phi_s[(ao + k) * kRowPad + lane] = P * f;
          q_s[(ao + k) * kRowPad + lane] = wt * u * P;
          gw = fma(u, gd, gw);
        }
        ao += sh.n_ao;
        rad += sh.n_prim;
      }
      __syncwarp();
      // coefficients of the chunk's AOs (angular factor applied here)
      const int n_c = ao * nmo;
      for (int o = lane; o < n_c; o += 32) {
        const int b = o / nmo, m = o - b * nmo;
        const double* x = phi_s + b * kRowPad;
        const double* y = wg_s + m * kRowPad;
        double a0 = 0.0, a1 = 0.0;
#pragma unroll
        for (int q = 0; q < 32; q += 2) {
          a0 = fma(x[q], y[q], a0);
          a1 = fma(x[q + 1], y[q + 1], a1);
        }
        my[off_c + b0 * nmo + o] = fma(ang[b0 + b], a0 + a1, my[off_c + b0 * nmo + o]);
      }
      // exponents of the chunk's primitives
      const int p1 = prim_start[b0 + ao];
      for (int o = prim_start[b0] + lane; o < p1; o += 32) {
        const double* x = q_s + (slot[o] >> 8) * kRowPad;
        const double* y = rd_s + (slot[o] & 0xff) * kRowPad;
        double a0 = 0.0, a1 = 0.0;
#pragma unroll
        for (int q = 0; q < 32; q += 2) {
          a0 = fma(x[q], y[q], a0);
          a1 = fma(x[q + 1], y[q + 1], a1);
        }
        my[o] += a0 + a1;
      }
      __syncwarp();
      s0 = s;
    }
    const double v = warp_sum(wt * gw);
    if (lane == 0) my[off_w] += v;
    __syncwarp();
  }
  flush_acc(acc, n_param, partial, ld_partial, col0 + blockIdx.x);
}

bool md_grad_supported(const WfDev& wf) {
  if (wf.bf_w != 0.0) return false;
  const int ns = wf.n_up > wf.n_down ? wf.n_up : wf.n_down;
  if (ns > kMdNS || wf.n_mo > kMdNM || wf.n_exc[0] > 128 || wf.n_exc[1] > 128) return false;
  return true;
}

// shared memory of k_md_rows with n warps per block
static size_t md_rows_smem_bytes(int n_prim, int n_param, int n) {
  return sizeof(double) * n * ((size_t)n_param + kRowsBuf) + ((sizeof(unsigned short) * (size_t)n_prim + 15) & ~size_t(15));
}

size_t md_grad_smem_bytes(const WfDev& wf, int n_param) {
  return gen_table_bytes(wf) + sizeof(double) * kMdWarps * (size_t)n_param;
}

// Scratch of launch_md_grad: Gamma [n_elec][n_mo][ldm] and the partial sums
// [n_param][2 x blocks].
size_t md_grad_scratch_bytes(const WfDev& wf, int64_t ldm, int n_param, int n_sm) {
  return sizeof(double) * ((size_t)wf.n_elec * wf.n_mo * ldm + (size_t)n_param * 2 * 4 * n_sm);
}

cudaError_t launch_md_grad(const WfDev& wf, const double* walkers, int64_t W, int64_t ldw, const Workspace& ws,
                           const double* e_loc, const double* stats, int n_prim, int n_param, double* scratch,
                           double* grad, cudaStream_t st, int weight) {
  int dev = 0, n_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
  const int nb = 4 * n_sm;
  double* gam = scratch;
  double* partial = scratch + (size_t)wf.n_elec * wf.n_mo * ws.ldm;
  const int64_t ldp = 2 * nb;
  // parameter blocks of qmc_param_layout: exponents (n_prim), MO
  // coefficients, CI weights, Jastrow b, backflow w
  const int off_d = n_prim + wf.n_ao * wf.n_mo;
  const size_t smem_a = sizeof(double) * kMdWarps * (size_t)n_param;
  cudaError_t e = cudaFuncSetAttribute(k_md_gamma, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_a);
  if (e != cudaSuccess) return e;
  k_md_gamma<<<nb, kMdThreads, smem_a, st>>>(wf, walkers, W, ldw, ws.mo, ws.nmp, ws.ldm, e_loc, stats, weight,
                                             n_param, off_d, gam, partial, ldp);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  // warps per block: four (two blocks of them per SM for CO's 1,008
  // parameters), fewer where a warp's parameter sums are too many
  int warps = kMdWarps;
  while (warps > 1 && md_rows_smem_bytes(n_prim, n_param, warps) > 227 * 1024) warps /= 2;
  const size_t smem_b = md_rows_smem_bytes(n_prim, n_param, warps);
  e = cudaFuncSetAttribute(k_md_rows, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_b);
  if (e != cudaSuccess) return e;
  k_md_rows<<<nb, 32 * warps, smem_b, st>>>(wf, walkers, W, ldw, gam, ws.ldm, e_loc, stats, weight, wf.ao_ang,
                                            wf.ao_prim, n_param, partial, ldp, nb);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return launch_row_sums(partial, n_param, (int)ldp, grad, st);
}

}  // namespace qmc
