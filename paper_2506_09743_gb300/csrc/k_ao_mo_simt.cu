// AO evaluation fused with the AO->MO contraction on the SIMT pipes.
//
// One thread per (walker, electron): evaluates every shell's radial factor
// once, every AO's value and kinetic channel, and accumulates
// Phi_{i,m} = sum_b phi_b C_{b,m} (Sec. 2.1, MO layer) for both channels in
// registers.  The MO table sits in shared memory and is read as a warp-wide
// broadcast.  Used by the FP64 and FP32 forms (the mixed forms run the
// contraction on tcgen05, k_ao_mo_tc.cu).
//
// FP64 form.  The kernel is bound by the FP64 pipe, so its instruction count is
// the time: complete s, p and d shells take closed forms that leave out what
// the general monomials multiply by zero and one (the operations that remain
// are those of the general path, with the same roundings), and 2 alpha and
// 4 alpha^2 of a primitive come from a table.  FAST takes the exponential of
// fp64_math.cuh (7 instructions) instead of the library's (about 19).
// CO, 16,384 walkers: 1,954 us with the general path, 1,560 us with the closed
// forms (the same bits); 65,536: 7.78 ms, 5.12 ms with FAST.
#include <type_traits>

#include "ao_eval.cuh"
#include "fp64_math.cuh"

namespace qmc {

namespace {

// kinetic channel f lap P + P RL + 2 gJ . grad of an AO from its gradient, in
// the general path's order of roundings (h = f lap P + P RL)
__device__ __forceinline__ double kin_from(double h, double gx, double gy, double gz, double gjx, double gjy,
                                           double gjz) {
  return fma(2.0, fma(gjz, gz, fma(gjx, gx, __dmul_rn(gjy, gy))), h);
}

}  // namespace

template <typename T, int NMO, int NCH, bool FAST>
__global__ void __launch_bounds__(128) k_ao_mo_simt(WfDev wf, const double* __restrict__ walkers, int64_t W,
                                                    int64_t ldw, const T* __restrict__ gradJ,
                                                    double* __restrict__ mo_out, int nmp, int64_t ldm) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  ShellDev* sh_s = reinterpret_cast<ShellDev*>(smem_raw);
  int* pow_s = reinterpret_cast<int*>(sh_s + wf.n_shell);
  T* C_s = reinterpret_cast<T*>(smem_raw + round_up(sizeof(ShellDev) * wf.n_shell + sizeof(int) * wf.n_ao, 16));
  constexpr bool F64 = std::is_same<T, double>::value;
  // FP64: per shell and primitive 2 alpha, 4 alpha^2, -2048 alpha / ln 2
  double* rad_s = reinterpret_cast<double*>(C_s + wf.n_ao * NMO);
  if (F64)
    for (int k = threadIdx.x; k < wf.n_shell * QMC_MAX_PRIM; k += blockDim.x) {
      const double al = wf.shells[k / QMC_MAX_PRIM].expo[k % QMC_MAX_PRIM];
      rad_s[3 * k] = 2.0 * al;
      rad_s[3 * k + 1] = __dmul_rn(4.0 * al, al);
      if (FAST) rad_s[3 * k + 2] = wf.nak[k];
    }
  const T* Cg = sizeof(T) == 8 ? reinterpret_cast<const T*>(wf.mo64) : reinterpret_cast<const T*>(wf.mo32);
  for (int k = threadIdx.x; k < wf.n_shell * (int)(sizeof(ShellDev) / 4); k += blockDim.x)
    reinterpret_cast<int*>(sh_s)[k] = reinterpret_cast<const int*>(wf.shells)[k];
  for (int k = threadIdx.x; k < wf.n_ao; k += blockDim.x) pow_s[k] = wf.ao_pow[k];
  for (int k = threadIdx.x; k < wf.n_ao * NMO; k += blockDim.x) {
    const int b = k / NMO, m = k % NMO;
    C_s[k] = m < wf.n_mo ? Cg[b * wf.n_mo + m] : T(0);
  }
  __syncthreads();

  const int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int i = blockIdx.y;
  if (w >= W) return;
  const double rx = walkers[(int64_t)(3 * i) * ldw + w];
  const double ry = walkers[(int64_t)(3 * i + 1) * ldw + w];
  const double rz = walkers[(int64_t)(3 * i + 2) * ldw + w];
  T gjx = T(0), gjy = T(0), gjz = T(0);
  if (NCH == 2) {
    gjx = gradJ[(int64_t)(3 * i) * ldm + w];
    gjy = gradJ[(int64_t)(3 * i + 1) * ldm + w];
    gjz = gradJ[(int64_t)(3 * i + 2) * ldm + w];
  }
  T acc0[NMO], acc1[NMO];
#pragma unroll
  for (int m = 0; m < NMO; ++m) { acc0[m] = T(0); acc1[m] = T(0); }

  int cur_atom = -1;
  T dx = T(0), dy = T(0), dz = T(0), r2 = T(0), rho = T(0), irho = T(0);
  T px[5], py[5], pz[5];
  bool have_pow = false;
  for (int s = 0; s < wf.n_shell; ++s) {
    const ShellDev& sh = sh_s[s];
    if (sh.atom != cur_atom) {
      cur_atom = sh.atom;
      displacement(rx, ry, rz, wf.atom_xyz[cur_atom], dx, dy, dz);
      // (the products are rounded before the sums, except with FAST: earlier
      // builds shared them with the power tables, and energies of expansions
      // keep those bits)
      if constexpr (FAST) r2 = dx * dx + dy * dy + dz * dz;
      else if constexpr (F64) r2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
      else r2 = __fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)), __fmul_rn(dz, dz));
      if (wf.any_sto) {  // Gaussians need r2 alone
        irho = T(1) / sqrt(r2);
        rho = r2 * irho;
      }
      have_pow = false;
    }
    T f, g1, f2;
    if constexpr (F64) {
      const double* rad = rad_s + 3 * QMC_MAX_PRIM * s;
      if (sh.kind == 0) {
        if (FAST) {
          f = sh.coef[0] * exp_scaled(rad[2], rho, wf.exp2_tab);
          for (int k = 0; k < sh.kn; ++k) f *= rho;
          const double q = (double)sh.kn * irho - sh.expo[0];
          g1 = q * f * irho;
          f2 = (q * q - (double)sh.kn * irho * irho) * f;
        } else {
          shell_radial(sh, r2, rho, irho, f, g1, f2, NCH == 2);
        }
      } else {
        f = 0.0;
        g1 = 0.0;
        f2 = 0.0;
        for (int p = 0; p < sh.n_prim; ++p) {
          const double a2 = rad[3 * p], a4 = rad[3 * p + 1];
          const double ex = FAST ? exp_scaled(rad[3 * p + 2], r2, wf.exp2_tab) : exp(-sh.expo[p] * r2);
          const double e = __dmul_rn(sh.coef[p], ex);
          f = __dadd_rn(f, e);
          if (NCH == 2) {
            g1 = fma(-a2, e, g1);
            f2 = fma(fma(a4, r2, -a2), e, f2);
          }
        }
      }
    } else {
      shell_radial(sh, r2, rho, irho, f, g1, f2, NCH == 2);
    }
    const T radial_lap = f2 + T(2 * (sh.l + 1)) * g1;
    if constexpr (F64) {
      if (sh.canon) {
        auto emit = [&](int b, double v, double kin) {
          const double* Cb = C_s + b * NMO;
#pragma unroll
          for (int m = 0; m < NMO; ++m) {
            const double c = Cb[m];
            acc0[m] += v * c;
            if (NCH == 2) acc1[m] += kin * c;
          }
        };
        const int b0 = sh.ao_first;
        if (sh.canon == 1) {
          emit(b0, f, NCH == 2 ? kin_from(radial_lap, __dmul_rn(g1, dx), __dmul_rn(g1, dy), __dmul_rn(g1, dz), gjx, gjy, gjz)
                               : 0.0);
          continue;
        }
        if (sh.canon == 2) {
          for (int k = 0; k < 3; ++k) {
            const int pw = pow_s[b0 + k], c = (pw & 15) ? 0 : ((pw >> 4) & 15) ? 1 : 2;
            const double x = c == 0 ? dx : c == 1 ? dy : dz;
            double kin = 0.0;
            if (NCH == 2) {
              const double t = __dmul_rn(x, g1);
              double gx = __dmul_rn(t, dx), gy = __dmul_rn(t, dy), gz = __dmul_rn(t, dz);
              if (c == 0) gx = fma(t, dx, f);
              else if (c == 1) gy = fma(t, dy, f);
              else gz = fma(t, dz, f);
              kin = kin_from(__dmul_rn(x, radial_lap), gx, gy, gz, gjx, gjy, gjz);
            }
            emit(b0 + k, __dmul_rn(x, f), kin);
          }
          continue;
        }
        const double fx = __dmul_rn(f, dx), fy = __dmul_rn(f, dy), fz = __dmul_rn(f, dz);
        for (int k = 0; k < 6; ++k) {
          const int pw = pow_s[b0 + k], a = pw & 15, bb = (pw >> 4) & 15, cc = (pw >> 8) & 15;
          double P, kin = 0.0;
          if (a == 2) {
            P = __dmul_rn(dx, dx);
            if (NCH == 2) {
              const double t = __dmul_rn(P, g1);
              kin = kin_from(fma(P, radial_lap, 2.0 * f), fma(t, dx, 2.0 * fx), __dmul_rn(t, dy), __dmul_rn(t, dz), gjx,
                             gjy, gjz);
            }
          } else if (bb == 2) {
            P = __dmul_rn(dy, dy);
            if (NCH == 2) {
              const double t = __dmul_rn(P, g1);
              kin = kin_from(fma(P, radial_lap, 2.0 * f), __dmul_rn(t, dx), fma(t, dy, 2.0 * fy), __dmul_rn(t, dz), gjx,
                             gjy, gjz);
            }
          } else if (cc == 2) {
            P = __dmul_rn(dz, dz);
            if (NCH == 2) {
              const double t = __dmul_rn(P, g1);
              kin = kin_from(fma(P, radial_lap, 2.0 * f), __dmul_rn(t, dx), __dmul_rn(t, dy), fma(t, dz, 2.0 * fz), gjx,
                             gjy, gjz);
            }
          } else if (cc == 0) {  // xy
            P = __dmul_rn(dx, dy);
            if (NCH == 2) {
              const double t = __dmul_rn(P, g1);
              kin = kin_from(__dmul_rn(P, radial_lap), fma(t, dx, fy), fma(t, dy, fx), __dmul_rn(t, dz), gjx, gjy, gjz);
            }
          } else if (bb == 0) {  // xz
            P = __dmul_rn(dx, dz);
            if (NCH == 2) {
              const double t = __dmul_rn(P, g1);
              kin = kin_from(__dmul_rn(P, radial_lap), fma(t, dx, fz), __dmul_rn(t, dy), fma(t, dz, fx), gjx, gjy, gjz);
            }
          } else {  // yz
            P = __dmul_rn(dy, dz);
            if (NCH == 2) {
              const double t = __dmul_rn(P, g1);
              kin = kin_from(__dmul_rn(P, radial_lap), __dmul_rn(t, dx), fma(t, dy, fz), fma(t, dz, fy), gjx, gjy, gjz);
            }
          }
          emit(b0 + k, __dmul_rn(P, f), kin);
        }
        continue;
      }
    }
    if (!have_pow) {
      pow_table(dx, px); pow_table(dy, py); pow_table(dz, pz);
      have_pow = true;
    }
    for (int k = 0; k < sh.n_ao; ++k) {
      const int b = sh.ao_first + k;
      T P, Px, Py, Pz, lapP;
      angular(pow_s[b], px, py, pz, P, Px, Py, Pz, lapP, NCH == 2);
      const T v = P * f;
      T kin = T(0);
      if (NCH == 2) {
        const T gx = f * Px + P * g1 * dx, gy = f * Py + P * g1 * dy, gz = f * Pz + P * g1 * dz;
        kin = f * lapP + P * radial_lap + T(2) * (gjx * gx + gjy * gy + gjz * gz);
      }
      const T* Cb = C_s + b * NMO;
#pragma unroll
      for (int m = 0; m < NMO; ++m) {
        const T c = Cb[m];
        acc0[m] += v * c;
        if (NCH == 2) acc1[m] += kin * c;
      }
    }
  }
  // walker-fastest FP64 MO layout [N][NCH][nmp][ldm] (FP32 results widened exactly)
  double* dst = mo_out + (size_t)i * NCH * nmp * ldm + w;
#pragma unroll
  for (int m = 0; m < NMO; ++m) {
    dst[(size_t)m * ldm] = widen(acc0[m]);
    if (NCH == 2) dst[(size_t)(nmp + m) * ldm] = widen(acc1[m]);
  }
}

template <typename T, bool FAST>
static cudaError_t launch_t(const WfDev& wf, const double* walkers, int64_t W, int64_t ldw, const Workspace& ws,
                            int nch, cudaStream_t st) {
  const dim3 block(128), grid((unsigned)((W + 127) / 128), (unsigned)wf.n_elec);
  const T* gj = static_cast<const T*>(ws.gradJ);
  double* mo = ws.mo;
  const size_t rad = sizeof(T) == 8 ? sizeof(double) * 3 * QMC_MAX_PRIM * (size_t)wf.n_shell : 0;
#define QMC_AOMO(NM)                                                                                        \
  if (wf.n_col <= NM) {                                                                                     \
    const size_t smem = round_up(sizeof(ShellDev) * wf.n_shell + sizeof(int) * wf.n_ao, 16) +              \
                        sizeof(T) * wf.n_ao * NM + rad;                                                     \
    if (nch == 2) {                                                                                         \
      auto kern = k_ao_mo_simt<T, NM, 2, FAST>;                                                             \
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);                   \
      kern<<<grid, block, smem, st>>>(wf, walkers, W, ldw, gj, mo, ws.nmp, ws.ldm);                         \
    } else {                                                                                                \
      auto kern = k_ao_mo_simt<T, NM, 1, FAST>;                                                             \
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);                   \
      kern<<<grid, block, smem, st>>>(wf, walkers, W, ldw, gj, mo, ws.nmp, ws.ldm);                         \
    }                                                                                                       \
    return cudaGetLastError();                                                                              \
  }
  if (ws.nmp != mo_row_pad(wf.n_mo, false)) return cudaErrorInvalidValue;
  // brackets of the columns that the determinant stage reads
  QMC_AOMO(2)
  QMC_AOMO(4)
  QMC_AOMO(8)
  QMC_AOMO(14)
  QMC_AOMO(16)
  QMC_AOMO(32)
#undef QMC_AOMO
  return cudaErrorInvalidValue;
}

// fast: the exponential of fp64_math.cuh in the FP64 form
cudaError_t launch_ao_mo_simt(const WfDev& wf, int prec, const double* walkers, int64_t W, int64_t ldw,
                              const Workspace& ws, int nch, bool fast, cudaStream_t st) {
  if (W == 0) return cudaSuccess;
  if (prec != QMC_FP64) return launch_t<float, false>(wf, walkers, W, ldw, ws, nch, st);
  return fast ? launch_t<double, true>(wf, walkers, W, ldw, ws, nch, st)
              : launch_t<double, false>(wf, walkers, W, ldw, ws, nch, st);
}

}  // namespace qmc
