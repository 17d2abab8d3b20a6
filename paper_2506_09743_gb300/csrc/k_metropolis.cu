// Metropolis-Hastings walker step (App. B): Gaussian proposal moving all
// electrons at once, acceptance min(1, |Psi'/Psi|^2) in log form.
//
// Random numbers: Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11) with
// key (seed lo, seed hi) and counter (block j, walker, step lo, step hi).
// Block j gives Gaussians 4j..4j+3 by Box-Muller on the word pairs
// (x0, x1), (x2, x3) with u(x) = (x + 0.5) 2^-32; block ceil(3N/4) word 0 is
// the acceptance uniform.  Both kernels regenerate their numbers from the
// counter, so nothing random is stored between them.  The step index is
// gstep plus, when gctr is not null, a device counter: a CUDA graph of one
// step is then replayed, and the kernels advance the counter themselves: the
// proposal reads gctr[0] and writes gctr[1] = gctr[0] + 1, the acceptance reads
// gctr[1] and writes it back to gctr[0] (each word has one writer, and its
// readers run in the kernel after it).  A one-thread kernel of its own took
// 1.5 us and a launch a step.
#include <cmath>
#include <mutex>
#include <vector>

#include "boxmuller.cuh"
#include "qmc_internal.cuh"

namespace qmc {

namespace {

__device__ double2 g_bm_sincos[kBmN];
__device__ double2 g_bm_log[kBmN];

__device__ __forceinline__ BmTables tables_here() { return BmTables{g_bm_sincos, g_bm_log}; }

}  // namespace

cudaError_t init_box_muller_tables() {
  static std::mutex mu;
  static std::vector<int> done;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lock(mu);
  for (int d : done)
    if (d == dev) return cudaSuccess;
  std::vector<double> sc(2 * kBmN), lg(2 * kBmN);
  const long double two_pi = 6.283185307179586476925286766559L;
  for (int j = 0; j < kBmN; ++j) {
    const long double a = two_pi * (long double)j / (long double)kBmN;
    sc[2 * j] = (double)sinl(a);
    sc[2 * j + 1] = (double)cosl(a);
    const long double m = 1.0L + (long double)j / (long double)kBmN;
    lg[2 * j] = (double)logl(m);
    lg[2 * j + 1] = (double)(1.0L / m);
  }
  e = cudaMemcpyToSymbol(g_bm_sincos, sc.data(), sizeof(double) * sc.size());
  if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_bm_log, lg.data(), sizeof(double) * lg.size());
  if (e == cudaSuccess) done.push_back(dev);
  return e;
}

cudaError_t box_muller_tables(BmTables* t) {
  void *a = nullptr, *b = nullptr;
  cudaError_t e = cudaGetSymbolAddress(&a, g_bm_sincos);
  if (e == cudaSuccess) e = cudaGetSymbolAddress(&b, g_bm_log);
  *t = BmTables{static_cast<const double2*>(a), static_cast<const double2*>(b)};
  return e;
}

// One thread per walker and Philox block (four coordinates).  The kernel is
// bound by the FP64 work of the Gaussians, about 30 instructions a pair; with
// one thread for a walker's whole vector a batch of 16,384 CO walkers filled
// 84% of the SM partitions with one warp each, a serial chain of 11 blocks.
__global__ void __launch_bounds__(128) k_propose(int n3, const double* __restrict__ walkers, int64_t W, int64_t ldw,
                                                 double* __restrict__ prop, int64_t ldm, double step, uint64_t seed,
                                                 uint64_t first_walker, uint64_t gstep,
                                                 unsigned long long* __restrict__ gctr) {
  const int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (w >= W) return;
  if (gctr) {
    gstep += gctr[0];
    if (w == 0 && blockIdx.y == 0) gctr[1] = gctr[0] + 1ull;
  }
  const uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
  const uint32_t wi = (uint32_t)(first_walker + (uint64_t)w);
  const int j = blockIdx.y;
  const u4 x = philox4x32_10(u4{(uint32_t)j, wi, (uint32_t)gstep, (uint32_t)(gstep >> 32)}, k0, k1);
  double z[4];
  box_muller4(tables_here(), x, z);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int k = 4 * j + q;
    if (k < n3) prop[(int64_t)k * ldm + w] = walkers[(int64_t)k * ldw + w] + step * z[q];
  }
}

__global__ void __launch_bounds__(128) k_accept(int n3, double* __restrict__ walkers, int64_t W, int64_t ldw,
                                                const double* __restrict__ prop, int64_t ldm,
                                                double* __restrict__ lp, const double* __restrict__ lp_new,
                                                uint64_t seed, uint64_t first_walker, uint64_t gstep,
                                                unsigned long long* __restrict__ gctr,
                                                int64_t* __restrict__ n_accept) {
  const int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (w >= W) return;
  if (gctr) {
    gstep += gctr[1] - 1ull;
    if (w == 0) gctr[0] = gctr[1];
  }
  const uint32_t wi = (uint32_t)(first_walker + (uint64_t)w);
  const int nblk = (n3 + 3) / 4;
  const u4 x = philox4x32_10(u4{(uint32_t)nblk, wi, (uint32_t)gstep, (uint32_t)(gstep >> 32)}, (uint32_t)seed,
                             (uint32_t)(seed >> 32));
  const double lnew = lp_new[w], lold = lp[w];
  if (log(u01(x.x)) < 2.0 * (lnew - lold)) {
    for (int k = 0; k < n3; ++k) walkers[(int64_t)k * ldw + w] = prop[(int64_t)k * ldm + w];
    lp[w] = lnew;
    if (n_accept) n_accept[w] += 1;
  }
}

// Initial walkers for the serving loop: electron i at R_home(i) + N(0, 1) per
// coordinate, Gaussians from the same Philox stream layout with the reserved
// step index 2^64 - 1 (never reached by a chain).
__global__ void __launch_bounds__(128) k_init_walkers(InitSpec spec, int64_t W, int64_t ldw,
                                                      double* __restrict__ walkers, uint64_t seed) {
  const int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (w >= W) return;
  const int n3 = 3 * spec.n_elec;
  for (int j = 0; 4 * j < n3; ++j) {
    const u4 x = philox4x32_10(u4{(uint32_t)j, (uint32_t)w, 0xFFFFFFFFu, 0xFFFFFFFFu}, (uint32_t)seed,
                               (uint32_t)(seed >> 32));
    double z[4];
    box_muller4(tables_here(), x, z);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int k = 4 * j + q;
      if (k < n3) walkers[(int64_t)k * ldw + w] = spec.home_xyz[k / 3][k % 3] + z[q];
    }
  }
}

// sum of the per-walker acceptance counts into out[0] (fixed order)
__global__ void k_sum_counts(const int64_t* __restrict__ c, int64_t W, double* __restrict__ out) {
  __shared__ long long red[256];
  long long s = 0;
  for (int64_t k = threadIdx.x; k < W; k += blockDim.x) s += c[k];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[0] = (double)red[0];
}

cudaError_t launch_init_walkers(const InitSpec& spec, int64_t W, int64_t ldw, double* walkers, uint64_t seed,
                                cudaStream_t st) {
  if (W == 0) return cudaSuccess;
  k_init_walkers<<<(unsigned)((W + 127) / 128), 128, 0, st>>>(spec, W, ldw, walkers, seed);
  return cudaGetLastError();
}

cudaError_t launch_sum_counts(const int64_t* counts, int64_t W, double* out, cudaStream_t st) {
  k_sum_counts<<<1, 256, 0, st>>>(counts, W, out);
  return cudaGetLastError();
}

cudaError_t launch_propose(const WfDev& wf, const double* walkers, int64_t W, int64_t ldw, const Workspace& ws,
                           double step, uint64_t seed, uint64_t first_walker, uint64_t gstep, uint64_t* gctr,
                           cudaStream_t st) {
  if (W == 0) return cudaSuccess;
  const dim3 grid((unsigned)((W + 127) / 128), (unsigned)((3 * wf.n_elec + 3) / 4));
  k_propose<<<grid, 128, 0, st>>>(3 * wf.n_elec, walkers, W, ldw, ws.prop, ws.ldm, step, seed, first_walker, gstep,
                                  reinterpret_cast<unsigned long long*>(gctr));
  return cudaGetLastError();
}

cudaError_t launch_accept(const WfDev& wf, double* walkers, int64_t W, int64_t ldw, const Workspace& ws,
                          uint64_t seed, uint64_t first_walker, uint64_t gstep, uint64_t* gctr,
                          int64_t* n_accept, cudaStream_t st) {
  if (W == 0) return cudaSuccess;
  k_accept<<<(unsigned)((W + 127) / 128), 128, 0, st>>>(3 * wf.n_elec, walkers, W, ldw, ws.prop, ws.ldm, ws.lp,
                                                         ws.lp_new, seed, first_walker, gstep,
                                                         reinterpret_cast<unsigned long long*>(gctr), n_accept);
  return cudaGetLastError();
}

}  // namespace qmc
