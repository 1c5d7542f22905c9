// Observables of the ICWF wavefunction (Eq. ansatz reconstructed on the grid) and the initial
// projection of Psi0 on the product basis.
//   obs          reduced densities rho_x, rho_R; <V>; BO projections chi^(n)(R) = int dx phi_n Psi;
//                kinetic energies by Parseval on the FFT of every grid line; final FP64 sums of
//                norm, energy, populations P_n and decoherence indicators D_nm (the quantities
//                the paper monitors in its two applications).
#include <cuda_runtime.h>

#include "icwf_internal.h"
#include "k_common.cuh"

namespace icwf {

// Deterministic block sum of one double per thread (blockDim.x = 256).
__device__ double block_sum(double v, double* red) {
  red[threadIdx.x] = v;
  __syncthreads();
  for (int s = 128; s > 0; s >>= 1) {
    if (threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
    __syncthreads();
  }
  const double r = red[0];
  __syncthreads();
  return r;
}

struct ObsArgs {
  const double2* Psi;
  const double* phi;
  int n_states;
  double* rho_x;
  double* rho_R;
  double2* proj;     // n_states x nR
  double* part;      // [0,nR): kinetic x per column; [nR,2nR): potential per column;
                     // [2nR, 2nR+nx): kinetic R per row
  const double2* twx;
  const double2* twR;
};

// Blocks [0, nR): column j (the x line at R_j); blocks [nR, nR+nx): row i (the R line at x_i).
__global__ void __launch_bounds__(256) k_obs_lines(JobView j, ObsArgs o) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double2* buf = (double2*)smem_raw;
  __shared__ double red[256];
  const bool col = blockIdx.x < (unsigned)j.nR;
  const int line = col ? blockIdx.x : blockIdx.x - j.nR;
  const int n = col ? j.nx : j.nR;
  const int logn = col ? j.logx : j.logR;
  double dens = 0.0, pot = 0.0;
  for (int e = threadIdx.x; e < n; e += blockDim.x) {
    const size_t idx = col ? (size_t)e * j.nR + line : (size_t)line * j.nR + e;
    const double2 v = o.Psi[idx];
    buf[e] = v;
    const double d = v.x * v.x + v.y * v.y;
    dens += d;
    if (col) pot += j.V[idx] * d;
  }
  __syncthreads();
  const double sd = block_sum(dens, red);
  if (col) {
    const double sp = block_sum(pot, red);
    if (threadIdx.x == 0) {
      o.rho_R[line] = j.dx * sd;
      o.part[j.nR + line] = j.dx * j.dR * sp;
    }
    for (int ns = 0; ns < o.n_states; ++ns) {
      const double* ph = o.phi + ((size_t)ns * j.nR + line) * j.nx;
      double pr = 0.0, pi = 0.0;
      for (int e = threadIdx.x; e < n; e += blockDim.x) {
        pr += ph[e] * buf[e].x;
        pi += ph[e] * buf[e].y;
      }
      const double sr = block_sum(pr, red);
      const double si = block_sum(pi, red);
      if (threadIdx.x == 0) o.proj[(size_t)ns * j.nR + line] = make_double2(j.dx * sr, j.dx * si);
    }
  } else {
    if (threadIdx.x == 0) o.rho_x[line] = j.dR * sd;
  }
  fft_dif(buf, col ? o.twx : o.twR, n, logn);
  double ek = 0.0;
  for (int mp = threadIdx.x; mp < n; mp += blockDim.x) {
    int m = (int)(__brev((unsigned)mp) >> (32 - logn));
    if (m >= n / 2) m -= n;
    ek += (buf[mp].x * buf[mp].x + buf[mp].y * buf[mp].y) * ((double)m * (double)m);
  }
  const double se = block_sum(ek, red);
  if (threadIdx.x == 0) {
    const double PI = 3.14159265358979323846;
    if (col) {
      const double g = 2.0 * PI / (j.nx * j.dx);
      o.part[line] = j.dR * (j.dx / j.nx) * se * g * g * 0.5 * j.inv_mx;
    } else {
      const double g = 2.0 * PI / (j.nR * j.dR);
      o.part[2 * j.nR + line] = j.dx * (j.dR / j.nR) * se * g * g * 0.5 * j.inv_mR;
    }
  }
}

// One CTA: out = {norm, ekx, ekR, epot}; pop[n]; decoh[n*ns + m].  A warp per sum (4 + ns + ns (ns + 1)
// / 2 of them), lanes striding over the line sums, so the sums run side by side without barriers
// (256 threads with a block reduction per sum, D_nm computed twice: 31 us at nR = 512 with cold
// caches; now 19).
constexpr int OF_WARPS = 32;
__global__ void __launch_bounds__(OF_WARPS * 32) k_obs_final(JobView j, ObsArgs o, double* out, double* pop,
                                                             double* decoh) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, ns = o.n_states;
  auto chi2 = [&](int n, int e) {
    const double2 v = o.proj[(size_t)n * j.nR + e];
    return v.x * v.x + v.y * v.y;
  };
  for (int q = warp; q < 4 + ns + ns * (ns + 1) / 2; q += OF_WARPS) {
    int n = 0, m = 0;
    if (q >= 4 + ns) {   // pair (n <= m)
      int t = q - 4 - ns;
      while (t >= ns - n) { t -= ns - n; ++n; }
      m = n + t;
    }
    const int len = q == 2 ? j.nx : j.nR;
    double s[4] = {0, 0, 0, 0};   // independent partial sums (FP64 latency)
    for (int e0 = lane; e0 < len; e0 += 128) {
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int e = e0 + 32 * k;
        if (e >= len) break;
        double v;
        if (q == 0) v = o.rho_R[e];
        else if (q == 1) v = o.part[e];
        else if (q == 2) v = o.part[2 * j.nR + e];
        else if (q == 3) v = o.part[j.nR + e];
        else if (q < 4 + ns) v = chi2(q - 4, e);
        else v = chi2(n, e) * chi2(m, e);
        s[k] += v;
      }
    }
    double t = (s[0] + s[1]) + (s[2] + s[3]);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
    if (lane != 0) continue;
    if (q == 0) out[0] = j.dR * t;
    else if (q < 4) out[q] = t;
    else if (q < 4 + ns) { if (pop) pop[q - 4] = j.dR * t; }
    else if (decoh) decoh[n * ns + m] = decoh[m * ns + n] = j.dR * t;
  }
}

void launch_obs_lines(const JobView& j, const double2* Psi, const double* phi, int n_states,
                      double* rho_x, double* rho_R, double2* proj, double* part, double* out,
                      double* pop, double* decoh, const double2* twx, const double2* twR,
                      cudaStream_t s) {
  ObsArgs o{Psi, phi, n_states, rho_x, rho_R, proj, part, twx, twR};
  const int nmax = j.nx > j.nR ? j.nx : j.nR;
  const size_t sm = (size_t)nmax * sizeof(double2);
  if (sm > 40 * 1024)
    cudaFuncSetAttribute(k_obs_lines, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  k_obs_lines<<<j.nR + j.nx, 256, sm, s>>>(j, o);
  k_obs_final<<<1, OF_WARPS * 32, 0, s>>>(j, o, out, pop, decoh);
}

// b_a = dx dR sum_i conj(psi_a(x_i)) sum_j Psi0[i, j] conj(chi_a(R_j)); one CTA per a, one warp
// per grid row i at a time.
__global__ void __launch_bounds__(256) k_init_projection(int N, int nx, int nR, double dx, double dR,
                                                         const double2* __restrict__ psi,
                                                         const double2* __restrict__ chi,
                                                         const double2* __restrict__ Psi0,
                                                         double2* __restrict__ b) {
  __shared__ double red[256];
  const int a = blockIdx.x;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const double2* ca = chi + (size_t)a * nR;
  const double2* pa = psi + (size_t)a * nx;
  double2 acc = make_double2(0, 0);
  for (int i = warp; i < nx; i += 8) {
    double2 t = make_double2(0, 0);
    const double2* row = Psi0 + (size_t)i * nR;
    for (int jj = lane; jj < nR; jj += 32) cfma(t, row[jj], cconj(ca[jj]));
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      t.x += __shfl_xor_sync(0xffffffffu, t.x, off);
      t.y += __shfl_xor_sync(0xffffffffu, t.y, off);
    }
    if (lane == 0) cfmac(acc, pa[i], t);
  }
  const double sr = block_sum(lane == 0 ? acc.x : 0.0, red);
  const double si = block_sum(lane == 0 ? acc.y : 0.0, red);
  if (threadIdx.x == 0) b[a] = make_double2(dx * dR * sr, dx * dR * si);
}

void launch_init_projection(int N, int nx, int nR, double dx, double dR, const double2* psi,
                            const double2* chi, const double2* Psi0, double2* b, cudaStream_t s) {
  k_init_projection<<<N, 256, 0, s>>>(N, nx, nR, dx, dR, psi, chi, Psi0, b);
}

}  // namespace icwf
