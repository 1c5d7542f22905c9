// Exact propagation of the two-coordinate wavefunction Psi(x, R) (Eq. TDSE without vector
// potential) by the second-order Strang split on the periodic cell-centred grid:
//   Psi <- e^{-i V dt/2} F^-1 e^{-i (kx^2/2m_x + kR^2/2m_R) dt} F e^{-i V dt/2} Psi.
// This is the reference the paper's figures compare the ICWF densities, populations and
// decoherence indicators with.  FP64; Psi row-major nx x nR (x slow).
//
// A step is two kernels, with one more at the end of a run of steps:
//   k_rows: per x row, inverse FFT along R of the step before (not at the start), the potential phase
//           (half of it at the start and the end, the whole between two steps), FFT along R;
//   k_cols: per group of CB adjacent R columns, FFT along x, the kinetic phase of (kx, kR) (both tables
//           bit-reversed, 1/n folded in), inverse FFT along x.
// Both turn around in registers: the last stages of one transform, the phase and the first stages of
// the other are one pass (fft_reg.cuh).
// Bound: FP64 instructions, 112 per point and step at 1024 x 512 (172 with radix-2 passes of eight
// instructions per butterfly, three kernels and both half phases).  50 steps and the observables there:
// 11.2 ms before, 7.45 now.
// Observables use per-row / per-CTA partial sums finished on the host in a fixed order.
#include <cuda_runtime.h>

#include <cmath>
#include <string>
#include <type_traits>
#include <vector>

#include "../../include/icwf_exact2d.h"
#include "icwf_internal.h"
#include "k_common.cuh"
#include "fft_reg.cuh"

namespace icwf {
namespace e2d {

constexpr int TPB = 256;
constexpr int MAX_STATES = 8;
// R columns per CTA of k_cols: a 32-byte sector; several CTAs per SM up to nx = 2048
constexpr int CB = 2;
using fftr::Tw;

__device__ __forceinline__ double block_sum(double v, double* red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __syncthreads();
  if (lane == 0) red[warp] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
  return s;   // valid in thread 0
}

// One x row per CTA: inverse FFT (INV), times ph (may be null), FFT (FWD).  in and out may alias.
template <int L, bool INV, bool FWD>
__global__ void __launch_bounds__(TPB) k_rows(const double2* in, double2* out, const double2* __restrict__ ph,
                                              const Tw* __restrict__ tf, const Tw* __restrict__ ti) {
  extern __shared__ __align__(16) double2 buf[];
  constexpr int n = 1 << L;
  const size_t base = (size_t)blockIdx.x * n;
  for (int j = threadIdx.x; j < n; j += blockDim.x) {
    double2 z = in[base + j];
    if (!INV && ph) z = cmul(ph[base + j], z);
    buf[fftr::pad(j)] = z;
  }
  __syncthreads();
  if (INV && FWD) {
    if (fftr::passes(L)) fftr::inv_pass<L, 3, 0>(buf, ti, 1);
    fftr::inv_passes<L, fftr::passes(L) - 1, 1>(buf, ti, 1);
    fftr::turn_space<L>(buf, tf, ti, [&](int j, double2 z) { return cmul(ph[base + j], z); });
    fftr::fwd_passes<L, 1, fftr::passes(L)>(buf, tf, 1);
    if (fftr::passes(L)) fftr::fwd_pass<L, 3, L - 3>(buf, tf, 1);
  } else if (INV) {
    fftr::inv_all<L>(buf, ti, 1);
  } else {
    fftr::fwd_all<L>(buf, tf, 1);
  }
  for (int j = threadIdx.x; j < n; j += blockDim.x) {
    double2 z = buf[fftr::pad(j)];
    if (INV && !FWD) z = cmul(ph[base + j], z);
    out[base + j] = z;
  }
}

// CB adjacent R columns per CTA (bit-reversed R frequencies after k_rows).  ENERGY false: FFT along x,
// multiply by kinx[m] kinR[col], inverse FFT along x, store.  ENERGY true: FFT along x and
// part[blockIdx.x] = sum |F|^2 (Tx[m] + TR[col]) (kinetic energy, not stored).
template <int L, bool ENERGY>
__global__ void __launch_bounds__(TPB) k_cols(double2* a, const double2* __restrict__ kinx,
                                              const double2* __restrict__ kinR, const Tw* __restrict__ tf,
                                              const Tw* __restrict__ ti, int nR, const double* __restrict__ Tx,
                                              const double* __restrict__ TR, double* part) {
  extern __shared__ __align__(16) double2 buf[];   // [CB][padded n]
  __shared__ double red[TPB / 32];
  constexpr int n = 1 << L;
  const int j0 = blockIdx.x * CB;
  for (int e = threadIdx.x; e < n * CB; e += blockDim.x) {
    const int i = e / CB, c = e % CB;
    buf[c * fftr::padded(n) + fftr::pad(i)] = a[(size_t)i * nR + j0 + c];
  }
  __syncthreads();
  fftr::fwd_passes<L, 0, fftr::passes(L)>(buf, tf, CB);
  if (!ENERGY) {
    double2 kr[CB];
#pragma unroll
    for (int c = 0; c < CB; ++c) kr[c] = kinR[j0 + c];
    fftr::turn_freq<L>(buf, tf, ti, CB, [&](int c, int m, double2 z) {
      double2 k = kr[0];
#pragma unroll
      for (int q = 1; q < CB; ++q) if (c == q) k = kr[q];
      return cmul(z, cmul(kinx[m], k));
    });
    fftr::inv_passes<L, fftr::passes(L) - 1, 0>(buf, ti, CB);
    for (int e = threadIdx.x; e < n * CB; e += blockDim.x) {
      const int i = e / CB, c = e % CB;
      a[(size_t)i * nR + j0 + c] = buf[c * fftr::padded(n) + fftr::pad(i)];
    }
  } else {
    fftr::fwd_pass<L, 3, L - 3>(buf, tf, CB);
    double s = 0.0;
    for (int e = threadIdx.x; e < n * CB; e += blockDim.x) {
      const int c = e >> L, m = e & (n - 1);
      const double2 z = buf[c * fftr::padded(n) + fftr::pad(m)];
      s += (z.x * z.x + z.y * z.y) * (Tx[m] + TR[j0 + c]);
    }
    s = block_sum(s, red);
    if (threadIdx.x == 0) part[blockIdx.x] = s;
  }
}

int smem_rows(int n) { return fftr::padded(n) * (int)sizeof(double2); }
int smem_cols(int n) { return CB * smem_rows(n); }
// a thread per group of eight points, up to TPB
int threads(int points) { return points / 8 < 32 ? 32 : (points / 8 > TPB ? TPB : points / 8); }

// f(std::integral_constant<int, L>) for L = log2 of a grid of 8 .. 4096 points
template <typename F>
void by_size(int L, const F& f) {
  switch (L) {
    case 3: f(std::integral_constant<int, 3>()); break;
    case 4: f(std::integral_constant<int, 4>()); break;
    case 5: f(std::integral_constant<int, 5>()); break;
    case 6: f(std::integral_constant<int, 6>()); break;
    case 7: f(std::integral_constant<int, 7>()); break;
    case 8: f(std::integral_constant<int, 8>()); break;
    case 9: f(std::integral_constant<int, 9>()); break;
    case 10: f(std::integral_constant<int, 10>()); break;
    case 11: f(std::integral_constant<int, 11>()); break;
    case 12: f(std::integral_constant<int, 12>()); break;
  }
}
template <bool INV, bool FWD>
void rows(int nx, int nR, int logR, const double2* in, double2* out, const double2* ph, const Tw* tf, const Tw* ti,
          cudaStream_t s) {
  by_size(logR, [&](auto L) {
    k_rows<L(), INV, FWD><<<nx, threads(nR), smem_rows(nR), s>>>(in, out, ph, tf, ti);
  });
}
template <bool ENERGY>
void cols(int nx, int nR, int logx, double2* a, const double2* kinx, const double2* kinR, const Tw* tf, const Tw* ti,
          const double* Tx, const double* TR, double* part, cudaStream_t s) {
  by_size(logx, [&](auto L) {
    k_cols<L(), ENERGY><<<nR / CB, threads(CB * nx), smem_cols(nx), s>>>(a, kinx, kinR, tf, ti, nR, Tx, TR, part);
  });
}
// the largest dynamic shared memory any handle uses, so that handles of different sizes can coexist
void attributes() {
  for (int l = 3; l <= 12; ++l)
    by_size(l, [&](auto L) {
      const int r = smem_rows(1 << L()), c = smem_cols(1 << L());
      cudaFuncSetAttribute(k_rows<L(), false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, r);
      cudaFuncSetAttribute(k_rows<L(), true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, r);
      cudaFuncSetAttribute(k_rows<L(), true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, r);
      cudaFuncSetAttribute(k_cols<L(), false>, cudaFuncAttributeMaxDynamicSharedMemorySize, c);
      cudaFuncSetAttribute(k_cols<L(), true>, cudaFuncAttributeMaxDynamicSharedMemorySize, c);
    });
}

// Per x row: dens[i] = sum_j |Psi|^2, pot[i] = sum_j |Psi|^2 V.
__global__ void __launch_bounds__(TPB) k_dens_rows(const double2* __restrict__ psi,
                                                   const double* __restrict__ V, int nR,
                                                   double* dens, double* pot) {
  __shared__ double red[TPB / 32];
  const size_t base = (size_t)blockIdx.x * nR;
  double s = 0.0, p = 0.0;
  for (int j = threadIdx.x; j < nR; j += blockDim.x) {
    const double2 z = psi[base + j];
    const double d = z.x * z.x + z.y * z.y;
    s += d;
    p += d * V[base + j];
  }
  s = block_sum(s, red);
  if (threadIdx.x == 0) dens[blockIdx.x] = s;
  p = block_sum(p, red);
  if (threadIdx.x == 0) pot[blockIdx.x] = p;
}

// Per R column j: dens[j] = sum_i |Psi|^2 and, for n < ns, proj[n][j] = sum_i phi[n][j][i] Psi[i][j].
__global__ void __launch_bounds__(TPB) k_cols_obs(const double2* __restrict__ psi, int nx, int nR,
                                                  const double* __restrict__ phi, int ns,
                                                  double* dens, double2* proj) {
  __shared__ double red[TPB / 32];
  const int j = blockIdx.x;
  double s = 0.0;
  double pr[MAX_STATES], pi[MAX_STATES];
#pragma unroll
  for (int n = 0; n < MAX_STATES; ++n) pr[n] = pi[n] = 0.0;
  for (int i = threadIdx.x; i < nx; i += blockDim.x) {
    const double2 z = psi[(size_t)i * nR + j];
    s += z.x * z.x + z.y * z.y;
#pragma unroll
    for (int n = 0; n < MAX_STATES; ++n) {
      if (n < ns) {
        const double f = phi[((size_t)n * nR + j) * nx + i];
        pr[n] += f * z.x;
        pi[n] += f * z.y;
      }
    }
  }
  s = block_sum(s, red);
  if (threadIdx.x == 0) dens[j] = s;
#pragma unroll
  for (int n = 0; n < MAX_STATES; ++n) {
    if (n < ns) {   // uniform over the block
      const double a = block_sum(pr[n], red);
      const double b = block_sum(pi[n], red);
      if (threadIdx.x == 0) proj[(size_t)n * nR + j] = make_double2(a, b);
    }
  }
}

int ilog2i(int n) {
  int l = 0;
  while ((1 << l) < n) ++l;
  return l;
}

// kin[mp] = e^{-i k^2 dt / 2m} / n and T[mp] = k^2 / 2m at bit-reversed position mp; tf, ti: forward
// twiddles by block, inverse ones by position.
void tables(int n, double d, double mass, double dt, std::vector<double2>& kin, std::vector<double>& T,
            std::vector<Tw>& tf, std::vector<Tw>& ti) {
  const int logn = ilog2i(n);
  const double PI = 3.14159265358979323846;
  kin.resize(n);
  T.resize(n);
  tf.resize(n / 2);
  ti.resize(n / 2);
  for (int mp = 0; mp < n; ++mp) {
    int m = 0;
    for (int b = 0; b < logn; ++b)
      if (mp & (1 << b)) m |= 1 << (logn - 1 - b);
    const int mm = m < n / 2 ? m : m - n;
    const double k = 2.0 * PI * (double)mm / ((double)n * d);
    const double e = k * k / (2.0 * mass);
    T[mp] = e;
    kin[mp] = make_double2(std::cos(-e * dt) / n, std::sin(-e * dt) / n);
  }
  // w = m (1 + i r), or -i m (1 + i r) i = m (1 + i r) with cos, sin of the angle minus 90 degrees
  auto entry = [](double angle, int form) {
    const double c = std::cos(angle), sn = std::sin(angle);
    return form ? Tw{sn, -c / sn} : Tw{c, sn / c};
  };
  for (int k = 0; k < n / 2; ++k) {
    double v = 0.0;
    for (int b = 0; b < logn - 1; ++b)
      if (k & (1 << b)) v += std::ldexp(1.0, -1 - b);
    tf[k] = entry(-PI * v, fftr::fwd_form(k));
    ti[k] = entry(2.0 * PI * (double)k / (double)n, fftr::inv_form(k, logn));
  }
}

}  // namespace e2d
}  // namespace icwf

using namespace icwf;

struct icwf_exact2d_ctx {
  int nx = 0, nR = 0, logx = 0, logR = 0, ns = 0;
  double dx = 0, dR = 0, dt = 0, t = 0;
  bool has_state = false;
  cudaStream_t stream = nullptr;
  std::vector<void*> allocs;
  double* V = nullptr;
  double2 *half = nullptr, *full = nullptr, *psi = nullptr, *work = nullptr;   // phases of V dt/2, V dt
  double2 *kinx = nullptr, *kinR = nullptr;
  e2d::Tw *tfx = nullptr, *tix = nullptr, *tfR = nullptr, *tiR = nullptr;
  double *Tx = nullptr, *TR = nullptr, *phi = nullptr;
  double *dens_x = nullptr, *pot = nullptr, *dens_R = nullptr, *part = nullptr;
  double2* proj = nullptr;
  std::string err;
};

namespace {

std::string g_err2;

icwf_status fail2(icwf_exact2d h, icwf_status st, const std::string& msg) {
  if (h) h->err = msg;
  else g_err2 = msg;
  return st;
}

template <typename T>
bool dalloc(icwf_exact2d h, T** p, size_t count) {
  void* q = nullptr;
  if (cudaMalloc(&q, count * sizeof(T)) != cudaSuccess) return false;
  h->allocs.push_back(q);
  *p = (T*)q;
  return true;
}

void release(icwf_exact2d h) {
  for (void* p : h->allocs) cudaFree(p);
  h->allocs.clear();
  if (h->stream) cudaStreamDestroy(h->stream);
  h->stream = nullptr;
}

icwf_status sync(icwf_exact2d h, const char* what) {
  const cudaError_t e = cudaStreamSynchronize(h->stream);
  if (e != cudaSuccess) return fail2(h, ICWF_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
  const cudaError_t l = cudaGetLastError();
  if (l != cudaSuccess) return fail2(h, ICWF_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(l));
  return ICWF_OK;
}

bool pow2_in(int n) { return n >= 8 && n <= 4096 && (n & (n - 1)) == 0; }

// copies ordered with the handle's (non-blocking) stream, complete on return
bool copy(icwf_exact2d h, void* dst, const void* src, size_t bytes, cudaMemcpyKind kind) {
  return cudaMemcpyAsync(dst, src, bytes, kind, h->stream) == cudaSuccess &&
         cudaStreamSynchronize(h->stream) == cudaSuccess;
}

}  // namespace

extern "C" {

icwf_status icwf_exact2d_create(const icwf_params* p, const double* V, icwf_exact2d* out) {
  if (!p || !V || !out) return fail2(nullptr, ICWF_ERR_ARG, "icwf_exact2d_create: null pointer");
  *out = nullptr;
  if (!pow2_in(p->nx) || !pow2_in(p->nR))
    return fail2(nullptr, ICWF_ERR_ARG, "icwf_exact2d_create: nx, nR must be powers of two in [8, 4096]");
  if (!(p->x_max > p->x_min) || !(p->R_max > p->R_min) || !(p->mass_x > 0) || !(p->mass_R > 0) ||
      !(p->dt > 0))
    return fail2(nullptr, ICWF_ERR_ARG, "icwf_exact2d_create: bad extents, masses or dt");
  icwf_exact2d h = new icwf_exact2d_ctx;
  h->nx = p->nx;
  h->nR = p->nR;
  h->logx = e2d::ilog2i(p->nx);
  h->logR = e2d::ilog2i(p->nR);
  h->dx = (p->x_max - p->x_min) / p->nx;
  h->dR = (p->R_max - p->R_min) / p->nR;
  h->dt = p->dt;
  const size_t NN = (size_t)h->nx * h->nR;
  if (cudaStreamCreateWithFlags(&h->stream, cudaStreamNonBlocking) != cudaSuccess) {
    delete h;
    return fail2(nullptr, ICWF_ERR_CUDA, "icwf_exact2d_create: cudaStreamCreate failed");
  }
  const int ncb = h->nR / e2d::CB;
  if (!dalloc(h, &h->V, NN) || !dalloc(h, &h->half, NN) || !dalloc(h, &h->full, NN) || !dalloc(h, &h->psi, NN) ||
      !dalloc(h, &h->work, NN) || !dalloc(h, &h->kinx, h->nx) || !dalloc(h, &h->kinR, h->nR) ||
      !dalloc(h, &h->tfx, h->nx / 2) || !dalloc(h, &h->tix, h->nx / 2) ||
      !dalloc(h, &h->tfR, h->nR / 2) || !dalloc(h, &h->tiR, h->nR / 2) ||
      !dalloc(h, &h->Tx, h->nx) || !dalloc(h, &h->TR, h->nR) || !dalloc(h, &h->dens_x, h->nx) ||
      !dalloc(h, &h->pot, h->nx) || !dalloc(h, &h->dens_R, h->nR) || !dalloc(h, &h->part, ncb) ||
      !dalloc(h, &h->proj, (size_t)e2d::MAX_STATES * h->nR)) {
    release(h);
    delete h;
    return fail2(nullptr, ICWF_ERR_OOM, "icwf_exact2d_create: cudaMalloc failed");
  }
  std::vector<double2> half(NN), full(NN), kx, kR;
  std::vector<e2d::Tw> fx, ix, fR, iR;
  std::vector<double> Tx, TR;
  for (size_t e = 0; e < NN; ++e) {
    half[e] = make_double2(std::cos(-0.5 * p->dt * V[e]), std::sin(-0.5 * p->dt * V[e]));
    full[e] = make_double2(std::cos(-p->dt * V[e]), std::sin(-p->dt * V[e]));
  }
  e2d::tables(h->nx, h->dx, p->mass_x, p->dt, kx, Tx, fx, ix);
  e2d::tables(h->nR, h->dR, p->mass_R, p->dt, kR, TR, fR, iR);
  const auto H2D = cudaMemcpyHostToDevice;
  bool ok = copy(h, h->V, V, NN * 8, H2D) && copy(h, h->half, half.data(), NN * 16, H2D) &&
            copy(h, h->full, full.data(), NN * 16, H2D) &&
            copy(h, h->kinx, kx.data(), kx.size() * 16, H2D) &&
            copy(h, h->kinR, kR.data(), kR.size() * 16, H2D) &&
            copy(h, h->tfx, fx.data(), fx.size() * 16, H2D) && copy(h, h->tix, ix.data(), ix.size() * 16, H2D) &&
            copy(h, h->tfR, fR.data(), fR.size() * 16, H2D) && copy(h, h->tiR, iR.data(), iR.size() * 16, H2D) &&
            copy(h, h->Tx, Tx.data(), Tx.size() * 8, H2D) &&
            copy(h, h->TR, TR.data(), TR.size() * 8, H2D);
  if (!ok) {
    release(h);
    delete h;
    return fail2(nullptr, ICWF_ERR_CUDA, "icwf_exact2d_create: upload failed");
  }
  e2d::attributes();
  *out = h;
  return ICWF_OK;
}

icwf_status icwf_exact2d_set_state(icwf_exact2d h, const double* psi) {
  if (!h || !psi) return fail2(h, ICWF_ERR_ARG, "icwf_exact2d_set_state: null pointer");
  const size_t NN = (size_t)h->nx * h->nR;
  if (!copy(h, h->psi, psi, NN * 16, cudaMemcpyHostToDevice))
    return fail2(h, ICWF_ERR_CUDA, "icwf_exact2d_set_state: upload failed");
  h->has_state = true;
  h->t = 0.0;
  return ICWF_OK;
}

icwf_status icwf_exact2d_set_projectors(icwf_exact2d h, int32_t n_states, const double* phi) {
  if (!h || !phi) return fail2(h, ICWF_ERR_ARG, "icwf_exact2d_set_projectors: null pointer");
  if (n_states < 1 || n_states > e2d::MAX_STATES)
    return fail2(h, ICWF_ERR_ARG, "icwf_exact2d_set_projectors: n_states must be in [1, 8]");
  const size_t n = (size_t)n_states * h->nR * h->nx;
  if (!h->phi && !dalloc(h, &h->phi, (size_t)e2d::MAX_STATES * h->nR * h->nx))
    return fail2(h, ICWF_ERR_OOM, "icwf_exact2d_set_projectors: cudaMalloc failed");
  if (!copy(h, h->phi, phi, n * 8, cudaMemcpyHostToDevice))
    return fail2(h, ICWF_ERR_CUDA, "icwf_exact2d_set_projectors: upload failed");
  h->ns = n_states;
  return ICWF_OK;
}

icwf_status icwf_exact2d_step(icwf_exact2d h, int32_t n_steps) {
  if (!h) return fail2(h, ICWF_ERR_ARG, "icwf_exact2d_step: null handle");
  if (n_steps < 0) return fail2(h, ICWF_ERR_ARG, "icwf_exact2d_step: n_steps < 0");
  if (!h->has_state) return fail2(h, ICWF_ERR_STATE, "icwf_exact2d_step: no state set");
  for (int s = 0; s < n_steps; ++s) {
    if (s == 0)
      e2d::rows<false, true>(h->nx, h->nR, h->logR, h->psi, h->psi, h->half, h->tfR, h->tiR, h->stream);
    else
      e2d::rows<true, true>(h->nx, h->nR, h->logR, h->psi, h->psi, h->full, h->tfR, h->tiR, h->stream);
    e2d::cols<false>(h->nx, h->nR, h->logx, h->psi, h->kinx, h->kinR, h->tfx, h->tix, nullptr, nullptr, nullptr,
                     h->stream);
  }
  if (n_steps > 0)
    e2d::rows<true, false>(h->nx, h->nR, h->logR, h->psi, h->psi, h->half, h->tfR, h->tiR, h->stream);
  const icwf_status st = sync(h, "icwf_exact2d_step");
  if (st == ICWF_OK) h->t += n_steps * h->dt;
  return st;
}

icwf_status icwf_exact2d_get_state(icwf_exact2d h, double* psi) {
  if (!h || !psi) return fail2(h, ICWF_ERR_ARG, "icwf_exact2d_get_state: null pointer");
  if (!h->has_state) return fail2(h, ICWF_ERR_STATE, "icwf_exact2d_get_state: no state set");
  if (!copy(h, psi, h->psi, (size_t)h->nx * h->nR * 16, cudaMemcpyDeviceToHost))
    return fail2(h, ICWF_ERR_CUDA, "icwf_exact2d_get_state: download failed");
  return ICWF_OK;
}

icwf_status icwf_exact2d_observables(icwf_exact2d h, icwf_obs* out) {
  if (!h || !out) return fail2(h, ICWF_ERR_ARG, "icwf_exact2d_observables: null pointer");
  if (!h->has_state) return fail2(h, ICWF_ERR_STATE, "icwf_exact2d_observables: no state set");
  const int nx = h->nx, nR = h->nR, ncb = nR / e2d::CB;
  e2d::k_dens_rows<<<nx, e2d::TPB, 0, h->stream>>>(h->psi, h->V, nR, h->dens_x, h->pot);
  e2d::k_cols_obs<<<nR, e2d::TPB, 0, h->stream>>>(h->psi, nx, nR, h->phi, h->ns, h->dens_R, h->proj);
  // kinetic energy: 2D FFT of Psi into work, then sum |F|^2 (Tx + TR) per column group
  e2d::rows<false, true>(nx, nR, h->logR, h->psi, h->work, nullptr, h->tfR, h->tiR, h->stream);
  e2d::cols<true>(nx, nR, h->logx, h->work, nullptr, nullptr, h->tfx, h->tix, h->Tx, h->TR, h->part, h->stream);
  icwf_status st = sync(h, "icwf_exact2d_observables");
  if (st != ICWF_OK) return st;
  std::vector<double> dx_(nx), pot(nx), dR_(nR), part(ncb);
  std::vector<double2> proj((size_t)h->ns * nR);
  const auto D2H = cudaMemcpyDeviceToHost;
  bool ok = copy(h, dx_.data(), h->dens_x, nx * 8, D2H) && copy(h, pot.data(), h->pot, nx * 8, D2H) &&
            copy(h, dR_.data(), h->dens_R, nR * 8, D2H) && copy(h, part.data(), h->part, ncb * 8, D2H) &&
            (h->ns == 0 || copy(h, proj.data(), h->proj, proj.size() * 16, D2H));
  if (!ok) return fail2(h, ICWF_ERR_CUDA, "icwf_exact2d_observables: download failed");
  double norm = 0.0, epot = 0.0, ekin = 0.0;
  for (int i = 0; i < nx; ++i) { norm += dx_[i]; epot += pot[i]; }
  for (int c = 0; c < ncb; ++c) ekin += part[c];
  norm *= h->dx * h->dR;
  epot *= h->dx * h->dR;
  ekin *= h->dx * h->dR / ((double)nx * nR);
  out->t = h->t;
  out->norm = norm;
  out->energy = norm > 0 ? (ekin + epot) / norm : 0.0;
  out->n_clamped = 0;
  out->n_states = h->ns;
  if (out->rho_x)
    for (int i = 0; i < nx; ++i) out->rho_x[i] = h->dR * dx_[i];
  if (out->rho_R)
    for (int j = 0; j < nR; ++j) out->rho_R[j] = h->dx * dR_[j];
  if (h->ns > 0) {
    std::vector<double> pn((size_t)h->ns * nR);
    for (int n = 0; n < h->ns; ++n)
      for (int j = 0; j < nR; ++j) {
        const double2 z = proj[(size_t)n * nR + j];
        const double re = h->dx * z.x, im = h->dx * z.y;
        pn[(size_t)n * nR + j] = re * re + im * im;
      }
    if (out->pop)
      for (int n = 0; n < h->ns; ++n) {
        double s = 0.0;
        for (int j = 0; j < nR; ++j) s += pn[(size_t)n * nR + j];
        out->pop[n] = h->dR * s;
      }
    if (out->decoh)
      for (int n = 0; n < h->ns; ++n)
        for (int m = 0; m < h->ns; ++m) {
          double s = 0.0;
          for (int j = 0; j < nR; ++j) s += pn[(size_t)n * nR + j] * pn[(size_t)m * nR + j];
          out->decoh[n * h->ns + m] = h->dR * s;
        }
  }
  return ICWF_OK;
}

icwf_status icwf_exact2d_destroy(icwf_exact2d h) {
  if (!h) return ICWF_OK;
  release(h);
  delete h;
  return ICWF_OK;
}

const char* icwf_exact2d_last_error(icwf_exact2d h) { return h ? h->err.c_str() : g_err2.c_str(); }

}  // extern "C"
