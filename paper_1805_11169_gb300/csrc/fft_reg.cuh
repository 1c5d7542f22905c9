// Batched FFTs of the exact propagator: columns of length n = 2^L in shared memory (padded by one
// element in eight), 2 to 4 radix-2 stages per pass in a thread's registers.
//
// FP64 instructions bound these transforms (an SM takes one warp's instruction per 19 cycles), so the
// butterflies a +- w b take six of them instead of eight (the fused multiply-add butterfly of Linzer
// and Feig, with the larger part of the twiddle factored out): with w = m (1 + i r), |r| <= 1,
//   u = p - r q, v = q + r p, (a.x +- m u, a.y +- m v),   p + i q = b or i b,
// where the second form (w = -i m (1 + i r) i) serves the angles whose sine is the larger part.  Both
// directions have the twiddle on the second operand: forward, natural to bit-reversed order, with one
// twiddle per block (e^{-i pi vdc(k)}, vdc: the bits of k mirrored behind the point); inverse,
// bit-reversed to natural order, with twiddles by position.  Multiplications by 1, +-i are left out,
// those by (1 +- i) / sqrt 2 have r = +-1.
#pragma once
#include <cuda_runtime.h>

namespace icwf {
namespace fftr {

struct Tw { double m, r; };   // multiplier and ratio; which form: fwd_form, inv_form

__host__ __device__ __forceinline__ int fwd_form(int k) { return (k ^ (k >> 1)) & 1; }
__host__ __device__ __forceinline__ int inv_form(int x, int L) { return ((x >> (L - 2)) ^ (x >> (L - 3))) & 1; }

__host__ __device__ __forceinline__ int pad(int i) { return i + (i >> 3); }
__host__ __device__ __forceinline__ int padded(int n) { return n + n / 8; }

// Stages before the last three (forward order): M = L - 3 of them in P passes of M / P or M / P + 1.
__host__ __device__ constexpr int passes(int L) { return L == 3 ? 0 : (L <= 7 ? 1 : (L <= 11 ? 2 : 3)); }
__host__ __device__ constexpr int pass_at(int L, int i) { return (L - 3) * i / (passes(L) ? passes(L) : 1); }

__device__ __forceinline__ double flip(double x) {   // -x by an integer operation
  return __hiloint2double(__double2hiint(x) ^ (int)0x80000000, __double2loint(x));
}
__device__ __forceinline__ double2 rot(double2 b, bool inv) {   // b times -i (forward) or i
  return inv ? make_double2(flip(b.y), b.x) : make_double2(b.y, flip(b.x));
}
__device__ __forceinline__ void fly1(double2& a, double2& b) {  // w = 1
  const double2 t = b;
  b = make_double2(a.x - t.x, a.y - t.y);
  a = make_double2(a.x + t.x, a.y + t.y);
}
__device__ __forceinline__ void fly(double2& a, double2& b, Tw w, int form) {
  const double p = form ? flip(b.y) : b.x, q = form ? b.x : b.y;
  const double u = fma(-w.r, q, p), v = fma(w.r, p, q);
  b = make_double2(fma(-w.m, u, a.x), fma(-w.m, v, a.y));
  a = make_double2(fma(w.m, u, a.x), fma(w.m, v, a.y));
}
constexpr double SQRT1_2 = 0.70710678118654752440;

// R forward stages from level l on the points i = 0 .. 2^R - 1 of block k (k = 0 if FIRST).
template <int R, bool FIRST>
__device__ __forceinline__ void fwd(double2 (&z)[1 << R], const Tw* __restrict__ tw, int k) {
#pragma unroll
  for (int t = 0; t < R; ++t) {
    const int d = 1 << (R - 1 - t);
#pragma unroll
    for (int bb = 0; bb < (1 << t); ++bb) {
      const bool odd = bb & 1;
      const int ke = ((FIRST ? 0 : k) << t) | (bb & ~1);   // odd block numbers: -i times the one before
      Tw w;
      if (!(FIRST && bb < 2)) {
        if (FIRST && bb < 4) w = Tw{-SQRT1_2, 1.0};        // k = 2: e^{-i pi / 4}
        else w = tw[ke];
      }
#pragma unroll
      for (int i = 0; i < d; ++i) {
        double2 &a = z[bb * 2 * d + i], &b = z[bb * 2 * d + d + i];
        if (odd) b = rot(b, false);
        if (FIRST && bb < 2) fly1(a, b);
        else fly(a, b, w, fwd_form(ke));
      }
    }
  }
}
// R inverse stages from span 2^s on the points j + i 2^s of a group (s = 0, j = 0 if FIRST), without
// the factor 1 / n.
template <int R, bool FIRST>
__device__ __forceinline__ void inv(double2 (&z)[1 << R], const Tw* __restrict__ tw, int j, int s, int L) {
#pragma unroll
  for (int t = 0; t < R; ++t) {
    const int d = 1 << t;
#pragma unroll
    for (int lo = 0; lo < d; ++lo) {
      const bool top = t > 0 && (lo >> (t - 1));           // a quarter turn beyond lo - d / 2
      const int le = top ? lo - d / 2 : lo;
      Tw w;
      int form = 0;
      if (!(FIRST && le == 0)) {
        const int x = ((FIRST ? 0 : j) + (le << (FIRST ? 0 : s))) << (L - 1 - (FIRST ? 0 : s) - t);
        w = tw[x];
        form = inv_form(x, L);
      }
#pragma unroll
      for (int i = 0; i < (1 << R); i += 2 * d) {
        double2 &a = z[i + lo], &b = z[i + lo + d];
        if (top) b = rot(b, true);
        if (FIRST && le == 0) fly1(a, b);
        else fly(a, b, w, form);
      }
    }
  }
}

// One pass over nb transforms; F sees the points in registers before (PRE) or after the stages.
template <int L, int R, int LEV>
__device__ __forceinline__ void fwd_pass(double2* buf, const Tw* __restrict__ tw, int nb) {
  constexpr int q = 1 << (L - LEV - R), G = 1 << (L - R);
  for (int g = threadIdx.x; g < nb * G; g += blockDim.x) {
    const int b = g >> (L - R), gg = g & (G - 1), k = gg / q, i0 = (k << (L - LEV)) + (gg & (q - 1));
    double2* p = buf + b * padded(1 << L);
    double2 z[1 << R];
#pragma unroll
    for (int i = 0; i < (1 << R); ++i) z[i] = p[pad(i0 + i * q)];
    fwd<R, LEV == 0>(z, tw, k);
#pragma unroll
    for (int i = 0; i < (1 << R); ++i) p[pad(i0 + i * q)] = z[i];
  }
  __syncthreads();
}
template <int L, int R, int S>
__device__ __forceinline__ void inv_pass(double2* buf, const Tw* __restrict__ tw, int nb) {
  constexpr int q = 1 << S, G = 1 << (L - R);
  for (int g = threadIdx.x; g < nb * G; g += blockDim.x) {
    const int b = g >> (L - R), gg = g & (G - 1), j = gg & (q - 1), i0 = ((gg >> S) << (S + R)) + j;
    double2* p = buf + b * padded(1 << L);
    double2 z[1 << R];
#pragma unroll
    for (int i = 0; i < (1 << R); ++i) z[i] = p[pad(i0 + i * q)];
    inv<R, S == 0>(z, tw, j, S, L);
#pragma unroll
    for (int i = 0; i < (1 << R); ++i) p[pad(i0 + i * q)] = z[i];
  }
  __syncthreads();
}
// The stages of all passes but the last three stages (forward), or after the first three (inverse);
// I from which pass, N up to which.
template <int L, int I, int N>
__device__ __forceinline__ void fwd_passes(double2* buf, const Tw* __restrict__ tw, int nb) {
  if constexpr (I < N) {
    fwd_pass<L, pass_at(L, I + 1) - pass_at(L, I), pass_at(L, I)>(buf, tw, nb);
    fwd_passes<L, I + 1, N>(buf, tw, nb);
  }
}
template <int L, int I, int N>   // the mirror image: pass I of the forward transform undone, down to N
__device__ __forceinline__ void inv_passes(double2* buf, const Tw* __restrict__ tw, int nb) {
  if constexpr (I >= N) {
    inv_pass<L, pass_at(L, I + 1) - pass_at(L, I), L - pass_at(L, I + 1)>(buf, tw, nb);
    inv_passes<L, I - 1, N>(buf, tw, nb);
  }
}
template <int L>
__device__ __forceinline__ void fwd_all(double2* buf, const Tw* __restrict__ tw, int nb) {
  fwd_passes<L, 0, passes(L)>(buf, tw, nb);
  fwd_pass<L, 3, L - 3>(buf, tw, nb);
}
template <int L>
__device__ __forceinline__ void inv_all(double2* buf, const Tw* __restrict__ tw, int nb) {
  inv_pass<L, 3, 0>(buf, tw, nb);
  inv_passes<L, passes(L) - 1, 0>(buf, tw, nb);
}
// Forward's last three stages, f(b, position, value) on every point, inverse's first three.
template <int L, typename F>
__device__ __forceinline__ void turn_freq(double2* buf, const Tw* __restrict__ tf, const Tw* __restrict__ ti, int nb,
                                          const F& f) {
  constexpr int G = 1 << (L - 3);
  for (int g = threadIdx.x; g < nb * G; g += blockDim.x) {
    const int b = g >> (L - 3), k = g & (G - 1);
    double2* p = buf + b * padded(1 << L);
    double2 z[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) z[i] = p[pad(8 * k + i)];
    fwd<3, L == 3>(z, tf, k);
#pragma unroll
    for (int i = 0; i < 8; ++i) z[i] = f(b, 8 * k + i, z[i]);
    inv<3, true>(z, ti, 0, 0, L);
#pragma unroll
    for (int i = 0; i < 8; ++i) p[pad(8 * k + i)] = z[i];
  }
  __syncthreads();
}
// Inverse's last pass, f on every point, forward's first pass (one transform).
template <int L, typename F>
__device__ __forceinline__ void turn_space(double2* buf, const Tw* __restrict__ tf, const Tw* __restrict__ ti,
                                           const F& f) {
  constexpr int R = passes(L) ? pass_at(L, 1) : 3, S = L - R, q = 1 << S;
  for (int j = threadIdx.x; j < q; j += blockDim.x) {
    double2 z[1 << R];
#pragma unroll
    for (int i = 0; i < (1 << R); ++i) z[i] = buf[pad(j + i * q)];
    inv<R, S == 0>(z, ti, j, S, L);
#pragma unroll
    for (int i = 0; i < (1 << R); ++i) z[i] = f(j + i * q, z[i]);
    fwd<R, true>(z, tf, 0);
#pragma unroll
    for (int i = 0; i < (1 << R); ++i) buf[pad(j + i * q)] = z[i];
  }
  __syncthreads();
}

}  // namespace fftr
}  // namespace icwf
