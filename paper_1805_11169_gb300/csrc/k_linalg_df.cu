// Coefficient solve of the mixed-precision modes (Eq. coeff) in double-float arithmetic.
//
// The regularised overlap S + eps I is factorised and the RK4 stage systems are solved with
// complex numbers stored as (re_hi, re_lo, im_hi, im_lo) FP32 quadruples (16 bytes, the size of a
// complex128), each part a double-float of ~48 significant bits (csrc/df64.cuh).  On this GPU the
// FP32 pipes have ~64x the FP64 throughput and a far shorter latency, and the Cholesky chain and
// the triangular-solve chains are latency-bound; S itself carries ~1e-6 relative rounding noise in
// these modes, far above the 48-bit arithmetic.  Dot products use compensated accumulation in the
// style of Ogita, Rump and Oishi's Dot2 (TwoProduct + TwoSum, errors summed separately), which
// returns them as accurately as if evaluated in twice the FP32 precision.
//
// Kernels: k_shift_mix_df (S -> S + eps I, converted); k_chol_df (the blocked Cholesky, one
// persistent launch with look-ahead, above 26 block columns several with the trailing updates between
// them on the tensor cores: diagonal updates, diagonal factors, panel slabs,
// trailing tiles and the inverses of the diagonal blocks as ticket-ordered tasks; the panel tasks
// also write L^H into the upper triangle); k_trsv_lower_df / k_trsv_upper_df (triangular solves above
// N = 2048, per-block kernels with global flags; k_solve.cu has the others).
#include <cuda_runtime.h>

#include <algorithm>

#include "cdf.cuh"
#include "icwf_internal.h"
#include "k_common.cuh"

namespace icwf {
namespace dfs {

constexpr int NB = 32;
constexpr unsigned WAIT_LIMIT = 1u << 22;

struct Batch {
  float4* m[2];
  float2* inv[2];   // 1/L_cc as double-floats
  float4* D[2];     // inverted diagonal blocks
};
// member of a two-entry parameter array without a dynamically indexed (local-memory) copy
template <typename T>
__device__ __forceinline__ T pick2(T const (&a)[2], unsigned i) { return i ? a[1] : a[0]; }

__device__ __forceinline__ cdf shfl_cdf(cdf v, int src) {
  cdf r;
  r.re.h = __shfl_sync(0xffffffffu, v.re.h, src);
  r.re.l = __shfl_sync(0xffffffffu, v.re.l, src);
  r.im.h = __shfl_sync(0xffffffffu, v.im.h, src);
  r.im.l = __shfl_sync(0xffffffffu, v.im.l, src);
  return r;
}

// ---------------------------------------------------------------------------- S + eps I

// One CTA per row r (no index division per element).
__global__ void k_shift_mix_df(int N, const double2* __restrict__ S0, const double2* __restrict__ S1,
                               double eps, double theta, float4* __restrict__ A) {
  const int r = blockIdx.x;
  for (int c = threadIdx.x; c < N; c += blockDim.x) {
    const size_t e = (size_t)r * N + c;
    double2 v;
    if (theta == 1.0) v = S1[e];
    else if (theta == 0.0) v = S0[e];
    else v = make_double2(0.5 * (S0[e].x + S1[e].x), 0.5 * (S0[e].y + S1[e].y));
    if (r == c) v.x += eps;
    A[e] = st4(cdf_make(df_from(v.x), df_from(v.y)));
  }
}

__device__ __forceinline__ void tri_index(int t, int& I, int& J) {
  int Jc = (int)((sqrt(8.0 * (double)t + 1.0) - 1.0) * 0.5);
  while (Jc * (Jc + 1) / 2 > t) --Jc;
  while ((Jc + 1) * (Jc + 2) / 2 <= t) ++Jc;
  J = Jc;
  I = t - Jc * (Jc + 1) / 2;
}

// ---------------------------------------------------------------------------- blocked factorisation
//
// Right-looking blocked Cholesky of up to two matrices in one persistent launch.  Every CTA is two
// groups of 256 threads with their own barriers and shared memory.  The first nbatch CTAs to arrive
// become the matrices' chain CTAs: chain m factors the diagonal blocks 0, 1, 2, ... of matrix m, alone
// on its SM.  All other groups take tickets for the remaining tasks, which are numbered block column
// by block column li (jb = li - 1 is the panel being applied):
//   [10 updates of diagonal block li] [some trailing tiles] [panel-li slabs of 8 rows] [the other
//   trailing tiles] [inverse of diagonal block li - 1].
// A task waits (bounded) on control words for exactly the data it reads, which come from smaller
// tickets or from a diagonal factor; a diagonal factor waits for updates whose tickets precede
// everything that waits for it.  So whatever is running can finish: progress needs only that the
// chains and one more CTA are resident.  The trailing tiles ahead of the slabs are as many as run
// while the diagonal factor does, so neither the slabs wait behind the whole trailing update nor the
// groups behind the factor.
// Why one launch: a launch per block column started every diagonal factor with a cold instruction
// cache (15-25 us each instead of 11) and kept the slabs behind all trailing tiles of their launch.
// All arithmetic is double-float with compensated (Dot2) accumulation; complex products in the
// updates use three real products (Karatsuba).

constexpr int CS_THREADS = 256;
constexpr int DIAG_TASKS = 10;                // 8 x 8 blocks of a diagonal block's lower triangle
constexpr int TS_ROWS = 8;                    // panel rows per slab task
constexpr unsigned CS_WAIT_LIMIT = 1u << 24;
constexpr int CS_SMEM = 6 * NB * NB * 8;      // largest task: trailing tile, 6 double-float planes
constexpr int CTA_THREADS = 2 * CS_THREADS;   // two groups
// shared memory requested per CTA: more than half an SM's, so that a chain CTA shares its SM with no
// other CTA of the launch
constexpr int CS_SMEM_LAUNCH = 116 * 1024;
static_assert(2 * CS_SMEM <= CS_SMEM_LAUNCH, "tasks need more shared memory than the launch asks for");
// Two-level form: while more than ONE_LAUNCH block columns are left, a launch factors PANEL of them and the
// trailing update from those runs on the tensor cores (launch_herk_df); the rest is one launch.  The
// FP32 tiles of a single launch bound its early steps (a 32 x 32 tile takes a group 12 us); the two
// launches of an update and a cold start of the diagonal factor cost about 30 us per panel.  All in
// panels / one launch, two matrices, us: 597 / 473 at N = 640, 788 / 652 at 769, 949 / 872 at 900, 1027 /
// 1076 at 1024, 1744 / 2667 at 1500, 2815 / 6059 at 2048; four columns cost 161 in panels and 219 in one
// launch from 29 blocks on, 178 and 162 from 25.
constexpr int PANEL = 4;
constexpr int ONE_LAUNCH = 26;
constexpr int AHEAD_TILES = 300;              // trailing tiles ahead of the slabs: one per group

// One group of CS_THREADS threads of a CTA.
struct Grp {
  int tid, bar;
  __device__ __forceinline__ void sync() const {
    asm volatile("bar.sync %0, %1;" ::"r"(bar), "n"(CS_THREADS) : "memory");
  }
};

__device__ __forceinline__ cdf ldcg4(const float4* p) { return ld4(__ldcg(p)); }
// a += x y for double-float reals (Dot2 step on the high parts, cross terms in FP32)
__device__ __forceinline__ void acc_prod_df(acc2& a, df x, df y) {
  acc_prod(a, x.h, y.h);
  acc_small(a, DF_FMA(x.h, y.l, DF_MUL(x.l, y.h)));
}
__device__ __forceinline__ acc2 acc_neg(acc2 a) { a.s = -a.s; a.c = -a.c; return a; }
// Karatsuba: x conj(w) from P1 = xr wr, P2 = xi wi, P3 = (xr + xi)(wr - wi)
__device__ __forceinline__ cdf kara_val(acc2 p1, acc2 p2, acc2 p3) {
  return cdf_make(acc_val(acc_merge(p1, p2)), acc_val(acc_merge(acc_merge(p3, acc_neg(p1)), p2)));
}

// until *f >= target, or with kBits until all bits of target are set
template <bool kBits = false>
__device__ __forceinline__ bool cs_wait(const unsigned* f, unsigned target, int* status) {
  const unsigned lim = wait_budget(status, CS_WAIT_LIMIT);
  for (unsigned it = 0; it < lim; ++it) {
    const unsigned v = ld_acquire(f);
    if (kBits ? (v & target) == target : v >= target) return true;
    if (it > 256) __nanosleep(128);
  }
  set_flag(status, ST_TIMEOUT);
  return false;
}
// all of this group's global writes, then a release increment of *f
__device__ __forceinline__ void cs_signal(const Grp& g, unsigned* f) {
  g.sync();
  if (g.tid == 0) {
    __threadfence();
    atomicAdd(f, 1u);
  }
}

// a -= x conj(y) with each part of a as an unevaluated sum whose low word is not renormalised: the two
// leading products of a part are added error-free, everything of second order goes to the low word.
// 24 FP32 operations per part, 16 of them on the longest chain.
__device__ __forceinline__ df df_sub2(df a, df x1, df y1, df x2, df y2) {   // a - x1 y1 - x2 y2
  const float p1 = DF_MUL(-x1.h, y1.h), p2 = DF_MUL(-x2.h, y2.h);
  const float e1 = DF_FMA(-x1.h, y1.h, -p1), e2 = DF_FMA(-x2.h, y2.h, -p2);
  float c = DF_FMA(-x1.h, y1.l, e1);
  c = DF_FMA(-x1.l, y1.h, c);
  float d = DF_FMA(-x2.h, y2.l, e2);
  d = DF_FMA(-x2.l, y2.h, d);
  const df t1 = two_sum(a.h, p1);
  const df t2 = two_sum(t1.h, p2);
  return df_make(t2.h, DF_ADD(DF_ADD(DF_ADD(a.l, t1.l), DF_ADD(c, d)), t2.l));
}
__device__ __forceinline__ void sub_mulc(cdf& a, cdf x, cdf y) {
  a.re = df_sub2(a.re, x.re, y.re, x.im, y.im);
  a.im = df_sub2(a.im, x.im, y.re, df_neg(x.re), y.im);
}
__device__ __forceinline__ cdf renorm(cdf a) {
  return cdf_make(fast_two_sum(a.re.h, a.re.l), fast_two_sum(a.im.h, a.im.l));
}

// One output per thread of an R x C block (R C = 256): returns A[orow][ocol] - sum_k X[r][k] conj(Y[c][k])
// with X = rows xrow0.., Y = rows yrow0.. of A over columns k0..k0+31.
template <int R, int C>
__device__ __forceinline__ cdf upd_one(const float4* A, int N, int xrow0, int yrow0, int k0,
                                       int orow, int ocol, bool ok, unsigned char* smem, const Grp& g) {
  df(*Xp)[R][NB] = (df(*)[R][NB])smem;                        // [3][R][32]
  df(*Yp)[NB][C] = (df(*)[NB][C])(smem + 3 * R * NB * 8);     // [3][32][C]
  const cdf a = ok ? ldcg4(A + (size_t)orow * N + ocol) : czero();   // issued first, used last
  for (int e = g.tid; e < R * NB; e += CS_THREADS) {
    const int r = e / NB, k = e % NB;
    cdf x = czero();
    if (xrow0 + r < N && k0 + k < N) x = ldcg4(A + (size_t)(xrow0 + r) * N + k0 + k);
    Xp[0][r][k] = x.re;
    Xp[1][r][k] = x.im;
    Xp[2][r][k] = df_add_sloppy(x.re, x.im);
  }
  for (int e = g.tid; e < C * NB; e += CS_THREADS) {
    const int k = e / C, c = e % C;
    cdf y = czero();
    if (yrow0 + c < N && k0 + k < N) y = ldcg4(A + (size_t)(yrow0 + c) * N + k0 + k);
    Yp[0][k][c] = y.re;
    Yp[1][k][c] = y.im;
    Yp[2][k][c] = df_add_sloppy(y.re, df_neg(y.im));
  }
  g.sync();
  const int r = g.tid / C, c = g.tid % C;
  acc2 p1 = acc_zero(), p2 = acc_zero(), p3 = acc_zero();
#pragma unroll 8
  for (int k = 0; k < NB; ++k) {
    acc_prod_df(p1, Xp[0][r][k], Yp[0][k][c]);
    acc_prod_df(p2, Xp[1][r][k], Yp[1][k][c]);
    acc_prod_df(p3, Xp[2][r][k], Yp[2][k][c]);
  }
  g.sync();
  return cdf_sub(a, kara_val(p1, p2, p3));
}

// 8 x 8 block (rb, cb), cb <= rb < 4, of diagonal block jp: A -= L_jp,jb L_jp,jb^H.  Each output's 32
// products are split over four lanes (8 each), whose sums meet by shuffles: the update sits on the
// factorisation's dependency chain, and ten such tasks take 2.5 us where three 16 x 16 ones took 4.
__device__ __forceinline__ void diag_update8(float4* A, int N, int jp, int jb, int rb, int cb, unsigned char* smem, const Grp& g) {
  cdf(*X)[NB + 1] = (cdf(*)[NB + 1])smem;                          // [8][33]
  cdf(*Y)[NB + 1] = (cdf(*)[NB + 1])(smem + 8 * (NB + 1) * 16);    // [8][33]
  const int r0 = jp * NB + rb * 8, c0 = jp * NB + cb * 8;
  {
    const int r = g.tid >> 5, k = g.tid & 31;
    X[r][k] = r0 + r < N ? ldcg4(A + (size_t)(r0 + r) * N + jb * NB + k) : czero();
    Y[r][k] = c0 + r < N ? ldcg4(A + (size_t)(c0 + r) * N + jb * NB + k) : czero();
  }
  const int o = g.tid >> 2, q = g.tid & 3, r = o >> 3, c = o & 7;
  const int gr = r0 + r, gc = c0 + c;
  const bool ok = gr < N && gc < N && gc <= gr;
  const cdf a = ok && q == 0 ? ldcg4(A + (size_t)gr * N + gc) : czero();
  g.sync();
  cdf s = a;
#pragma unroll
  for (int k = 0; k < 8; ++k) sub_mulc(s, X[r][q + 4 * k], Y[c][q + 4 * k]);
  s = renorm(s);
#pragma unroll
  for (int off = 1; off < 4; off <<= 1) {
    cdf t;
    t.re.h = __shfl_xor_sync(0xffffffffu, s.re.h, off);
    t.re.l = __shfl_xor_sync(0xffffffffu, s.re.l, off);
    t.im.h = __shfl_xor_sync(0xffffffffu, s.im.h, off);
    t.im.l = __shfl_xor_sync(0xffffffffu, s.im.l, off);
    s = cdf_make(df_add_sloppy(s.re, t.re), df_add_sloppy(s.im, t.im));
  }
  if (ok && q == 0) A[(size_t)gr * N + gc] = st4(s);
}

// Trailing tile (rb, cb), cb <= rb: A_rc -= L_r,jb L_c,jb^H, 2 x 2 outputs per thread.
__device__ __forceinline__ void herk_tile(float4* A, int N, int jb, int rb, int cb,
                                          unsigned char* smem, const Grp& g) {
  df(*Rp)[NB][NB] = (df(*)[NB][NB])smem;                      // [plane][row][k]
  df(*Cp)[NB][NB] = (df(*)[NB][NB])(smem + 3 * NB * NB * 8);  // [plane][k][col]
  const int k0 = jb * NB;
  for (int e = g.tid; e < NB * NB; e += CS_THREADS) {
    const int r = e / NB, m = e % NB;
    cdf a = czero();
    if (rb * NB + r < N && k0 + m < N) a = ldcg4(A + (size_t)(rb * NB + r) * N + k0 + m);
    Rp[0][r][m] = a.re;
    Rp[1][r][m] = a.im;
    Rp[2][r][m] = df_add_sloppy(a.re, a.im);
    // transposed walk for the column tile: conflict-free shared-memory stores
    const int m2 = e / NB, r2 = e % NB;
    cdf b = czero();
    if (cb * NB + r2 < N && k0 + m2 < N) b = ldcg4(A + (size_t)(cb * NB + r2) * N + k0 + m2);
    Cp[0][m2][r2] = b.re;
    Cp[1][m2][r2] = b.im;
    Cp[2][m2][r2] = df_add_sloppy(b.re, df_neg(b.im));
  }
  g.sync();
  const int tx = g.tid & 15, ty = g.tid >> 4;
  acc2 acc[3][2][2];
#pragma unroll
  for (int p = 0; p < 3; ++p)
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
      for (int c = 0; c < 2; ++c) acc[p][r][c] = acc_zero();
#pragma unroll 4
  for (int m = 0; m < NB; ++m) {
#pragma unroll
    for (int p = 0; p < 3; ++p) {
      const df a0 = Rp[p][ty][m], a1 = Rp[p][ty + 16][m];
      const df b0 = Cp[p][m][tx], b1 = Cp[p][m][tx + 16];
      acc_prod_df(acc[p][0][0], a0, b0);
      acc_prod_df(acc[p][0][1], a0, b1);
      acc_prod_df(acc[p][1][0], a1, b0);
      acc_prod_df(acc[p][1][1], a1, b1);
    }
  }
#pragma unroll
  for (int r = 0; r < 2; ++r)
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int gr = rb * NB + ty + 16 * r, gc = cb * NB + tx + 16 * c;
      if (gr < N && gc < N && gc <= gr) {
        float4* p = A + (size_t)gr * N + gc;
        *p = st4(cdf_sub(ldcg4(p), kara_val(acc[0][r][c], acc[1][r][c], acc[2][r][c])));
      }
    }
}

// Factor diagonal block jp in place: L L^H = A_jp,jp (lower triangle), reciprocal pivots to inv.
// Warp w owns columns 4w .. 4w + 3 in registers, lane = row, and the columns flow through shared
// memory without a barrier: a warp subtracts column k's products as soon as flag k is up, then factors
// its own four columns (pivot by shuffle, y = 1/sqrt(d) with one refinement step, scaling, the next
// columns updated by shuffles), raises their flags, writes them out and sets its bit of *done, so that
// the slabs below follow the factor column by column.
// What bounds it is the pivots' dependency chain (shuffle, reciprocal square root, scaling, hand-over,
// update; about 300 cycles each).  With a barrier and a hand-over per pivot, and a column's updates
// spread over all warps, the block took 14 us; with a panel of 8 columns in one warp 14.6 (its 230
// instructions per pivot, not their latency).
constexpr int PB = 4;                       // columns per warp
__device__ __forceinline__ void flag_wait(const volatile int* f, int* status) {
  int it = 0;
  while (!*f && ++it < (1 << 20)) {
  }
  if (it == (1 << 20)) set_flag(status, ST_TIMEOUT);
  __threadfence_block();
}

// columns c0 + J .. c0 + 3 (lane = row); L[c * 32 + r] and flag[c] receive the finished ones
template <int J>
__device__ __forceinline__ void panel_steps(cdf (&a)[PB], df (&y)[PB], int c0, cdf* L, volatile int* flag, bool& bad) {
  const int lane = threadIdx.x & 31, c = c0 + J;
  const cdf v = renorm(a[J]);
  df d;
  d.h = __shfl_sync(0xffffffffu, v.re.h, c);
  d.l = __shfl_sync(0xffffffffu, v.re.l, c);
  const bool ok = d.h > 0.f;
  bad = bad || !ok;
  d = ok ? d : df_make(1.f, 0.f);
  y[J] = df_rsqrt1(d);
  cdf l = cdf_scale(v, y[J]);
  l = lane == c ? cdf_make(df_mul(d, y[J]), df_make(0.f, 0.f)) : l;
  l = lane < c ? czero() : l;
  L[c * NB + lane] = l;
  __syncwarp();
  if (lane == 0) {
    __threadfence_block();
    flag[c] = 1;
  }
  a[J] = l;
  if constexpr (J + 1 < PB) {
#pragma unroll
    for (int q = J + 1; q < PB; ++q) sub_mulc(a[q], l, shfl_cdf(l, c0 + q));
    panel_steps<J + 1>(a, y, c0, L, flag, bad);
  }
}

__device__ __forceinline__ void potrf_task(int N, float4* A, float2* inv, int jp, int* status, unsigned* done,
                                           unsigned char* smem, const Grp& g) {
  cdf* L = (cdf*)smem;                       // L[c * 32 + r]
  volatile int* flag = (volatile int*)(L + NB * NB);
  const int warp = g.tid >> 5, lane = g.tid & 31;
  const int r0 = jp * NB, c0 = warp * PB;
  const df zero = df_make(0.f, 0.f), one = df_make(1.f, 0.f);
  cdf a[PB];
#pragma unroll
  for (int j = 0; j < PB; ++j) {
    a[j] = cdf_make(lane == c0 + j ? one : zero, zero);   // rows past the matrix: identity
    if (lane >= c0 + j && r0 + lane < N) a[j] = ldcg4(A + (size_t)(r0 + lane) * N + r0 + c0 + j);
  }
  g.sync();                                  // the previous block's columns have been read
  if (g.tid < NB) flag[g.tid] = 0;
  g.sync();
  // all but the last earlier column; that one joins the warp's own (its products for the first own
  // column are the ones on the chain, the others fill the pivot's latency)
#pragma unroll 1
  for (int k = 0; k + 1 < c0; ++k) {
    flag_wait(flag + k, status);
    const cdf lr = L[k * NB + lane];
#pragma unroll
    for (int j = 0; j < PB; ++j) sub_mulc(a[j], lr, L[k * NB + c0 + j]);
  }
  if (c0 > 0) {
    flag_wait(flag + c0 - 1, status);
    const cdf lr = L[(c0 - 1) * NB + lane];
#pragma unroll
    for (int j = 0; j < PB; ++j) sub_mulc(a[j], lr, L[(c0 - 1) * NB + c0 + j]);
  }
  df y[PB];
  bool bad = false;
  panel_steps<0>(a, y, c0, L, flag, bad);
#pragma unroll
  for (int j = 0; j < PB; ++j) {
    if (lane >= c0 + j && r0 + lane < N) A[(size_t)(r0 + lane) * N + r0 + c0 + j] = st4(a[j]);
    if (lane == 0 && r0 + c0 + j < N) inv[r0 + c0 + j] = make_float2(y[j].h, y[j].l);
  }
  if (bad && lane == 0) set_flag(status, ST_CHOL);
  __threadfence();
  __syncwarp();
  if (lane == 0) atomicOr(done, 1u << warp);
}

// D = L^{-1} of diagonal block jp (final), by 2 x 2 blocks of 16:
//   D11 = L11^{-1}, D22 = L22^{-1} (forward substitution of the unit vectors, one column per
//   half-warp, compensated accumulation), then D21 = -D22 (L21 D11) as two 16 x 16 products.
__device__ __forceinline__ void trtri_task(int N, const float4* A, const float2* inv, float4* D,
                                           int jp, unsigned char* smem, const Grp& g) {
  constexpr int H = NB / 2;
  cdf(*Ls)[NB + 1] = (cdf(*)[NB + 1])smem;                                  // [32][33]
  cdf(*Ds)[NB + 1] = (cdf(*)[NB + 1])(smem + NB * (NB + 1) * 16);           // [32][33]
  cdf(*Ts)[H + 1] = (cdf(*)[H + 1])(smem + 2 * NB * (NB + 1) * 16);         // [16][17]
  df* ys = (df*)(smem + 2 * NB * (NB + 1) * 16 + H * (H + 1) * 16);
  const int warp = g.tid >> 5, lane = g.tid & 31;
  const int r0 = jp * NB;
  const df zero = df_make(0.f, 0.f), one = df_make(1.f, 0.f);
  for (int e = g.tid; e < NB * NB; e += CS_THREADS) {
    const int r = e / NB, c = e % NB;
    Ls[r][c] = (c < r && r0 + r < N) ? ldcg4(A + (size_t)(r0 + r) * N + r0 + c) : czero();
  }
  if (g.tid < NB) {
    const float2 v = r0 + g.tid < N ? __ldcg(inv + r0 + g.tid) : make_float2(1.f, 0.f);
    ys[g.tid] = df_make(v.x, v.y);
  }
  g.sync();
  // the 32 unit-vector solves (block b, column j) in two passes of 16 half-warps; rows above j
  // come out as zero by themselves (right-hand side and accumulator are zero there)
  const int hl = lane & (H - 1);
#pragma unroll 1
  for (int pass = 0; pass < 2; ++pass) {
    const int sp = 2 * warp + (lane >> 4) + H * pass;
    const int b = sp / H, j = sp % H, o = b * H;
    cacc acc = cacc_zero();
    cdf dv = czero();
    for (int k = 0; k < H; ++k) {
      const cdf v = cdf_scale(cdf_sub(cdf_make(k == j ? one : zero, zero), cacc_val(acc)), ys[o + k]);
      cdf bk;
      bk.re.h = __shfl_sync(0xffffffffu, v.re.h, k, H);
      bk.re.l = __shfl_sync(0xffffffffu, v.re.l, k, H);
      bk.im.h = __shfl_sync(0xffffffffu, v.im.h, k, H);
      bk.im.l = __shfl_sync(0xffffffffu, v.im.l, k, H);
      if (hl == k) dv = bk;
      if (hl > k) cacc_mul(acc, Ls[o + hl][o + k], bk);
    }
    Ds[o + hl][o + j] = dv;
    Ds[o + hl][H - o + j] = czero();      // the other 16 columns of these rows: D12 = 0 / D21 later
  }
  g.sync();
  // T = L21 D11, then D21 = -D22 T
  const int r = g.tid / H, c = g.tid % H;
  cacc t = cacc_zero();
#pragma unroll 4
  for (int m = 0; m < H; ++m) cacc_mul(t, Ls[H + r][m], Ds[m][c]);
  Ts[r][c] = cacc_val(t);
  g.sync();
  cacc u = cacc_zero();
#pragma unroll 4
  for (int m = 0; m < H; ++m) cacc_mul(u, Ds[H + r][H + m], Ts[m][c]);
  const cdf d21 = cacc_val(u);
  Ds[H + r][c] = cdf_make(df_neg(d21.re), df_neg(d21.im));
  g.sync();
  for (int e = g.tid; e < NB * NB; e += CS_THREADS) {
    const int rr = e / NB, cc = e % NB;
    if (r0 + rr < N) D[((size_t)jp * NB + rr) * NB + cc] = st4(Ds[rr][cc]);
  }
}

// Control words of one factorisation (zeroed before its launch), per matrix m:
//   ticket[p], role[p]               counters of the worker tasks and of the CTAs of launch p
//   diag  [li][m]                    finished 8 x 8 updates of diagonal block li
//   pdone [li][m]                    bit w: columns 4w.. of diagonal factor li published
//   slabdone[m][l][b]                finished 8-row panel slabs of block column l in row block b
//   tilecnt [m][r][c]                trailing updates applied to tile (r, c)
struct CholCtl {
  unsigned* w;
  int T, N;
  __device__ CholCtl(unsigned* ctl, int n) : w(ctl), T((n + NB - 1) / NB), N(n) {}
  // launches start PANEL block columns apart
  __device__ unsigned* ticket(int lo) const { return w + 2 * (lo / PANEL); }
  __device__ unsigned* role(int lo) const { return w + 2 * (lo / PANEL) + 1; }
  __device__ unsigned* diag(int li, int m) const { return w + (T + 2) + 2 * li + m; }
  __device__ unsigned* pdone(int li, int m) const { return w + 3 * (T + 2) + 2 * li + m; }
  __device__ unsigned* sd(int m, int l, int b) const { return w + 5 * (T + 2) + ((size_t)m * (T + 1) + l) * T + b; }
  __device__ unsigned* tc(int m, int r, int c) const {
    return w + 5 * (T + 2) + 2 * (size_t)(T + 1) * T + ((size_t)m * T + r) * T + c;
  }
  __device__ unsigned slabs_in(int b) const {
    const int rows = N - b * NB < NB ? N - b * NB : NB;
    return (unsigned)((rows + TS_ROWS - 1) / TS_ROWS);
  }
};

// column c is one of the eight from k0
constexpr int SB = 8;   // columns a slab takes at a time
__device__ __forceinline__ bool lane_of(int c, int k0) { return (c & ~(SB - 1)) == k0; }

// threads 0..2 wait (bounded) for one control word each, then fence; the caller synchronises the group
__device__ __forceinline__ void wait_counts(const Grp& g, const unsigned* f0, unsigned t0, const unsigned* f1,
                                            unsigned t1, const unsigned* f2, unsigned t2, int* status) {
  if (g.tid < 3) {
    const unsigned* f = g.tid == 0 ? f0 : (g.tid == 1 ? f1 : f2);
    const unsigned t = g.tid == 0 ? t0 : (g.tid == 1 ? t1 : t2);
    if (t > 0) {
      cs_wait(f, t, status);
      __threadfence();
    }
  }
}
// thread 0 waits (bounded) until *f >= target, then fences; the caller synchronises the group
__device__ __forceinline__ void wait_count(const Grp& g, const unsigned* f, unsigned target, int* status) {
  if (g.tid == 0 && target > 0) {
    cs_wait(f, target, status);
    __threadfence();
  }
}

// Tasks of block column li besides its diagonal factor, per matrix, in a launch over the block columns
// [lo, hi): the updates from its own columns to the columns up to hi.
struct StepTasks {
  int diag, herk, slab, inv, tiles;   // tiles: of the whole trailing triangle
  __host__ __device__ StepTasks(int N, int lo, int hi, int li) {
    const int T = (N + NB - 1) / NB, rt = T - li - 1, rows = N - (li + 1) * NB, w = hi - 1 - li;
    diag = (li > lo && li < hi) ? DIAG_TASKS : 0;
    tiles = rt * (rt + 1) / 2;
    herk = (li > lo && w > 0) ? w * rt - w * (w - 1) / 2 : 0;
    slab = (li < hi && rows > 0) ? (rows + TS_ROWS - 1) / TS_ROWS : 0;
    inv = li > lo ? 1 : 0;
  }
  __host__ __device__ int count() const { return diag + herk + slab + inv; }
};

// Task t of block column li (all matrices).
__device__ __forceinline__ void chol_task(const Grp& g, int N, const Batch& mb, int nb, int lo, int li, int t, const StepTasks& st,
                                          const CholCtl& cc, int* status, unsigned char* sm) {
  const int jp = li, jb = li - 1;
  const unsigned before = (unsigned)(li > lo ? jb - lo : 0);   // earlier updates of a tile in this launch
  if (t < nb * st.diag) {
    // 8 x 8 block (rb, cb) of diagonal block jp: A -= L_jp,jb L_jp,jb^H; needs panel jb on the rows
    // of block jp and the earlier trailing updates of the diagonal tile
    const int m = t % nb;
    int cb, rb;
    tri_index(t / nb, cb, rb);
    wait_counts(g, cc.sd(m, jb, jp), cc.slabs_in(jp), cc.tc(m, jp, jp), before, nullptr, 0, status);
    g.sync();
    diag_update8(pick2(mb.m, m), N, jp, jb, rb, cb, sm, g);
    cs_signal(g, cc.diag(li, m));
    return;
  }
  t -= nb * st.diag;
  // trailing tiles, the slabs after the first AHEAD_TILES of them
  const int ahead = nb * st.herk < AHEAD_TILES ? nb * st.herk : AHEAD_TILES;
  const bool slab = t >= ahead && t < ahead + nb * st.slab;
  if (t < nb * (st.herk + st.slab) && !slab) {
    if (t >= ahead) t -= nb * st.slab;
    const int m = t % nb;
    // block columns from the left (the next steps need them first), rows from the diagonal
    int I, J;
    tri_index(st.tiles - 1 - t / nb, I, J);
    const int rb = cc.T - 1 - I, cb = cc.T - 1 - J;
    // panel jb on both row blocks, and the tile's earlier updates
    wait_counts(g, cc.sd(m, jb, rb), cc.slabs_in(rb), cc.sd(m, jb, cb), cc.slabs_in(cb), cc.tc(m, rb, cb),
                before, status);
    g.sync();
    herk_tile(pick2(mb.m, m), N, jb, rb, cb, sm, g);
    cs_signal(g, cc.tc(m, rb, cb));
    return;
  }
  if (slab) {
    // panel slab: rows i0..i0+7 of block column jp.  a = A - L_i,jb L_jp,jb^H, then x L^H = a by
    // substitution along the row (warp = row, lane = column): x_m = (a_m - sum_k<m x_k conj(L_mk)) / L_mm
    t -= ahead;
    const int m = t % nb, sl = t / nb;
    float4* A = pick2(mb.m, m);
    const float2* inv = pick2(mb.inv, m);
    const int i0 = (jp + 1) * NB + sl * TS_ROWS;
    const int r = g.tid / NB, c = g.tid % NB;
    const bool ok = i0 + r < N;
    const int bi = i0 / NB;
    if (li > lo) {
      // panel jb on these rows and on the rows of block jp, and the tile's earlier updates
      wait_counts(g, cc.sd(m, jb, bi), cc.slabs_in(bi), cc.sd(m, jb, jp), cc.slabs_in(jp), cc.tc(m, bi, jp),
                  before, status);
      g.sync();
    }
    cdf a;
    if (li > lo) a = upd_one<TS_ROWS, NB>(A, N, i0, jp * NB, jb * NB, i0 + r, jp * NB + c, ok, sm, g);
    else a = ok ? ldcg4(A + (size_t)(i0 + r) * N + jp * NB + c) : czero();
    // with L' = L diag(y) (y_k = 1 / L_kk) and x = z diag(y): z_k = a_k - sum_j<k z_j conj(L'_kj), so
    // the chain carries no scaling.  Eight columns at a time, as the diagonal factor publishes them:
    // only the last eight are left when it finishes.
    cdf z = czero();
    df yc = df_make(0.f, 0.f);
#pragma unroll 1
    for (int k0 = 0; k0 < NB; k0 += SB) {
      if (g.tid == 0) {
        cs_wait<true>(cc.pdone(li, m), (1u << ((k0 + SB) / PB)) - 1u, status);
        __threadfence();
      }
      g.sync();
      cdf lk[SB];
      const float4* lp = A + (size_t)(jp * NB + c) * N + jp * NB + k0;
      const float2 yv = lane_of(c, k0) ? __ldcg(inv + jp * NB + c) : make_float2(0.f, 0.f);
#pragma unroll
      for (int k = 0; k < SB; ++k) lk[k] = k0 + k < c ? ldcg4(lp + k) : czero();
      if (lane_of(c, k0)) yc = df_make(yv.x, yv.y);
#pragma unroll
      for (int k = 0; k < SB; ++k) {
        df y;
        y.h = __shfl_sync(0xffffffffu, yv.x, k0 + k);
        y.l = __shfl_sync(0xffffffffu, yv.y, k0 + k);
        lk[k] = cdf_scale(lk[k], y);
      }
#pragma unroll
      for (int k = 0; k < SB; ++k) {
        a = renorm(a);
        const cdf zk = shfl_cdf(a, k0 + k);
        if (c == k0 + k) z = zk;
        sub_mulc(a, zk, lk[k]);   // lk = 0 for c <= k
      }
    }
    if (ok) {
      const cdf x = cdf_scale(z, yc);
      A[(size_t)(i0 + r) * N + jp * NB + c] = st4(x);
      // L^H in the (otherwise unused) upper triangle: the backward solve reads it by rows
      A[(size_t)(jp * NB + c) * N + i0 + r] = st4(cdf_make(x.re, df_neg(x.im)));
    }
    cs_signal(g, cc.sd(m, li, bi));
    return;
  }
  t -= nb * (st.herk + st.slab);
  {
    // inverse of the previous diagonal block (final once its factor is published), for the solves
    const int m = t;
    if (g.tid == 0) {
      cs_wait<true>(cc.pdone(li - 1, m), (1u << (NB / PB)) - 1u, status);
      __threadfence();
    }
    g.sync();
    trtri_task(N, pick2(mb.m, m), pick2(mb.inv, m), pick2(mb.D, m), jp - 1, sm, g);
  }
}

__global__ void __launch_bounds__(CTA_THREADS, 1) k_chol_df(int N, Batch mb, int nb, int lo, int hi, unsigned* ctl, int* status) {
  extern __shared__ __align__(16) unsigned char smem_all[];
  __shared__ unsigned s_role, s_t[2];
  const CholCtl cc(ctl, N);
  if (threadIdx.x == 0) s_role = atomicAdd(cc.role(lo), 1u);
  __syncthreads();
  const int half = threadIdx.x / CS_THREADS;
  const Grp g{(int)threadIdx.x % CS_THREADS, 1 + half};
  unsigned char* sm = smem_all + half * CS_SMEM;
  if ((int)s_role < nb) {
    if (half) return;
    const int m = (int)s_role;
    for (int li = lo; li < hi; ++li) {
      if (li > lo) wait_count(g, cc.diag(li, m), (unsigned)DIAG_TASKS, status);
      g.sync();
      potrf_task(N, pick2(mb.m, m), pick2(mb.inv, m), li, status, cc.pdone(li, m), sm, g);
    }
    return;
  }
  int li = lo;
  unsigned base = 0;
  StepTasks st(N, lo, hi, lo);
  while (true) {
    if (g.tid == 0) s_t[half] = atomicAdd(cc.ticket(lo), 1u);
    g.sync();
    const unsigned t = s_t[half];
    g.sync();   // shared memory of the previous task and s_t are free after this
    while (li <= hi && t - base >= (unsigned)(nb * st.count())) {
      base += nb * st.count();
      st = StepTasks(N, lo, hi, ++li);
    }
    if (li > hi) return;
    chol_task(g, N, mb, nb, lo, li, (int)(t - base), st, cc, status, sm);
  }
}

// ---------------------------------------------------------------------------- triangular solves

constexpr int TW = 8;
constexpr int CW = 4;
constexpr int CPW = NB / CW;

__device__ __forceinline__ bool wait_flag(const unsigned* f, unsigned epoch, int* status) {
  const unsigned lim = wait_budget(status, WAIT_LIMIT);
  for (unsigned it = 0; it < lim; ++it) {
    if (ld_acquire(f) == epoch) return true;
    if (it > 4096) __nanosleep(64);
  }
  set_flag(status, ST_TIMEOUT);
  return false;
}
__device__ __forceinline__ void named_sync(int id, int n) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}
__device__ __forceinline__ void fence_acq_rel_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }

// Forward solve L z = y (z published as double-floats, consumers wait on per-block flags).
// Same schedule as the FP64 kernel: warps CW.. accumulate the older blocks, warps 0..CW-1 share the
// critical block jb-1 and the diagonal product with D_jb.
__global__ void __launch_bounds__(TW * 32) k_trsv_lower_df(int N, const float4* __restrict__ L,
                                                          const float4* __restrict__ D,
                                                          const double2* __restrict__ y,
                                                          float4* __restrict__ z, unsigned* flags,
                                                          unsigned* ticket, unsigned epoch,
                                                          int* status) {
  __shared__ cacc part[TW][NB];
  __shared__ cdf Ds[NB][NB + 1];
  __shared__ cdf vsh[NB];
  __shared__ int s_jb;
  if (threadIdx.x == 0) s_jb = (int)atomicAdd(ticket, 1u);
  __syncthreads();
  const int jb = s_jb;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r0 = jb * NB;
  for (int e = threadIdx.x; e < NB * NB; e += blockDim.x) {
    const int r = e / NB, c = e % NB;
    Ds[r][c] = (r0 + r < N) ? ld4(D[((size_t)jb * NB + r) * NB + c]) : czero();
  }
  const bool row_ok = r0 + lane < N;
  const float4* Lrow = L + (size_t)(row_ok ? r0 + lane : 0) * N;
  cacc acc = cacc_zero();
  for (int m = warp - CW; warp >= CW && m < jb - 1; m += TW - CW) {
    if (lane == 0) wait_flag(flags + m, epoch, status);
    __syncwarp();
    const cdf zm = ldcg4(z + m * NB + lane);
#pragma unroll 8
    for (int c = 0; c < NB; ++c) cacc_mul(acc, ld4(__ldg(Lrow + m * NB + c)), shfl_cdf(zm, c));
  }
  if (warp >= CW) part[warp][lane] = acc;
  const int mc = jb - 1;
  cdf lv[CPW];
#pragma unroll
  for (int q = 0; q < CPW; ++q)
    lv[q] = (warp < CW && mc >= 0) ? ld4(__ldg(Lrow + mc * NB + warp * CPW + q)) : czero();
  // the right-hand side, converted off the chain
  const double2 yv = (warp == 0 && row_ok) ? y[r0 + lane] : make_double2(0.0, 0.0);
  const cdf yc = cdf_make(df_from(yv.x), df_from(yv.y));
  __syncthreads();
  if (warp >= CW) return;
  cacc p = cacc_zero();
  if (mc >= 0) {
    if (lane == 0) wait_flag(flags + mc, epoch, status);
    __syncwarp();
    const cdf zm = ldcg4(z + mc * NB + lane);
#pragma unroll
    for (int q = 0; q < CPW; ++q) cacc_mul(p, lv[q], shfl_cdf(zm, warp * CPW + q));
  }
  part[warp][lane] = p;
  named_sync(1, CW * 32);
  if (warp == 0) {
    cacc s = part[0][lane];
#pragma unroll
    for (int w = 1; w < TW; ++w) s = cacc_merge(s, part[w][lane]);
    vsh[lane] = row_ok ? cdf_sub(yc, cacc_val(s)) : czero();
  }
  named_sync(1, CW * 32);
  cacc o = cacc_zero();
#pragma unroll
  for (int q = 0; q < CPW; ++q) {
    const int c = warp * CPW + q;
    cacc_mul(o, Ds[lane][c], vsh[c]);
  }
  part[warp][lane] = o;
  named_sync(1, CW * 32);
  if (warp == 0) {
    cacc s = part[0][lane];
#pragma unroll
    for (int w = 1; w < CW; ++w) s = cacc_merge(s, part[w][lane]);
    if (row_ok) z[r0 + lane] = st4(cacc_val(s));
    fence_acq_rel_gpu();
    __syncwarp();
    if (lane == 0) st_release(flags + jb, epoch);
  }
}

// Backward solve L^H w = z (double-floats), out = w or -i w in FP64.
__global__ void __launch_bounds__(TW * 32) k_trsv_upper_df(int N, const float4* __restrict__ L,
                                                          const float4* __restrict__ D,
                                                          const float4* __restrict__ z,
                                                          double2* __restrict__ w_out, bool minus_i,
                                                          float4* __restrict__ wbuf, unsigned* flags,
                                                          unsigned* ticket, unsigned epoch,
                                                          int* status) {
  __shared__ cacc part[TW][NB];
  __shared__ cdf Ds[NB][NB + 1];
  __shared__ cdf vsh[NB];
  __shared__ int s_jb;
  const int nblk = (N + NB - 1) / NB;
  if (threadIdx.x == 0) s_jb = nblk - 1 - (int)atomicAdd(ticket, 1u);
  __syncthreads();
  const int jb = s_jb;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r0 = jb * NB;
  for (int e = threadIdx.x; e < NB * NB; e += blockDim.x) {
    const int r = e / NB, c = e % NB;
    Ds[r][c] = (r0 + r < N) ? ld4(D[((size_t)jb * NB + r) * NB + c]) : czero();
  }
  const bool col_ok = r0 + lane < N;
  cacc acc = cacc_zero();
  for (int m = nblk - 1 - (warp - CW); warp >= CW && m >= jb + 2; m -= TW - CW) {
    if (lane == 0) wait_flag(flags + m, epoch, status);
    __syncwarp();
    const cdf wm = (m * NB + lane < N) ? ldcg4(wbuf + m * NB + lane) : czero();
#pragma unroll 8
    for (int c = 0; c < NB; ++c) {
      const cdf l = (m * NB + c < N && col_ok) ? ld4(__ldg(L + (size_t)(m * NB + c) * N + r0 + lane))
                                                 : czero();
      cacc_cmul(acc, l, shfl_cdf(wm, c));
    }
  }
  if (warp >= CW) part[warp][lane] = acc;
  const int mc = jb + 1;
  cdf lv[CPW];
#pragma unroll
  for (int q = 0; q < CPW; ++q) {
    const int c = warp * CPW + q;
    lv[q] = (warp < CW && mc < nblk && mc * NB + c < N && col_ok)
                ? ld4(__ldg(L + (size_t)(mc * NB + c) * N + r0 + lane))
                : czero();
  }
  const cdf zc = (warp == 0 && col_ok) ? ld4(z[r0 + lane]) : czero();
  __syncthreads();
  if (warp >= CW) return;
  cacc p = cacc_zero();
  if (mc < nblk) {
    if (lane == 0) wait_flag(flags + mc, epoch, status);
    __syncwarp();
    const cdf wm = (mc * NB + lane < N) ? ldcg4(wbuf + mc * NB + lane) : czero();
#pragma unroll
    for (int q = 0; q < CPW; ++q) cacc_cmul(p, lv[q], shfl_cdf(wm, warp * CPW + q));
  }
  part[warp][lane] = p;
  named_sync(1, CW * 32);
  if (warp == 0) {
    cacc s = part[0][lane];
#pragma unroll
    for (int w = 1; w < TW; ++w) s = cacc_merge(s, part[w][lane]);
    vsh[lane] = col_ok ? cdf_sub(zc, cacc_val(s)) : czero();
  }
  named_sync(1, CW * 32);
  // w_r = sum_c conj(D_cr) v_c
  cacc o = cacc_zero();
#pragma unroll
  for (int q = 0; q < CPW; ++q) {
    const int c = warp * CPW + q;
    cacc_cmul(o, Ds[c][lane], vsh[c]);
  }
  part[warp][lane] = o;
  named_sync(1, CW * 32);
  if (warp == 0) {
    cacc s = part[0][lane];
#pragma unroll
    for (int w = 1; w < CW; ++w) s = cacc_merge(s, part[w][lane]);
    const cdf wv = cacc_val(s);
    if (col_ok) wbuf[r0 + lane] = st4(wv);
    fence_acq_rel_gpu();
    __syncwarp();
    if (lane == 0) st_release(flags + jb, epoch);
    if (col_ok) {
      const double re = df_to(wv.re), im = df_to(wv.im);
      w_out[r0 + lane] = minus_i ? make_double2(im, -re) : make_double2(re, im);
    }
  }
}

}  // namespace dfs

// ---------------------------------------------------------------------------- launchers

void launch_shift_mix_df(int N, const double2* S0, const double2* S1, double eps, double theta,
                         void* A, cudaStream_t s) {
  dfs::k_shift_mix_df<<<N, 256, 0, s>>>(N, S0, S1, eps, theta, (float4*)A);
}

cudaError_t cholesky_df_attributes() {
  return cudaFuncSetAttribute(dfs::k_chol_df, cudaFuncAttributeMaxDynamicSharedMemorySize, dfs::CS_SMEM_LAUNCH);
}

int launch_cholesky_df(int N, void* const* A, void* const* inv, void* const* D, int nbatch,
                       unsigned* ctl, void* herk_scratch, int* status, cudaStream_t s) {
  using namespace dfs;
  Batch mb;
  for (int q = 0; q < 2; ++q) {
    const int k = (nbatch > 1 && q == 1) ? 1 : 0;
    mb.m[q] = (float4*)A[k];
    mb.inv[q] = (float2*)inv[k];
    mb.D[q] = (float4*)D[k];
  }
  const int T = (N + NB - 1) / NB;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaMemsetAsync(ctl, 0, chol_ctl_words(N) * sizeof(unsigned), s);
  int launches = 0;
  for (int lo = 0, hi; lo < T; lo = hi) {
    hi = herk_scratch && T - lo > ONE_LAUNCH ? lo + PANEL : T;
    // chain CTAs and two groups per worker CTA, no more workers than the widest step has tasks
    int widest = 1;
    for (int li = lo; li <= hi; ++li) widest = std::max(widest, nbatch * StepTasks(N, lo, hi, li).count());
    const int grid = std::min(std::max(sms, nbatch + 1), nbatch + (widest + 1) / 2);
    k_chol_df<<<grid, CTA_THREADS, CS_SMEM_LAUNCH, s>>>(N, mb, nbatch, lo, hi, ctl, status);
    ++launches;
    if (hi < T) launches += launch_herk_df(N, lo * NB, hi * NB, A, nbatch, herk_scratch, status, s);
  }
  return launches + launch_near_products(N, A, D, nbatch, true, s);
}

int chol_panel(int N) { return (N + dfs::NB - 1) / dfs::NB > dfs::ONE_LAUNCH ? dfs::PANEL : 0; }
size_t chol_ctl_words(int N) {
  const size_t T = (N + dfs::NB - 1) / dfs::NB;
  return 5 * (T + 2) + 2 * (T + 1) * T + 2 * T * T;
}

int launch_chol_solve_df(int N, const void* L, const void* D, const double2* y, void* work,
                          double2* out, bool minus_i, unsigned* flags, unsigned* tickets,
                          unsigned epoch, int* status, cudaStream_t s) {
  using namespace dfs;
  if (launch_cluster_solve(N, L, D, y, out, minus_i, true, status, s)) return 1;
  const int nblk = (N + NB - 1) / NB;
  // block flags and tickets (which follow them) start from zero in every solve, so a captured
  // launch sequence can be replayed with the same epoch
  cudaMemsetAsync(flags, 0, (2 * (size_t)nblk + 2) * sizeof(unsigned), s);
  (void)tickets;
  float4* zb = (float4*)work;
  k_trsv_lower_df<<<nblk, TW * 32, 0, s>>>(N, (const float4*)L, (const float4*)D, y, zb, flags,
                                            flags + 2 * nblk, epoch, status);
  k_trsv_upper_df<<<nblk, TW * 32, 0, s>>>(N, (const float4*)L, (const float4*)D, zb, out, minus_i,
                                            zb + N, flags + nblk, flags + 2 * nblk + 1, epoch, status);
  return 2;
}

}  // namespace icwf
