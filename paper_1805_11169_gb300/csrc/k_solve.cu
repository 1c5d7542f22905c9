// Triangular solves of the coefficient equation for N <= 2048, both passes in one launch of one
// 16-CTA thread-block cluster, in double-float (mixed modes) or FP64 arithmetic.
//
// Kernels: k_near_products (beside the factorisation), k_cluster_solve.
#include <cuda_runtime.h>

#include "cdf.cuh"
#include "icwf_internal.h"
#include "k_common.cuh"

namespace icwf {
namespace slv {

constexpr int NB = 32;         // block size of the factorisation
constexpr int CL = 16;         // CTAs per cluster
constexpr int ROWS = NB / CL;  // rows of every block that a CTA owns
constexpr int WARPS = 16;
constexpr int MAX_BLOCKS = 64; // largest size: 4 blocks per warp
constexpr unsigned long long CWAIT_NS = 2000000000ull;

// Double-float arithmetic: 16-byte elements, compensated accumulators; the factor's upper triangle holds
// L^H.
struct Df {
  using E = float4;
  using V = cdf;
  using Acc = dfs::cacc;
  using Part = dfs::acc2;   // one component of an accumulator
  static constexpr bool UPPER = true;
  __device__ static V load(E e) { return dfs::ld4(e); }
  __device__ static E store(V v) { return dfs::st4(v); }
  __device__ static V zero() { return dfs::czero(); }
  __device__ static Acc acc_zero() { return dfs::cacc_zero(); }
  __device__ static void mul(Acc& a, V x, V y) { dfs::cacc_mul(a, x, y); }
  __device__ static void cmul(Acc& a, V x, V y) { dfs::cacc_cmul(a, x, y); }
  __device__ static V val(const Acc& a) { return dfs::cacc_val(a); }
  __device__ static V neg(V v) {
    return cdf_make(df_make(-v.re.h, -v.re.l), df_make(-v.im.h, -v.im.l));
  }
  __device__ static V conj(V v) { return cdf_make(v.re, df_make(-v.im.h, -v.im.l)); }
  __device__ static V sub(V a, V b) { return cdf_sub(a, b); }
  __device__ static V from(double2 y) { return cdf_make(df_from(y.x), df_from(y.y)); }
  __device__ static double2 to(V v) { return make_double2(df_to(v.re), df_to(v.im)); }
  __device__ static Part part(const Acc& a, bool im) {
    Part p;
    p.s = im ? a.im.s : a.re.s;
    p.c = im ? a.im.c : a.re.c;
    return p;
  }
  __device__ static Part add_shfl(Part a, Part give, int o) {
    Part b;
    b.s = __shfl_xor_sync(0xffffffffu, give.s, o);
    b.c = __shfl_xor_sync(0xffffffffu, give.c, o);
    return dfs::acc_merge(a, b);
  }
  __device__ static V join(Part p, bool im, int o) {
    const df a = dfs::acc_val(p);
    const df b = df_make(__shfl_xor_sync(0xffffffffu, a.h, o), __shfl_xor_sync(0xffffffffu, a.l, o));
    return im ? cdf_make(b, a) : cdf_make(a, b);
  }
};

// FP64 arithmetic; L^H is read from the lower triangle.
struct F64 {
  using E = double2;
  using V = double2;
  using Acc = double2;
  using Part = double;
  static constexpr bool UPPER = false;
  __device__ static V load(E e) { return e; }
  __device__ static E store(V v) { return v; }
  __device__ static V zero() { return make_double2(0.0, 0.0); }
  __device__ static Acc acc_zero() { return zero(); }
  __device__ static void mul(Acc& a, V x, V y) { cfma(a, x, y); }
  __device__ static void cmul(Acc& a, V x, V y) { cfmac(a, x, y); }
  __device__ static V val(const Acc& a) { return a; }
  __device__ static V neg(V v) { return make_double2(-v.x, -v.y); }
  __device__ static V conj(V v) { return cconj(v); }
  __device__ static V sub(V a, V b) { return csub(a, b); }
  __device__ static V from(double2 y) { return y; }
  __device__ static double2 to(V v) { return v; }
  __device__ static Part part(const Acc& a, bool im) { return im ? a.y : a.x; }
  __device__ static Part add_shfl(Part a, Part give, int o) { return a + __shfl_xor_sync(0xffffffffu, give, o); }
  __device__ static V join(Part p, bool im, int o) {
    const double b = __shfl_xor_sync(0xffffffffu, p, o);
    return im ? make_double2(b, p) : make_double2(p, b);
  }
};

// ---------------------------------------------------------------------------- neighbour products

// Negated products of the inverted diagonal blocks with the two blocks next to them, per block row m:
//   P[0] = -D_m L[m, m-1], P[1] = -D_m L[m, m-2] (forward), P[2] = -D_m^H L^H[m, m+1],
//   P[3] = -D_m^H L^H[m, m+2] (backward), each stored as rows of 32 like D.
// grid (4 x block rows, 4, matrices): 8 rows per CTA, warp = row, lane = column, so that two warps share
// a scheduler and the 32 terms of an entry run at latency, not at issue rate (32 rows per CTA, double
// floats: 9 us for two matrices at N = 64, now 5).  The triangular factor's zeros are skipped.  With the
// products a solve's chain has one 32 x 32 product per block instead of two.
constexpr int NPR = 8;
template <class T>
__global__ void __launch_bounds__(NPR * 32) k_near_products(int N, const typename T::E* __restrict__ L0,
                                                            const typename T::E* __restrict__ L1,
                                                            const typename T::E* __restrict__ D0,
                                                            const typename T::E* __restrict__ D1,
                                                            typename T::E* __restrict__ P0,
                                                            typename T::E* __restrict__ P1) {
  using V = typename T::V;
  __shared__ V Ds[NPR][NB + 1], Bs[NB][NB + 1];
  const int per = NB / NPR, nb = gridDim.x / per, m = blockIdx.x / per, which = blockIdx.y;
  const typename T::E* L = blockIdx.z ? L1 : L0;
  const typename T::E* D = blockIdx.z ? D1 : D0;
  typename T::E* P = (blockIdx.z ? P1 : P0) + (size_t)which * nb * NB * NB;
  const bool fwd = which < 2;
  const int j = fwd ? m - 1 - which : m + 1 + (which - 2);
  if (j < 0 || j >= nb) return;
  const int w = threadIdx.x >> 5, c = threadIdx.x & 31, r0 = (blockIdx.x % per) * NPR, r = r0 + w;
  if (fwd) {
    const int row = m * NB + r;
    Ds[w][c] = row < N ? T::load(D[(size_t)row * NB + c]) : T::zero();
  } else {   // D^H's rows r0.. are D's columns
    const int k = threadIdx.x / NPR, q = threadIdx.x % NPR;
    Ds[q][k] = m * NB + k < N ? T::load(D[(size_t)(m * NB + k) * NB + r0 + q]) : T::zero();
  }
#pragma unroll
  for (int i = 0; i < NB / NPR; ++i) {
    const int k = w + NPR * i;
    if (fwd || T::UPPER) {
      const int row = m * NB + k, col = j * NB + c;
      Bs[k][c] = row < N && col < N ? T::load(L[(size_t)row * N + col]) : T::zero();
    } else {   // L[j, m], entry (k, c): L^H[m, j] is its conjugate transpose
      const int row = j * NB + k, col = m * NB + c;
      Bs[c][k] = row < N && col < N ? T::conj(T::load(L[(size_t)row * N + col])) : T::zero();
    }
  }
  __syncthreads();
  typename T::Acc s = T::acc_zero();
  if (fwd) {
    for (int k = 0; k <= r; ++k) T::mul(s, Ds[w][k], Bs[k][c]);
  } else {
    for (int k = r; k < NB; ++k) T::cmul(s, Ds[w][k], Bs[k][c]);
  }
  P[(size_t)(m * NB + r) * NB + c] = T::store(T::neg(T::val(s)));
}

// ---------------------------------------------------------------------------- cluster primitives

__device__ __forceinline__ uint32_t s_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ unsigned long long gtime_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t map_rank(uint32_t local, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(rank));
  return r;
}
__device__ __forceinline__ void bar_init(uint64_t* b, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(s_u32(b)), "r"(count) : "memory");
}
__device__ __forceinline__ void bar_expect(uint64_t* b, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(s_u32(b)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool bar_try(uint64_t* b) {   // phase 0; may wait a while by itself
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], 0;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(s_u32(b))
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool bar_test(uint64_t* b) {  // phase 0, immediate
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], 0;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(s_u32(b))
      : "memory");
  return ok != 0;
}
// store 16 bytes into CTA `rank`'s shared memory (the address is this CTA's twin of it) and complete 16
// bytes of the transaction count of that CTA's barrier `bar`
template <class E>
__device__ __forceinline__ void st_async16(E v, const void* dst_local, uint64_t* bar_local, uint32_t rank) {
  const uint4 u = *reinterpret_cast<const uint4*>(&v);
  const uint32_t dst = map_rank(s_u32(dst_local), rank);
  const uint32_t bar = map_rank(s_u32(bar_local), rank);
  asm volatile(
      "st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];"
      ::"r"(dst), "r"(u.x), "r"(u.y), "r"(u.z), "r"(u.w), "r"(bar)
      : "memory");
}

// ---------------------------------------------------------------------------- cluster solve
//
// Every CTA owns two rows of every block of 32 (CTA k: rows 2k and 2k + 1); within a CTA, warp w owns the
// blocks w, w + 16, ... in the order of the pass, half a warp per row, two columns per lane, with the
// blocks' partial sums in registers.  Every CTA keeps the whole forward solution z and backward solution
// w, in its shared memory.  Forward, with t the order of the blocks (backward alike, from the last block,
// with L^H, D^H and the other P):
//   z_m = D_m s_m - D_m L[m, m-2] z_{m-2} - D_m L[m, m-1] z_{m-1},  s_m = y_m - sum_{j <= m-3} L_mj z_j.
// On the arrival of z_t the warp of block
//   t + 1 adds its product (P[0] z_t), sums over the lanes and sends its two entries of z_{t+1} to the 16
//         CTAs, one 16-byte store per lane: the chain;
//   t + 2 adds P[1] z_t and, s_{t+2} having arrived, D s_{t+2} (per lane, no sum over lanes yet);
//   t + 3 adds L z_t, sums and sends its two entries of s_{t+3};
//   later ones add L z_t.
// A message is 32 st.async per CTA that complete the transaction count of the receiver's barrier of that
// block, so a warp waits on local barriers only and there is no CTA barrier in a pass.
//
// Bound: the chain's latency per block (two products, a sum over 16 lanes, an exchange through
// distributed shared memory), and in FP64 the FP64 pipe.  Rows of every block on every CTA spread the
// chain's product and the later rows' products evenly: with whole blocks dealt to the CTAs, one SM's
// 32 x 32 product (635 cycles in double-float, 2150 in FP64) was on the chain.
// Per step of four solves, before / now, us: double-float 84 / 48 at N = 100, 256 / 121 at 512, 662 / 264
// at 1024, 2330 / 1027 at 2048 (8 CTAs, whole blocks, D on the chain); FP64 250 / 57 at N = 100, 766 / 181
// at 500, 1770 / 437 at 1024 (a CTA per block row, flags in global memory, two launches).  Above N = 2048
// that form stays (64 blocks fill the warps' registers and 133 KB of shared memory).

struct Layout {   // shared memory; arrays of nblk * 32 elements and nblk barriers each
  int nblk;
  unsigned char* base;
  template <class E> __device__ E* vec(int k) const { return (E*)base + (size_t)k * nblk * NB; }   // z, w, s, s'
  __device__ uint64_t* bars(int k) const { return (uint64_t*)(base + (size_t)4 * nblk * NB * 16) + k * nblk; }
  __device__ int* abort_flag() const { return (int*)(bars(4)); }
};
constexpr size_t smem_bytes(int nblk) { return (size_t)4 * nblk * (NB * 16 + 8) + 16; }

// Bounded wait for a block's barrier.  An overridden poll budget (icwf_set_wait_limit) that runs out
// raises the timeout flag; the wait itself goes on, since stores of other CTAs must not outlive the
// launch.  The timer and the abort flag are looked at every 64th poll: they would lengthen the usual
// short wait.
__device__ __forceinline__ void block_wait(uint64_t* b, volatile int* abort_flag, unsigned budget, int* status) {
  if (budget != ~0u) {
    unsigned n = 0;
    while (n < budget && !bar_test(b)) ++n;
    if (n == budget && !bar_test(b)) set_flag(status, ST_TIMEOUT);
  }
  unsigned long long t0 = 0;
  for (unsigned it = 1; !bar_try(b); ++it) {
    if (it & 63u) continue;
    if (*abort_flag) return;
    const unsigned long long t = gtime_ns();
    if (t0 == 0) t0 = t;
    if (t - t0 > CWAIT_NS) {
      *abort_flag = 1;
      set_flag(status, ST_TIMEOUT);
      return;
    }
  }
}

// Sum over the 16 lanes of a row, to all of them.  The first step splits the components over the halves,
// so that every step merges one of them; merges are symmetric in their operands.
template <class T>
__device__ __forceinline__ typename T::V row_sum(const typename T::Acc& a) {
  const bool im = threadIdx.x & 8;
  typename T::Part p = T::add_shfl(T::part(a, im), T::part(a, !im), 8);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) p = T::add_shfl(p, p, o);
  return T::join(p, im, 8);
}

// One pass.  NI: blocks per warp.
template <class T, int NI, bool FWD>
__device__ __forceinline__ void pass(const Layout& lay, int N, int rank, const typename T::E* __restrict__ L,
                                     const typename T::E* __restrict__ D, const typename T::E* __restrict__ P,
                                     const double2* __restrict__ y, double2* __restrict__ out, bool minus_i,
                                     unsigned budget, int* status) {
  using E = typename T::E;
  using V = typename T::V;
  const int nblk = lay.nblk, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rb = ROWS * rank + (lane >> 4), c0 = 2 * (lane & 15);   // this lane's row and columns of a block
  E* sol = lay.vec<E>(FWD ? 0 : 1);
  E* svec = lay.vec<E>(FWD ? 2 : 3);
  uint64_t* zbar = lay.bars(FWD ? 0 : 1);
  uint64_t* sbar = lay.bars(FWD ? 2 : 3);
  volatile int* abort_flag = lay.abort_flag();
  const E* P1 = P + (FWD ? (size_t)0 : (size_t)2 * nblk * NB * NB);
  const E* P2 = P1 + (size_t)nblk * NB * NB;
  auto blk = [&](int t) { return FWD ? t : nblk - 1 - t; };
  // operand of block order tau (> t) for z_t: L (L^H) or a neighbour product; FP64's L^H conjugated at use
  auto load_k = [&](int tau, int t, V (&k)[2]) {
    const int row = blk(tau) * NB + rb, col = blk(t) * NB + c0;
    if (tau - t < 3) {
      const E* p = (tau - t == 1 ? P1 : P2) + (size_t)row * NB + c0;
      k[0] = T::load(__ldg(p));
      k[1] = T::load(__ldg(p + 1));
      return;
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const bool in = row < N && col + q < N;
      if (FWD || T::UPPER) k[q] = in ? T::load(__ldg(L + (size_t)row * N + col + q)) : T::zero();
      else k[q] = in ? T::load(__ldg(L + (size_t)(col + q) * N + row)) : T::zero();
    }
  };
  typename T::Acc acc[NI];
  V k[NI][2], kd[2], rhs[NI];
#pragma unroll
  for (int i = 0; i < NI; ++i) {
    const int tau = warp + WARPS * i;
    acc[i] = T::acc_zero();
    if (tau >= nblk) continue;
    const int row = blk(tau) * NB + rb;
    if (FWD) rhs[i] = T::from(row < N ? y[row] : make_double2(0.0, 0.0));
    if (tau > 0) load_k(tau, 0, k[i]);
  }
  if (warp >= nblk) return;
  const int last = warp + WARPS * ((nblk - 1 - warp) / WARPS);   // the warp's last block
  // t < 0: the first three blocks have no products before their D s
#pragma unroll 1
  for (int t = -3; t < last; ++t) {
    V z[2];
    if (t >= 0) {
      block_wait(zbar + blk(t), abort_flag, budget, status);
      const E* zp = sol + blk(t) * NB + c0;
      z[0] = T::load(zp[0]);
      z[1] = T::load(zp[1]);
    }
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      const int tau = warp + WARPS * i, d = tau - t;
      if (tau >= nblk || d < 1) continue;
      if (t < 0 && d > 3) continue;
      const int b = blk(tau);
      if (t >= 0) {
        if (FWD || T::UPPER || d < 3) {
          T::mul(acc[i], k[i][0], z[0]);
          T::mul(acc[i], k[i][1], z[1]);
        } else {
          T::cmul(acc[i], k[i][0], z[0]);
          T::cmul(acc[i], k[i][1], z[1]);
        }
        // the next block's operand, on its way while the warp waits for that block
        if (d > 1) load_k(tau, t + 1, k[i]);
      }
      if (d > 3) continue;
      if (d == 3) {
        // D's operand; then s
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const int rd = b * NB + (FWD ? rb : c0 + q);
          kd[q] = rd < N ? T::load(__ldg(D + (size_t)rd * NB + (FWD ? c0 + q : rb))) : T::zero();
        }
        V r;
        if (FWD) {
          r = rhs[i];
        } else {   // the forward solution
          block_wait(lay.bars(0) + b, abort_flag, budget, status);
          r = T::load(lay.vec<E>(0)[b * NB + rb]);
        }
        const V s = t >= 0 ? T::sub(r, row_sum<T>(acc[i])) : r;
        st_async16(T::store(s), svec + b * NB + rb, sbar + b, lane & 15);
        acc[i] = T::acc_zero();
      } else if (d == 2) {
        block_wait(sbar + b, abort_flag, budget, status);
        const E* sp = svec + b * NB + c0;
        if (FWD) {
          T::mul(acc[i], kd[0], T::load(sp[0]));
          T::mul(acc[i], kd[1], T::load(sp[1]));
        } else {
          T::cmul(acc[i], kd[0], T::load(sp[0]));
          T::cmul(acc[i], kd[1], T::load(sp[1]));
        }
      } else {
        const V v = row_sum<T>(acc[i]);
        st_async16(T::store(v), sol + b * NB + rb, zbar + b, lane & 15);
        if (!FWD && (lane & 15) == 0 && b * NB + rb < N) {
          const double2 o = T::to(v);
          out[b * NB + rb] = minus_i ? make_double2(o.y, -o.x) : o;
        }
      }
    }
  }
}

template <class T, int NI>
__global__ void __launch_bounds__(WARPS * 32, 1)
k_cluster_solve(int N, const typename T::E* __restrict__ L, const typename T::E* __restrict__ D,
                const typename T::E* __restrict__ P, const double2* __restrict__ y, double2* __restrict__ out,
                bool minus_i, int* status) {
  extern __shared__ __align__(128) unsigned char csm[];
  Layout lay;
  lay.nblk = (N + NB - 1) / NB;
  lay.base = csm;
  const int rank = (int)cluster_rank();
  const unsigned budget = wait_budget(status, ~0u);
  for (int e = threadIdx.x; e < 4 * lay.nblk; e += WARPS * 32) {
    bar_init(lay.bars(0) + e, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    bar_expect(lay.bars(0) + e, NB * 16u);
  }
  if (threadIdx.x == 0) *lay.abort_flag() = 0;
  __syncthreads();
  cluster_sync();
  pass<T, NI, true>(lay, N, rank, L, D, P, y, out, minus_i, budget, status);
  pass<T, NI, false>(lay, N, rank, L, D, P, y, out, minus_i, budget, status);
  // every store into this CTA has landed before it ends
  for (int e = threadIdx.x; e < 4 * lay.nblk; e += WARPS * 32)
    block_wait(lay.bars(0) + e, lay.abort_flag(), ~0u, status);
  __syncthreads();
  cluster_sync();
  if (*(volatile int*)lay.abort_flag()) {
    // a wait gave up: stores of other CTAs may still be landing in this CTA's shared memory, which must
    // not end before they complete; they take microseconds, so linger
    const unsigned long long t0 = gtime_ns();
    while (gtime_ns() - t0 < 200000ull) {
    }
  }
}

size_t near_offset(int N) { return (size_t)((N + NB - 1) / NB) * NB * NB; }

template <class T>
int near_products(int N, void* const* L, void* const* D, int nbatch, cudaStream_t s) {
  using E = typename T::E;
  const int nb = (N + NB - 1) / NB, k = nbatch > 1 ? 1 : 0;
  if (nb > MAX_BLOCKS || nb < 2) return 0;
  E *d0 = (E*)D[0], *d1 = (E*)D[k];
  k_near_products<T><<<dim3(nb * (NB / NPR), 4, nbatch), NPR * 32, 0, s>>>(
      N, (const E*)L[0], (const E*)L[k], d0, d1, d0 + near_offset(N), d1 + near_offset(N));
  return 1;
}

template <class T, int NI>
cudaError_t attributes() {
  const cudaError_t e = cudaFuncSetAttribute(k_cluster_solve<T, NI>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)smem_bytes(NI * WARPS));
  return e != cudaSuccess ? e
                          : cudaFuncSetAttribute(k_cluster_solve<T, NI>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
}

template <class T, int NI>
void launch(int N, const void* L, const void* D, const double2* y, double2* out, bool minus_i, int* status,
            cudaStream_t s) {
  using E = typename T::E;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = CL;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(CL);
  cfg.blockDim = dim3(WARPS * 32);
  cfg.dynamicSmemBytes = smem_bytes((N + NB - 1) / NB);
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, k_cluster_solve<T, NI>, N, (const E*)L, (const E*)D, (const E*)D + near_offset(N), y, out,
                     minus_i, status);
}

template <class T>
void launch_by_size(int N, const void* L, const void* D, const double2* y, double2* out, bool minus_i, int* status,
                    cudaStream_t s) {
  const int nb = (N + NB - 1) / NB;
  if (nb <= WARPS) launch<T, 1>(N, L, D, y, out, minus_i, status, s);
  else if (nb <= 2 * WARPS) launch<T, 2>(N, L, D, y, out, minus_i, status, s);
  else launch<T, 4>(N, L, D, y, out, minus_i, status, s);
}

}  // namespace slv

cudaError_t cluster_solve_attributes() {
  using namespace slv;
  for (cudaError_t e : {attributes<Df, 1>(), attributes<Df, 2>(), attributes<Df, 4>(), attributes<F64, 1>(),
                        attributes<F64, 2>(), attributes<F64, 4>()})
    if (e != cudaSuccess) return e;
  return cudaSuccess;
}

// The neighbour products follow the N x 32 inverted diagonal blocks in the D buffer, whole blocks each.
size_t diag_inv_bytes(int N) { return 5 * slv::near_offset(N) * 16; }

int launch_near_products(int N, void* const* L, void* const* D, int nbatch, bool df, cudaStream_t s) {
  return df ? slv::near_products<slv::Df>(N, L, D, nbatch, s) : slv::near_products<slv::F64>(N, L, D, nbatch, s);
}

bool launch_cluster_solve(int N, const void* L, const void* D, const double2* y, double2* out, bool minus_i,
                          bool df, int* status, cudaStream_t s) {
  using namespace slv;
  if ((N + NB - 1) / NB > MAX_BLOCKS) return false;
  if (df) launch_by_size<Df>(N, L, D, y, out, minus_i, status, s);
  else launch_by_size<F64>(N, L, D, y, out, minus_i, status, s);
  return true;
}

}  // namespace icwf
