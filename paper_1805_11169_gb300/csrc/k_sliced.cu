// Matrix elements (Eq. M, W, W1, W2) as Grams of sliced operands on the sm_103a tensor cores, and their
// combination into S and Heff: both in the FP64 mode, S in the mixed modes (their Heff is made of
// floating-point products, k_assemble_tc.cu).
//
// Slicing.  A CWF column (weighted by u_g(x) for the rank-k terms) is scaled by a power of two 2^-e so
// that its components lie in (-1, 1) and is cut into D balanced integers d_p, value = 2^e sum_p d_p
// 2^-(b0 + beta p), stored exactly as BF16; products of digits are integers, so the sums over the grid
// are exact in FP32 as long as they stay below 2^24.  b0 = 6, beta = 7 in the FP64 mode (D = 8: 55 bits
// below the largest component), b0 = beta = 6 with D = 4 for the mixed modes' overlap (24 bits: S is
// then the exact Gram of fixed-point CWFs and positive semidefinite; b0 = beta = 5 on 4096-point grids).
//
// Products.  conj(a) b = sum over piece pairs (p, q); the pairs with p + q < L are kept and every level
// l = p + q has its own FP32 accumulator in TMEM.  With the T kets' pieces stored one after the
// other, [b_0; b_1; ...] is a single operand of up to 256 rows, so one MMA takes piece p of 128 bras
// against all pieces q < L - p at once and lands on the adjacent accumulators of levels p, p + 1, ...:
// M = 128, N up to 256, where the tensor cores and not the shared-memory operand reads are the bound.
// (One MMA per pair, N = 64, measured 88-115 cycles where the tensor pipe needs 32.)
// L = D keeps products down to the pieces' own truncation; the overlap keeps all 2D - 1 levels.
//
// Digits are only as many as a term needs: term g of the interaction is at most v_g = s_g max|u_g|
// max|w_g| anywhere on the grid, so it takes D_g = ceil((56 + log2(v_g / max v)) / 7) digits, and every
// term is cut 2^-56 below the largest one.  That is below the factors' own rounding (the SVD leaves 2^-53
// of s_1, spread over the grid), also for a term that sits on a few grid points, where s_g alone says
// little.  At the paper's scale (21 terms) it is 23 digit pairs on average instead of 36.
//
// Level sums (digits) are combined as 64-bit integers, in units of 2^-F of level 0, and converted
// once: no FP64 instruction in the loop (FP64 runs at 1/61 of FP32 here).  The accumulators are drained
// into the integers every `drain` K slices, before a leading level could pass 2^24 (drain_slices).
//
// Layout.  Operands are written by k_slices in the order the MMA reads them: tiles of 128 bra rows (T
// ket rows) x 16 grid points in the 32-byte-swizzled K-major form, [tile][K slice][Re, Im][piece],
// so that a pipeline stage is two or three contiguous bulk copies.
//
// k_gram_sliced: persistent CTAs (320 threads, one per SM) take units (Gram, 128-bra x T-ket tile) by
// a ticket, the most expensive first; warp 8 copies stages, warp 9 issues the MMAs, warps 0..7 drain
// TMEM (warp w: lanes 32 (w mod 4).., column half w div 4).  Ring geometry follows the unit's D.
// Every wait is bounded (2 s): a timeout raises the status flag, drains what is in flight, returns.
//
// Bound: an MMA of M = 128 takes max(N / 2, operand bytes / 128) cycles (measured over N = 32..256), so
// the wide operands of all pieces at once keep it on the tensor pipe's side; the copies' writes into
// shared memory come on top.
// Measured (GB300; ms per assembly, before -> now): FP64 mode, N = 1024, 22 terms on 1024 x 512, 144 (FP64
// FMAs) -> 4.0, the tensor pipe busy 63-66% of k_gram_sliced; N = 16, 64 terms on 128 x 64, 13.1 (one CTA)
// -> 0.11; N = 256, 21 terms on 512 x 256, 17.7 -> 0.32; reconstruction at N = 1024 in the FP64 mode
// 4.3 -> 0.22.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "df64.cuh"
#include "icwf_internal.h"
#include "k_common.cuh"
#include "sliced.cuh"
#include "tc_ptx.cuh"

namespace icwf {
namespace sl {

using namespace tc;

constexpr int RING_BYTES = 220 * 1024;
constexpr int MAX_SLOTS = 6;
constexpr int UNIT_RING = 4;
constexpr int MAX_GRAMS = 256;         // Grams of one launch
constexpr int SMEM_BYTES = RING_BYTES + 1024 /*align*/ + 512 /*barriers, unit ring*/ + MAX_GRAMS * 4;
static_assert(SMEM_BYTES <= 227 * 1024, "shared memory per CTA exceeded");
constexpr int EPI_WARPS = 8, TMA_WARP = 8, MMA_WARP = 9, THREADS = 320;
constexpr int COL_IM = 256;            // TMEM: Re levels at [0, 256), Im levels at [256, 512)
constexpr int EX_BAD = 0x40000000;     // exponent of a row with a non-finite component

// the double-float trailing update's panel and digits (see k_herk_slices)
constexpr int HERK_COLS = 128, HERK_KS = HERK_COLS / 16, HERK_D = 7, HERK_B0 = 6, HERK_BETA = 7;

// bytes of a pipeline stage (one K slice): both planes' pieces of 128 bras and T kets
__host__ __device__ inline int stage_bytes(int d, int t) { return 2 * d * (MT + t) * ROW_BYTES; }
__host__ __device__ inline int ring_slots(int d, int t) {
  const int s = RING_BYTES / stage_bytes(d, t);
  return s < MAX_SLOTS ? s : MAX_SLOTS;
}

// One Gram (one side, one weight) of a launch.
struct Gram {
  const unsigned char* A;   // bras: 128-row tiles, da pieces stored per plane
  const unsigned char* B;   // kets: T-row tiles with d pieces per plane, or NULL: rows of A
  const int* ea;            // scale exponents of the bras and kets
  const int* eb;
  double2* out;             // tiles [ket][bra] as in Tri
  int ks, da, d, l, t;      // K slices; pieces stored / used; levels; kets per unit
  int drain;                // K slices per accumulation
  int b0, beta, fbits;      // digit weights; fraction bits of the integer accumulators
  int unit0;                // first unit
  int cols;                 // 0: upper-triangle tiles of `rows` trajectories; else a rectangular product
  int rows;                 //    of rows x cols elements, out row-major
};

struct GramArgs {
  const Gram* grams;
  double2* out;             // overrides the Grams' outputs if not NULL
  int ngrams, units, N;
  float4* herk[2];          // if set: Gram i's conj(bra) ket is subtracted from the double-floats
  int R0;                   //    herk[i][(R0 + ket) N + R0 + bra], bra <= ket, R0 + ket < N
  unsigned* ticket;
  int* status;
};

// Where unit v of Gram g reads and writes: bra tile, ket tile (of T rows), first output element, the
// output's strides along bras and kets, and how many of each are stored.
struct UnitAt {
  int I, J, bt;             // bra tile; 128-ket tile and T-ket tile
  size_t out;
  int sr, sc, nr, nc;
};
__device__ __forceinline__ UnitAt unit_at(const Gram& g, int v) {
  UnitAt u;
  const int qn = MT / g.t;
  if (g.cols == 0) {
    const Tri tri(g.rows);
    int tile, part;
    tri.unit(v, g.t, tile, part);
    tri_tile(tile, u.I, u.J);
    u.bt = u.J * qn + part;
    u.out = tri.at(tile) + (size_t)part * g.t * tri.br;
    u.sr = 1;
    u.sc = tri.br;
    u.nr = tri.br;
    u.nc = (tile < tri.full ? MT : tri.kl) - part * g.t;
  } else {
    const int nt = (g.cols + g.t - 1) / g.t;
    u.I = v / nt;
    u.bt = v % nt;
    u.J = u.bt / qn;
    u.out = (size_t)u.I * MT * g.cols + (size_t)u.bt * g.t;
    u.sr = g.cols;
    u.sc = 1;
    u.nr = g.rows - u.I * MT;
    u.nc = g.cols - u.bt * g.t;
  }
  return u;
}

// dst (shared) <- src (global), both 16-byte aligned, completing on bar
__device__ __forceinline__ void bulk_load(void* dst, const void* src, int bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ int gram_of(const int* unit0, int n, int u) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (unit0[mid] <= u) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// sum += the levels' exact integers of 8 columns (Re at col, Im at col + COL_IM) in units 2^-fbits
__device__ __forceinline__ void drain8(uint32_t col, int L, int t, int beta, int fbits,
                                       long long (&re)[8], long long (&im)[8]) {
#pragma unroll 1
  for (int lv = 0; lv < L; ++lv) {
    float vr[8], vi[8];
    tmem_ld8(col + lv * t, vr);
    tmem_ld8(col + COL_IM + lv * t, vi);
    tmem_wait_ld();
    const int sh = fbits - beta * lv;
    if (sh >= 32) {   // only the upper word changes
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        re[e] += (long long)((unsigned long long)(unsigned)(__float2int_rn(vr[e]) << (sh - 32)) << 32);
        im[e] += (long long)((unsigned long long)(unsigned)(__float2int_rn(vi[e]) << (sh - 32)) << 32);
      }
    } else if (sh >= 0) {   // one 32 x 32 + 64 bit multiply-add per sum
      const unsigned w = 1u << sh;
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        re[e] += (long long)__float2int_rn(vr[e]) * (long long)w;
        im[e] += (long long)__float2int_rn(vi[e]) * (long long)w;
      }
    } else {
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        re[e] += __float2int_rn(vr[e]) >> -sh;
        im[e] += __float2int_rn(vi[e]) >> -sh;
      }
    }
  }
}

// x 2^k for a normal x: one multiplication in the usual range
__device__ __forceinline__ float scaled(float x, int k) {
  return (unsigned)(k + 126) < 253u ? x * __uint_as_float((unsigned)(k + 127) << 23) : ldexpf(x, k);
}

// the first n of 8 kets
// (xb: the warp's lanes hold the exponents of its kets; these are kets l0..)
__device__ __forceinline__ void store8(double2* out, int sc, int n, int xb, int l0, int ea, int shift,
                                       const long long (&re)[8], const long long (&im)[8]) {
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    const int x = __shfl_sync(0xffffffffu, xb, l0 + e);
    if (e >= n) continue;
    double2 z = make_double2(fixed_to_f64(re[e], ea + x + shift), fixed_to_f64(im[e], ea + x + shift));
    if (ea == EX_BAD || x == EX_BAD) z.x = z.y = __longlong_as_double(0x7FF8000000000000ll);
    out[(size_t)e * sc] = z;
  }
}

// Subtraction of 8 kets' sums from the rows r..r + 7 of A, lane = bra (column c of A), a: the old values.
// The levels (exact integers) are added from the smallest up in double-float arithmetic.
__device__ __forceinline__ void herk_load8(const float4* __restrict__ A, int N, int r, int c, float4 (&a)[8]) {
#pragma unroll
  for (int e = 0; e < 8; ++e)
    a[e] = r + e < N && c <= r + e ? A[(size_t)(r + e) * N + c] : make_float4(0.f, 0.f, 0.f, 0.f);
}
template <int L, int BETA>
__device__ __forceinline__ void herk_levels8(uint32_t col, int t, df (&re)[8], df (&im)[8]) {
#pragma unroll
  for (int lv = L - 1; lv >= 0; --lv) {
    float vr[8], vi[8];
    tmem_ld8(col + lv * t, vr);
    tmem_ld8(col + COL_IM + lv * t, vi);
    tmem_wait_ld();
    const float w = __int_as_float((127 - BETA * lv) << 23);
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      if (lv == L - 1) {
        re[e] = df_make(vr[e] * w, 0.f);
        im[e] = df_make(vi[e] * w, 0.f);
      } else {
        re[e] = df_add_f(re[e], vr[e] * w);
        im[e] = df_add_f(im[e], vi[e] * w);
      }
    }
  }
}
__device__ __forceinline__ void herk_store8(float4* __restrict__ A, int N, int r, int c, int xb, int l0, int ea,
                                            int shift, const float4 (&a)[8], const df (&re)[8], const df (&im)[8]) {
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    const int x = __shfl_sync(0xffffffffu, xb, l0 + e), k = ea + x + shift;
    df vr = df_make(scaled(re[e].h, k), scaled(re[e].l, k)), vi = df_make(scaled(im[e].h, k), scaled(im[e].l, k));
    if (ea == EX_BAD || x == EX_BAD) vr.h = vi.h = __int_as_float(0x7FC00000);
    vr = df_sub(df_make(a[e].x, a[e].y), vr);
    vi = df_sub(df_make(a[e].z, a[e].w), vi);
    if (r + e < N && c <= r + e) A[(size_t)(r + e) * N + c] = make_float4(vr.h, vr.l, vi.h, vi.l);
  }
}

// The issuer's view of the stage ring.
struct MmaRing {
  unsigned char* ring;
  uint64_t *full, *empty;
  volatile int* abort_flag;
  int* status;
  int bytes, slots, slot;
  unsigned pf;              // phase bits of the slots' next full wait
};

// D[tmem] += A B^T (or = with acc = 0) from the low words of the operand descriptors; the high word,
// which holds the strides and the swizzle, is the same for all of them.
constexpr uint32_t DESC_HI = (uint32_t)((8 * ROW_BYTES) >> 4) | (1u << 14) | (6u << 29);
__device__ __forceinline__ uint32_t desc_lo(uint32_t saddr) { return ((saddr & 0x3FFFFu) >> 4) | (1u << 16); }
__device__ __forceinline__ void mma_add(uint32_t d, uint32_t a, uint32_t b, uint32_t id) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 x, y;\n\tsetp.ne.b32 p, 1, 0;\n\tmov.b64 x, {%1, %4};\n\t"
      "mov.b64 y, {%2, %4};\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], x, y, %3, p;\n\t}" ::"r"(d),
      "r"(a), "r"(b), "r"(id), "n"(DESC_HI));
}
__device__ __forceinline__ void mma_set(uint32_t d, uint32_t a, uint32_t b, uint32_t id, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 x, y;\n\tsetp.ne.b32 p, %5, 0;\n\tmov.b64 x, {%1, %4};\n\t"
      "mov.b64 y, {%2, %4};\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], x, y, %3, p;\n\t}" ::"r"(d),
      "r"(a), "r"(b), "r"(id), "n"(DESC_HI), "r"(acc));
}

// One accumulation over n K slices of D pieces and L levels.  One thread issues every MMA of the CTA,
// so it must need fewer cycles per MMA than the tensor cores (96 on average at D = 2): unrolled over
// the pieces, addresses and instruction descriptors computed once per accumulation, 32-bit
// descriptor arithmetic, and the next slice's barrier polled before this slice's MMAs.  (Looping
// over the pieces took 130 cycles per MMA, unrolled with 64-bit descriptors 104.)
template <int D, int L>
__device__ __forceinline__ bool issue_slices(MmaRing& r, uint32_t tmem, int t, uint32_t id0, int n) {
  constexpr uint32_t AT = (MT * ROW_BYTES) >> 4, AQ = D * AT;
  const uint32_t bt = (uint32_t)(t * ROW_BYTES) >> 4, bq = D * bt;
  const uint32_t ring = desc_lo(smem_u32(r.ring)), step = (uint32_t)r.bytes >> 4;
  uint32_t col[D], id[D], idn[D];
#pragma unroll
  for (int p = 0; p < D; ++p) {
    col[p] = tmem + p * t;
    id[p] = id0 + idesc_n((L - p < D ? L - p : D) * t);
    idn[p] = id[p] | IDESC_NEG_A;
  }
  bool ready = mbar_test(r.full + r.slot, (r.pf >> r.slot) & 1u);
  for (int s = 0; s < n; ++s) {
    if (!ready && !mbar_wait(r.full + r.slot, (r.pf >> r.slot) & 1u, r.abort_flag, r.status)) return false;
    r.pf ^= 1u << r.slot;
    const int cur = r.slot;
    r.slot = cur + 1 == r.slots ? 0 : cur + 1;
    if (s + 1 < n) ready = mbar_test(r.full + r.slot, (r.pf >> r.slot) & 1u);
    fence_after();
    const uint32_t ap = ring + cur * step, bp = ap + 2 * AQ;
    if (s == 0) {
#pragma unroll
      for (int p = 0; p < D; ++p) {
        const uint32_t a = ap + p * AT, re = col[p], im = re + COL_IM;
        if (p > 0 && L - p >= D) {
          // the top level of this piece starts here: its own, overwriting MMAs
          const uint32_t b = bp + (D - 1) * bt, i1 = id0 + idesc_n(t), i2 = id0 + idesc_n((D - 1) * t);
          const uint32_t c = (D - 1) * t;
          mma_set(re + c, a, b, i1, 0u);
          mma_set(im + c, a, b + bq, i1, 0u);
          mma_add(re + c, a + AQ, b + bq, i1);
          mma_add(im + c, a + AQ, b, i1 | IDESC_NEG_A);
          mma_add(re, a, bp, i2);
          mma_add(im, a, bp + bq, i2);
          mma_add(re, a + AQ, bp + bq, i2);
          mma_add(im, a + AQ, bp, i2 | IDESC_NEG_A);
        } else {
          mma_set(re, a, bp, id[p], p > 0);
          mma_set(im, a, bp + bq, id[p], p > 0);
          mma_add(re, a + AQ, bp + bq, id[p]);
          mma_add(im, a + AQ, bp, idn[p]);
        }
      }
    } else {
#pragma unroll
      for (int p = 0; p < D; ++p) {
        // Re += P P + Q Q, Im += P Q - Q P
        const uint32_t a = ap + p * AT, re = col[p], im = re + COL_IM;
        mma_add(re, a, bp, id[p]);
        mma_add(im, a, bp + bq, id[p]);
        mma_add(re, a + AQ, bp + bq, id[p]);
        mma_add(im, a + AQ, bp, idn[p]);
      }
    }
    mma_commit(r.empty + cur);
  }
  return true;
}

__global__ void __launch_bounds__(THREADS, 1) k_gram_sliced(GramArgs args) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* ring = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* full = (uint64_t*)(ring + RING_BYTES);
  uint64_t* empty = full + MAX_SLOTS;
  uint64_t* acc_full = empty + MAX_SLOTS;
  uint64_t* acc_empty = acc_full + 1;
  uint64_t* ufull = acc_empty + 1;
  uint64_t* uempty = ufull + UNIT_RING;
  uint64_t* drain = uempty + UNIT_RING;
  int* uring = (int*)(drain + 1);
  uint32_t* tmem_slot = (uint32_t*)(uring + UNIT_RING);
  volatile int* abort_flag = (volatile int*)(tmem_slot + 1);
  int* unit0 = (int*)(ring + RING_BYTES + 512);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int* status = args.status;

  for (int i = threadIdx.x; i < args.ngrams; i += THREADS) unit0[i] = args.grams[i].unit0;
  if (threadIdx.x == 0) {
    for (int s = 0; s < MAX_SLOTS; ++s) { mbar_init(full + s, 1); mbar_init(empty + s, 1); }
    for (int s = 0; s < UNIT_RING; ++s) {
      mbar_init(ufull + s, 1);
      mbar_init(uempty + s, 1 + EPI_WARPS * 32);
    }
    mbar_init(acc_full, 1);
    mbar_init(acc_empty, EPI_WARPS * 32);
    mbar_init(drain, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tmem_slot;

  // phase bits of the ring slots: the producer's next wait on empty, the issuer's on full
  if (warp == TMA_WARP) {
    if (lane == 0) {
      unsigned pe = (1u << MAX_SLOTS) - 1;   // a fresh barrier passes a wait on parity 1
      unsigned filled = 0;                   // slots filled at least once
      int slot = 0, geo = -1;
      bool ok = true;
      for (unsigned n = 0; ok; ++n) {
        const int u = (int)atomicAdd(args.ticket, 1u);
        const int us = n & (UNIT_RING - 1);
        if (!mbar_wait(uempty + us, ((n / UNIT_RING) & 1u) ^ 1u, abort_flag, status)) break;
        const bool last = u >= args.units;
        uring[us] = last ? -1 : u;
        mbar_arrive(ufull + us);
        if (last) break;
        const Gram& g = args.grams[gram_of(unit0, args.ngrams, u)];
        const int d = g.d, t = g.t, da = g.da, ks = g.ks;
        const UnitAt at = unit_at(g, u - g.unit0);
        const int bytes = stage_bytes(d, t), slots = ring_slots(d, t);
        if (bytes != geo) {
          // another ring geometry: every copy and MMA of the old one must be done
          for (int s = 0; s < MAX_SLOTS && ok; ++s)
            ok = mbar_wait(empty + s, (pe >> s) & 1u, abort_flag, status);
          if (!ok) break;
          geo = bytes;
          slot = 0;
        }
        const size_t a_slice = (size_t)2 * da * MT * ROW_BYTES, b_slice = (size_t)2 * d * t * ROW_BYTES;
        const unsigned char* ap = g.A + (size_t)at.I * ks * a_slice;
        const unsigned char* bp = g.B ? g.B + (size_t)at.bt * ks * b_slice
                                      : g.A + (size_t)at.J * ks * a_slice +
                                            (size_t)(at.bt * t - at.J * MT) * ROW_BYTES;
        const bool own_b = g.B != nullptr;
        for (int s = 0; s < ks; ++s) {
          if (!(ok = mbar_wait(empty + slot, (pe >> slot) & 1u, abort_flag, status))) break;
          pe ^= 1u << slot;
          filled |= 1u << slot;
          unsigned char* st = ring + slot * bytes;
          uint64_t* bar = full + slot;
          mbar_expect_tx(bar, bytes);
          const int pa = d * MT * ROW_BYTES;
          bulk_load(st, ap, pa, bar);
          bulk_load(st + pa, ap + (size_t)da * MT * ROW_BYTES, pa, bar);
          unsigned char* sb = st + 2 * pa;
          if (own_b) {
            bulk_load(sb, bp, (int)b_slice, bar);
            bp += b_slice;
          } else {
            for (int pl = 0; pl < 2; ++pl)
              for (int p = 0; p < d; ++p)
                bulk_load(sb + (pl * d + p) * t * ROW_BYTES,
                          bp + (size_t)(pl * da + p) * MT * ROW_BYTES, t * ROW_BYTES, bar);
            bp += a_slice;
          }
          ap += a_slice;
          slot = slot + 1 == slots ? 0 : slot + 1;
        }
      }
      if (*abort_flag) {
        // copies that may still be landing: the last fill of every slot (bounded)
        for (int s = 0; s < MAX_SLOTS; ++s) {
          if (!((filled >> s) & 1u)) continue;
          const unsigned long long t0 = gtime();
          while (!mbar_test(full + s, (pe >> s) & 1u) && gtime() - t0 < WAIT_NS) {
          }
        }
      }
    }
  } else if (warp == MMA_WARP) {
    if (lane == 0) {
      unsigned pf = 0, chunk = 0;
      int slot = 0, geo = -1;
      bool ok = true;
      for (unsigned n = 0; ok; ++n) {
        const int us = n & (UNIT_RING - 1);
        if (!mbar_wait(ufull + us, (n / UNIT_RING) & 1u, abort_flag, status)) break;
        const int u = *(volatile int*)(uring + us);
        mbar_arrive(uempty + us);
        if (u < 0) break;
        const Gram& g = args.grams[gram_of(unit0, args.ngrams, u)];
        const int d = g.d, t = g.t, L = g.l, ks = g.ks, dr = g.drain;
        const int bytes = stage_bytes(d, t), slots = ring_slots(d, t);
        if (bytes != geo) { geo = bytes; slot = 0; }
        const uint32_t id0 = idesc_mn(0, MT, 0);
        for (int s0 = 0; s0 < ks && ok; s0 += dr) {
          if (!(ok = mbar_wait(acc_empty, (chunk & 1u) ^ 1u, abort_flag, status))) break;
          fence_after();
          ++chunk;
          const int s1 = s0 + dr < ks ? s0 + dr : ks;
          MmaRing rg{ring, full, empty, abort_flag, status, bytes, slots, slot, pf};
          const int n = s1 - s0;
          if (L > d) ok = issue_slices<4, 7>(rg, tmem, t, id0, n);
          else if (d == 2) ok = issue_slices<2, 2>(rg, tmem, t, id0, n);
          else if (d == 3) ok = issue_slices<3, 3>(rg, tmem, t, id0, n);
          else if (d == 4) ok = issue_slices<4, 4>(rg, tmem, t, id0, n);
          else if (d == 5) ok = issue_slices<5, 5>(rg, tmem, t, id0, n);
          else if (d == 6) ok = issue_slices<6, 6>(rg, tmem, t, id0, n);
          else if (d == 7) ok = issue_slices<7, 7>(rg, tmem, t, id0, n);
          else ok = issue_slices<8, 8>(rg, tmem, t, id0, n);
          slot = rg.slot;
          pf = rg.pf;
          if (ok) mma_commit(acc_full);
        }
      }
      mma_commit(drain);   // every MMA issued by this CTA
    }
  } else {
    // ---------------- epilogue: lane = bra row, each column half by one warp of the quarter ----
    const int quarter = warp & 3, half = warp >> 2;
    const int row = quarter * 32 + lane;
    const uint32_t base = tmem + ((uint32_t)(quarter * 32) << 16);
    unsigned chunk = 0;
    bool ok = true;
    for (unsigned n = 0; ok; ++n) {
      const int us = n & (UNIT_RING - 1);
      // (a wait that ends by abort ends for every lane of the warp: the flag stays up)
      ok = mbar_wait(ufull + us, (n / UNIT_RING) & 1u, abort_flag, status);
      if (!__all_sync(0xffffffffu, ok)) break;
      const int u = *(volatile int*)(uring + us);
      mbar_arrive(uempty + us);
      if (u < 0) break;
      const Gram& g = args.grams[gram_of(unit0, args.ngrams, u)];
      const int t = g.t, L = g.l;
      const UnitAt at = unit_at(g, u - g.unit0);
      const int nch = (g.ks + g.drain - 1) / g.drain;
      const int ea = g.ea[at.I * MT + row];
      const int c0 = half * (t / 2);                    // this warp's first ket of the unit
      // exponents of this warp's kets, one per lane (up to 64 kets), off the accumulators' wait
      const int* eb = g.eb + at.bt * t + c0;
      const int xb0 = lane < t / 2 ? eb[lane] : 0, xb1 = 32 + lane < t / 2 ? eb[32 + lane] : 0;
      const size_t o = at.out + (size_t)row * at.sr + (size_t)c0 * at.sc;
      const int sc = at.sc;
      const int nk = row < at.nr ? at.nc - c0 : 0;      // kets this lane stores, from c0 on
      const uint32_t col = base + half * (t / 2);
      if (args.herk[0]) {
        float4* A = args.ngrams > 1 && u >= unit0[1] ? args.herk[1] : args.herk[0];
        const int r = args.R0 + at.bt * t + c0, c = args.R0 + at.I * MT + row;
#pragma unroll 1
        for (int h = 0; h < 2 && ok; ++h) {
          float4 a[8];   // on their way while the MMAs run and the levels are read
          herk_load8(A, args.N, r + 8 * h, c, a);
          if (h == 0) {
            ok = __all_sync(0xffffffffu, mbar_wait(acc_full, chunk & 1u, abort_flag, status));
            if (!ok) break;
            ++chunk;
            fence_after();
          }
          df re[8], im[8];
          herk_levels8<HERK_D, HERK_BETA>(col + 8 * h, t, re, im);
          if (h == 1) {
            fence_before();
            mbar_arrive(acc_empty);
          }
          herk_store8(A, args.N, r + 8 * h, c, xb0, 8 * h, ea, -2 * HERK_B0, a, re, im);
        }
      } else {
        double2* out = (args.out ? args.out : g.out) + o;
        const int shift = -2 * g.b0 - g.fbits;
        if (t == 32) {
          long long re[2][8], im[2][8];
#pragma unroll
          for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int e = 0; e < 8; ++e) re[h][e] = im[h][e] = 0;
          for (int c = 0; c < nch && ok; ++c, ++chunk) {
            ok = __all_sync(0xffffffffu, mbar_wait(acc_full, chunk & 1u, abort_flag, status));
            if (!ok) break;
            fence_after();
            drain8(col, L, t, g.beta, g.fbits, re[0], im[0]);
            drain8(col + 8, L, t, g.beta, g.fbits, re[1], im[1]);
            fence_before();
            mbar_arrive(acc_empty);
          }
          if (!ok) break;
          store8(out, sc, nk, xb0, 0, ea, shift, re[0], im[0]);
          store8(out + (size_t)8 * sc, sc, nk - 8, xb0, 8, ea, shift, re[1], im[1]);
        } else {
          // one accumulation (the plan drains only units of 32 kets)
          ok = __all_sync(0xffffffffu, mbar_wait(acc_full, chunk & 1u, abort_flag, status));
          if (!ok) break;
          ++chunk;
          fence_after();
#pragma unroll 1
          for (int c8 = 0; c8 < t / 2; c8 += 8) {
            long long re[8], im[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) re[e] = im[e] = 0;
            drain8(col + c8, L, t, g.beta, g.fbits, re, im);
            store8(out + (size_t)c8 * sc, sc, nk - c8, c8 < 32 ? xb0 : xb1, c8 & 31, ea, shift, re, im);
          }
          fence_before();
          mbar_arrive(acc_empty);
        }
      }
    }
  }

  // ---------------- teardown ----------------
  __syncthreads();
  if (warp == MMA_WARP && lane == 0) {
    // an abort can leave MMAs in flight: let them retire before TMEM is released (bounded)
    const unsigned long long t0 = gtime();
    while (!mbar_test(drain, 0u) && gtime() - t0 < WAIT_NS) {
    }
  }
  fence_before();
  __syncthreads();
  fence_after();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
}

// ---------------------------------------------------------------------------- operands

// Operands of up to SLICE_GROUP terms in the same format: rows = CWF columns of one side, weighted by
// w[i] of each term if given (complex128 CWFs only).
constexpr int SLICE_GROUP = 4;
struct Slice {
  const void* src;          // complex128 or complex64, row r at src + r n
  const double* w;          // ng weights of n points each
  unsigned char* out;       // term q at out + q ostride, its exponents at ex + q estride
  int* ex;                  // rpad exponents
  size_t ostride, estride;
  int ng, n, ks, rows, rpad, R;   // terms, points, K slices, rows (and padded to tiles of R rows)
  int d, b0, beta;
};

// 8 consecutive points of one row: `part` 0 or 1 of their K slice
__device__ __forceinline__ unsigned char* slice_at(const Slice& s, int row, int c8, int plane, int p) {
  const int tile = row / s.R, r = row - tile * s.R;
  return s.out + ((((size_t)tile * s.ks + (c8 >> 1)) * 2 + plane) * s.d + p) * ((size_t)s.R * ROW_BYTES) +
         swizzle32(r, c8 & 1);
}

// Digits of 8 FP64 values |x| < 2^e: integers round(x 2^(b0 + beta (D - 1) - e)) cut from the bottom
// into balanced base-2^beta digits (the top one at most 2^b0), stored exactly as BF16.
template <int D>
__device__ __forceinline__ void emit_f64(const Slice& s, int row, int c8, int plane, const double (&x)[8], int e) {
  uint32_t pk[D][4];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    int dg[D];
    digits_of<D>(x[k], s.b0 + s.beta * (D - 1) - e, dg);
#pragma unroll
    for (int p = 0; p < D; ++p) {
      const uint32_t h = __float_as_uint(small_int_to_float(dg[p])) >> 16;
      if (k & 1) pk[p][k >> 1] |= h << 16;
      else pk[p][k >> 1] = h;
    }
  }
#pragma unroll
  for (int p = 0; p < D; ++p)
    *(uint4*)slice_at(s, row, c8, plane, p) = make_uint4(pk[p][0], pk[p][1], pk[p][2], pk[p][3]);
}

// Digits of 8 FP32 values by exact FP32 steps: d = rint(v), v = (v - d) 2^beta.
__device__ __forceinline__ void emit_f32_digits(const Slice& s, int row, int c8, int plane, const float (&x)[8],
                                                float f1, float f2) {
  float v[8];
  const float B = (float)(1 << s.beta);
#pragma unroll
  for (int k = 0; k < 8; ++k) v[k] = x[k] * f1 * f2;
  for (int p = 0; p < s.d; ++p) {
    uint32_t pk[4];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const float r = rintf(v[k]);
      v[k] = (v[k] - r) * B;
      const uint32_t h = __float_as_uint(r) >> 16;
      if (k & 1) pk[k >> 1] |= h << 16;
      else pk[k >> 1] = h;
    }
    *(uint4*)slice_at(s, row, c8, plane, p) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
  }
}

// Components of 8 points of a row (zero past the row's end and in padding rows); 16-byte loads (rows
// are 8 or more points, so every chunk starts on a 16-byte boundary).
__device__ __forceinline__ void load8(const Slice& s, int row, int c8, float (&re)[8], float (&im)[8]) {
  const float4* p = (const float4*)((const float2*)s.src + (size_t)row * s.n + 8 * c8);
  const bool in = row < s.rows && 8 * c8 < s.n;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float4 z = in ? p[k] : make_float4(0.f, 0.f, 0.f, 0.f);
    re[2 * k] = z.x; im[2 * k] = z.y; re[2 * k + 1] = z.z; im[2 * k + 1] = z.w;
  }
}
__device__ __forceinline__ void load8(const Slice& s, int row, int c8, double (&re)[8], double (&im)[8]) {
  const double2* p = (const double2*)s.src + (size_t)row * s.n + 8 * c8;
  const bool in = row < s.rows && 8 * c8 < s.n;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const double2 z = in ? p[k] : make_double2(0.0, 0.0);
    re[k] = z.x; im[k] = z.y;
  }
}
__device__ __forceinline__ void weight8(const Slice&, int, int, float (&)[8], float (&)[8]) {}
__device__ __forceinline__ void weight8(const Slice& s, int q, int c8, double (&re)[8], double (&im)[8]) {
  if (!s.w || 8 * c8 >= s.n) return;
  const double2* w = (const double2*)(s.w + (size_t)q * s.n + 8 * c8);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const double2 f = w[k];
    re[2 * k] *= f.x; im[2 * k] *= f.x;
    re[2 * k + 1] *= f.y; im[2 * k + 1] *= f.y;
  }
}
__device__ __forceinline__ unsigned long long max8(unsigned long long m, const double (&re)[8], const double (&im)[8]) {
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const unsigned long long a = abs_bits(re[k]), b = abs_bits(im[k]);
    m = m > a ? m : a;
    m = m > b ? m : b;
  }
  return m;
}
__device__ __forceinline__ unsigned long long max8(unsigned long long m, const float (&re)[8], const float (&im)[8]) {
  unsigned x = (unsigned)m;
#pragma unroll
  for (int k = 0; k < 8; ++k)
    x = max(x, max(__float_as_uint(re[k]) & 0x7FFFFFFFu, __float_as_uint(im[k]) & 0x7FFFFFFFu));
  return x;
}

// Largest magnitude (as bits) of one row over its tpr threads (a power of two; rows of fewer than 32
// threads share a warp).
__device__ __forceinline__ unsigned long long row_max(unsigned long long m, int tpr, unsigned long long* red) {
  for (int o = (tpr < 32 ? tpr : 32) >> 1; o > 0; o >>= 1) {
    const unsigned long long x = __shfl_xor_sync(0xffffffffu, m, o);
    m = m > x ? m : x;
  }
  if (tpr > 32) {
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    __syncthreads();
    const int w0 = ((int)threadIdx.x / tpr) * (tpr >> 5);
    for (int w = 0; w < tpr >> 5; ++w) m = m > red[w0 + w] ? m : red[w0 + w];
  }
  return m;
}

// digits of 8 points of row `row`
__device__ __forceinline__ void emit8(const Slice& s, int row, int c, int e, const double (&re)[8],
                                      const double (&im)[8]) {
  switch (s.d) {
    case 2: emit_f64<2>(s, row, c, 0, re, e); emit_f64<2>(s, row, c, 1, im, e); break;
    case 3: emit_f64<3>(s, row, c, 0, re, e); emit_f64<3>(s, row, c, 1, im, e); break;
    case 4: emit_f64<4>(s, row, c, 0, re, e); emit_f64<4>(s, row, c, 1, im, e); break;
    case 5: emit_f64<5>(s, row, c, 0, re, e); emit_f64<5>(s, row, c, 1, im, e); break;
    case 6: emit_f64<6>(s, row, c, 0, re, e); emit_f64<6>(s, row, c, 1, im, e); break;
    case 7: emit_f64<7>(s, row, c, 0, re, e); emit_f64<7>(s, row, c, 1, im, e); break;
    default: emit_f64<8>(s, row, c, 0, re, e); emit_f64<8>(s, row, c, 1, im, e); break;
  }
}
__device__ __forceinline__ void emit8(const Slice& s, int row, int c, int e, const float (&re)[8],
                                      const float (&im)[8]) {
  // 2^k in two factors, each a normal number
  const int k2 = s.b0 - e;
  const float f1 = scaled(1.f, k2 / 2), f2 = scaled(1.f, k2 - k2 / 2);
  emit_f32_digits(s, row, c, 0, re, f1, f2);
  emit_f32_digits(s, row, c, 1, im, f1, f2);
}

// Operands in slices, grid (row groups, operand groups): a row's 8-point chunks are spread over
// min(2 ks, 256) threads, and a thread keeps its chunk (all of its work up to 2048 points) for every
// term of the group: what bounds this kernel is the load/store unit's passes over scattered 32-byte
// rows.
template <typename T>
__device__ __forceinline__ void slice_rows(Slice s, unsigned long long (&red)[2][8]) {
  constexpr bool F64 = sizeof(T) == 8;
  const int c8n = 2 * s.ks, tpr = c8n < 256 ? c8n : 256, rpb = 256 / tpr;
  if ((int)blockIdx.x * rpb >= s.rpad) return;
  const int row = (int)blockIdx.x * rpb + (int)threadIdx.x / tpr, t0 = (int)threadIdx.x % tpr;
  T zr[8], zi[8];
  load8(s, row, t0, zr, zi);
  for (int q = 0; q < s.ng; ++q) {
    T re[8], im[8];
    unsigned long long m = 0;
    for (int c = t0 + tpr; c < c8n; c += tpr) {
      load8(s, row, c, re, im);
      weight8(s, q, c, re, im);
      m = max8(m, re, im);
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) { re[k] = zr[k]; im[k] = zi[k]; }
    weight8(s, q, t0, re, im);
    m = max8(m, re, im);
    // magnitudes order like their bit patterns, NaN above infinity
    m = row_max(m, tpr, red[q & 1]);
    const bool bad = m >= (F64 ? 0x7FF0000000000000ull : 0x7F800000ull);
    int e = 0;
    if (!bad) {
      if constexpr (F64) e = exponent_above_f64(m);
      else e = m ? ilogbf(__uint_as_float((unsigned)m)) + 1 : 0;
    }
    if (row < s.rpad) {
      if (t0 == 0) s.ex[row] = bad ? EX_BAD : e;
      for (int c = t0; c < c8n; c += tpr) {
        if (c != t0) {
          load8(s, row, c, re, im);
          weight8(s, q, c, re, im);
        }
        if (bad) {
#pragma unroll
          for (int k = 0; k < 8; ++k) re[k] = im[k] = 0;
        }
        emit8(s, row, c, e, re, im);
      }
    }
    s.out += s.ostride;
    s.ex += s.estride;
  }
}

template <typename T>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 4 : 2) k_slices(const Slice* __restrict__ list,
                                                                        unsigned* ticket) {
  __shared__ unsigned long long red[2][8];
  const Slice s = list[blockIdx.y];
  if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *ticket = 0;   // the Gram launch's
  slice_rows<T>(s, red);
}

// An operand of Psi(x_i, R_j) = sum_a C_a psi_a(x_i) chi_a(R_j): rows = grid points, K = trajectories.
// Row r, point a is C_a src[a n + r], conjugated (the Grams conjugate their bras), or src[a n + r]
// without C.
struct SliceT {
  const void* src;
  const double2* C;
  unsigned char* out;
  int* ex;
  int n, ks, N, rpad, R, d, f32;
};

// 8 rows per CTA (a 1024-point side fills the chip): lane = row + 8 x group, a warp's four groups and
// the CTA's warps take every 64th set of 8 trajectories, twice: for the rows' largest components
// (bounded by (|Re C| + |Im C|) max(|Re|, |Im|)), then for the digits.
constexpr int ST_WARPS = 16, ST_ROWS = 8, ST_GROUPS = 4;
__global__ void __launch_bounds__(ST_WARPS * 32) k_slices_t(SliceT sx, SliceT sR, unsigned* ticket) {
  __shared__ unsigned long long red[ST_WARPS * ST_GROUPS][ST_ROWS];
  const SliceT q = blockIdx.y ? sR : sx;
  if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *ticket = 0;   // the Gram launch's
  const int r = threadIdx.x & (ST_ROWS - 1), grp = threadIdx.x / ST_ROWS;
  const int row = (int)blockIdx.x * ST_ROWS + r;
  if ((int)blockIdx.x * ST_ROWS >= q.rpad) return;
  auto at = [&](int a) {
    double2 z = make_double2(0.0, 0.0);
    if (a < q.N && row < q.n)
      z = q.f32 ? to_d(((const float2*)q.src)[(size_t)a * q.n + row])
                : ((const double2*)q.src)[(size_t)a * q.n + row];
    return z;
  };
  unsigned long long m = 0;
  for (int c = grp; c < 2 * q.ks; c += ST_WARPS * ST_GROUPS) {
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int a = 8 * c + k;
      const double2 z = at(a);
      unsigned long long x = abs_bits(z.x), y = abs_bits(z.y);
      x = x > y ? x : y;
      if (q.C && a < q.N) x = abs_bits(bits_f64(x) * (fabs(q.C[a].x) + fabs(q.C[a].y)));
      m = m > x ? m : x;
    }
  }
  red[grp][r] = m;
  __syncthreads();
#pragma unroll 8
  for (int w = 0; w < ST_WARPS * ST_GROUPS; ++w) m = m > red[w][r] ? m : red[w][r];
  const bool bad = m >= 0x7FF0000000000000ull;
  const int e = bad ? 0 : exponent_above_f64(m);
  if (grp == 0) q.ex[row] = bad ? EX_BAD : e;
  Slice s;
  s.out = q.out; s.ks = q.ks; s.R = q.R; s.d = q.d; s.b0 = 6; s.beta = 7;
  for (int c = grp; c < 2 * q.ks; c += ST_WARPS * ST_GROUPS) {
    double re[8], im[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int a = 8 * c + k;
      double2 z = at(a);
      if (q.C && a < q.N) z = cconj(cmul(q.C[a], z));
      re[k] = bad ? 0.0 : z.x;
      im[k] = bad ? 0.0 : z.y;
    }
    if (q.d == 8) {
      emit_f64<8>(s, row, c, 0, re, e);
      emit_f64<8>(s, row, c, 1, im, e);
    } else {
      emit_f64<5>(s, row, c, 0, re, e);
      emit_f64<5>(s, row, c, 1, im, e);
    }
  }
}

// ---------------------------------------------------------------------------- S and Heff

// Heff_ab = sum_g s_g (A_g - u_g(x_b) S1)(B_g - w_g(R_b) S2) - V(x_b, R_b) S_ab over the terms
// [g0, g1) of this launch; `first` starts the sums at zero (else they continue from H), `last`
// subtracts the pinned potential and writes S.  The raw Grams of the terms carry s_g dx and dR already
// (folded into the operands' weights), those of the overlap don't.
struct HeffArgs {
  int N, g0, g1, first, last;
  const double2 *S1, *S2;   // raw Grams of the overlap
  const double2 *A, *B;     // Grams of the terms g0.., one after the other
  double dx, dR;
  const double *sig, *px, *pR, *d;
  double2 *S, *H;
  int split;                // term groups (blockIdx.z); > 1: partial sums meet in `part`
  double2* part;            // [group][direct, mirrored], a Gram's storage each
  unsigned* done;           // [tile][patch]: groups finished (zero between launches)
};

// Threads of one 32 x 32 patch of a 128 x 128 upper-triangle tile: lane = bra, 4 kets each.  Bound: 8
// FP64 instructions per term, element and side (0.4 ms at N = 1024 and 22 terms).  With fewer patches
// than SMs the terms are split over CTAs as well (16 trajectories, 64 terms: 202 us without, 50 us
// with).
constexpr int HG = 16;   // terms staged at a time

// A 32 x 32 patch of S, bras from a0 and kets from b0, lane = bra, sv[e]: ket b0 + ty + 8 e.  Each pair is
// stored once, from its a <= b side, so that S is exactly Hermitian.
__device__ __forceinline__ void store_s(double2* S, int N, bool mirror, int a0, int b0, const double2 (&sv)[4],
                                        double2 (&tr)[32][33]) {
  const int lane = threadIdx.x & 31, ty = threadIdx.x >> 5, a = a0 + lane;
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const int b = b0 + ty + 8 * e;
    tr[lane][ty + 8 * e] = sv[e];
    if (a < N && b < N && (mirror || a < b)) S[(size_t)b * N + a] = cconj(sv[e]);
  }
  __syncthreads();
#pragma unroll
  for (int e = 0; e < 4; ++e) {   // rows of S: lane = ket
    const int ao = a0 + ty + 8 * e, bo = b0 + lane;
    if (ao < N && bo < N && (mirror || ao <= bo)) S[(size_t)ao * N + bo] = tr[ty + 8 * e][lane];
  }
}

__global__ void __launch_bounds__(256) k_heff(HeffArgs p) {
  __shared__ double2 tr[32][33];
  // the terms' factor values at the 32 bras and 32 kets
  __shared__ double uxs[HG][64], wRs[HG][64];
  __shared__ int s_last;
  int I, J;
  tri_tile(blockIdx.y, I, J);
  const int N = p.N, lane = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int ar = (blockIdx.x & 3) * 32 + lane, br = (blockIdx.x >> 2) * 32 + ty;
  const int a = I * MT + ar, b0 = J * MT + br;
  if (I * MT + (int)(blockIdx.x & 3) * 32 >= N || J * MT + (int)(blockIdx.x >> 2) * 32 >= N) return;
  const bool mirror = I != J, a_ok = a < N;
  const Tri tri(N);
  const size_t gs = tri.size(), at0 = tri.at(blockIdx.y) + (size_t)br * tri.br + ar, step = (size_t)8 * tri.br;
  double2 s1[4], s2[4], h[4], ht[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    s1[e] = cscale(p.S1[at0 + e * step], p.dx);
    s2[e] = cscale(p.S2[at0 + e * step], p.dR);
    h[e] = ht[e] = make_double2(0.0, 0.0);
    const int b = b0 + 8 * e;
    if (!p.first && blockIdx.z == 0 && a_ok && b < N) {
      h[e] = p.H[(size_t)a * N + b];
      if (mirror) ht[e] = p.H[(size_t)b * N + a];
    }
  }
  const int as = I * MT + (int)(blockIdx.x & 3) * 32, bs = J * MT + (int)(blockIdx.x >> 2) * 32;
  const int z0 = p.g0 + (int)((long long)(p.g1 - p.g0) * blockIdx.z / p.split);
  const int z1 = p.g0 + (int)((long long)(p.g1 - p.g0) * (blockIdx.z + 1) / p.split);
  for (int g = z0; g < z1; ++g) {
    const int gl = (g - z0) & (HG - 1);
    if (gl == 0) {
      __syncthreads();
      for (int i = threadIdx.x; i < HG * 64; i += 256) {
        const int gi = g + (i >> 6), c = i & 63, t = c < 32 ? as + c : bs + c - 32;
        if (gi < z1) {
          uxs[i >> 6][c] = t < N ? p.sig[gi] * p.px[(size_t)gi * N + t] : 0.0;
          wRs[i >> 6][c] = t < N ? p.pR[(size_t)gi * N + t] : 0.0;
        }
      }
      __syncthreads();
    }
    const double2* A = p.A + (size_t)(g - p.g0) * gs + at0;
    const double2* B = p.B + (size_t)(g - p.g0) * gs + at0;
    const double uxa = uxs[gl][lane], wRa = wRs[gl][lane];
    double2 xs[4], ys[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) { xs[e] = A[e * step]; ys[e] = B[e * step]; }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const double2 x = xs[e], y = ys[e];
      const double uxb = uxs[gl][32 + ty + 8 * e], wRb = wRs[gl][32 + ty + 8 * e];
      const double atr = x.x - uxb * s1[e].x, ati = x.y - uxb * s1[e].y;
      const double btr = y.x - wRb * s2[e].x, bti = y.y - wRb * s2[e].y;
      h[e].x = fma(atr, btr, fma(-ati, bti, h[e].x));
      h[e].y = fma(atr, bti, fma(ati, btr, h[e].y));
      if (mirror) {
        // entry (b, a): conj(A) - u(x_a) conj(S1), conj(B) - w(R_a) conj(S2)
        const double mtr = x.x - uxa * s1[e].x, mti = x.y - uxa * s1[e].y;
        const double ntr = y.x - wRa * s2[e].x, nti = y.y - wRa * s2[e].y;
        ht[e].x = fma(mtr, ntr, fma(-mti, nti, ht[e].x));
        ht[e].y = fma(-mtr, nti, fma(-mti, ntr, ht[e].y));
      }
    }
  }
  if (p.split > 1) {
    // few tiles: the terms are spread over CTAs; the last one to finish a patch adds the groups' sums
    // in their order (so the result does not depend on timing) and goes on
    double2* mine = p.part + blockIdx.z * 2 * gs + at0;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      mine[e * step] = h[e];
      if (mirror) mine[gs + e * step] = ht[e];
    }
    __threadfence();
    __syncthreads();
    unsigned* cnt = p.done + blockIdx.y * 16 + blockIdx.x;
    if (threadIdx.x == 0) s_last = atomicAdd(cnt, 1u) == (unsigned)p.split - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    if (threadIdx.x == 0) *cnt = 0;
#pragma unroll
    for (int e = 0; e < 4; ++e) h[e].x = h[e].y = ht[e].x = ht[e].y = 0;
    for (int z = 0; z < p.split; ++z) {
      const double2* q = p.part + z * 2 * gs + at0;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const double2 v = __ldcg(q + e * step);
        h[e].x += v.x; h[e].y += v.y;
        if (mirror) {
          const double2 w = __ldcg(q + gs + e * step);
          ht[e].x += w.x; ht[e].y += w.y;
        }
      }
    }
  }
  double2 sv[4];
  const double da = a_ok && p.last ? p.d[a] : 0.0;
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const int b = b0 + 8 * e;
    const bool in = a_ok && b < N;
    double2 hd = h[e], hm = ht[e];
    if (p.last) {
      sv[e] = cmul(s1[e], s2[e]);
      if (a == b) sv[e].y = 0.0;
      const double db = in ? p.d[b] : 0.0;
      hd = make_double2(hd.x - db * sv[e].x, hd.y - db * sv[e].y);
      hm = make_double2(hm.x - da * sv[e].x, hm.y + da * sv[e].y);
    }
    tr[lane][ty + 8 * e] = hd;
    if (mirror && in) p.H[(size_t)b * N + a] = hm;
  }
  __syncthreads();
  // rows of H: lane = ket
  const int ao = I * MT + (blockIdx.x & 3) * 32 + ty, bo = J * MT + (blockIdx.x >> 2) * 32 + lane;
#pragma unroll
  for (int e = 0; e < 4; ++e)
    if (ao + 8 * e < N && bo < N) p.H[(size_t)(ao + 8 * e) * N + bo] = tr[ty + 8 * e][lane];
  if (!p.last) return;
  __syncthreads();
  store_s(p.S, N, mirror, I * MT + (int)(blockIdx.x & 3) * 32, J * MT + (int)(blockIdx.x >> 2) * 32, sv, tr);
}

// S = S1 o S2 alone (the mixed modes), patches as above.
__global__ void __launch_bounds__(256) k_overlap(int N, const double2* __restrict__ S1, const double2* __restrict__ S2,
                                                 double dx, double dR, double2* __restrict__ S) {
  __shared__ double2 tr[32][33];
  int I, J;
  tri_tile(blockIdx.y, I, J);
  const int lane = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int ac = (int)(blockIdx.x & 3) * 32, bc = (int)(blockIdx.x >> 2) * 32;
  if (I * MT + ac >= N || J * MT + bc >= N) return;
  const Tri tri(N);
  const size_t at0 = tri.at(blockIdx.y) + (size_t)(bc + ty) * tri.br + ac + lane;
  double2 sv[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const size_t at = at0 + (size_t)8 * e * tri.br;
    sv[e] = cmul(cscale(S1[at], dx), cscale(S2[at], dR));
    if (I * MT + ac + lane == J * MT + bc + ty + 8 * e) sv[e].y = 0.0;
  }
  store_s(S, N, I != J, I * MT + ac, J * MT + bc, sv, tr);
}

// ---------------------------------------------------------------------------- plan

size_t al(size_t b) { return (b + 1023) & ~(size_t)1023; }
int ilog2_ceil(int n) { int l = 0; while ((1 << l) < n) ++l; return l; }

// Terms of one batch: as many as fit BATCH_BYTES of operands and Grams (at least one).  A batch is three
// launches and a last wave, so more memory is faster: at 512 / 128 / 64 / 32 MB a handle of N = 1024 on
// 1024 x 512 has 606 / 210 / 147 / 147 MB of work space and takes 6.7 / 7.3 / 7.6 / 7.6 ms for a step and
// the observables, one of N = 256 on 512 x 256 1.97 / 2.04 / 2.15 / 2.44 ms for two.  128 MB keeps the work
// space near the size of the handle's own state.
constexpr size_t BATCH_BYTES = (size_t)128 << 20;

int tiles_of(int N) { return Tri(N).tiles(); }
int kets_per_unit(int N, int most) { return N <= 32 && most > 32 ? 32 : (N <= 64 && most > 64 ? 64 : most); }

// K slices per accumulation of D digits (b0 = 6, beta = 7).  The leading D - 4 levels stay below 2^24
// whatever the digits are: (l + 1) pairs x 2 products x 2^12 x 16 points per slice.  The level after
// them could round only if its digits were all large and of one sign; its worst case, 2^-43 of the
// largest possible sum at 1024 points, is that of an FP64 sum of as many products.
int drain_slices(int d) {
  if (d <= 4) return 1 << 20;
  int s = 1;
  while (2 * s * 16 * (d - 4) <= (1 << 11)) s *= 2;
  return s;
}

// Digits of a term of relative size r (of its largest value on the grid, to the largest of all terms).
int term_digits(double r) {
  if (!(r > 0)) return 2;
  const int d = (int)std::ceil((56.0 + std::log2(r)) / 7.0);
  return d < 2 ? 2 : (d > 8 ? 8 : d);
}

// ---------------------------------------------------------------------------- trailing update
//
// The double-float Cholesky's trailing update over a panel of HERK_COLS columns as one Gram of the
// panel's rows: HERK_D digits (48 bits below a row's largest component, the precision of a double-float)
// and the pairs up to 2^-48 of the leading one; the epilogue subtracts in double-float.
// Bound: the tensor pipe, 8 slices of 2000 cycles per unit (128 x 32 elements; 2330 measured), and at few
// units the serial rest: 7300 cycles to the first MMA, 11000 from the last one to the stores.  (With the
// 64-bit integer sums of the other Grams and A read after them that was 24000.)
struct HerkSlices {
  const float4* A[2];
  unsigned char* out[2];
  int* ex[2];
  int N, k0, R0, rpad;
  Gram* grams;
  Gram g[2];
  int ng;
  unsigned* ticket;
};

// Digits of the panel's rows from R0 on, 16 threads per row with 8 columns each; rows past N: zeros.
// Also resets the Gram launch's ticket and writes its table.
__global__ void __launch_bounds__(256) k_herk_slices(HerkSlices p) {
  const int m = blockIdx.y, row = blockIdx.x * 16 + (threadIdx.x >> 4), c8 = threadIdx.x & 15;
  if (blockIdx.x == 0 && m == 0 && threadIdx.x == 0) {
    *p.ticket = 0;
    for (int i = 0; i < p.ng; ++i) p.grams[i] = i ? p.g[1] : p.g[0];
  }
  const float4* A = m ? p.A[1] : p.A[0];
  unsigned char* out = m ? p.out[1] : p.out[0];
  const int r = p.R0 + row;
  float4 v[8];
  unsigned mx = 0;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    v[k] = r < p.N ? A[(size_t)r * p.N + p.k0 + 8 * c8 + k] : make_float4(0.f, 0.f, 0.f, 0.f);
    mx = max(mx, max(__float_as_uint(v[k].x) & 0x7FFFFFFFu, __float_as_uint(v[k].z) & 0x7FFFFFFFu));
  }
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  const bool bad = mx >= 0x7F800000u;
  const int e = mx == 0 || bad ? 0 : max((int)(mx >> 23), 1) - 126;
  if (c8 == 0) (m ? p.ex[1] : p.ex[0])[row] = bad ? EX_BAD : e;
  const int q = HERK_B0 + HERK_BETA * (HERK_D - 1) - e;
#pragma unroll
  for (int plane = 0; plane < 2; ++plane) {
    uint32_t pk[HERK_D][4];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const float h = plane ? v[k].z : v[k].x, l = plane ? v[k].w : v[k].y;
      int dg[HERK_D];
      cut_digits<HERK_D>(bad ? 0 : fixed_of_f32(h, q) + fixed_of_f32(l, q), dg);
#pragma unroll
      for (int d = 0; d < HERK_D; ++d) {
        const uint32_t b = __float_as_uint(small_int_to_float(dg[d])) >> 16;
        if (k & 1) pk[d][k >> 1] |= b << 16;
        else pk[d][k >> 1] = b;
      }
    }
    const int tile = row / MT, rr = row - tile * MT;
#pragma unroll
    for (int d = 0; d < HERK_D; ++d)
      *(uint4*)(out + ((((size_t)tile * HERK_KS + (c8 >> 1)) * 2 + plane) * HERK_D + d) * (MT * ROW_BYTES) +
                swizzle32(rr, c8 & 1)) = make_uint4(pk[d][0], pk[d][1], pk[d][2], pk[d][3]);
  }
}

size_t herk_rows(int N) { return (size_t)(N + MT - 1) / MT * MT; }
size_t herk_operand(int N) { return herk_rows(N) * HERK_COLS * 2 * HERK_D * 2; }

}  // namespace sl

cudaError_t sliced_attributes() {
  return cudaFuncSetAttribute(sl::k_gram_sliced, cudaFuncAttributeMaxDynamicSharedMemorySize, sl::SMEM_BYTES);
}

size_t herk_df_bytes(int N) {
  using namespace sl;
  return chol_panel(N) == 0 ? 0 : 1024 + 2 * (herk_rows(N) * sizeof(int) + herk_operand(N));
}

int launch_herk_df(int N, int k0, int R0, void* const* A, int nb, void* scratch, int* status, cudaStream_t s) {
  using namespace sl;
  static_assert(2 * sizeof(Gram) <= 768, "table");
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  unsigned char* b = (unsigned char*)scratch;
  HerkSlices p{};
  p.N = N; p.k0 = k0; p.R0 = R0; p.ng = nb;
  p.rpad = (N - R0 + MT - 1) / MT * MT;
  p.ticket = (unsigned*)b;
  p.grams = (Gram*)(b + 256);
  const int tiles = p.rpad / MT, units = tiles * (tiles + 1) / 2 * (MT / 32);
  GramArgs ga{};
  for (int m = 0; m < 2; ++m) {
    const int k = m < nb ? m : 0;
    p.A[m] = (const float4*)A[k];
    p.ex[m] = (int*)(b + 1024) + k * herk_rows(N);
    p.out[m] = b + 1024 + 2 * herk_rows(N) * sizeof(int) + k * herk_operand(N);
    Gram& g = p.g[m];
    g.A = p.out[m];
    g.ea = g.eb = p.ex[m];
    g.rows = p.rpad;
    g.ks = g.drain = HERK_KS;
    g.da = g.d = g.l = HERK_D;
    g.t = 32;
    g.b0 = HERK_B0;
    g.beta = HERK_BETA;
    g.unit0 = m * units;
    ga.herk[m] = (float4*)A[k];
  }
  k_herk_slices<<<dim3(p.rpad / 16, nb), 256, 0, s>>>(p);
  ga.grams = p.grams;
  ga.ngrams = nb;
  ga.units = nb * units;
  ga.N = N;
  ga.R0 = R0;
  ga.ticket = p.ticket;
  ga.status = status;
  k_gram_sliced<<<std::min(ga.units, sms), THREADS, SMEM_BYTES, s>>>(ga);
  return 2;
}

// Layout of the scratch and tables of one handle's assembly.  Built twice: once to size the arena
// (base NULL), once to fill it.
struct AsmPlan::Impl {
  struct Batch { int slice0, nslice, gram0, ngram, units, g0, g1, rowgroups; size_t A, B; };
  std::vector<sl::Slice> slices;
  std::vector<sl::Gram> grams;
  std::vector<Batch> batches;
  std::vector<double> Uw, Ww;            // FP64 mode: weights u_g s_g dx and w_g dR
  size_t work = 0;                       // start of the region below, which every stage uses for itself
  size_t part = 0, o_done = 0;           // split term sums of k_heff
  int split = 1;
  size_t bytes = 0, o_slices = 0, o_grams = 0, o_uw = 0, o_ww = 0, o_ticket = 0;
  size_t S1 = 0, S2 = 0;
  size_t r_xa = 0, r_xe = 0, r_Rb = 0, r_Re = 0;   // reconstruction operands (in the batch scratch)
  int rec_gram = 0, rec_units = 0, rec_d = 0;
  unsigned char* base = nullptr;
  int precision = 0;
  bool f64 = false, split_s = false;
  int sms = 152;
};

AsmPlan::AsmPlan() {}
AsmPlan::~AsmPlan() { delete impl; }

size_t AsmPlan::layout(const AsmShape& q, const JobView* j, void* base, size_t work_min) {
  using namespace sl;
  delete impl;
  impl = new Impl;
  Impl& m = *impl;
  const bool f64 = q.precision == ICWF_FP64, split_s = !f64 && q.overlap_split;
  m.precision = q.precision;
  m.f64 = f64;
  m.split_s = split_s;
  m.base = (unsigned char*)base;
  const int N = q.N, K = q.K;
  const int rp = (N + MT - 1) / MT * MT, tiles = tiles_of(N);
  const int n[2] = {q.nx, q.nR}, ks[2] = {(q.nx + 15) / 16, (q.nR + 15) / 16};
  size_t off = 0;
  auto take = [&](size_t b) { const size_t o = off; off += al(b); return o; };
  const size_t out_b = Tri(N).size() * sizeof(double2);
  m.o_ticket = take(256);
  const int dS = f64 ? 8 : 4;
  auto op_bytes = [&](int side, int rows, int d) { return (size_t)rows * ks[side] * 2 * d * ROW_BYTES; };
  auto padded = [&](int r) { return (N + r - 1) / r * r; };   // rows of an operand in tiles of r
  std::vector<int> dg(K, 0);
  std::vector<std::pair<int, int>> ranges;   // batches of terms (FP64 mode)
  size_t batch_max = 0;
  if (f64) {
    m.o_uw = take((size_t)K * q.nx * 8);
    m.o_ww = take((size_t)K * q.nR * 8);
    // few tiles leave SMs idle in k_heff: spread the terms over up to 16 groups of 4 or more
    const int patches = tiles_of(N) == 1 ? ((N + 31) / 32) * ((N + 31) / 32) : tiles * 16;
    m.split = std::max(1, std::min({16, 304 / patches, K / 4}));
    m.o_done = take((size_t)tiles * 16 * 4);
    const double top = *std::max_element(q.peak, q.peak + K);
    for (int g = 0; g < K; ++g) dg[g] = term_digits(top > 0 ? q.peak[g] / top : 0.0);
  } else if (!split_s) {
    ranges.push_back({0, 0});   // the overlap alone
  }
  // kets per unit of a term of d digits
  auto kets = [&](int side, int d) {
    const int t = drain_slices(d) < ks[side] ? 32 : (d <= 2 ? 128 : (d <= 4 ? 64 : 32));
    return kets_per_unit(N, t);
  };
  for (int g = 0; f64 && g < K;) {
    size_t b = 0;
    int e = g;
    while (e < K && 2 * (e - g) + 4 < MAX_GRAMS) {
      size_t add = 2 * al(out_b);
      for (int s = 0; s < 2; ++s) {
        const int r = padded(kets(s, dg[e]));
        add += al(op_bytes(s, r, dg[e])) + al((size_t)r * 4);
      }
      if (e > g && b + add > BATCH_BYTES) break;
      b += add;
      ++e;
    }
    batch_max = std::max(batch_max, b);
    ranges.push_back({g, e});
    g = e;
  }
  // One region for the stages that follow each other: the assembly's operands and Grams (mixed modes: of
  // the overlap), the mixed modes' split operands, the reconstruction's operands, and what the
  // caller runs in between (work_min bytes).
  m.work = off;
  m.S1 = take(out_b);
  m.S2 = take(out_b);
  // digits of the CWFs: the operands of S and the bras of every term
  size_t sa[2] = {0, 0}, se[2] = {0, 0};
  for (int s = 0; s < 2; ++s) {
    sa[s] = take(op_bytes(s, rp, dS));
    se[s] = take((size_t)rp * 4);
  }
  if (m.split > 1) m.part = take((size_t)m.split * 2 * out_b);
  const int rxp = (q.nx + MT - 1) / MT * MT, rRp = (q.nR + MT - 1) / MT * MT, ksN = (N + 15) / 16;
  m.rec_d = f64 ? 8 : 5;
  auto rec_op = [&](int rows) { return (size_t)rows * ksN * 2 * m.rec_d * ROW_BYTES; };
  const size_t rec_bytes = al(rec_op(rxp)) + al(rec_op(rRp)) + al((size_t)rxp * 4) + al((size_t)rRp * 4);
  const size_t scratch = take(batch_max);
  size_t work_bytes = split_s ? 0 : off - m.work;
  if (!f64) work_bytes = std::max(work_bytes, heff_tc_scratch_bytes(N, q.nx, q.nR, K));
  off = m.work + al(std::max({work_bytes, rec_bytes, work_min}));
  m.r_xa = m.work;
  m.r_Rb = m.r_xa + al(rec_op(rxp));
  m.r_xe = m.r_Rb + al(rec_op(rRp));
  m.r_Re = m.r_xe + al((size_t)rxp * 4);
  auto ptr = [&](size_t o) { return m.base + o; };
  for (size_t r = 0; r < ranges.size(); ++r) {
    const int g0 = ranges[r].first, g1 = ranges[r].second;
    Impl::Batch b{};
    b.slice0 = (int)m.slices.size();
    b.gram0 = (int)m.grams.size();
    b.g0 = g0;
    b.g1 = g1;
    auto add_slice = [&](int side, const double* w, size_t out, size_t ex, int R, int d, int b0, int beta) {
      Slice s{};
      s.src = j ? (side ? j->chi : j->psi) : nullptr;
      s.w = w;
      s.ng = 1;
      s.out = ptr(out);
      s.ex = (int*)ptr(ex);
      s.n = n[side]; s.ks = ks[side]; s.rows = N; s.rpad = padded(R); s.R = R;
      s.d = d; s.b0 = b0; s.beta = beta;
      m.slices.push_back(s);
    };
    auto add_gram = [&](int side, size_t A, size_t eA, int da, const unsigned char* B, const int* eB, int d, int l,
                        int t, int drain, int b0, int beta, size_t out) {
      Gram x{};
      x.A = ptr(A);
      x.B = B;
      x.ea = (int*)ptr(eA);
      x.eb = eB ? eB : (int*)ptr(eA);
      x.out = (double2*)ptr(out);
      x.ks = ks[side]; x.da = da; x.d = d; x.l = l; x.t = t; x.drain = drain;
      x.b0 = b0; x.beta = beta;
      x.rows = N;
      // |sum| <= 2 K 2^(2 b0) units of level 0
      x.fbits = 62 - (1 + ilog2_ceil(16 * ks[side]) + 2 * b0);
      m.grams.push_back(x);
    };
    for (int s = 0; s < 2; ++s) {
      if (r > 0) break;   // bras and the overlap once per assembly
      const int bd = f64 ? 6 : (n[s] <= 2048 ? 6 : 5), beta = f64 ? 7 : bd;
      add_slice(s, nullptr, sa[s], se[s], MT, dS, bd, beta);
      const int L = f64 ? dS : 2 * dS - 1;
      add_gram(s, sa[s], se[s], dS, nullptr, nullptr, dS, L, 32, f64 ? drain_slices(dS) : 1 << 20, bd, beta,
               s ? m.S2 : m.S1);
    }
    size_t so = scratch;
    auto tmp = [&](size_t bytes) { const size_t o = so; so += al(bytes); return o; };
    // the Grams of one side are consecutive (k_heff walks them with a fixed stride)
    b.A = tmp((size_t)(g1 - g0) * out_b);
    b.B = tmp((size_t)(g1 - g0) * out_b);
    int grp[2] = {-1, -1};
    for (int g = g0; g < g1; ++g)
      for (int s = 0; s < 2; ++s) {
        const int d = dg[g];
        const int dr = drain_slices(d), t = kets(s, d);
        const size_t o = tmp(op_bytes(s, padded(t), d)), oe = tmp((size_t)padded(t) * 4);
        const double* w = (const double*)ptr(s ? m.o_ww : m.o_uw) + (size_t)g * n[s];
        // consecutive terms in the same format share a group (their operands are evenly spaced)
        Slice* last = grp[s] >= 0 ? &m.slices[grp[s]] : nullptr;
        if (last && last->ng < SLICE_GROUP && last->d == d && last->R == t) {
          const size_t os = (size_t)(ptr(o) - last->out), es = (size_t)((int*)ptr(oe) - last->ex);
          if (last->ng == 1) { last->ostride = os; last->estride = es; }
          if (os == last->ng * last->ostride && es == last->ng * last->estride) ++last->ng;
          else last = nullptr;
        } else {
          last = nullptr;
        }
        if (!last) {
          grp[s] = (int)m.slices.size();
          add_slice(s, w, o, oe, t, d, 6, 7);
        }
        add_gram(s, sa[s], se[s], dS, ptr(o), (int*)ptr(oe), d, d, t, dr, 6, 7,
                 (s ? b.B : b.A) + (size_t)(g - g0) * out_b);
      }
    b.nslice = (int)m.slices.size() - b.slice0;
    b.ngram = (int)m.grams.size() - b.gram0;
    // the most expensive units first (tensor time of a unit: levels' pairs x kets x slices)
    auto cost = [](const Gram& x) {
      int pairs = 0;
      for (int p = 0; p < x.d; ++p) pairs += std::min(x.d, x.l - p);
      return (long long)pairs * x.t * x.ks;
    };
    std::stable_sort(m.grams.begin() + b.gram0, m.grams.end(),
                     [&](const Gram& x, const Gram& y) { return cost(x) > cost(y); });
    for (int i = 0; i < b.ngram; ++i) {
      Gram& x = m.grams[b.gram0 + i];
      x.unit0 = b.units;
      b.units += Tri(N).units(x.t);
    }
    for (int i = 0; i < b.nslice; ++i) {
      const Slice& s = m.slices[b.slice0 + i];
      const int tpr = std::min(2 * s.ks, 256), rpb = 256 / tpr;
      b.rowgroups = std::max(b.rowgroups, (s.rpad + rpb - 1) / rpb);
    }
    m.batches.push_back(b);
  }
  {
    Gram x{};
    x.A = ptr(m.r_xa); x.B = ptr(m.r_Rb);
    x.ea = (int*)ptr(m.r_xe); x.eb = (int*)ptr(m.r_Re);
    x.ks = ksN; x.da = x.d = x.l = m.rec_d; x.t = 32; x.drain = drain_slices(m.rec_d);
    x.b0 = 6; x.beta = 7;
    x.fbits = 62 - (1 + ilog2_ceil(16 * ksN) + 12);
    x.rows = q.nx; x.cols = q.nR;
    m.rec_gram = (int)m.grams.size();
    m.rec_units = rxp / MT * ((q.nR + 31) / 32);
    m.grams.push_back(x);   // its output is an argument of the launch
  }
  m.o_slices = take(m.slices.size() * sizeof(Slice));
  m.o_grams = take(m.grams.size() * sizeof(Gram));
  m.bytes = off;
  return m.bytes;
}

void* AsmPlan::work() const { return impl->base + impl->work; }

bool AsmPlan::upload(const AsmShape& q, const double* U, const double* W, cudaStream_t s) {
  using namespace sl;
  Impl& m = *impl;
  const size_t nu = (size_t)q.K * q.nx, nw = (size_t)q.K * q.nR;
  if (m.f64) {
    m.Uw.resize(nu);
    m.Ww.resize(nw);
    for (int g = 0; g < q.K; ++g) {
      for (int i = 0; i < q.nx; ++i) m.Uw[(size_t)g * q.nx + i] = U[(size_t)g * q.nx + i] * (q.sig[g] * q.dx);
      for (int i = 0; i < q.nR; ++i) m.Ww[(size_t)g * q.nR + i] = W[(size_t)g * q.nR + i] * q.dR;
    }
    if (cudaMemcpyAsync(m.base + m.o_uw, m.Uw.data(), nu * 8, cudaMemcpyHostToDevice, s) != cudaSuccess ||
        cudaMemcpyAsync(m.base + m.o_ww, m.Ww.data(), nw * 8, cudaMemcpyHostToDevice, s) != cudaSuccess ||
        cudaMemsetAsync(m.base + m.o_done, 0, (size_t)tiles_of(q.N) * 16 * 4, s) != cudaSuccess)
      return false;
  } else if (!heff_tc_ready()) {
    return false;
  }
  if (cudaMemcpyAsync(m.base + m.o_slices, m.slices.data(), m.slices.size() * sizeof(Slice), cudaMemcpyHostToDevice,
                      s) != cudaSuccess ||
      cudaMemcpyAsync(m.base + m.o_grams, m.grams.data(), m.grams.size() * sizeof(Gram), cudaMemcpyHostToDevice,
                      s) != cudaSuccess)
    return false;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&m.sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return false;
  return cudaStreamSynchronize(s) == cudaSuccess;
}

int AsmPlan::launch(const JobView& j, double2* S, double2* H, cudaStream_t s) const {
  using namespace sl;
  const Impl& m = *impl;
  const int tiles = tiles_of(j.N);
  for (const auto& b : m.batches) {
    const Slice* sl0 = (const Slice*)(m.base + m.o_slices) + b.slice0;
    unsigned* ticket = (unsigned*)(m.base + m.o_ticket);
    if (m.f64) k_slices<double><<<dim3(b.rowgroups, b.nslice), 256, 0, s>>>(sl0, ticket);
    else k_slices<float><<<dim3(b.rowgroups, b.nslice), 256, 0, s>>>(sl0, ticket);
    GramArgs ga{};
    ga.grams = (const Gram*)(m.base + m.o_grams) + b.gram0;
    ga.out = nullptr;
    ga.ngrams = b.ngram;
    ga.units = b.units;
    ga.N = j.N;
    ga.ticket = (unsigned*)(m.base + m.o_ticket);
    ga.status = j.status;
    k_gram_sliced<<<std::min(b.units, m.sms), THREADS, SMEM_BYTES, s>>>(ga);
    if (!m.f64) {
      k_overlap<<<dim3(16, tiles), 256, 0, s>>>(j.N, (const double2*)(m.base + m.S1), (const double2*)(m.base + m.S2),
                                                j.dx, j.dR, S);
      break;
    }
    HeffArgs ha;
    ha.N = j.N; ha.g0 = b.g0; ha.g1 = b.g1;
    ha.first = b.g0 == 0;
    ha.last = b.g1 == j.K;
    ha.S1 = (const double2*)(m.base + m.S1); ha.S2 = (const double2*)(m.base + m.S2);
    ha.A = (const double2*)(m.base + b.A); ha.B = (const double2*)(m.base + b.B);
    ha.dx = j.dx; ha.dR = j.dR;
    ha.sig = j.sig; ha.px = j.px; ha.pR = j.pR; ha.d = j.d;
    ha.S = S; ha.H = H;
    ha.split = std::max(1, std::min(m.split, (b.g1 - b.g0) / 4));
    ha.part = (double2*)(m.base + m.part);
    ha.done = (unsigned*)(m.base + m.o_done);
    k_heff<<<dim3(16, tiles, ha.split), 256, 0, s>>>(ha);
  }
  int launches = 3 * (int)m.batches.size();
  // the overlap's operands are no longer needed
  if (!m.f64) launches += launch_heff_tc(j, m.precision, m.split_s ? S : nullptr, H, m.base + m.work, s);
  return launches;
}

// Psi[i nR + j] = sum_a C_a psi_a(x_i) chi_a(R_j) as a sliced product over the trajectories: 8 digits
// in the FP64 mode, 5 in the mixed modes, whose terms carry FP32 rounding.  Digits are cut below the largest
// component of an operand's row, so a sum is good to 2^-55 (2^-34) of max_a |C_a psi_a(x_i)| max_a
// |chi_a(R_j)|, which is more than the largest term where different trajectories give the two maxima: far
// out in the tails of Psi.
int AsmPlan::reconstruct(const JobView& j, const double2* C, double2* Psi, cudaStream_t s) const {
  using namespace sl;
  const Impl& m = *impl;
  const int rxp = (j.nx + MT - 1) / MT * MT, rRp = (j.nR + MT - 1) / MT * MT;
  SliceT sx{}, sR{};
  sx.src = j.psi; sx.C = C;
  sx.out = m.base + m.r_xa; sx.ex = (int*)(m.base + m.r_xe);
  sx.n = j.nx; sx.ks = (j.N + 15) / 16; sx.N = j.N; sx.rpad = rxp; sx.R = MT; sx.d = m.rec_d; sx.f32 = !m.f64;
  sR = sx;
  sR.src = j.chi; sR.C = nullptr;
  sR.out = m.base + m.r_Rb; sR.ex = (int*)(m.base + m.r_Re);
  sR.n = j.nR; sR.rpad = rRp; sR.R = 32;
  k_slices_t<<<dim3(std::max(rxp, rRp) / ST_ROWS, 2), ST_WARPS * 32, 0, s>>>(sx, sR, (unsigned*)(m.base + m.o_ticket));
  GramArgs ga{};
  ga.grams = (const Gram*)(m.base + m.o_grams) + m.rec_gram;
  ga.out = Psi;
  ga.ngrams = 1;
  ga.units = m.rec_units;
  ga.N = j.N;
  ga.ticket = (unsigned*)(m.base + m.o_ticket);
  ga.status = j.status + STATUS_OBS;
  k_gram_sliced<<<std::min(ga.units, m.sms), THREADS, SMEM_BYTES, s>>>(ga);
  return 2;
}

}  // namespace icwf
