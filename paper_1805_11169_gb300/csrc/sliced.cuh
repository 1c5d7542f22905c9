// Number formats and index arithmetic of the sliced Grams (k_sliced.cu): digits of FP64 numbers by
// integer operations, their integer sums back to FP64, the operand swizzle and the triangular tile
// index.  Host and device code.
#pragma once
#include <math.h>
#include <stddef.h>
#include <stdint.h>
#include <string.h>

#if defined(__CUDACC__)
#define SL_HD __host__ __device__ __forceinline__
#else
#define SL_HD inline
#endif

namespace icwf {
namespace sl {

constexpr int MT = 128;          // bras (and kets) per output tile
constexpr int ROW_BYTES = 32;    // one operand row of a K slice: 16 values of 2 bytes

// Byte offset of the 8-point half `part` of row r inside an operand tile: rows of 32 bytes, the two
// 16-byte halves swapped in every second group of four rows (the 32-byte swizzle: address bit 4 is
// XORed with bit 7; tiles start on 256-byte boundaries).
SL_HD int swizzle32(int r, int part) { return r * ROW_BYTES + ((part ^ ((r >> 2) & 1)) << 4); }

// Upper-triangle tile (I <= J) number t, column by column.
SL_HD void tri_tile(int t, int& I, int& J) {
  int c = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
  while (c * (c + 1) / 2 > t) --c;
  while ((c + 1) * (c + 2) / 2 <= t) ++c;
  J = c;
  I = t - c * (c + 1) / 2;
}

// Storage of a Hermitian Gram of N trajectories: 128 x 128 tiles [ket][bra] of the upper triangle, column
// by column; those of the last column hold only the kets that there are, in whole 32s, and a single tile
// only such bras.
struct Tri {
  int T, full;    // row blocks; tiles before the last column
  int kl, br;     // kets of the last column's tiles; bras of a row of a tile
  SL_HD explicit Tri(int N)
      : T((N + MT - 1) / MT), full(T * (T - 1) / 2), kl((N - (T - 1) * MT + 31) / 32 * 32), br(T == 1 ? kl : MT) {}
  SL_HD int tiles() const { return full + T; }
  SL_HD size_t at(int tile) const {
    return tile <= full ? (size_t)tile * MT * MT : (size_t)full * MT * MT + (size_t)(tile - full) * kl * br;
  }
  SL_HD size_t size() const { return at(tiles()); }
  // units of t kets: of a tile, of all tiles, and the tile and part of unit v
  SL_HD int units_last(int t) const { return (kl + t - 1) / t; }
  SL_HD int units(int t) const { return full * (MT / t) + T * units_last(t); }
  SL_HD void unit(int v, int t, int& tile, int& part) const {
    const int q = MT / t, f = full * q, l = units_last(t);
    tile = v < f ? v / q : full + (v - f) / l;
    part = v < f ? v % q : (v - f) % l;
  }
};

SL_HD unsigned long long f64_bits(double x) {
#if defined(__CUDA_ARCH__)
  return (unsigned long long)__double_as_longlong(x);
#else
  unsigned long long u;
  memcpy(&u, &x, 8);
  return u;
#endif
}
SL_HD double bits_f64(unsigned long long u) {
#if defined(__CUDA_ARCH__)
  return __longlong_as_double((long long)u);
#else
  double x;
  memcpy(&x, &u, 8);
  return x;
#endif
}
SL_HD int clz64(unsigned long long u) {
#if defined(__CUDA_ARCH__)
  return __clzll((long long)u);
#else
  return u ? __builtin_clzll(u) : 64;
#endif
}
SL_HD unsigned long long abs_bits(double x) { return f64_bits(x) & 0x7FFFFFFFFFFFFFFFull; }

// The smallest e with |x| < 2^e for a finite |x| given by its bits (0 for zero).
SL_HD int exponent_above_f64(unsigned long long mbits) {
  const int E = (int)(mbits >> 52);
  if (E) return E - 1022;
  return mbits ? -1074 + (64 - clz64(mbits)) : 0;
}

// round(x 2^q) for |x| 2^q < 2^62, half away from zero.
SL_HD long long fixed_of(double x, int q) {
  const unsigned long long u = f64_bits(x);
  const int E = (int)((u >> 52) & 0x7FFu);
  const unsigned long long frac = u & 0xFFFFFFFFFFFFFull;
  const unsigned long long mant = E ? (frac | (1ull << 52)) : frac;   // |x| = mant 2^p2
  const int s = (E ? E - 1075 : -1074) + q;
  unsigned long long r;
  if (s >= 0) r = mant << s;
  else if (s <= -54) r = 0;   // below half a unit
  else r = (mant + (1ull << (-s - 1))) >> (-s);
  return (u >> 63) ? -(long long)r : (long long)r;
}

// The same of an FP32 number.
SL_HD long long fixed_of_f32(float x, int q) {
#if defined(__CUDA_ARCH__)
  const uint32_t u = __float_as_uint(x);
#else
  uint32_t u;
  memcpy(&u, &x, 4);
#endif
  const uint32_t E = (u >> 23) & 0xFFu;
  const unsigned long long mant = (u & 0x7FFFFFu) | (E ? 0x800000u : 0u);
  const int s = (E ? (int)E - 150 : -149) + q;
  unsigned long long r;
  if (s >= 0) r = mant << s;
  else if (s <= -25) r = 0;
  else r = (mant + (1ull << (-s - 1))) >> (-s);
  return u >> 31 ? -(long long)r : (long long)r;
}

// D balanced base-2^7 digits of X, most significant first: the lower ones in [-64, 63], the first takes
// what is left (|d_0| <= 64 when |X| <= 2^(6 + 7 (D - 1))).
template <int D>
SL_HD void cut_digits(long long X, int (&dg)[D]) {
#if defined(__CUDACC__)
#pragma unroll
#endif
  for (int p = D - 1; p > 0; --p) {
    const int d = (int)((X + 64) & 127) - 64;
    dg[p] = d;
    X = (X - d) >> 7;
  }
  dg[0] = (int)X;
}
// digits of round(x 2^q)
template <int D>
SL_HD void digits_of(double x, int q, int (&dg)[D]) {
  cut_digits<D>(fixed_of(x, q), dg);
}

// An integer of at most 22 bits as a float: added to the bits of 1.5 2^23, whose unit is 1.
SL_HD float small_int_to_float(int d) {
  const uint32_t b = 0x4B400000u + (uint32_t)d;
  float f;
#if defined(__CUDA_ARCH__)
  f = __uint_as_float(b);
#else
  memcpy(&f, &b, 4);
#endif
  return f - 12582912.0f;
}

// x 2^sh rounded once to FP64, by integer operations.
SL_HD double fixed_to_f64(long long x, int sh) {
  if (x == 0) return 0.0;
  const unsigned long long neg = x < 0 ? 1ull << 63 : 0ull;
  unsigned long long u = x < 0 ? 0ull - (unsigned long long)x : (unsigned long long)x;
  const int z = clz64(u);
  u <<= z;
  const unsigned long long m = (u >> 11) + ((u >> 10) & 1ull);   // 53 bits, half up
  const int E = 1023 + 63 - z + sh;                              // biased exponent of 2^52-scaled m
  if (E <= 1 || E >= 2046) return ldexp((double)x, sh);
  return bits_f64(neg | ((((unsigned long long)(E - 1)) << 52) + m));
}

}  // namespace sl
}  // namespace icwf
