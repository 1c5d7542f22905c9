// Complex double-floats as stored by the double-float solver, (re_hi, re_lo, im_hi, im_lo) in 16 bytes,
// and complex dot products in compensated (Dot2) accumulation.
#pragma once
#include <cuda_runtime.h>

#include "df64.cuh"

namespace icwf {
namespace dfs {

__device__ __forceinline__ cdf ld4(const float4 v) {
  return cdf_make(df_make(v.x, v.y), df_make(v.z, v.w));
}
__device__ __forceinline__ float4 st4(cdf z) { return make_float4(z.re.h, z.re.l, z.im.h, z.im.l); }
__device__ __forceinline__ cdf czero() { return cdf_make(df_make(0.f, 0.f), df_make(0.f, 0.f)); }

// Compensated accumulator: value = s + c.
struct acc2 {
  float s, c;
};
__device__ __forceinline__ void acc_prod(acc2& a, float x, float y) {
  const float p = DF_MUL(x, y);
  const float e = DF_FMA(x, y, -p);
  const df t = two_sum(a.s, p);
  a.s = t.h;
  a.c = DF_ADD(a.c, DF_ADD(t.l, e));
}
__device__ __forceinline__ void acc_small(acc2& a, float x) { a.c = DF_ADD(a.c, x); }
__device__ __forceinline__ df acc_val(acc2 a) { return two_sum(a.s, a.c); }
__device__ __forceinline__ acc2 acc_zero() { acc2 a; a.s = 0.f; a.c = 0.f; return a; }
__device__ __forceinline__ acc2 acc_merge(acc2 a, acc2 b) {
  const df t = two_sum(a.s, b.s);
  acc2 r;
  r.s = t.h;
  r.c = DF_ADD(DF_ADD(a.c, b.c), t.l);
  return r;
}

struct cacc {
  acc2 re, im;
};
__device__ __forceinline__ cacc cacc_zero() { cacc z; z.re = acc_zero(); z.im = acc_zero(); return z; }
__device__ __forceinline__ cacc cacc_merge(cacc a, cacc b) {
  cacc r; r.re = acc_merge(a.re, b.re); r.im = acc_merge(a.im, b.im); return r;
}
__device__ __forceinline__ cdf cacc_val(cacc a) { return cdf_make(acc_val(a.re), acc_val(a.im)); }
// a += x * y
__device__ __forceinline__ void cacc_mul(cacc& a, cdf x, cdf y) {
  acc_prod(a.re, x.re.h, y.re.h);
  acc_prod(a.re, -x.im.h, y.im.h);
  acc_small(a.re, DF_FMA(x.re.h, y.re.l, DF_MUL(x.re.l, y.re.h)));
  acc_small(a.re, -DF_FMA(x.im.h, y.im.l, DF_MUL(x.im.l, y.im.h)));
  acc_prod(a.im, x.re.h, y.im.h);
  acc_prod(a.im, x.im.h, y.re.h);
  acc_small(a.im, DF_FMA(x.re.h, y.im.l, DF_MUL(x.re.l, y.im.h)));
  acc_small(a.im, DF_FMA(x.im.h, y.re.l, DF_MUL(x.im.l, y.re.h)));
}
// a += conj(x) * y
__device__ __forceinline__ void cacc_cmul(cacc& a, cdf x, cdf y) {
  acc_prod(a.re, x.re.h, y.re.h);
  acc_prod(a.re, x.im.h, y.im.h);
  acc_small(a.re, DF_FMA(x.re.h, y.re.l, DF_MUL(x.re.l, y.re.h)));
  acc_small(a.re, DF_FMA(x.im.h, y.im.l, DF_MUL(x.im.l, y.im.h)));
  acc_prod(a.im, x.re.h, y.im.h);
  acc_prod(a.im, -x.im.h, y.re.h);
  acc_small(a.im, DF_FMA(x.re.h, y.im.l, DF_MUL(x.re.l, y.im.h)));
  acc_small(a.im, -DF_FMA(x.im.h, y.re.l, DF_MUL(x.im.l, y.re.h)));
}

}  // namespace dfs
}  // namespace icwf
