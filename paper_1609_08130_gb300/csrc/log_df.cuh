// log_df.cuh -- the natural logarithm in pairs of FP32 numbers (df.cuh).
//
// Tang's table-driven method (P. T. P. Tang, ACM Trans. Math. Softw. 16(4),
// 1990): x = 2^e m, c the centre of m's interval of width 1/128,
// t = m / c - 1 with 1/c rounded to 12 bits (|t| < 2^-7.9), log x = e ln 2 +
// log c + log(1 + t); the leading terms as pairs, the cubic and higher ones in
// FP32 (below 2^-24 of the rest).  Absolute error about 2^-48 max(1, |log x|).
#pragma once
#include "df.cuh"

namespace rss {

// lt: 1/c and log c (a pair) of the 128 intervals; et: (e - shift) ln 2 (a
// pair) by the biased exponent.
struct LogTables {
  float4 lt[128];
  float2 et[256];
};
// Entry `i` of both tables (i < 256; the first 128 threads fill lt).
__device__ __forceinline__ void log_tables_entry(LogTables *T, int i, int shift) {
  if (i < 128) {
    const double c = 1.0 + (double)(2 * i + 1) * (1.0 / 256.0);
    const double ic = rint(4096.0 / c) * (1.0 / 4096.0), lc = -log(ic);
    const float h = (float)lc;
    T->lt[i] = make_float4((float)ic, h, (float)(lc - (double)h), 0.f);
  }
  const double ev = (double)(i - 127 - shift) * 0.69314718055994530942;
  const float h = (float)ev;
  T->et[i] = make_float2(h, (float)(ev - (double)h));
}

// log of r2 > 0, a normal FP32 pair
__device__ __forceinline__ Df log_df(Df r2, const float4 *lt, const float2 *et) {
  const unsigned u = __float_as_uint(r2.h);
  const float4 T = lt[(u >> 16) & 127];
  const float2 E = et[u >> 23];
  const float mh = __uint_as_float((u & 0x7fffffu) | 0x3f800000u);
  const float ml = r2.l * __uint_as_float(0x7f000000u - (u & 0x7f800000u));
  const float p = __fmul_rn(mh, T.x), pe = __fmaf_rn(mh, T.x, -p);
  const float th = __fadd_rn(p, -1.f);  // exact
  const float tl = __fmaf_rn(ml, T.x, pe);
  const float sq = __fmul_rn(th, th), se = __fmaf_rn(th, th, -sq);
  float pol = __fmaf_rn(th, -1.f / 6.f, 0.2f);
  pol = __fmaf_rn(th, pol, -0.25f);
  pol = __fmaf_rn(th, pol, 1.f / 3.f);
  float lo = __fmaf_rn(-0.5f, se, __fmul_rn(__fmul_rn(sq, th), pol));
  // tl's share: tl (1 - th + th^2 - th^3 - tl / 2)
  const float g = __fmaf_rn(0.5f, tl, __fmaf_rn(sq, th, __fmaf_rn(-th, th, th)));
  lo = __fadd_rn(lo, __fmaf_rn(-g, tl, tl));
  const Df ab = quick_two_sum(th, -0.5f * sq);
  const Df uv = two_sum(E.x, T.y);
  const Df w = two_sum(uv.h, ab.h);
  lo = __fadd_rn(__fadd_rn(lo, __fadd_rn(E.y, T.z)), __fadd_rn(__fadd_rn(uv.l, ab.l), w.l));
  return quick_two_sum(w.h, lo);
}

}  // namespace rss
