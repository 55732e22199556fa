// log_tf.cuh -- the natural logarithm in three FP32 parts (tf.cuh).
//
// Tang's table-driven method (P. T. P. Tang, ACM Trans. Math. Softw. 16(4),
// 1990): x = 2^e m, c the centre of m's interval of width 1/512, ic = 1/c
// rounded to FP32, t = m ic - 1 (|t| < 2^-9.9), log x = e ln 2 - log ic +
// log(1 + t).  e ln 2 and -log ic are in three parts, the first two multiples of
// 2^-13 and 2^-34, so that their sums are exact; t in two parts and its rounding
// errors; t^2 / 2 as a product and its error; the cubic and higher terms
// (below 2^-31) in FP32.  Absolute error about 2^-56 max(1, |log x|).
#pragma once
#include "tf.cuh"

namespace rss {

constexpr int LOG_CELLS = 512;
constexpr float LOG_M = 0x1.8p-11f;  // the anchor of the second parts, in lt's

// lt: 1/c and -log(1/c) (the second part plus LOG_M) of the intervals; et:
// (e - shift) ln 2 by the biased exponent.
struct LogTables {
  float4 lt[LOG_CELLS];
  float4 et[256];
};

// k ln 2 in the parts of et, |k| < 2^11: ln 2 as a number of 33 bits and the rest
__device__ __forceinline__ float4 log_tables_exponent(int k) {
  const double a = (double)k * 0x1.62e42feep-1, b = (double)k * 0x1.a39ef35793c76p-33;
  const double h = rint(a * 0x1p13) * 0x1p-13, m = rint((a - h + b) * 0x1p34) * 0x1p-34;
  return make_float4((float)h, (float)m, (float)((a - h - m) + b), 0.f);
}

// log of x > 0, a normal FP32 leading part
__device__ __forceinline__ Tf log_tf(Tf x, const float4 *lt, const float4 *et) {
  const unsigned u = __float_as_uint(x.h);
  const float4 T = lt[(u >> 14) & (LOG_CELLS - 1)];
  const float4 E = et[u >> 23];
  const float mh = __uint_as_float((u & 0x7fffffu) | 0x3f800000u);
  const float sc = __uint_as_float(0x7f000000u - (u & 0x7f800000u));
  const float mm = x.m * sc, ml = x.l * sc;
  const float p = __fmul_rn(mh, T.x), pe = __fmaf_rn(mh, T.x, -p);
  const float q = __fmul_rn(mm, T.x), qe = __fmaf_rn(mm, T.x, -q);
  const float th = __fadd_rn(p, -1.f), tl = __fadd_rn(pe, q);  // th exact
  const float sq = __fmul_rn(th, th), se = __fmaf_rn(th, th, -sq);
  // th^3 (1/3 - th / 4 + th^2 / 5); -se / 2 and tl's share tl (-th + th^2 - th^3 - tl / 2)
  const float pol = __fmaf_rn(th, __fmaf_rn(th, 0.2f, -0.25f), 1.f / 3.f);
  float lo = __fmaf_rn(-0.5f, se, __fmaf_rn(ml, T.x, qe));
  lo = __fmaf_rn(tl, __fmaf_rn(-0.5f, tl, __fmaf_rn(-th, __fmaf_rn(th, th, -th), -th)), lo);
  const Df w = two_sum(__fadd_rn(E.x, T.y), th);
  Anchored A{__fadd_rn(E.y, T.z), __fadd_rn(lo, __fadd_rn(E.z, T.w))};
  A.add(w.l);
  A.add(-0.5f * sq);
  A.add(__fmul_rn(__fmul_rn(sq, th), pol));
  A.add(pe);
  A.add(q);
  const Df s = quick_two_sum(w.h, __fadd_rn(A.s, -LOG_M));
  return {s.h, s.l, A.low};
}

}  // namespace rss
