// log_table.h -- the intervals' table of log_tf.cuh, made on the host: 1/c
// rounded to FP32 and -log of that in three parts, from the logarithm to about
// 2^-100 (a series in pairs of FP64 numbers), since FP64's own log would leave
// 2^-54.  The same bits on every host: additions, products and FMAs only.
#pragma once
#include <cmath>

namespace rss {

namespace log_table_detail {
struct Dd {
  double h, l;
};
inline Dd two_sum(double a, double b) {
  const double s = a + b, t = s - a;
  return {s, (a - (s - t)) + (b - t)};
}
inline Dd add(Dd a, Dd b) {
  const Dd s = two_sum(a.h, b.h);
  const double l = s.l + (a.l + b.l), h = s.h + l;
  return {h, l - (h - s.h)};
}
inline Dd mul(Dd a, Dd b) {
  const double p = a.h * b.h, e = std::fma(a.h, b.h, -p) + (a.h * b.l + a.l * b.h), h = p + e;
  return {h, e - (h - p)};
}
inline Dd div(Dd a, Dd b) {
  const double q = a.h / b.h;
  const Dd r = add(a, mul(Dd{-q, 0.0}, b));
  return add(Dd{q, 0.0}, Dd{(r.h + r.l) / b.h, 0.0});
}
// log x = 2 (z + z^3 / 3 + z^5 / 5 + ...), z = (x - 1) / (x + 1), for x in (1/2, 1]
inline Dd log(double x) {
  const Dd z = div(two_sum(x, -1.0), two_sum(x, 1.0)), z2 = mul(z, z);
  Dd s{0.0, 0.0};
  for (int k = 32; k >= 0; k--) s = add(mul(s, z2), div(Dd{1.0, 0.0}, Dd{2.0 * k + 1.0, 0.0}));
  s = mul(s, z);
  return {2.0 * s.h, 2.0 * s.l};
}
}  // namespace log_table_detail

// Entry i of `cells`: {1/c, the parts of -log(1/c)}, the second plus `anchor`.
inline void log_table_entry(int i, int cells, float anchor, float out[4]) {
  const float ic = (float)(2.0 * cells / (2.0 * cells + 2.0 * i + 1.0));
  const log_table_detail::Dd g = log_table_detail::log((double)ic);
  const double h = std::nearbyint(-g.h * 0x1p13) * 0x1p-13;
  const log_table_detail::Dd r = log_table_detail::add({-g.h - h, 0.0}, {-g.l, 0.0});
  const double m = std::nearbyint(r.h * 0x1p34) * 0x1p-34;
  out[0] = ic;
  out[1] = (float)h;
  out[2] = (float)(m + (double)anchor);
  out[3] = (float)((r.h - m) + r.l);
}

}  // namespace rss
