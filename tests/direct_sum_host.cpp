// The three-part arithmetic of the direct sum (tf.cuh, log_tf.cuh,
// log_table.h) compiled for the host, against the host's long double: prints
// one "name value" line a check, each the largest error seen in units of
// 2^-53.  rsqrtf is the correctly rounded one moved by up to two units in the
// last place, since the device's is approximate.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>

#define __device__
#define __forceinline__ inline
struct float2 {
  float x, y;
};
struct float4 {
  float x, y, z, w;
};
static inline float4 make_float4(float a, float b, float c, float d) { return {a, b, c, d}; }
static inline float __fadd_rn(float a, float b) { return a + b; }
static inline float __fmul_rn(float a, float b) { return a * b; }
static inline float __fmaf_rn(float a, float b, float c) { return fmaf(a, b, c); }
static inline unsigned __float_as_uint(float f) {
  unsigned u;
  memcpy(&u, &f, 4);
  return u;
}
static inline float __uint_as_float(unsigned u) {
  float f;
  memcpy(&f, &u, 4);
  return f;
}
static int g_ulps = 0;
static inline float rsqrtf(float x) {
  return __uint_as_float(__float_as_uint((float)(1.0 / std::sqrt((double)x))) + g_ulps);
}

#include "log_table.h"
#include "log_tf.cuh"

using namespace rss;
typedef long double Ld;

static uint64_t g_state = 1;
static uint64_t next() {  // splitmix64
  uint64_t z = g_state += 0x9e3779b97f4a7c15ull;
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}
static double uniform() { return (double)(next() >> 11) * 0x1p-53; }
static Ld value(Tf a) { return (Ld)a.h + a.m + a.l; }
static Tf split(double s) {
  const float h = (float)s, m = (float)(s - h);
  return {h, m, (float)(s - h - m)};
}
static void report(const char *name, Ld worst) { printf("%s %.6g\n", name, (double)(worst * 0x1p53L)); }

// coordinates below 2^40 in the parts of the direct sum
static void parts(double x, float *o) {
  const double h = std::rint(x * 0x1p-17) * 0x1p17, l = std::rint((x - h) * 0x1p7) * 0x1p-7;
  o[0] = (float)h, o[1] = (float)l, o[2] = (float)((x - h) - l);
}
template <int DIM> static Ld dist_error(double scale) {
  Ld worst = 0;
  for (int t = 0; t < 200000; t++) {
    float d[3 * DIM];
    Ld ref = 0;
    for (int i = 0; i < DIM; i++) {
      // one point anywhere, the other about `scale` of the box away
      const double a = 0x1p24 + uniform() * 0x1.8p39, b = std::fabs(a + (uniform() - 0.5) * scale * 0x1p40);
      float pa[3], pb[3];
      parts(a, pa), parts(b, pb);
      for (int p = 0; p < 3; p++) d[3 * i + p] = pa[p] - pb[p];
      ref += ((Ld)a - b) * ((Ld)a - b);
    }
    if (ref < 0x1p-20L) continue;
    worst = std::fmax(worst, fabsl(value(dist2_tf<DIM>(d)) / ref - 1));
  }
  return worst;
}

int main() {
  static float4 lt[LOG_CELLS], et[256];
  Ld worst = 0;
  for (int i = 0; i < LOG_CELLS; i++) {
    float o[4];
    log_table_entry(i, LOG_CELLS, LOG_M, o);
    lt[i] = {o[0], o[1], o[2], o[3]};
    worst = std::fmax(worst, fabsl((Ld)o[1] + ((Ld)o[2] - LOG_M) + o[3] + logl((Ld)o[0])));
  }
  report("table", worst);
  worst = 0;
  for (int shift = -1800; shift <= 1800; shift += 360)
    for (int i = 0; i < 256; i++) {
      const int k = i - 127 - shift;
      if (k <= -2048 || k >= 2048) continue;
      const float4 e = log_tables_exponent(k);
      const Ld ref = k * 0.693147180559945309417232121458176568L;
      worst = std::fmax(worst, fabsl((Ld)e.x + e.y + e.z - ref) / std::fmax((Ld)1, fabsl(ref)));
    }
  report("exponent", worst);
  for (int i = 0; i < 256; i++) et[i] = log_tables_exponent(i - 127);

  report("dist2", std::fmax(std::fmax(dist_error<2>(1.0), dist_error<2>(1e-4)), dist_error<2>(0x1p-37)));
  report("dist3", std::fmax(std::fmax(dist_error<3>(1.0), dist_error<3>(1e-4)), dist_error<3>(0x1p-37)));

  Ld wl = 0, wr = 0;
  for (int t = 0; t < 600000; t++) {
    // every exponent of a scaled r^2 and every table interval; near 1 in turn
    double x = (1.0 + uniform()) * std::ldexp(1.0, (int)(next() % 143) - 60);
    if (t & 1) x = 1.0 + (uniform() - 0.5) * 0x1p-6;
    const Tf s = split(x);
    const Ld ref = logl((Ld)x);
    wl = std::fmax(wl, fabsl(value(log_tf(s, lt, et)) - ref) / std::fmax((Ld)1, fabsl(ref)));
    g_ulps = (int)(next() % 5) - 2;
    wr = std::fmax(wr, fabsl(value(rsqrt_tf(s)) * sqrtl((Ld)x) - 1));
  }
  report("log", wl);
  report("rsqrt", wr);

  // sums of 256 products, against the sum of their magnitudes
  Ld wa = 0;
  for (int t = 0; t < 4000; t++) {
    Tf s{0.f, 0.f, 0.f};
    Ld ref = 0, mag = 0;
    const bool positive = t & 1;
    for (int i = 0; i < 256; i++) {
      const double a = (uniform() + 1e-3) * std::ldexp(1.0, (int)(next() % 8)), x = uniform() - (positive ? 0.0 : 0.5);
      add_mul_tf(s, split(a), split(x));
      ref += (Ld)a * x;
      mag += fabsl((Ld)a * x);
    }
    wa = std::fmax(wa, fabsl(value(s) - ref) / mag);
  }
  report("sum", wa);
  return 0;
}
