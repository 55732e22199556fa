// tf.cuh -- numbers as unevaluated sums of three FP32 numbers, for sums that
// have to be as accurate as FP64 ones.
//
// A pair (df.cuh) carries 48 bits; here the rounding errors of a pair's second
// part are kept as well, in a third part that plain FP32 arithmetic carries
// along, so a value is good to about 2^-56.  No divisions, no FP64: an FP64
// operation occupies this part's FP64 pipe for about 64 cycles a warp.
// Algorithms: T. J. Dekker, "A floating-point technique for extending the
// available precision" (1971), with exact products by FMA; sums of several
// small terms are split at a constant (Anchored) as in S. M. Rump, T. Ogita
// and S. Oishi, "Accurate floating-point summation" (2008).
#pragma once
#include "df.cuh"

namespace rss {

// h + m normalised, l of the size of m's rounding error or somewhat more
struct Tf {
  float h, m, l;
};

// A sum of terms that together stay below 2^(k-2): M = 1.5 2^k fixes a grid of
// 2^(k-23); the terms' multiples of it add up exactly in s, what is left over
// (below 2^(k-24) a term) in low.
struct Anchored {
  float s, low;
  __device__ __forceinline__ void add(float a) {
    const float t = __fadd_rn(s, a);
    low = __fadd_rn(low, __fadd_rn(a, -__fadd_rn(t, -s)));
    s = t;
  }
};

// Squared distance: d[3 i ..] are coordinate i's difference in three parts, the
// first two exact, each at least as large as the next or zero.
template <int DIM> __device__ __forceinline__ Tf dist2_tf(const float (&d)[3 * DIM]) {
  float p[DIM], e[DIM], q[DIM], w = 0.f;
#pragma unroll
  for (int i = 0; i < DIM; i++) {
    const Df t = quick_two_sum(d[3 * i], d[3 * i + 1]);
    const Df u = quick_two_sum(t.l, d[3 * i + 2]);
    const Df z = quick_two_sum(t.h, u.h);  // the difference is z.h + z.l + u.l
    const float g = __fadd_rn(z.h, z.h);
    p[i] = __fmul_rn(z.h, z.h);
    e[i] = __fmaf_rn(z.h, z.h, -p[i]);
    q[i] = __fmul_rn(g, z.l);
    const float r = __fmaf_rn(z.l, z.l, __fmaf_rn(g, u.l, __fmaf_rn(g, z.l, -q[i])));
    w = i == 0 ? r : __fadd_rn(w, r);
  }
  Df P = two_sum(p[0], p[1]);
  const float low01 = P.l;
  if (DIM == 3) P = two_sum(P.h, p[DIM - 1]);
  // the small terms are below 2^-21 P.h together: a grid of 2^-42 of P.h's power of two
  const float M = __uint_as_float(((__float_as_uint(P.h) & 0x7f800000u) - (19u << 23)) | 0x400000u);
  Anchored A{M, w};
  A.add(low01);
  if (DIM == 3) A.add(P.l);
#pragma unroll
  for (int i = 0; i < DIM; i++) {
    A.add(e[i]);
    A.add(q[i]);
  }
  const Df R = quick_two_sum(P.h, __fadd_rn(A.s, -M));
  return {R.h, R.l, A.low};
}

// 1 / sqrt(d): FP32 seed y, residual r = 1 - d y^2 (|r| < 2^-20) to about
// 2^-66, then y (1 + r / 2 + 3 r^2 / 8)
__device__ __forceinline__ Tf rsqrt_tf(Tf d) {
  const float y = rsqrtf(d.h);
  const float p = __fmul_rn(y, y), pe = __fmaf_rn(y, y, -p);
  const float P = __fmul_rn(d.h, p), Pe = __fmaf_rn(d.h, p, -P);
  const float g = __fmul_rn(d.h, pe), ge = __fmaf_rn(d.h, pe, -g);
  const float k = __fmul_rn(d.m, p), ke = __fmaf_rn(d.m, p, -k);
  constexpr float M = 0x1.8p-18f;
  Anchored A{__fadd_rn(M, __fadd_rn(1.f, -P)), 0.f};  // exact: 1 - P is a multiple of 2^-24
  A.add(-Pe);
  A.add(-g);
  A.add(-k);
  const float r = __fadd_rn(A.s, -M);
  const float low = __fadd_rn(A.low, -__fmaf_rn(d.m, pe, __fmaf_rn(d.l, p, __fadd_rn(ge, ke))));
  const float c = 0.5f * y, q = __fmul_rn(c, r);
  float v = __fmaf_rn(c, r, -q);
  v = __fmaf_rn(c, low, v);
  v = __fmaf_rn(__fmul_rn(0.75f * c, r), r, v);
  const Df s = quick_two_sum(y, q);
  return {s.h, s.l, v};
}

// s += a x.  Every rounding error of the terms of size 2^-24 goes into s.l.
__device__ __forceinline__ void add_mul_tf(Tf &s, Tf a, Tf x) {
  const float p = __fmul_rn(a.h, x.h), e = __fmaf_rn(a.h, x.h, -p);
  const float q = __fmul_rn(a.h, x.m), f = __fmaf_rn(a.h, x.m, -q);
  const float k = __fmul_rn(a.m, x.h), g = __fmaf_rn(a.m, x.h, -k);
  const float w = __fmaf_rn(a.m, x.m, __fmaf_rn(a.h, x.l, __fmaf_rn(a.l, x.h, __fadd_rn(f, g))));
  const Df r = two_sum(s.h, p);
  const Df b = two_sum(e, q);
  const Df c = two_sum(k, r.l);
  const Df t = two_sum(b.h, c.h);
  const Df u = two_sum(s.m, t.h);
  s.h = r.h;
  s.m = u.h;
  s.l = __fadd_rn(s.l, __fadd_rn(w, __fadd_rn(__fadd_rn(b.l, c.l), __fadd_rn(t.l, u.l))));
}

}  // namespace rss
