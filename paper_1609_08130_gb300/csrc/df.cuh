// df.cuh -- numbers as unevaluated sums of two FP32 numbers (48 bits).
//
// An FP64 operation occupies this part's FP64 pipe for about 64 cycles per
// warp (2.15 per clock and SM measured); a pair operation is 3 to 13 FP32
// instructions at 128 per clock and SM.  Algorithms: Dekker, "A floating-point
// technique for extending the available precision" (1971); exact products by
// FMA.  The _rn intrinsics keep the compiler from contracting or reassociating
// them.
#pragma once
#ifdef __CUDACC__
#include <cuda_runtime.h>
#endif

namespace rss {

struct Df {
  float h, l;
};
__device__ __forceinline__ Df two_sum(float a, float b) {
  const float s = __fadd_rn(a, b), bb = __fadd_rn(s, -a);
  return {s, __fadd_rn(__fadd_rn(a, -__fadd_rn(s, -bb)), __fadd_rn(b, -bb))};
}
// |a| >= |b| or a == 0
__device__ __forceinline__ Df quick_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  return {s, __fadd_rn(b, -__fadd_rn(s, -a))};
}
__device__ __forceinline__ Df mul(Df a, Df b) {
  const float p = __fmul_rn(a.h, b.h);
  float e = __fmaf_rn(a.h, b.h, -p);
  e = __fmaf_rn(a.h, b.l, e);
  e = __fmaf_rn(a.l, b.h, e);
  return quick_two_sum(p, e);
}
// s + a b, the low part left unnormalised
__device__ __forceinline__ Df add_mul(Df s, Df a, Df b) {
  const float p = __fmul_rn(a.h, b.h);
  float e = __fmaf_rn(a.h, b.h, -p);
  e = __fmaf_rn(a.h, b.l, e);
  e = __fmaf_rn(a.l, b.h, e);
  const Df t = two_sum(s.h, p);
  return {t.h, __fadd_rn(s.l, __fadd_rn(t.l, e))};
}
__device__ __forceinline__ Df sub_mul(Df s, Df a, Df b) { return add_mul(s, Df{-a.h, -a.l}, b); }
__device__ __forceinline__ Df add(Df a, Df b) {
  const Df t = two_sum(a.h, b.h);
  return quick_two_sum(t.h, __fadd_rn(t.l, __fadd_rn(a.l, b.l)));
}
// 1 / sqrt(d): FP32 seed y, residual r = 1 - d y^2 as a pair, then
// y (1 + r / 2 + 3 r^2 / 8)
__device__ __forceinline__ Df rsqrt_df(Df d) {
  const float y = rsqrtf(d.h);
  const float p = __fmul_rn(y, y);
  const Df t = mul(d, {p, __fmaf_rn(y, y, -p)});
  const Df r = quick_two_sum(__fadd_rn(1.f, -t.h), -t.l);
  const float c = 0.5f * y, q = __fmul_rn(c, r.h);
  float e = __fmaf_rn(c, r.h, -q);
  e = __fmaf_rn(c, r.l, e);
  e = __fmaf_rn(0.75f * c, r.h * r.h, e);
  const Df s = quick_two_sum(y, q);
  return quick_two_sum(s.h, __fadd_rn(s.l, e));
}

}  // namespace rss
