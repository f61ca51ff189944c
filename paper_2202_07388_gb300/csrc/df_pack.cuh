// Double-float arithmetic on two lanes: every binary32 operation of the
// double-float formulas (oq_device.cuh) as one packed two-lane instruction
// (FADD2 / FMUL2 / FFMA2 of sm_100-class GPUs), in the same order, so each
// lane's result is bit for bit the scalar one.  A packed instruction occupies
// the binary32 pipe as long as two scalar ones; it halves the issue slots and
// the parallelism that hides the latency of the dependent chains (measured: 4
// warps per SM with 4 independent chains reach 100 of 128 lane operations per
// clock packed, 16 warps are needed scalar).
#pragma once
#include "oq_device.cuh"

namespace oq {
namespace df2 {

typedef float2 F2;
__device__ __forceinline__ F2 bc(float a) { return make_float2(a, a); }
__device__ __forceinline__ F2 add(F2 a, F2 b) { return __fadd2_rn(a, b); }
// RN(a - b): the product b * (-1) is exact, so one rounding as in a subtraction
__device__ __forceinline__ F2 sub(F2 a, F2 b) { return __ffma2_rn(b, bc(-1.f), a); }
__device__ __forceinline__ F2 mul(F2 a, F2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ F2 neg(F2 a) { return make_float2(-a.x, -a.y); }

// lane k (k = 0, 1) holds hi.k + lo.k
struct D2 {
  F2 hi, lo;
};
struct C2 {
  D2 re, im;
};
__device__ __forceinline__ D2 dneg(D2 x) { return D2{neg(x.hi), neg(x.lo)}; }
__device__ __forceinline__ C2 cneg(C2 z) { return C2{dneg(z.re), dneg(z.im)}; }

// the error-free transformations and double-float operations of
// oq_device.cuh, lane by lane
__device__ __forceinline__ D2 two_sum(F2 a, F2 b) {
  const F2 s = add(a, b);
  const F2 bb = sub(s, a);
  return D2{s, add(sub(a, sub(s, bb)), sub(b, bb))};
}
__device__ __forceinline__ D2 fast_two_sum(F2 a, F2 b) {
  const F2 s = add(a, b);
  return D2{s, sub(b, sub(s, a))};
}
__device__ __forceinline__ D2 dadd(D2 x, D2 y) {
  const D2 s = two_sum(x.hi, y.hi);
  return fast_two_sum(s.hi, add(s.lo, add(x.lo, y.lo)));
}
// x + y without the final renormalisation: the two-sum of the high parts
// and the low parts added to its error (8 operations instead of dadd's 11).
// The low part may exceed ulp(hi)/2 by a few ulp; a product or another lazy sum
// takes such a value as it is, and dnorm restores the normal form.
__device__ __forceinline__ D2 add_lazy(D2 x, D2 y) {
  const D2 s = two_sum(x.hi, y.hi);
  return D2{s.hi, add(s.lo, add(x.lo, y.lo))};
}
__device__ __forceinline__ D2 dnorm(D2 x) { return fast_two_sum(x.hi, x.lo); }
// x * 2^k for a power of two s = 2^k: exact, both parts scaled
__device__ __forceinline__ D2 dscale(D2 x, float s) { return D2{mul(x.hi, bc(s)), mul(x.lo, bc(s))}; }
// a * b + c (both factors per lane)
__device__ __forceinline__ D2 dfma(D2 a, D2 b, D2 c) {
  const F2 p = mul(a.hi, b.hi);
  F2 e = fma2(a.hi, b.hi, neg(p));
  e = fma2(a.hi, b.lo, e);
  e = fma2(a.lo, b.hi, e);
  const D2 s = two_sum(c.hi, p);
  return fast_two_sum(s.hi, add(s.lo, add(c.lo, e)));
}

// A dot product accumulated lazily: s is the running sum of the high products (each
// added by a two-sum), e collects the two-sum errors and the low parts; one
// renormalisation at the end.  One factor is shared by the two lanes.
struct Acc {
  F2 s, e;
};
__device__ __forceinline__ void acc_first(Acc& a, dfloat x, D2 y) {
  const F2 xh = bc(x.hi), xl = bc(x.lo);
  a.s = mul(xh, y.hi);
  F2 e = fma2(xh, y.hi, neg(a.s));
  e = fma2(xh, y.lo, e);
  a.e = fma2(xl, y.hi, e);
}
__device__ __forceinline__ void acc_add(Acc& a, dfloat x, D2 y) {
  const F2 xh = bc(x.hi), xl = bc(x.lo);
  const F2 p = mul(xh, y.hi);
  F2 e = fma2(xh, y.hi, neg(p));
  e = fma2(xh, y.lo, e);
  e = fma2(xl, y.hi, e);
  const D2 t = two_sum(a.s, p);
  a.s = t.hi;
  a.e = add(a.e, add(t.lo, e));
}
__device__ __forceinline__ D2 acc_get(const Acc& a) { return fast_two_sum(a.s, a.e); }

// z * i^c for c in 0..3: a swap of the parts for odd c and sign flips, all by selects
__device__ __forceinline__ C2 rot_ic(const C2& z, int c) {
  const bool sw = c & 1;
  D2 re = sw ? z.im : z.re, im = sw ? z.re : z.im;
  if (c == 1 || c == 2) re = dneg(re);
  if (c >= 2) im = dneg(im);
  return C2{re, im};
}
// acc_first, acc_add with both factors per lane
__device__ __forceinline__ void acc_first(Acc& a, D2 x, D2 y) {
  a.s = mul(x.hi, y.hi);
  F2 e = fma2(x.hi, y.hi, neg(a.s));
  e = fma2(x.hi, y.lo, e);
  a.e = fma2(x.lo, y.hi, e);
}
__device__ __forceinline__ void acc_add(Acc& a, D2 x, D2 y) {
  const F2 p = mul(x.hi, y.hi);
  F2 e = fma2(x.hi, y.hi, neg(p));
  e = fma2(x.hi, y.lo, e);
  e = fma2(x.lo, y.hi, e);
  const D2 t = two_sum(a.s, p);
  a.s = t.hi;
  a.e = add(a.e, add(t.lo, e));
}
// both parts times an exact per-lane factor (+-1)
__device__ __forceinline__ D2 dsign(D2 x, F2 s) { return D2{mul(x.hi, s), mul(x.lo, s)}; }

}  // namespace df2
}  // namespace oq
