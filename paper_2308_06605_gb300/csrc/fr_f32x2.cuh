// Pairs of FP32 and double-float values with the packed FP32 instructions of sm_100 and later: one
// instruction, two lanes.
//
// A packed instruction does no more FMAs per cycle than two scalar ones (a dependent double-float sum runs
// at 32.8 against 30.7 T operations/s, plain FMA chains at 37 both ways), but takes one issue slot instead
// of two, and the double-float volume kernels are bound by issue (76 % of the slots, FP32 pipe 59 %).
#pragma once

#include <cuda_runtime.h>

#include "df32.cuh"

namespace frx {

struct f2 {
  float2 v;
};
__device__ __forceinline__ f2 mkf2(float x, float y) { return f2{make_float2(x, y)}; }
__device__ __forceinline__ f2 dupf(float x) { return mkf2(x, x); }
__device__ __forceinline__ f2 operator-(f2 a) { return mkf2(-a.v.x, -a.v.y); }
__device__ __forceinline__ f2 padd(f2 a, f2 b) { return f2{__fadd2_rn(a.v, b.v)}; }
__device__ __forceinline__ f2 pmul(f2 a, f2 b) { return f2{__fmul2_rn(a.v, b.v)}; }
__device__ __forceinline__ f2 pfma(f2 a, f2 b, f2 c) { return f2{__ffma2_rn(a.v, b.v, c.v)}; }
__device__ __forceinline__ f2 psub(f2 a, f2 b) { return pfma(b, dupf(-1.f), a); }
__device__ __forceinline__ f2 pabs(f2 a) { return mkf2(::fabsf(a.v.x), ::fabsf(a.v.y)); }

__device__ __forceinline__ f2 operator+(f2 a, f2 b) { return padd(a, b); }
__device__ __forceinline__ f2 operator-(f2 a, f2 b) { return psub(a, b); }
__device__ __forceinline__ f2 operator*(f2 a, f2 b) { return pmul(a, b); }
__device__ __forceinline__ f2 muladd(f2 c, f2 a, f2 b) { return pfma(a, b, c); }
__device__ __forceinline__ f2 scale2(f2 x, float f) { return pmul(x, dupf(f)); }
__device__ __forceinline__ f2 reciprocal(f2 x) { return mkf2(1.f / x.v.x, 1.f / x.v.y); }
__device__ __forceinline__ f2 dot3(f2 a0, f2 b0, f2 a1, f2 b1, f2 a2, f2 b2) {
  return pfma(a2, b2, pfma(a1, b1, pmul(a0, b0)));
}

struct __align__(16) d2 {      // one 16-byte shared-memory access
  f2 hi, lo;
};
__device__ __forceinline__ d2 mkd2(f2 hi, f2 lo) { return d2{hi, lo}; }
__device__ __forceinline__ d2 dup(df32 x) { return d2{dupf(x.hi), dupf(x.lo)}; }
__device__ __forceinline__ d2 pack(df32 a, df32 b) { return d2{mkf2(a.hi, b.hi), mkf2(a.lo, b.lo)}; }
__device__ __forceinline__ df32 lane0(d2 x) { return df(x.hi.v.x, x.lo.v.x); }
__device__ __forceinline__ df32 lane1(d2 x) { return df(x.hi.v.y, x.lo.v.y); }

// The same error-free transformations as the scalar ones, lane by lane.
__device__ __forceinline__ d2 fast_two_sum(f2 a, f2 b) {
  const f2 s = padd(a, b);
  return d2{s, psub(b, psub(s, a))};
}
__device__ __forceinline__ d2 two_sum(f2 a, f2 b) {
  const f2 s = padd(a, b), bb = psub(s, a);
  return d2{s, padd(psub(a, psub(s, bb)), psub(b, bb))};
}
// a b - p, and the cross terms, on top of it.
__device__ __forceinline__ f2 perr(d2 a, d2 b, f2 p) {
  return pfma(a.lo, b.hi, pfma(a.hi, b.lo, pfma(a.hi, b.hi, -p)));
}
__device__ __forceinline__ d2 operator-(d2 x) { return d2{-x.hi, -x.lo}; }
__device__ __forceinline__ d2 operator+(d2 x, d2 y) {
  const d2 s = two_sum(x.hi, y.hi);
  return fast_two_sum(s.hi, padd(s.lo, padd(x.lo, y.lo)));
}
__device__ __forceinline__ d2 operator-(d2 x, d2 y) { return x + (-y); }
__device__ __forceinline__ d2 operator*(d2 x, d2 y) {
  const f2 p = pmul(x.hi, y.hi);
  return fast_two_sum(p, perr(x, y, p));
}
__device__ __forceinline__ d2 muladd(d2 c, d2 a, d2 b) {
  const f2 p = pmul(a.hi, b.hi);
  const d2 s = two_sum(c.hi, p);
  return fast_two_sum(s.hi, padd(s.lo, padd(c.lo, perr(a, b, p))));
}
__device__ __forceinline__ d2 scale2(d2 x, float f) { return d2{scale2(x.hi, f), scale2(x.lo, f)}; }
__device__ __forceinline__ d2 scale2(d2 x, f2 f) { return d2{pmul(x.hi, f), pmul(x.lo, f)}; }
__device__ __forceinline__ d2 dot3(d2 a0, d2 b0, d2 a1, d2 b1, d2 a2, d2 b2) {
  const f2 p0 = pmul(a0.hi, b0.hi), p1 = pmul(a1.hi, b1.hi), p2 = pmul(a2.hi, b2.hi);
  const f2 e0 = perr(a0, b0, p0), e1 = perr(a1, b1, p1), e2 = perr(a2, b2, p2);
  const d2 s = two_sum(p0, p1), t = two_sum(s.hi, p2);
  return fast_two_sum(t.hi, padd(padd(padd(e0, e1), padd(e2, s.lo)), t.lo));
}
__device__ __forceinline__ d2 reciprocal(d2 x) {
  const f2 y = mkf2(rcp_newton(x.hi.v.x), rcp_newton(x.hi.v.y));
  const f2 e = pfma(-x.lo, y, pfma(-x.hi, y, dupf(1.f)));
  return fast_two_sum(y, pmul(y, pfma(e, e, e)));
}

template <> struct Dot<f2> {
  f2 s;
  __device__ __forceinline__ Dot() : s(dupf(0.f)) {}
  __device__ __forceinline__ explicit Dot(f2 x) : s(x) {}
  __device__ __forceinline__ Dot(f2 c, f2 x) : s(pmul(c, x)) {}
  __device__ __forceinline__ void add(f2 c, f2 x) { s = pfma(c, x, s); }
  __device__ __forceinline__ f2 raw() const { return s; }
};
template <> struct Dot<d2> {
  f2 s, e;
  __device__ __forceinline__ Dot() : s(dupf(0.f)), e(dupf(0.f)) {}
  __device__ __forceinline__ explicit Dot(d2 x) : s(x.hi), e(x.lo) {}
  __device__ __forceinline__ Dot(d2 c, d2 x) {
    s = pmul(c.hi, x.hi);
    e = perr(c, x, s);
  }
  __device__ __forceinline__ void add(d2 c, d2 x) {
    const f2 p = pmul(c.hi, x.hi), err = perr(c, x, p);
    const d2 t = two_sum(s, p);
    s = t.hi;
    e = padd(e, padd(t.lo, err));
  }
  __device__ __forceinline__ void plus(d2 x) {
    const d2 t = two_sum(s, x.hi);
    s = t.hi;
    e = padd(e, padd(t.lo, x.lo));
  }
  __device__ __forceinline__ d2 raw() const { return fast_two_sum(s, e); }
};

}  // namespace frx
