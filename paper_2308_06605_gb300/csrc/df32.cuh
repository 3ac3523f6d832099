// df32: a value represented as the unevaluated sum hi + lo of two FP32 numbers (|lo| <= ulp(hi)/2),
// about 48 significant bits, computed entirely on the FP32 pipe.
//
// Error-free transformations used (published methods):
//   two_sum      Knuth, TAOCP vol. 2, 4.2.2: s = fl(a + b) and the exact rounding error e.
//   fast_two_sum Dekker 1971 ("A floating-point technique for extending the available
//                precision"), valid for |a| >= |b|.
//   two_prod     exact product error with one fused multiply-add: e = fma(a, b, -fl(a b)).
// Double-word addition, multiplication, division and square root follow the "sloppy" variants
// of Hida, Li & Bailey (2001, "Algorithms for quad-double precision floating point
// arithmetic"): relative error of a few 2^-44 with respect to the operands' magnitudes, which is
// the scale every tolerance of this library is stated against.
// Plain products use __fmul_rn/__fadd_rn so the compiler cannot contract them into FMAs, which
// would break the error-free transformations.
#pragma once

#include <cuda_runtime.h>

#include <cmath>

namespace frx {

using ::sqrt;   // keep the double overload visible next to sqrt(df32)

struct df32 {
  float hi, lo;
};

__host__ __device__ __forceinline__ df32 df(float hi, float lo) {
  df32 r;
  r.hi = hi;
  r.lo = lo;
  return r;
}

// Host-side split of a double into hi + lo (for uploading operators and geometry).
inline df32 df_split_host(double d) {
  const float hi = (float)d;
  return df(hi, (float)(d - (double)hi));
}

__device__ __forceinline__ df32 df_from(double d) {
  const float hi = __double2float_rn(d);
  return df(hi, __double2float_rn(d - (double)hi));
}

__device__ __forceinline__ df32 fast_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  return df(s, __fadd_rn(b, __fsub_rn(a, s)));
}

__device__ __forceinline__ df32 two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return df(s, e);
}

// FP32 to FP64 is exact, and the conversion instruction occupies the FP64 pipe (one warp instruction in 64 cycles per
// scheduler), so normal numbers are converted on the integer pipe: the mantissa is shifted and the
// exponent rebiased, same bits.  Zeros, subnormals, infinities and NaN take the instruction, behind a real branch (as
// a select the compiler issues the conversions always).  Correction at 48^3 p = 4 0.810 -> 0.757 ms per launch,
// interface fluxes of inviscid double-float 40^3 p = 3 0.164 -> 0.126, with the Roe flux 0.195 -> 0.174 (15^3 channel,
// p = 5); viscous Rusanov, bound by FP32 issue, 0.682 -> 0.691.  The same for FP64 to FP32 in df_from gained 4 % in
// the last RK44 stage and lost 7 % in the SSP stages: not done.
__device__ __forceinline__ bool is_normal(float x) { return (__float_as_uint(x) << 1) - 0x01000000u < 0xfe000000u; }
__device__ __forceinline__ double widen_normal(float x) {
  const int b = __float_as_int(x);
  return __hiloint2double(((b >> 3) & 0x8fffffff) + 0x38000000, b << 29);
}
__device__ __forceinline__ double to_double(df32 x) {
  if (is_normal(x.hi) && is_normal(x.lo)) return widen_normal(x.hi) + widen_normal(x.lo);
  return (double)x.hi + (double)x.lo;
}
__device__ __forceinline__ double to_double(double x) { return x; }

__device__ __forceinline__ df32 operator+(df32 x, df32 y) {
  df32 s = two_sum(x.hi, y.hi);
  const float e = __fadd_rn(s.lo, __fadd_rn(x.lo, y.lo));
  return fast_two_sum(s.hi, e);
}

__device__ __forceinline__ df32 operator-(df32 x) { return df(-x.hi, -x.lo); }
__device__ __forceinline__ df32 operator-(df32 x, df32 y) { return x + (-y); }

__device__ __forceinline__ df32 operator*(df32 x, df32 y) {
  const float p = __fmul_rn(x.hi, y.hi);
  float e = __fmaf_rn(x.hi, y.hi, -p);
  e = __fmaf_rn(x.hi, y.lo, e);
  e = __fmaf_rn(x.lo, y.hi, e);
  return fast_two_sum(p, e);
}

__device__ __forceinline__ df32 operator/(df32 x, df32 y) {
  const float q1 = __fdiv_rn(x.hi, y.hi);
  const df32 r = x - y * df(q1, 0.f);
  const float q2 = __fdiv_rn(r.hi, y.hi);
  return fast_two_sum(q1, q2);
}

__device__ __forceinline__ df32 &operator+=(df32 &x, df32 y) { return x = x + y; }
__device__ __forceinline__ df32 &operator-=(df32 &x, df32 y) { return x = x - y; }
__device__ __forceinline__ df32 &operator*=(df32 &x, df32 y) { return x = x * y; }

// 1/x by Newton-Raphson iteration from the hardware's approximation: y (FP32, one step), then the
// correction y (e + e^2) with e = 1 - x y taken from both parts of x.  10 FP32 instructions and no branch
// (the quotient above: two IEEE divisions with their slow paths).  |e| < 2^-23, so the four roundings of the
// correction (two in e, the sum e + e^2, the product with y) are 2^-48 of 1/x at most each: relative error below
// 2^-46.  1/0 and 1/inf come out as NaN.
__device__ __forceinline__ float rcp_newton(float x) {
  float y;
  asm("rcp.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return __fmaf_rn(y, __fmaf_rn(-x, y, 1.f), y);
}
__device__ __forceinline__ df32 reciprocal(df32 x) {
  const float y = rcp_newton(x.hi);
  const float e = __fmaf_rn(-x.lo, y, __fmaf_rn(-x.hi, y, 1.f));
  return fast_two_sum(y, __fmul_rn(y, __fmaf_rn(e, e, e)));
}
__device__ __forceinline__ double reciprocal(double x) { return 1.0 / x; }
__device__ __forceinline__ float reciprocal(float x) { return 1.f / x; }

__device__ __forceinline__ df32 sqrt(df32 x) {
  if (x.hi <= 0.f) return df(0.f, 0.f);
  const float s = __fsqrt_rn(x.hi);
  const float r = __fadd_rn(__fmaf_rn(-s, s, x.hi), x.lo);
  return fast_two_sum(s, __fmul_rn(r, rcp_newton(__fmul_rn(2.f, s))));
}

// Sum of products sum_i c_i x_i.  For double: FMAs.  For df32: the leading parts are summed with
// two_sum and every rounding error (of the products via two_prod and the cross terms, and of the
// sums) is collected in one FP32 error term, normalised once by get() -- the usual compensated
// dot product (Ogita, Rump & Oishi 2005, "Accurate sum and dot product"), 12 FP32 instructions
// per term instead of 18 for a double-float multiply followed by an add.
template <typename T> struct Dot;

template <> struct Dot<double> {
  double s;
  __device__ __forceinline__ Dot() : s(0.0) {}
  __device__ __forceinline__ Dot(double c, double x) : s(c * x) {}
  __device__ __forceinline__ explicit Dot(double x) : s(x) {}
  __device__ __forceinline__ void add(double c, double x) { s = fma(c, x, s); }
  __device__ __forceinline__ void plus(double x) { s += x; }
  __device__ __forceinline__ void join(const Dot &o) { s += o.s; }
  __device__ __forceinline__ double get() const { return s; }
  __device__ __forceinline__ double raw() const { return s; }
};

template <> struct Dot<float> {
  float s;
  __device__ __forceinline__ Dot() : s(0.f) {}
  __device__ __forceinline__ Dot(float c, float x) : s(c * x) {}
  __device__ __forceinline__ explicit Dot(float x) : s(x) {}
  __device__ __forceinline__ void add(float c, float x) { s = fmaf(c, x, s); }
  __device__ __forceinline__ void plus(float x) { s += x; }
  __device__ __forceinline__ float get() const { return s; }
  __device__ __forceinline__ float raw() const { return s; }
};

template <> struct Dot<df32> {
  float s, e;
  __device__ __forceinline__ Dot() : s(0.f), e(0.f) {}
  __device__ __forceinline__ explicit Dot(df32 x) : s(x.hi), e(x.lo) {}
  // The first term by itself: 4 instructions instead of 12.
  __device__ __forceinline__ Dot(df32 c, df32 x) {
    s = __fmul_rn(c.hi, x.hi);
    e = __fmaf_rn(c.lo, x.hi, __fmaf_rn(c.hi, x.lo, __fmaf_rn(c.hi, x.hi, -s)));
  }
  __device__ __forceinline__ void add(df32 c, df32 x) {
    const float p = __fmul_rn(c.hi, x.hi);
    float err = __fmaf_rn(c.hi, x.hi, -p);
    err = __fmaf_rn(c.hi, x.lo, err);
    err = __fmaf_rn(c.lo, x.hi, err);
    const float t = __fadd_rn(s, p);
    const float bb = __fsub_rn(t, s);
    const float r = __fadd_rn(__fsub_rn(s, __fsub_rn(t, bb)), __fsub_rn(p, bb));
    s = t;
    e = __fadd_rn(e, __fadd_rn(r, err));
  }
  __device__ __forceinline__ void plus(df32 x) {
    const df32 t = two_sum(s, x.hi);
    s = t.hi;
    e = __fadd_rn(e, __fadd_rn(t.lo, x.lo));
  }
  // Another sum on top of this one (8 instructions).
  __device__ __forceinline__ void join(const Dot &o) {
    const df32 t = two_sum(s, o.s);
    s = t.hi;
    e = __fadd_rn(e, __fadd_rn(t.lo, o.e));
  }
  __device__ __forceinline__ df32 get() const {
    const df32 r = two_sum(s, e);
    return fast_two_sum(r.hi, r.lo);
  }
  // The same value s + e with one fast_two_sum: normalised when |s| >= |e|; under cancellation
  // (|e| > |s|) an unevaluated pair whose sum is the dot product to the same absolute error.
  __device__ __forceinline__ df32 raw() const { return fast_two_sum(s, e); }
};

// a0 b0 + a1 b1 + a2 b2.  df32: the leading products by two two_sums, every error in one term
// (31 FP32 instructions; three Dot terms started from zero take 39).
__device__ __forceinline__ double dot3(double a0, double b0, double a1, double b1, double a2, double b2) {
  return fma(a2, b2, fma(a1, b1, a0 * b0));
}
__device__ __forceinline__ float dot3(float a0, float b0, float a1, float b1, float a2, float b2) {
  return fmaf(a2, b2, fmaf(a1, b1, a0 * b0));
}
__device__ __forceinline__ df32 dot3(df32 a0, df32 b0, df32 a1, df32 b1, df32 a2, df32 b2) {
  const float p0 = __fmul_rn(a0.hi, b0.hi), p1 = __fmul_rn(a1.hi, b1.hi), p2 = __fmul_rn(a2.hi, b2.hi);
  const float e0 = __fmaf_rn(a0.lo, b0.hi, __fmaf_rn(a0.hi, b0.lo, __fmaf_rn(a0.hi, b0.hi, -p0)));
  const float e1 = __fmaf_rn(a1.lo, b1.hi, __fmaf_rn(a1.hi, b1.lo, __fmaf_rn(a1.hi, b1.hi, -p1)));
  const float e2 = __fmaf_rn(a2.lo, b2.hi, __fmaf_rn(a2.hi, b2.lo, __fmaf_rn(a2.hi, b2.hi, -p2)));
  const df32 s = two_sum(p0, p1), t = two_sum(s.hi, p2);
  return fast_two_sum(t.hi, __fadd_rn(__fadd_rn(__fadd_rn(e0, e1), __fadd_rn(e2, s.lo)), t.lo));
}

// c + a b (df32: 15 FP32 instructions, against 18 for the product and the sum by themselves).
__device__ __forceinline__ double muladd(double c, double a, double b) { return fma(a, b, c); }
__device__ __forceinline__ float muladd(float c, float a, float b) { return fmaf(a, b, c); }
__device__ __forceinline__ df32 muladd(df32 c, df32 a, df32 b) {
  const float p = __fmul_rn(a.hi, b.hi);
  const float e = __fmaf_rn(a.lo, b.hi, __fmaf_rn(a.hi, b.lo, __fmaf_rn(a.hi, b.hi, -p)));
  const df32 s = two_sum(c.hi, p);
  return fast_two_sum(s.hi, __fadd_rn(s.lo, __fadd_rn(c.lo, e)));
}

// x times a power of two (exact).
__device__ __forceinline__ double scale2(double x, float f) { return x * (double)f; }
__device__ __forceinline__ float scale2(float x, float f) { return x * f; }
__device__ __forceinline__ df32 scale2(df32 x, float f) { return df(__fmul_rn(x.hi, f), __fmul_rn(x.lo, f)); }

__device__ __forceinline__ df32 fabs(df32 x) { return x.hi < 0.f ? -x : x; }
__device__ __forceinline__ bool operator<(df32 x, df32 y) { return x.hi < y.hi || (x.hi == y.hi && x.lo < y.lo); }
__device__ __forceinline__ df32 fmax(df32 x, df32 y) { return x < y ? y : x; }
using ::fabs;
using ::fmax;

// Scalar-type helpers so templated kernels read the same for double and df32.
template <typename T> __device__ __forceinline__ T from_double(double d);
template <> __device__ __forceinline__ double from_double<double>(double d) { return d; }
template <> __device__ __forceinline__ df32 from_double<df32>(double d) { return df_from(d); }
template <> __device__ __forceinline__ float from_double<float>(double d) { return __double2float_rn(d); }

// Arithmetic of the viscous branch (gradients, gradient traces, stress and heat flux): the element
// arithmetic T, or, with FP32_VISCOUS on the double-float path (FR_PREC_MIXED_VF32), plain FP32.
// These terms are scaled by the viscosity, so their FP32 rounding enters the residual in
// proportion to 1/Re (the gradients are taken of the perturbation from the element's first point,
// so large state values do not cancel in FP32).
template <typename T, bool FP32_VISCOUS> struct GradOf { using type = T; };
template <> struct GradOf<df32, true> { using type = float; };
template <typename TG> __device__ __forceinline__ TG to_g(double x);
template <> __device__ __forceinline__ double to_g<double>(double x) { return x; }
template <typename TG> __device__ __forceinline__ TG to_g(df32 x);
template <> __device__ __forceinline__ float to_g<float>(df32 x) { return __fadd_rn(x.hi, x.lo); }
template <> __device__ __forceinline__ df32 to_g<df32>(df32 x) { return x; }
template <typename T> __device__ __forceinline__ T from_g(double x);
template <> __device__ __forceinline__ double from_g<double>(double x) { return x; }
template <typename T> __device__ __forceinline__ T from_g(float x);
template <> __device__ __forceinline__ df32 from_g<df32>(float x) { return df(x, 0.f); }
template <typename T> __device__ __forceinline__ T from_g(df32 x);
template <> __device__ __forceinline__ df32 from_g<df32>(df32 x) { return x; }

}  // namespace frx
