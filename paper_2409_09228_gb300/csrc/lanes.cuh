// Lane types for the fused kernel: float (one track per thread), F2 (two
// tracks per thread, held in the two halves of a float2), F1 (one track,
// rounded as in a pair), and double (the
// FP64 variant, one track per thread).
//
// The per-track math is written once as templates over the lane type.  With
// F2 every add, multiply and fused multiply-add is one packed sm_100+
// instruction (__fadd2_rn / __fmul2_rn / __ffma2_rn, each component rounded
// exactly like the scalar operation), so one issue slot carries the FP32 work
// of two tracks; loads and stores become 64-bit.  Operations without a packed
// form (reciprocal, rsqrt, comparisons) run per component.  Comparisons give
// masks (bool or M2) that all()/any()/sel() consume.
#pragma once

#include <cuda_runtime.h>

namespace fitk {

struct F2 {
  float2 v;
  __device__ __forceinline__ F2() {}
  __device__ __forceinline__ F2(float a) : v(make_float2(a, a)) {}  // broadcast
  __device__ __forceinline__ F2(float a, float b) : v(make_float2(a, b)) {}
  __device__ __forceinline__ explicit F2(float2 a) : v(a) {}
};

struct M2 {
  bool x, y;
};

// One track whose every operation rounds as a lane of F2's does: no product
// is contracted with a sum that the code does not write as fma (a float's
// are).  For calls too small to fill the SMs with pairs of tracks, with the
// pairs' results.
struct F1 {
  float v;
  __device__ __forceinline__ F1() {}
  __device__ __forceinline__ F1(float a) : v(a) {}
};

// ---- arithmetic ----------------------------------------------------------
__device__ __forceinline__ F2 operator+(F2 a, F2 b) { return F2(__fadd2_rn(a.v, b.v)); }
__device__ __forceinline__ F2 operator-(F2 a) { return F2(-a.v.x, -a.v.y); }
__device__ __forceinline__ F2 operator-(F2 a, F2 b) { return F2(__fadd2_rn(a.v, (-b).v)); }
__device__ __forceinline__ F2 operator*(F2 a, F2 b) { return F2(__fmul2_rn(a.v, b.v)); }
__device__ __forceinline__ F2& operator+=(F2& a, F2 b) { return a = a + b; }
__device__ __forceinline__ F2& operator-=(F2& a, F2 b) { return a = a - b; }
__device__ __forceinline__ F2& operator*=(F2& a, F2 b) { return a = a * b; }

__device__ __forceinline__ F1 operator+(F1 a, F1 b) { return F1(__fadd_rn(a.v, b.v)); }
__device__ __forceinline__ F1 operator-(F1 a) { return F1(-a.v); }
__device__ __forceinline__ F1 operator-(F1 a, F1 b) { return F1(__fadd_rn(a.v, -b.v)); }
__device__ __forceinline__ F1 operator*(F1 a, F1 b) { return F1(__fmul_rn(a.v, b.v)); }
__device__ __forceinline__ F1& operator+=(F1& a, F1 b) { return a = a + b; }

__device__ __forceinline__ float fma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ F1 fma(F1 a, F1 b, F1 c) { return F1(__fmaf_rn(a.v, b.v, c.v)); }
__device__ __forceinline__ F2 fma(F2 a, F2 b, F2 c) { return F2(__ffma2_rn(a.v, b.v, c.v)); }

// Division and square root where a couple of ulp are far below the fit's
// tolerance: the approximate reciprocal, square root and rsqrt (MUFU) instead
// of the IEEE sequences.
__device__ __forceinline__ float frcp(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ F1 frcp(F1 x) { return F1(frcp(x.v)); }
__device__ __forceinline__ F2 frcp(F2 x) { return F2(frcp(x.v.x), frcp(x.v.y)); }
__device__ __forceinline__ float fdiv(float a, float b) { return __fdividef(a, b); }
// a * (1/b): the reciprocals per lane, the product packed
__device__ __forceinline__ F1 fdiv(F1 a, F1 b) { return a * frcp(b); }
__device__ __forceinline__ F2 fdiv(F2 a, F2 b) { return a * frcp(b); }
// Approximate square root and reciprocal square root (one MUFU operation
// each, relative error ~2^-23); NaN for x < 0, which every caller either
// excludes by its own test or sends down a failing branch.  Subnormal
// inputs flush to zero (.ftz): the fit's quantities are far from 1e-38, and
// the subnormal-safe forms cost a test and two multiplies around each MUFU.
__device__ __forceinline__ float fsqrt(float x) {
  float r;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ F1 fsqrt(F1 x) { return F1(fsqrt(x.v)); }
__device__ __forceinline__ F2 fsqrt(F2 x) { return F2(fsqrt(x.v.x), fsqrt(x.v.y)); }
__device__ __forceinline__ float frsqrt(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ F1 frsqrt(F1 x) { return F1(frsqrt(x.v)); }
__device__ __forceinline__ F2 frsqrt(F2 x) { return F2(frsqrt(x.v.x), frsqrt(x.v.y)); }
__device__ __forceinline__ float fabs_(float x) { return fabsf(x); }
__device__ __forceinline__ F1 fabs_(F1 x) { return F1(fabsf(x.v)); }
__device__ __forceinline__ F2 fabs_(F2 x) { return F2(fabsf(x.v.x), fabsf(x.v.y)); }
__device__ __forceinline__ float fmax_(float a, float b) { return fmaxf(a, b); }
__device__ __forceinline__ F1 fmax_(F1 a, F1 b) { return F1(fmaxf(a.v, b.v)); }
__device__ __forceinline__ F2 fmax_(F2 a, F2 b) { return F2(fmaxf(a.v.x, b.v.x), fmaxf(a.v.y, b.v.y)); }
__device__ __forceinline__ float floor_(float x) { return floorf(x); }
__device__ __forceinline__ F1 floor_(F1 x) { return F1(floorf(x.v)); }
__device__ __forceinline__ F2 floor_(F2 x) { return F2(floorf(x.v.x), floorf(x.v.y)); }
__device__ __forceinline__ float copysign_(float a, float b) { return copysignf(a, b); }
__device__ __forceinline__ F1 copysign_(F1 a, F1 b) { return F1(copysignf(a.v, b.v)); }
__device__ __forceinline__ F2 copysign_(F2 a, F2 b) {
  return F2(copysignf(a.v.x, b.v.x), copysignf(a.v.y, b.v.y));
}

// ---- masks ---------------------------------------------------------------
__device__ __forceinline__ bool le(float a, float b) { return a <= b; }
__device__ __forceinline__ bool le(F1 a, F1 b) { return a.v <= b.v; }
__device__ __forceinline__ bool lt(F1 a, F1 b) { return a.v < b.v; }
__device__ __forceinline__ bool pos(F1 x) { return 0.f < x.v; }
__device__ __forceinline__ bool neg(F1 x) { return x.v < 0.f; }
__device__ __forceinline__ bool nonpos(F1 x) { return x.v <= 0.f; }
__device__ __forceinline__ bool finite_(F1 x) { return isfinite(x.v); }
__device__ __forceinline__ F1 sel(bool m, F1 a, F1 b) { return m ? a : b; }
__device__ __forceinline__ M2 le(F2 a, F2 b) { return {a.v.x <= b.v.x, a.v.y <= b.v.y}; }
__device__ __forceinline__ bool lt(float a, float b) { return a < b; }
__device__ __forceinline__ M2 lt(F2 a, F2 b) { return {a.v.x < b.v.x, a.v.y < b.v.y}; }
// x > 0, x < 0 and x <= 0 (in double on the integer pipe, see below)
__device__ __forceinline__ bool pos(float x) { return 0.f < x; }
__device__ __forceinline__ M2 pos(F2 x) { return {0.f < x.v.x, 0.f < x.v.y}; }
__device__ __forceinline__ bool neg(float x) { return x < 0.f; }
__device__ __forceinline__ M2 neg(F2 x) { return {x.v.x < 0.f, x.v.y < 0.f}; }
__device__ __forceinline__ bool nonpos(float x) { return x <= 0.f; }
__device__ __forceinline__ M2 nonpos(F2 x) { return {x.v.x <= 0.f, x.v.y <= 0.f}; }
__device__ __forceinline__ bool finite_(float a) { return isfinite(a); }
__device__ __forceinline__ M2 finite_(F2 a) { return {(bool)isfinite(a.v.x), (bool)isfinite(a.v.y)}; }
__device__ __forceinline__ bool all(bool m) { return m; }
__device__ __forceinline__ bool all(M2 m) { return m.x && m.y; }
__device__ __forceinline__ bool any(bool m) { return m; }
__device__ __forceinline__ bool any(M2 m) { return m.x || m.y; }
__device__ __forceinline__ bool not_(bool m) { return !m; }
__device__ __forceinline__ M2 not_(M2 m) { return {!m.x, !m.y}; }
__device__ __forceinline__ bool and_(bool a, bool b) { return a && b; }
__device__ __forceinline__ M2 and_(M2 a, M2 b) { return {a.x && b.x, a.y && b.y}; }
__device__ __forceinline__ bool or_(bool a, bool b) { return a || b; }
__device__ __forceinline__ M2 or_(M2 a, M2 b) { return {a.x || b.x, a.y || b.y}; }
__device__ __forceinline__ float sel(bool m, float a, float b) { return m ? a : b; }
__device__ __forceinline__ F2 sel(M2 m, F2 a, F2 b) {
  return F2(m.x ? a.v.x : b.v.x, m.y ? a.v.y : b.v.y);
}

// ---- double (the FP64 variant, one track per thread) -----------------------
// A warp's FP64 operation holds its SM's FP64 pipe for 16 cycles, so the FP64
// kernels are bound by the count of these alone (the pipe is 89 % busy).  Reciprocal and
// reciprocal square root take a coarse start from the MUFU (rcp.approx.ftz.f64,
// rsqrt.approx.ftz.f64: about 2^-19) and one correction of third order
// (Householder, "The Numerical Treatment of a Single Nonlinear Equation",
// 1970): with e = 1 - x y, 1/x = y / (1 - e) = y (1 + e + e^2 + ...), and with
// e = 1 - x y^2, x^(-1/2) = y (1 - e)^(-1/2) = y (1 + e/2 + 3 e^2/8 + ...).
// What is dropped is below 2^-58, so they are good to 0.51 and 1.0 ulp (1 / x
// and 1 / sqrt(x) of IEEE operations to 0.5 and 1.5), in 3 and 5 operations.
// Quotient and square root end with Newton's step from the result's residual,
// which an fma gives without rounding: 0.5 ulp, as the IEEE operations.
// A zero, subnormal, huge, negative (roots) or non-finite argument goes to
// those.
__device__ __forceinline__ double fma(double a, double b, double c) { return ::fma(a, b, c); }
// 2^-500 <= |x| < 2^500, on the integer pipe; positive: also x > 0
__device__ __forceinline__ bool mid_range(double x, bool positive) {
  const int hi = positive ? __double2hiint(x) : __double2hiint(x) & 0x7fffffff;
  return (unsigned)(hi - 0x20b00000) < 0x3e800000u;
}
static __device__ __noinline__ double ieee_rcp(double x) { return 1.0 / x; }
static __device__ __noinline__ double ieee_div(double a, double b) { return a / b; }
static __device__ __noinline__ double ieee_sqrt(double x) { return ::sqrt(x); }
// Comparisons with zero by the upper word (a subnormal counts as zero; a NaN
// as neither sign, but as x <= 0, whose callers test another value too).
__device__ __forceinline__ bool pos(double x) { return (unsigned)(__double2hiint(x) - 1) < 0x7ff00000u; }
__device__ __forceinline__ bool neg(double x) {
  return (unsigned)__double2hiint(x) - 0x80000001u < 0x7ff00000u;
}
__device__ __forceinline__ bool nonpos(double x) { return !pos(x); }
__device__ __forceinline__ double frcp(double x) {
  if (!mid_range(x, false)) return ieee_rcp(x);
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = ::fma(-x, y, 1.0);
  return ::fma(::fma(e, e, e), y, y);
}
// a (1/b), with the quotient's remainder folded back
__device__ __forceinline__ double fdiv(double a, double b) {
  if (!mid_range(b, false)) return ieee_div(a, b);
  const double y = frcp(b), q = a * y;
  return ::fma(::fma(-b, q, a), y, q);
}
__device__ __forceinline__ double frsqrt(double x) {
  if (!mid_range(x, true)) return ieee_rcp(ieee_sqrt(x));
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = ::fma(-(x * y), y, 1.0);
  return ::fma(::fma(e, 0.375, 0.5), e * y, y);
}
__device__ __forceinline__ double fsqrt(double x) {  // NaN for x < 0, as in FP32
  if (!mid_range(x, true)) return ieee_sqrt(x);
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  y = ::fma(::fma(-(x * y), y, 1.0), 0.5 * y, y);  // Newton: 2^-38
  const double r = x * y;
  return ::fma(::fma(-r, r, x), 0.5 * y, r);
}
// |x| < the double whose upper word is hi (a positive one), on the integer pipe
__device__ __forceinline__ bool below_hi(double x, int hi) {
  return (__double2hiint(x) & 0x7fffffff) < hi;
}
__device__ __forceinline__ double fabs_(double x) { return ::fabs(x); }
__device__ __forceinline__ double floor_(double x) { return ::floor(x); }
__device__ __forceinline__ double fmax_(double a, double b) { return ::fmax(a, b); }
__device__ __forceinline__ double copysign_(double a, double b) { return ::copysign(a, b); }
__device__ __forceinline__ bool le(double a, double b) { return a <= b; }
__device__ __forceinline__ bool lt(double a, double b) { return a < b; }
__device__ __forceinline__ bool finite_(double a) {
  return (__double2hiint(a) & 0x7ff00000) != 0x7ff00000;
}
__device__ __forceinline__ double sel(bool m, double a, double b) { return m ? a : b; }

// ---- lanes ---------------------------------------------------------------
// exact: the type's propagation takes crossing_start's exact form itself; the
// others leave such a track to the float path.
template <class T>
struct Lanes;
template <>
struct Lanes<float> {
  static constexpr int n = 1;
  static constexpr bool exact = true;
  using M = bool;
  __device__ __forceinline__ static float get(float a, int) { return a; }
  __device__ __forceinline__ static bool get(bool m, int) { return m; }
};
template <>
struct Lanes<double> {
  static constexpr int n = 1;
  static constexpr bool exact = true;
  using M = bool;
  __device__ __forceinline__ static double get(double a, int) { return a; }
  __device__ __forceinline__ static bool get(bool m, int) { return m; }
};
template <>
struct Lanes<F1> {
  static constexpr int n = 1;
  static constexpr bool exact = false;
  using M = bool;
  __device__ __forceinline__ static float get(F1 a, int) { return a.v; }
  __device__ __forceinline__ static bool get(bool m, int) { return m; }
};
template <>
struct Lanes<F2> {
  static constexpr int n = 2;
  static constexpr bool exact = false;
  using M = M2;
  __device__ __forceinline__ static float get(F2 a, int i) { return i ? a.v.y : a.v.x; }
  __device__ __forceinline__ static bool get(M2 m, int i) { return i ? m.y : m.x; }
};

// Streaming loads and stores of lane-consecutive tracks (p points at the
// first track; for F2 it is 8-byte aligned).
__device__ __forceinline__ void ld(float& d, const float* p) { d = __ldcs(p); }
__device__ __forceinline__ void ld(F1& d, const float* p) { d = F1(__ldcs(p)); }
__device__ __forceinline__ void ld(F2& d, const float* p) {
  d = F2(__ldcs(reinterpret_cast<const float2*>(p)));
}
__device__ __forceinline__ void ld(double& d, const double* p) { d = __ldcs(p); }
__device__ __forceinline__ void st(double* p, double v) { *p = v; }
__device__ __forceinline__ void st(float* p, float v) { *p = v; }
__device__ __forceinline__ void st(float* p, F1 v) { *p = v.v; }
__device__ __forceinline__ void st(float* p, F2 v) { *reinterpret_cast<float2*>(p) = v.v; }

}  // namespace fitk
