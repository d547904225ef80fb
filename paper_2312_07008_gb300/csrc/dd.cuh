// Double-float ("dd") arithmetic: a value is hi + lo with two float32s,
// |lo| <= ulp(hi)/2, about 48 significant bits.  GB300 runs float32 at many
// times its float64 rate, so the elementwise stages of the fast form (the
// Eq. A7 regulariser, the 2-RDM dressing, the digit staging) use these
// operations.  The error-free transformations are Knuth's TwoSum and the
// fused-multiply-add TwoProduct; additions and products follow the standard
// double-float construction (Dekker 1971).
#pragma once
#include <cuda_runtime.h>

#include "f32x2.cuh"

namespace dsrg {

// The operations are written for float32 and for packed pairs of it (f32x2: two
// values at once, half the instructions).
__device__ __forceinline__ float fl_add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float fl_sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float fl_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float fl_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float fl_neg(float a) { return -a; }
__device__ __forceinline__ f32x2 fl_add(f32x2 a, f32x2 b) { return f2_add(a, b); }
__device__ __forceinline__ f32x2 fl_sub(f32x2 a, f32x2 b) { return f2_sub(a, b); }
__device__ __forceinline__ f32x2 fl_mul(f32x2 a, f32x2 b) { return f2_mul(a, b); }
__device__ __forceinline__ f32x2 fl_fma(f32x2 a, f32x2 b, f32x2 c) { return f2_fma(a, b, c); }
__device__ __forceinline__ f32x2 fl_neg(f32x2 a) { return f2_mul(a, f2_set(-1.0f, -1.0f)); }

// the components of a T: 1 of float, 2 of f32x2
template <class T>
struct FlCount;
template <>
struct FlCount<float> {
  static constexpr int N = 1;
};
template <>
struct FlCount<f32x2> {
  static constexpr int N = 2;
};
__device__ __forceinline__ void fl_get(float x, float (&v)[1]) { v[0] = x; }
__device__ __forceinline__ void fl_get(f32x2 x, float (&v)[2]) { f2_get(x, &v[0], &v[1]); }
__device__ __forceinline__ float fl_pack(const float (&v)[1]) { return v[0]; }
__device__ __forceinline__ f32x2 fl_pack(const float (&v)[2]) { return f2_set(v[0], v[1]); }
template <class T>
__device__ __forceinline__ T fl_set(float x) {
  if constexpr (FlCount<T>::N == 1) return x;
  else return f2_set(x, x);
}

template <class T>
struct ddt {
  T hi, lo;
};
using dd = ddt<float>;
using dd2 = ddt<f32x2>;

__device__ __forceinline__ dd dd_make(float h) { return {h, 0.0f}; }
template <class T>
__device__ __forceinline__ ddt<T> dd_splat(dd a) {
  return {fl_set<T>(a.hi), fl_set<T>(a.lo)};
}

template <class T>
__device__ __forceinline__ ddt<T> two_sum(T a, T b) {
  const T s = fl_add(a, b);
  const T bb = fl_sub(s, a);
  const T e = fl_add(fl_sub(a, fl_sub(s, bb)), fl_sub(b, bb));
  return {s, e};
}

template <class T>
__device__ __forceinline__ ddt<T> quick_two_sum(T a, T b) {  // |a| >= |b|
  const T s = fl_add(a, b);
  return {s, fl_sub(b, fl_sub(s, a))};
}

template <class T>
__device__ __forceinline__ ddt<T> two_prod(T a, T b) {
  const T p = fl_mul(a, b);
  return {p, fl_fma(a, b, fl_neg(p))};
}

template <class T>
__device__ __forceinline__ ddt<T> dd_add(ddt<T> a, ddt<T> b) {
  ddt<T> s = two_sum(a.hi, b.hi);
  const ddt<T> t = two_sum(a.lo, b.lo);
  s.lo = fl_add(s.lo, t.hi);
  s = quick_two_sum(s.hi, s.lo);
  s.lo = fl_add(s.lo, t.lo);
  return quick_two_sum(s.hi, s.lo);
}

__device__ __forceinline__ dd dd_neg(dd a) { return {-a.hi, -a.lo}; }

// a + b with an absolute error of a few units of 2^-48 max(|a|, |b|) (no
// relative accuracy when the high parts cancel); for sums whose terms keep
// their sign or whose cancellation the caller does not need resolved.
template <class T>
__device__ __forceinline__ ddt<T> dd_add_fast(ddt<T> a, ddt<T> b) {
  ddt<T> s = two_sum(a.hi, b.hi);
  s.lo = fl_add(s.lo, fl_add(a.lo, b.lo));
  return quick_two_sum(s.hi, s.lo);
}
template <class T>
__device__ __forceinline__ ddt<T> dd_sub_fast(ddt<T> a, ddt<T> b) {
  const T s = fl_sub(a.hi, b.hi), bb = fl_sub(a.hi, s);  // TwoSum of a.hi and -b.hi
  const T e = fl_sub(fl_sub(a.hi, fl_add(s, bb)), fl_sub(b.hi, bb));
  return quick_two_sum(s, fl_add(e, fl_sub(a.lo, b.lo)));
}
__device__ __forceinline__ dd dd_sub(dd a, dd b) { return dd_add(a, dd_neg(b)); }

// a + b and a - b of the same accuracy where |a| >= |b| or a = 0
template <class T>
__device__ __forceinline__ ddt<T> dd_add_ordered(ddt<T> a, ddt<T> b) {
  const T s = fl_add(a.hi, b.hi), e = fl_sub(b.hi, fl_sub(s, a.hi));
  return quick_two_sum(s, fl_add(e, fl_add(a.lo, b.lo)));
}
template <class T>
__device__ __forceinline__ ddt<T> dd_sub_ordered(ddt<T> a, ddt<T> b) {
  const T s = fl_sub(a.hi, b.hi), e = fl_sub(fl_sub(a.hi, s), b.hi);
  return quick_two_sum(s, fl_add(e, fl_sub(a.lo, b.lo)));
}

template <class T>
__device__ __forceinline__ ddt<T> dd_add_f(ddt<T> a, T b) {
  ddt<T> s = two_sum(a.hi, b);
  s.lo = fl_add(s.lo, a.lo);
  return quick_two_sum(s.hi, s.lo);
}

template <class T>
__device__ __forceinline__ ddt<T> dd_mul(ddt<T> a, ddt<T> b) {
  ddt<T> p = two_prod(a.hi, b.hi);
  p.lo = fl_fma(a.hi, b.lo, p.lo);
  p.lo = fl_fma(a.lo, b.hi, p.lo);
  return quick_two_sum(p.hi, p.lo);
}

template <class T>
__device__ __forceinline__ ddt<T> dd_mul_f(ddt<T> a, T b) {
  ddt<T> p = two_prod(a.hi, b);
  p.lo = fl_fma(a.lo, b, p.lo);
  return quick_two_sum(p.hi, p.lo);
}

// 1 / b by Newton's iteration r + r (1 - b r) with fused multiply-adds (Markstein,
// IBM J. Res. Dev. 34, 1990): from the hardware's approximation to float32, where
// 1 - b.hi r is exact, and from there to double-float: relative error about 2^-46.
__device__ __forceinline__ float fl_recip_approx(float b) {
  float r;
  asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(b));
  return r;
}
__device__ __forceinline__ f32x2 fl_recip_approx(f32x2 b) {
  float x, y;
  f2_get(b, &x, &y);
  return f2_set(fl_recip_approx(x), fl_recip_approx(y));
}
template <class T>
__device__ __forceinline__ ddt<T> dd_recip(ddt<T> b) {
  const T one = fl_set<T>(1.0f), nh = fl_neg(b.hi);
  T r = fl_recip_approx(b.hi);
  r = fl_fma(r, fl_fma(nh, r, one), r);
  const T e = fl_sub(fl_fma(nh, r, one), fl_mul(b.lo, r));
  return quick_two_sum(r, fl_mul(r, e));
}

__device__ __forceinline__ dd dd_from_double(double x) {
  const float h = __double2float_rn(x);
  return {h, __double2float_rn(x - (double)h)};
}

__device__ __forceinline__ double dd_to_double(dd a) { return (double)a.hi + (double)a.lo; }

}  // namespace dsrg
