// The Eq. A7 regulariser in double-float arithmetic, shared by the
// elementwise epilogue kernel and the fused epilogue of the contraction
// kernel.
//
// With x = s Delta^2 >= 0, y = exp(-x):
//   tau = nu (1 - y) / Delta,  kappa = 2 nu - Delta tau = nu (1 + y).
// exp(-x) follows the table method of Tang (ACM TOMS 15, 1989): x = n ln 2 / 64
// + u with |u| <= ln 2 / 128 (Cody and Waite's reduction: ln 2 / 64 in three
// parts), exp(-x) = 2^-q 2^-j/64 exp(-u), n = 64 q + j, and exp(-u) from its
// Taylor series.  With T' = 2^-q 2^-j/64,
//   y = T' - T' (1 - e^-u),   1 - y = (1 - T') + T' (1 - e^-u),
// and 1 - T' from a table where q = 0, so that the small-Delta branch of Eq. A7
// (R -> s Delta) keeps its relative accuracy without a separate series.  For
// x > 40, y < 5e-18 is dropped.
#pragma once
#include "dd.cuh"

namespace dsrg {

struct RegTables {
  dd T[64];  // 2^-j/64
  dd C[64];  // 1 - 2^-j/64
};

// ln 2 / 64 = REG_L1 + REG_L2 + REG_L3: n REG_L1 is exact for n < 2^12
constexpr double REG_STEP = 0.69314718055994530942 / 64.0;
constexpr float REG_L1 = 2839.0f / 262144.0f;
constexpr float REG_L2 = (float)(REG_STEP - (double)REG_L1);
constexpr float REG_L3 = (float)(REG_STEP - (double)REG_L1 - (double)REG_L2);
constexpr double REG_SIXTH = 1.0 / 6.0;
constexpr float REG_ROUND = 12582912.0f;  // 1.5 2^23: x + REG_ROUND has the rounded x in its low bits

// R1 = (1 - exp(-s Delta^2)) / Delta and y = exp(-s Delta^2), double-float, of
// one value (T = float) or two (f32x2).  About 170 instructions either way.
template <class T>
__device__ __forceinline__ void regularize(ddt<T> delta, dd s, const RegTables& R, ddt<T>* r1, ddt<T>* y) {
  constexpr int N = FlCount<T>::N;
  ddt<T> x = dd_mul(dd_splat<T>(s), dd_mul(delta, delta));
  float xh[N], dh[N];
  fl_get(x.hi, xh);
  fl_get(delta.hi, dh);
  bool big[N], tiny[N], all_big = true, special = false;
#pragma unroll
  for (int c = 0; c < N; ++c) {
    big[c] = xh[c] > 40.0f;
    tiny[c] = xh[c] < 1e-20f || dh[c] == 0.0f;  // R1 = s Delta (1 - x/2 + ...), y = 1 - x: the x terms are below the precision
    all_big &= big[c];
    special |= big[c] || tiny[c];
  }
  if (all_big) {
    *y = {fl_set<T>(0.0f), fl_set<T>(0.0f)};
    *r1 = dd_recip(delta);
    return;
  }
  ddt<T> d = delta;
  if (special) {  // any values in range: replaced at the end
    float a[N], b[N], e[N], f[N];
    fl_get(x.lo, a);
    fl_get(delta.lo, b);
#pragma unroll
    for (int c = 0; c < N; ++c) {
      const bool sp = big[c] || tiny[c];
      xh[c] = sp ? 1.0f : xh[c];
      a[c] = sp ? 0.0f : a[c];
      e[c] = tiny[c] ? 1.0f : dh[c];
      f[c] = tiny[c] ? 0.0f : b[c];
    }
    x = {fl_pack(xh), fl_pack(a)};
    d = {fl_pack(e), fl_pack(f)};
  }
  // x = n ln 2 / 64 + u: the high part is exact after one fused multiply-add
  const T tn = fl_fma(x.hi, fl_set<T>((float)(1.0 / REG_STEP)), fl_set<T>(REG_ROUND));
  const T n = fl_sub(tn, fl_set<T>(REG_ROUND));
  const T h1 = fl_fma(n, fl_set<T>(-REG_L1), x.hi);
  const T h2 = fl_mul(n, fl_set<T>(-REG_L2));
  const T e2 = fl_fma(n, fl_set<T>(REG_L2), h2);
  ddt<T> u = two_sum(h1, h2);
  u.lo = fl_add(u.lo, fl_fma(n, fl_set<T>(-REG_L3), fl_sub(x.lo, e2)));
  u = quick_two_sum(u.hi, u.lo);
  // 1 - e^-u = u - u^2 (1/2 - u/6 + (u^2/24 - u^3/120 + u^4/720))   (|u| <= 0.0055);
  // u/6 in double-float, the terms in the inner brackets (< 1.3e-6) in float
  constexpr float S1 = (float)REG_SIXTH, S2 = (float)(REG_SIXTH - (double)S1);
  const T tail = fl_mul(fl_mul(u.hi, u.hi), fl_fma(u.hi, fl_fma(u.hi, fl_set<T>(1.0f / 720.0f), fl_set<T>(-1.0f / 120.0f)),
                                                   fl_set<T>(1.0f / 24.0f)));
  const T a = fl_mul(u.hi, fl_set<T>(-S1));
  const T al = fl_fma(u.hi, fl_set<T>(S2), fl_fma(u.lo, fl_set<T>(S1), fl_fma(u.hi, fl_set<T>(S1), a)));
  ddt<T> w = quick_two_sum(fl_set<T>(0.5f), a);
  w.lo = fl_add(w.lo, fl_sub(tail, al));
  const ddt<T> omp = dd_sub_ordered(u, dd_mul(dd_mul(u, u), w));
  // T' = 2^-q T_j, 1 - y = (1 - T') + T' (1 - e^-u), y = T' - T' (1 - e^-u)
  float nb[N], th[N], tl[N];
  fl_get(tn, nb);
  bool first = false;
  int ni[N];
#pragma unroll
  for (int c = 0; c < N; ++c) {
    ni[c] = __float_as_int(nb[c]) - __float_as_int(REG_ROUND);
    first |= ni[c] < 64;
    const dd t = R.T[ni[c] & 63];
    const float sc = __int_as_float((127 - (ni[c] >> 6)) << 23);
    th[c] = t.hi * sc;
    tl[c] = t.lo * sc;
  }
  const ddt<T> tq = {fl_pack(th), fl_pack(tl)};
  ddt<T> omt = dd_sub_ordered(ddt<T>{fl_set<T>(1.0f), fl_set<T>(0.0f)}, tq);
  if (first) {  // q = 0: from the table, without cancellation
    float ch[N], cl[N];
    fl_get(omt.hi, ch);
    fl_get(omt.lo, cl);
#pragma unroll
    for (int c = 0; c < N; ++c)
      if (ni[c] < 64) {
        const dd t = R.C[ni[c] & 63];
        ch[c] = t.hi;
        cl[c] = t.lo;
      }
    omt = {fl_pack(ch), fl_pack(cl)};
  }
  const ddt<T> z = dd_mul(tq, omp);
  *y = dd_sub_ordered(tq, z);
  *r1 = dd_mul(dd_add_ordered(omt, z), dd_recip(d));
  if (special) {
    float yh[N], yl[N], rh[N], rl[N], bh[N], bl[N], dl[N];
    const ddt<T> rec = dd_recip(d);
    fl_get(y->hi, yh);
    fl_get(y->lo, yl);
    fl_get(r1->hi, rh);
    fl_get(r1->lo, rl);
    fl_get(rec.hi, bh);
    fl_get(rec.lo, bl);
    fl_get(delta.lo, dl);
#pragma unroll
    for (int c = 0; c < N; ++c) {
      const dd sd = dd_mul(s, dd{dh[c], dl[c]});
      yh[c] = big[c] ? 0.0f : (tiny[c] ? 1.0f : yh[c]);
      yl[c] = big[c] || tiny[c] ? 0.0f : yl[c];
      rh[c] = big[c] ? bh[c] : (tiny[c] ? sd.hi : rh[c]);
      rl[c] = big[c] ? bl[c] : (tiny[c] ? sd.lo : rl[c]);
    }
    *y = {fl_pack(yh), fl_pack(yl)};
    *r1 = {fl_pack(rh), fl_pack(rl)};
  }
}

}  // namespace dsrg
