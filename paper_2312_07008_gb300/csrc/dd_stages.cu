// Elementwise stages of the fast form in double-float arithmetic:
//   - the Eq. A7 regulariser applied to the contraction tiles (tau, kappa),
//     regularizer.cuh,
//   - the 2-RDM dressing of the vv classes with the energy partials.
// Their float64 counterparts are gemm_f64.cu (fused epilogue) and dress.cu.
#include "dd.cuh"
#include "regularizer.cuh"
#include "dress_common.cuh"
#include "kernels.h"

namespace dsrg {

namespace {

using namespace dressc;

// Filled once per device (float64 exp2 / expm1, then split); kernels copy it
// to shared memory.
__device__ RegTables g_reg;

__global__ void reg_tables_fill_kernel() {
  for (int j = threadIdx.x; j < 64; j += blockDim.x) {
    g_reg.T[j] = dd_from_double(exp2(-j / 64.0));
    g_reg.C[j] = dd_from_double(-expm1(-j * 0.69314718055994530942 / 64.0));
  }
}

__device__ __forceinline__ void reg_tables_load(RegTables& R) {
  const float* src = reinterpret_cast<const float*>(&g_reg);
  float* dst = reinterpret_cast<float*>(&R);
  for (int k = threadIdx.x; k < (int)(sizeof(RegTables) / sizeof(float)); k += blockDim.x) dst[k] = src[k];
}

__global__ void eps_dd_kernel(int n, const double* __restrict__ eps, float2* __restrict__ out) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n) {
    const dd v = dd_from_double(eps[k]);
    out[k] = make_float2(v.hi, v.lo);
  }
}

constexpr int EPI_ROWS = 8;  // rows a of one pair per block

// tau / kappa (vv, double-float) and t^{ij}_{ex} (va / av, float64) from the
// double-float contraction tiles nu[slot][a][b].  One block per EPI_ROWS rows
// of one pair.
__global__ void __launch_bounds__(256) pair_epilogue_dd_kernel(Geometry g, const double* __restrict__ eps,
                                                               const float2* __restrict__ eps_dd,
                                                               const int2* __restrict__ pairs,
                                                               const float2* __restrict__ nu,
                                                               float2* __restrict__ tau, float2* __restrict__ kap,
                                                               double* __restrict__ ts) {
  __shared__ RegTables R;
  __shared__ float2 s_ca[EPI_ROWS];
  reg_tables_load(R);
  const int a0 = blockIdx.x * EPI_ROWS, slot = blockIdx.y;
  const int na = g.na, nv = g.nv, np = g.np;
  const int2 pr = pairs[slot];
  const int i = pr.x, j = pr.y;
  const double* ep = eps + g.nc;
  // Delta = (eps_i + eps_j - eps_a) - eps_b, the row part rounded once to double-float
  if (threadIdx.x < EPI_ROWS && a0 + threadIdx.x < np) {
    const dd ca = dd_from_double(eps[i] + eps[j] - ep[a0 + threadIdx.x]);
    s_ca[threadIdx.x] = make_float2(ca.hi, ca.lo);
  }
  __syncthreads();
  const dd s = dd_from_double(g.s);
  const int rows = min(EPI_ROWS, np - a0);
  for (int ra = 0; ra < rows; ++ra)
  for (int b = threadIdx.x; b < np; b += blockDim.x) {
    const int a = a0 + ra;
    const bool av = a >= na, bv = b >= na;
    if (!av && !bv) continue;
    if (ts == nullptr && !(av && bv)) continue;
    const float2 nn = nu[((long)slot * np + a) * np + b];
    const dd n = {nn.x, nn.y};
    const float2 eb = eps_dd[g.nc + b];
    const float2 ca2 = s_ca[a - a0];
    const dd delta = dd_sub(dd{ca2.x, ca2.y}, dd{eb.x, eb.y});
    dd r1, y;
    regularize(delta, s, R, &r1, &y);
    const dd t = dd_mul(n, r1);
    if (av && bv) {
      const dd k = dd_mul(n, dd_add_f(y, 1.0f));
      const long o = ((long)slot * nv + (a - na)) * nv + (b - na);
      tau[o] = make_float2(t.hi, t.lo);
      kap[o] = make_float2(k.hi, k.lo);
    } else if (av) {
      ts[(((long)i * g.nh + j) * nv + (a - na)) * na + b] = dd_to_double(t);
    } else if (i != j) {
      ts[(((long)j * g.nh + i) * nv + (b - na)) * na + a] = dd_to_double(t);
    }
  }
}

__device__ __forceinline__ dd ld(const float2* p, long i) {
  const float2 v = p[i];
  return {v.x, v.y};
}

// acc + c s without renormalisation: the product's high part is added error-free
// (TwoSum), its low parts and both errors to the low word in float32.  nh = -s.hi.
template <class T>
__device__ __forceinline__ void dd_fma_into(ddt<T>& acc, ddt<T> c, ddt<T> s, T nh) {
  const T p = fl_mul(c.hi, s.hi);
  const T ne = fl_fma(c.hi, nh, p);  // minus the product's error
  const ddt<T> t = two_sum(acc.hi, p);
  acc.lo = fl_sub(fl_add(fl_fma(c.lo, s.hi, fl_fma(c.hi, s.lo, acc.lo)), t.lo), ne);
  acc.hi = t.hi;
}
__device__ __forceinline__ dd dd_fma_acc(dd acc, dd c, dd s) {
  dd_fma_into(acc, c, s, -s.hi);
  return quick_two_sum(acc.hi, acc.lo);
}

// What the staging of the dressed matrices needs of a row: the largest |hi| of
// all its elements (digit planes: rowmax, atomics), or a bound of each tile's
// norm (residues: rowpart[matrix][tile column][row], strides for tiles of GT).
// Float64 atomics per row instead took more time than the dressing itself (the
// SM has two float64 lanes; opdm pass of nvir 1200: 67 ms).
__device__ __forceinline__ bool square_in_range(float s) { return s > 1e-30f && s < 1e38f; }

// Norms of eight of a warp's rows of 32 elements each (v: this lane's |hi|; row
// of value i: lane 4 i's result): the lanes halve the values before they halve
// themselves (9 shuffles).  Where a square would leave float32's range, the
// largest element times 32^1/2.
__device__ __forceinline__ float row_norms8(const float (&v)[8]) {
  const int lane = threadIdx.x & 31;
  float x[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) x[i] = v[i] * v[i];
#pragma unroll
  for (int h = 4, o = 16; h > 0; h >>= 1, o >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < h; ++i) x[i] = (up ? x[i + h] : x[i]) + __shfl_xor_sync(0xffffffffu, up ? x[i] : x[i + h], o);
  }
  x[0] += __shfl_xor_sync(0xffffffffu, x[0], 2);
  x[0] += __shfl_xor_sync(0xffffffffu, x[0], 1);
  float n = sqrtf(x[0]);
  if (__any_sync(0xffffffffu, !square_in_range(x[0]))) {
    const int mine = lane >> 2;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float m = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(v[i])));
      if (mine == i) n = m * 5.6568546f;  // above 32^1/2
    }
  }
  return n;
}

// Core pairs.  With P = tau + tau^T and Q = tau - tau^T (and the same of kappa)
// the pair (m, n) contributes E = <P, P_k> / 2 + 3 <Q, Q_k> / 2 and the dressed
// matrices sqrt(lambda) sigma = P and sqrt(3) Q; the pair (m, m) E = <tau, kappa>
// and sqrt(2) tau.  One pass over the upper 32 x 32 tiles, four elements and
// their transposes per thread, no coefficients: the general kernel spent about
// 200 instructions on an element (dressing of an opdm pass of nvir 1200: 54.3 ms,
// now 48.5; nvir 300 with 6 active: 0.82, now 0.70).  Bound by memory: 16 bytes
// read and 16 written per element.
constexpr int CT = 32;
__global__ void __launch_bounds__(256, 4) dress_core_dd_kernel(int nv, const DressDesc* __restrict__ desc,
                                                               const float2* __restrict__ tau,
                                                               const float2* __restrict__ kap, float2* __restrict__ sig,
                                                               double* __restrict__ sig_sign, double* __restrict__ e_part,
                                                               int want_sig, unsigned* __restrict__ rowmax,
                                                               float* __restrict__ rowpart) {
  __shared__ float2 sT[CT][CT + 1], sK[CT][CT + 1];
  __shared__ double red[8];
  const DressDesc D = desc[blockIdx.y];
  const bool diag = D.kind == GROUP_CC_DIAG;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nt = (nv + CT - 1) / CT, nup = nt * (nt + 1) / 2;
  const long nv2 = (long)nv * nv;
  const float2* T = tau + (long)D.slot * nv2;
  const float2* K = kap + (long)D.slot * nv2;
  float2* S0 = want_sig ? sig + (long)D.out * nv2 : nullptr;
  const dd root3 = dd_from_double(1.7320508075688772935), root2 = dd_from_double(1.4142135623730950488);
  dd eP = dd_make(0.0f), eQ = dd_make(0.0f);
  // rows R0 + warp + 8 r of both outputs, over tile column tcol
  auto magnitudes = [&](const float (&mag)[8], int R0, int tcol) {
    if (rowpart) {
      const float n = row_norms8(mag);
      const int i = lane >> 2, row = R0 + warp + 8 * (i & 3);
      if ((lane & 3) == 0 && row < nv && !(diag && i >= 4))
        rowpart[((long)(D.out + (i >> 2)) * ((nv + GT - 1) / GT) + tcol) * nv + row] = n;
    } else {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int row = R0 + warp + 8 * (i & 3);
        const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(mag[i]));
        if (lane == 0 && row < nv && !(diag && i >= 4)) atomicMax(rowmax + (long)(D.out + (i >> 2)) * nv + row, m);
      }
    }
  };
  int te = 0, base = 0;
  for (int t = blockIdx.x; t < nup; t += gridDim.x) {
    while (t >= base + (nt - te)) {
      base += nt - te;
      ++te;
    }
    const int tf = te + (t - base), E0 = te * CT, F0 = tf * CT;
    const bool upper = te != tf;
    const float w = upper ? 1.0f : 0.5f;
    float2 a[4], b[4];
    __syncthreads();  // the last tile's shared elements are read
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int e = E0 + warp + 8 * r, f = F0 + lane, fr = F0 + warp + 8 * r, ec = E0 + lane;
      const bool in = e < nv && f < nv, ok = fr < nv && ec < nv;
      a[r] = in ? T[(long)e * nv + f] : make_float2(0.f, 0.f);
      b[r] = in ? K[(long)e * nv + f] : make_float2(0.f, 0.f);
      sT[warp + 8 * r][lane] = ok ? T[(long)fr * nv + ec] : make_float2(0.f, 0.f);
      sK[warp + 8 * r][lane] = ok ? K[(long)fr * nv + ec] : make_float2(0.f, 0.f);
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int er = warp + 8 * r;
      const float2 xt = sT[lane][er], xk = sK[lane][er];
      const dd ta = {a[r].x, a[r].y}, tb = {xt.x, xt.y}, ka = {b[r].x, b[r].y}, kb = {xk.x, xk.y};
      dd p = dd_add_fast(ta, tb), q = dd_sub_fast(ta, tb);
      const dd kp = dd_add_fast(ka, kb), kq = dd_sub_fast(ka, kb);
      eP = dd_fma_acc(eP, dd{p.hi * w, p.lo * w}, kp);  // w = 1 or 1/2: exact
      eQ = dd_fma_acc(eQ, dd{q.hi * w, q.lo * w}, kq);
      if (want_sig) {
        if (diag) p = dd_mul(root2, ta);
        else q = dd_mul(root3, q);
        // the transposed positions of this element: read by no other thread
        a[r] = make_float2(p.hi, p.lo);
        b[r] = make_float2(q.hi, q.lo);
      }
    }
    if (!want_sig) continue;
    float mag[8];
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int er = warp + 8 * r, e = E0 + er, f = F0 + lane;
      const bool in = e < nv && f < nv;
      if (in) {
        S0[(long)e * nv + f] = a[r];
        if (!diag) S0[nv2 + (long)e * nv + f] = b[r];
      }
      sT[er][lane] = a[r];
      sK[er][lane] = b[r];
      mag[r] = in ? fabsf(a[r].x) : 0.0f;
      mag[4 + r] = in ? fabsf(b[r].x) : 0.0f;
    }
    magnitudes(mag, E0, tf);
    if (!upper) continue;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 4; ++r) {  // rows f: S[f][e] = P, -Q
      const int fr = warp + 8 * r, f = F0 + fr, e = E0 + lane;
      const bool in = f < nv && e < nv;
      const float2 p = sT[lane][fr], q = sK[lane][fr];
      if (in) {
        S0[(long)f * nv + e] = p;
        if (!diag) S0[nv2 + (long)f * nv + e] = make_float2(-q.x, -q.y);
      }
      mag[r] = in ? fabsf(p.x) : 0.0f;
      mag[4 + r] = in ? fabsf(q.x) : 0.0f;
    }
    magnitudes(mag, F0, te);
  }
  // over the upper tiles: <P, P_k> + 3 <Q, Q_k>; the pair (m, m) has <P, P_k> = 4 <tau, kappa>, half of it upper
  double pd = diag ? 0.5 * dd_to_double(eP) : dd_to_double(eP) + 3.0 * dd_to_double(eQ);
  for (int o = 16; o > 0; o >>= 1) pd += __shfl_down_sync(0xffffffffu, pd, o);
  if (lane == 0) red[warp] = pd;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int v = 0; v < 8; ++v) s += red[v];
    e_part[(long)blockIdx.y * gridDim.x + blockIdx.x] = s;
  }
  if (want_sig && blockIdx.x == 0 && threadIdx.x < (diag ? 1 : 2)) sig_sign[D.out + threadIdx.x] = 1.0;
}

// Double-float form of the group dressing (same structure as dress.cu).  Bound
// by the float32 pipe and the latency of its chains: 12 operations per slot and
// output for each of tau and kappa, which share the coefficient and go through
// packed pairs.  nvir 600, 40 core and 10 active orbitals, with the core pairs'
// kernel: 7.48 -> 6.98 ms (a third block per SM: 7.24 with two, 7.73 with four).
template <int OCT>
__global__ void __launch_bounds__(GNT, 3)
    dress_dd_kernel(int nv, int na, const DressDesc* __restrict__ desc, DressAux aux,
                    const float2* __restrict__ tau, const float2* __restrict__ kap, float2* __restrict__ sig,
                    double* __restrict__ sig_sign, double* __restrict__ e_part, int want_sig,
                    unsigned* __restrict__ rowmax, float* __restrict__ rowpart) {
  constexpr int NS = MAXSLOT;
  // double-float coefficients, every word twice: {hi, hi, lo, lo} multiplies a
  // (tau, kappa) pair
  __shared__ float4 cf2[NS * OCT];
  __shared__ double lam[OCT], sgn[OCT], dg[NS];
  __shared__ dd lamw[OCT], sqd[OCT];
  __shared__ float sgnf[OCT], dgf[NS];  // float copies: no float64 op in the loops
  // transposed tiles double-buffered: one barrier per slot
  __shared__ float2 tT[2][GT][GT + 1], tK[2][GT][GT + 1], sA[GT][GT + 1];
  __shared__ double red[GNT / 32];
  const DressDesc D = desc[blockIdx.y];
  // the float64 coefficients fill the lower half; each thread's, from the back
  double(*cd)[OCT] = reinterpret_cast<double(*)[OCT]>(cf2);
  group_coefficients<OCT>(D, aux, na, cd, lam, sgn, dg);
  const int oc = D.o_count;
  for (int base = (D.nslots * OCT - 1) / GNT * GNT; base >= 0; base -= GNT) {
    const int idx = base + threadIdx.x;
    const bool in = idx < D.nslots * OCT;
    const dd v = in ? dd_from_double(cd[idx / OCT][idx % OCT]) : dd_make(0.0f);
    __syncthreads();  // read before the places of this pass, which start at 2 base, are written
    if (in) cf2[idx] = make_float4(v.hi, v.hi, v.lo, v.lo);
    __syncthreads();
  }
  for (int o = threadIdx.x; o < oc; o += blockDim.x) {
    lamw[o] = dd_from_double(0.5 * lam[o]);
    sqd[o] = dd_from_double(sqrt(fabs(lam[o])));
    sgnf[o] = sgn[o] > 0.0 ? 1.0f : -1.0f;
  }
  for (int u = threadIdx.x; u < D.nslots; u += blockDim.x) dgf[u] = (float)dg[u];
  __syncthreads();
  const int ntd = (nv + GT - 1) / GT;
  const int nup = ntd * (ntd + 1) / 2;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const long nv2 = (long)nv * nv;
  const int ns = D.nslots;
  unsigned posmask = 0;  // bit o: output o is symmetric (sgn +1)
#pragma unroll
  for (int o = 0; o < OCT; ++o)
    if (o < oc && sgnf[o] > 0.0f) posmask |= 1u << o;
  // upper tile t -> (te, tf), te <= tf; t only grows, so the row search
  // resumes where the last one ended (row_te starts at tile row_base)
  int row_te = 0, row_base = 0;
  auto decode = [&](int t, int* te_, int* tf_) {
    while (t >= row_base + (ntd - row_te)) {
      row_base += ntd - row_te;
      ++row_te;
    }
    *te_ = row_te;
    *tf_ = row_te + (t - row_base);
  };
  // this thread's operands of slot u in tile (te, tf): tau and kappa at (e, f)
  // and at (f, e) (the latter staged transposed through shared memory)
  float2 na_ = make_float2(0.f, 0.f), nb_ = na_, nt_ = na_, nk_ = na_;
  auto fetch = [&](int te, int tf, int u) {
    const float2* T = tau + (long)(D.slot + u) * nv2;
    const float2* K = kap + (long)(D.slot + u) * nv2;
    const int e = te * GT + ty, f = tf * GT + tx;
    const bool in = e < nv && f < nv;
    na_ = in ? T[(long)e * nv + f] : make_float2(0.f, 0.f);
    nb_ = in ? K[(long)e * nv + f] : make_float2(0.f, 0.f);
    const int fr = tf * GT + ty, ec = te * GT + tx;
    const bool ok = fr < nv && ec < nv;
    nt_ = ok ? T[(long)fr * nv + ec] : make_float2(0.f, 0.f);
    nk_ = ok ? K[(long)fr * nv + ec] : make_float2(0.f, 0.f);
  };
  dd part = dd_make(0.0f);
  // one row's 16 elements of a tile (16 lanes share ty), as row_norms8
  auto magnitude = [&](float v, long mat, int tcol, int row) {
    if (rowpart) {
      float x = v * v;
#pragma unroll
      for (int w = 8; w > 0; w >>= 1) x += __shfl_xor_sync(0xffffffffu, x, w);
      float n = sqrtf(x);
      if (__any_sync(0xffffffffu, !square_in_range(x))) {
        n = v;
#pragma unroll
        for (int w = 8; w > 0; w >>= 1) n = fmaxf(n, __shfl_xor_sync(0xffffffffu, n, w));
        n *= 4.0f;
      }
      if (tx == 0 && row < nv) rowpart[(mat * ((nv + GT - 1) / GT) + tcol) * nv + row] = n;
    } else if (rowmax) {
#pragma unroll
      for (int w = 8; w > 0; w >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, w));
      if (tx == 0 && row < nv) atomicMax(rowmax + mat * nv + row, __float_as_uint(v));
    }
  };
  int t = blockIdx.x, te = 0, tf = 0, buf = 0;
  if (t < nup) {
    decode(t, &te, &tf);
    fetch(te, tf, 0);
  }
  while (t < nup) {
    const int tn = t + gridDim.x;
    int ten = 0, tfn = 0;
    if (tn < nup) decode(tn, &ten, &tfn);
    const int E0 = te * GT, F0 = tf * GT;
    const int e = E0 + ty, f = F0 + tx;
    const bool inside = e < nv && f < nv;
    const float w = (te == tf) ? 1.0f : 2.0f;
    dd2 acc[OCT];  // outputs of tau and of kappa, packed: half the instructions
#pragma unroll
    for (int o = 0; o < OCT; ++o) acc[o] = {f2_set(0.f, 0.f), f2_set(0.f, 0.f)};
    for (int u = 0; u < ns; ++u) {
      tT[buf][ty][tx] = nt_;
      tK[buf][ty][tx] = nk_;
      const dd2 a = {f2_set(na_.x, nb_.x), f2_set(na_.y, nb_.y)};
      // the next slot's (or the next tile's first slot's) loads fly during
      // this slot's arithmetic
      if (u + 1 < ns) fetch(te, tf, u + 1);
      else if (tn < nup) fetch(ten, tfn, 0);
      __syncthreads();
      // c T + c sgn dg T^T = c (T + sgn dg T^T) with sgn = +-1, dg in {0, 1}:
      // the two signed combinations are formed once per slot
      const float du = dgf[u];
      const float2 xt = tT[buf][tx][ty], xk = tK[buf][tx][ty];
      const f32x2 du2 = f2_set(du, du);
      const dd2 at = {f2_mul(du2, f2_set(xt.x, xk.x)), f2_mul(du2, f2_set(xt.y, xk.y))};
      const dd2 sp = dd_add_fast(a, at), sm = dd_sub_fast(a, at);
      const f32x2 np = fl_neg(sp.hi), nm = fl_neg(sm.hi);
      const float4* cu = cf2 + u * OCT;
#pragma unroll
      for (int o = 0; o < OCT; ++o) {
        if (o < oc) {
          const float4 c = cu[o];
          const bool pos = (posmask >> o) & 1u;
          dd_fma_into(acc[o], dd2{f2_set(c.x, c.y), f2_set(c.z, c.w)}, pos ? sp : sm, pos ? np : nm);
        }
      }
      buf ^= 1;
    }
#pragma unroll
    for (int o = 0; o < OCT; ++o) {
      if (o < oc) {
        dd at, ak;
        acc[o] = quick_two_sum(acc[o].hi, acc[o].lo);
        f2_get(acc[o].hi, &at.hi, &ak.hi);
        f2_get(acc[o].lo, &at.lo, &ak.lo);
        if (inside) part = dd_add(part, dd_mul_f(dd_mul(lamw[o], dd_mul(at, ak)), w));
        if (want_sig) {
          const dd v = dd_mul(sqd[o], at);
          const long mat = D.out + D.o_begin + o;
          float2* S = sig + mat * nv2;
          if (inside) S[(long)e * nv + f] = make_float2(v.hi, v.lo);
          magnitude(inside ? fabsf(v.hi) : 0.0f, mat, tf, e);
          if (te != tf) {
            sA[ty][tx] = make_float2(v.hi, v.lo);
            __syncthreads();
            const int fr = F0 + ty, ec = E0 + tx;
            const float sg = sgnf[o];
            const bool ok = fr < nv && ec < nv;
            if (ok) S[(long)fr * nv + ec] = make_float2(sg * sA[tx][ty].x, sg * sA[tx][ty].y);
            magnitude(ok ? fabsf(sA[tx][ty].x) : 0.0f, mat, te, fr);
            __syncthreads();
          }
        }
      }
    }
    t = tn;
    te = ten;
    tf = tfn;
  }
  double pd = dd_to_double(part);
  for (int o = 16; o > 0; o >>= 1) pd += __shfl_down_sync(0xffffffffu, pd, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = pd;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int wv = 0; wv < GNT / 32; ++wv) s += red[wv];
    e_part[(long)blockIdx.y * gridDim.x + blockIdx.x] = s;
  }
  if (want_sig && blockIdx.x == 0 && threadIdx.x < oc)
    sig_sign[D.out + D.o_begin + threadIdx.x] = (lam[threadIdx.x] >= 0.0) ? 1.0 : -1.0;
}

// n regulariser values for tests: r1[k] = R1(delta[k]), y[k] = exp(-s delta^2)
__global__ void regularize_test_kernel(int n, const double* delta, double s, double* r1, double* y) {
  __shared__ RegTables R;
  reg_tables_load(R);
  __syncthreads();
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
    // this value beside another one of the list, as the pairs of the epilogue
    const dd p = dd_from_double(delta[k]), q = dd_from_double(delta[n - 1 - k]);
    dd2 r, z;
    regularize(dd2{f2_set(p.hi, q.hi), f2_set(p.lo, q.lo)}, dd_from_double(s), R, &r, &z);
    dd a, b;
    float other;
    f2_get(r.hi, &a.hi, &other);
    f2_get(r.lo, &a.lo, &other);
    f2_get(z.hi, &b.hi, &other);
    f2_get(z.lo, &b.lo, &other);
    r1[k] = dd_to_double(a);
    y[k] = dd_to_double(b);
  }
}

}  // namespace

int eps_to_dd(int n, const double* eps, float2* out, cudaStream_t st) {
  if (n <= 0) return DSRG_FNO_OK;
  eps_dd_kernel<<<ceil_div(n, 256), 256, 0, st>>>(n, eps, out);
  DSRG_LAUNCH_CHECK();
  return DSRG_FNO_OK;
}

// The regulariser table of the current device, filled on first use.
static int ensure_reg_tables() {
  static std::mutex mu;
  static bool ready[64] = {};
  int dev = 0;
  DSRG_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return DSRG_FNO_ERR_UNSUPPORTED;
  std::lock_guard<std::mutex> lk(mu);
  if (!ready[dev]) {
    // on a private stream, waited for: later kernels of every stream see it
    cudaStream_t s0;
    DSRG_CUDA(cudaStreamCreateWithFlags(&s0, cudaStreamNonBlocking));
    reg_tables_fill_kernel<<<1, 64, 0, s0>>>();
    DSRG_LAUNCH_CHECK();
    DSRG_CUDA(cudaStreamSynchronize(s0));
    DSRG_CUDA(cudaStreamDestroy(s0));
    ready[dev] = true;
  }
  return DSRG_FNO_OK;
}

// Device address of the current device's regulariser tables (filled first).
int reg_tables_device(const RegTables** out) {
  DSRG_TRY(ensure_reg_tables());
  void* p = nullptr;
  DSRG_CUDA(cudaGetSymbolAddress(&p, g_reg));
  *out = static_cast<const RegTables*>(p);
  return DSRG_FNO_OK;
}

__global__ void hole_particle_dd_kernel(Geometry g, const double* __restrict__ eps, float2* __restrict__ out) {
  const long R = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (R >= (long)g.nh * g.np) return;
  const int i = (int)(R / g.np), a = (int)(R - (long)i * g.np);
  const dd v = dd_from_double(eps[i] - eps[g.nc + a]);
  out[R] = make_float2(v.hi, v.lo);
}

// hp[i np + a] = eps_i - eps_a (hole i, particle a) in double-float: the
// denominator Delta^{ij}_{ab} = hp[i a] + hp[j b] of the fused epilogue.
int hole_particle_dd(const Geometry& g, const double* eps, float2* out, cudaStream_t st) {
  const long n = (long)g.nh * g.np;
  if (n <= 0) return DSRG_FNO_OK;
  hole_particle_dd_kernel<<<ceil_div(n, 256), 256, 0, st>>>(g, eps, out);
  DSRG_LAUNCH_CHECK();
  return DSRG_FNO_OK;
}

int pair_epilogue_dd(const Geometry& g, const double* eps, const float2* eps_dd, const int2* pairs, int npairs,
                     const float2* nu, float2* tau, float2* kap, double* ts, cudaStream_t st) {
  if (npairs <= 0) return DSRG_FNO_OK;
  DSRG_TRY(ensure_reg_tables());
  dim3 grid(ceil_div(g.np, EPI_ROWS), npairs);
  pair_epilogue_dd_kernel<<<grid, 256, 0, st>>>(g, eps, eps_dd, pairs, nu, tau, kap, ts);
  DSRG_LAUNCH_CHECK();
  return DSRG_FNO_OK;
}

int dress_dd(const Geometry& g, const DressDesc* d_desc, int ndesc, int ncc, const DressAux& aux,
             const float2* tau, const float2* kap, float2* sig, double* sig_sign, double* e_part, bool want_sig,
             unsigned* rowmax, float* rowpart, cudaStream_t st) {
  if (ncc > 0) {
    dim3 grid(DRESS_TILE_BLOCKS, ncc);
    dress_core_dd_kernel<<<grid, 256, 0, st>>>(g.nv, d_desc, tau, kap, sig, sig_sign, e_part, want_sig ? 1 : 0, rowmax,
                                               rowpart);
    DSRG_LAUNCH_CHECK();
  }
  if (ndesc > ncc) {
    dim3 grid(DRESS_TILE_BLOCKS, ndesc - ncc);
    dress_dd_kernel<DRESS_OC><<<grid, GNT, 0, st>>>(g.nv, g.na, d_desc + ncc, aux, tau, kap, sig, sig_sign,
                                                    e_part + (long)ncc * DRESS_TILE_BLOCKS, want_sig ? 1 : 0,
                                                    rowmax, rowpart);
    DSRG_LAUNCH_CHECK();
  }
  return DSRG_FNO_OK;
}

int regularize_test(int n, const double* delta, double s, double* r1, double* y, cudaStream_t st) {
  if (n <= 0) return DSRG_FNO_OK;
  DSRG_TRY(ensure_reg_tables());
  regularize_test_kernel<<<ceil_div(n, 256), 256, 0, st>>>(n, delta, s, r1, y);
  DSRG_LAUNCH_CHECK();
  return DSRG_FNO_OK;
}

}  // namespace dsrg
