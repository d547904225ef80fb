// Pieces of the divide-and-conquer eigensolver of a symmetric tridiagonal
// matrix that work on one node or one root (eig_dc.cu launches them).  They
// compile for the host too, where a test replays the whole solve.
//
// Method: Cuppen (Numer. Math. 36, 1981) with the deflation of Dongarra and
// Sorensen (SIAM J. Sci. Stat. Comput. 8, 1987), the secular equation by the
// rational iteration of Li ("Solving secular equations stably and
// efficiently", 1994), and vectors from the recomputed z of Gu and Eisenstat
// (SIAM J. Matrix Anal. Appl. 16, 1995), which makes them orthogonal to
// working precision however close the roots are.
#pragma once
#include <math.h>

namespace dsrg {
namespace dc {

#ifdef __CUDACC__
#define DC_HD __host__ __device__ __forceinline__
#else
#define DC_HD inline
#endif

constexpr double DC_EPS = 1.1102230246251565e-16;  // 2^-53
constexpr int DC_LEAF = 8;                         // largest leaf

// levels of the tree over n rows, leaves of at most DC_LEAF
DC_HD int dc_levels(int n) {
  int l = 0;
  while ((n + (1 << l) - 1) >> l > DC_LEAF) ++l;
  return l;
}
// first row of node t on level l (the nodes of level l + 1 halve them)
DC_HD int dc_bound(int n, int l, int t) { return (int)(((long)t * n) >> l); }

// rows of the largest node of level l (a node is at most one row longer than another)
DC_HD int dc_node_rows(int n, int l) { return (n + (1 << l) - 1) >> l; }
// shared memory of the deflation on level l: sorted d and z, keys, order, type and
// flag of every row of a node
constexpr int DC_DEFLATE_ROW_BYTES = 8 + 8 + 8 + 4 + 1 + 1;
DC_HD int dc_deflate_bytes(int n, int l) { return DC_DEFLATE_ROW_BYTES * dc_node_rows(n, l); }

// 1 / x, 1 / sqrt(x) and sqrt(x) from a float32 estimate r and the binomial series in
// what it leaves, e = 1 - x r and 1 - x r^2: 1 / x = r (1 - e)^-1 = r (1 + e + e^2 +
// ...), 1 / sqrt(x) = r (1 - e)^-1/2 = r (1 + e / 2 + 3 e^2 / 8 + ...), up to e^2.  With
// |e| below 2^-22 and 2^-20 the rest is under 2^-60, the roundings leave relative
// errors of 1, 3/2 and 5/2 units of 2^-53.  Chains of 3 to 5 float64 instructions
// where the library's take 15 to 30; an SM has two float64 lanes, and a chain of
// float64 operations is what most steps of the solver wait for.
DC_HD double dc_rcp(double x) {
#ifdef __CUDA_ARCH__
  const float f = __double2float_rn(x), a = fabsf(f);
  if (!(a > 1e-37f && a < 1e37f)) return 1.0 / x;
  const double r = (double)__frcp_rn(f), e = fma(-x, r, 1.0);
  return fma(r, fma(e, e, e), r);
#else
  return 1.0 / x;
#endif
}
DC_HD double dc_rsqrt(double x) {
#ifdef __CUDA_ARCH__
  const float f = __double2float_rn(x);
  if (!(f > 1e-36f && f < 1e37f)) return 1.0 / sqrt(x);
  const double r = (double)rsqrtf(f), e = fma(-x * r, r, 1.0);
  return fma(r * e, fma(e, 0.375, 0.5), r);
#else
  return 1.0 / sqrt(x);
#endif
}
DC_HD double dc_sqrt(double x) {
#ifdef __CUDA_ARCH__
  const float f = __double2float_rn(x);
  if (!(f > 1e-36f && f < 1e37f)) return sqrt(x);
  return x * dc_rsqrt(x);
#else
  return sqrt(x);
#endif
}

// The lanes that share one root or one node: a serial one (host) and a warp.
struct SerialLane {
  DC_HD int id() const { return 0; }
  DC_HD int count() const { return 1; }
  DC_HD double sum(double x) const { return x; }
  DC_HD void sum4(double&, double&, double&, double&) const {}
  DC_HD double prod(double x) const { return x; }
};

#ifdef __CUDACC__
struct WarpLane {
  __device__ __forceinline__ int id() const { return threadIdx.x & 31; }
  __device__ __forceinline__ int count() const { return 32; }
  __device__ __forceinline__ double sum(double x) const {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
  }
  // four sums at once: the lanes halve the values before they halve themselves
  // (6 additions instead of 20)
  __device__ __forceinline__ void sum4(double& a, double& b, double& c, double& d) const {
    const bool h = threadIdx.x & 16, g = threadIdx.x & 8;
    const double u = (h ? c : a) + __shfl_xor_sync(0xffffffffu, h ? a : c, 16);
    const double v = (h ? d : b) + __shfl_xor_sync(0xffffffffu, h ? b : d, 16);
    double x = (g ? v : u) + __shfl_xor_sync(0xffffffffu, g ? u : v, 8);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    a = __shfl_sync(0xffffffffu, x, 0);
    b = __shfl_sync(0xffffffffu, x, 8);
    c = __shfl_sync(0xffffffffu, x, 16);
    d = __shfl_sync(0xffffffffu, x, 24);
  }
  __device__ __forceinline__ double prod(double x) const {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x *= __shfl_xor_sync(0xffffffffu, x, o);
    return x;
  }
};
#endif

// Deflation of one node.  d, z, type: eigenvalues of both children in
// ascending order, their entries of the unit coupling vector (weight rho > 0)
// and 1 or 3 for a column with rows of the first or of the second child;
// order: their columns (node-local).  Columns whose z is negligible, or whose
// d is so close to the next one's that rotating the two columns makes one z
// zero at a cost below tol, keep their d as an eigenvalue.  Out: kcol, kd, kz,
// ktype of the K kept columns (ascending d; type 2: rows of both children),
// dcol, dval of the m - K others, and the rotations in the order to apply
// (p' = c p + s q, q' = c q - s p on columns p, q).
struct Rotation {
  int p, q;
  double c, s;
};
// flag[r]: dc_flag of column r and the one before it, formed beforehand (in
// parallel): the serial scan tests a pair itself only after a rotation or a
// deflation has come between.
DC_HD bool dc_close(double dp, double zp, double dc, double zc, double tol) {
  return fabs((dc - dp) * zp * zc) <= tol * (zp * zp + zc * zc);
}
DC_HD unsigned char dc_flag(int r, const double* d, const double* z, double rho, double tol) {
  const bool small = !(rho * fabs(z[r]) > tol);
  const bool close = r > 0 && dc_close(d[r - 1], z[r - 1], d[r], z[r], tol);
  return (unsigned char)((small ? 1 : 0) | (close ? 2 : 0));
}
DC_HD int dc_deflate(int m, const int* order, const double* d, const double* z, const unsigned char* flag,
                     const unsigned char* type, double rho, double tol, int* kcol, double* kd, double* kz, unsigned char* ktype, int* dcol, double* dval, Rotation* rot, int* nrot) {
  int K = 0, nd = 0, nr = 0, prev = -1;
  double dp = 0.0, zp = 0.0;
  int tp = 0;
  bool as_sorted = true;  // dp, zp are the sorted column prev's own
  for (int r = 0; r < m; ++r) {
    double dc = d[r], zc = z[r];
    int tc = type[r];
    if (flag[r] & 1) {
      dcol[nd] = order[r];
      dval[nd++] = dc;
      continue;
    }
    if (prev >= 0) {
      // the rotation leaves (dc - dp) zp zc / (zp^2 + zc^2) off the diagonal
      const double w2 = zp * zp + zc * zc;
      const bool close = as_sorted && prev == r - 1 ? (flag[r] & 2) != 0 : dc_close(dp, zp, dc, zc, tol);
      as_sorted = !close;
      if (close) {
        const double w = sqrt(w2), co = zc / w, si = -zp / w;
        rot[nr++] = Rotation{order[prev], order[r], co, si};
        if (tc != tp) tc = 2;
        dcol[nd] = order[prev];
        dval[nd++] = dp * co * co + dc * si * si;
        dc = dp * si * si + dc * co * co;
        zc = w;
      } else {
        kcol[K] = order[prev];
        kd[K] = dp;
        kz[K] = zp;
        ktype[K++] = (unsigned char)tp;
      }
    }
    prev = r;
    dp = dc;
    zp = zc;
    tp = tc;
  }
  if (prev >= 0) {
    kcol[K] = order[prev];
    kd[K] = dp;
    kz[K] = zp;
    ktype[K++] = (unsigned char)tp;
  }
  *nrot = nr;
  return K;
}

// Root j of 1 + rho sum_i z_i^2 / (d_i - x) = 0 (d ascending and distinct):
// x = d[*base] + *eta with the nearer pole as base, eta to full relative
// accuracy.
template <typename Lane>
DC_HD void dc_secular(int K, int j, const double* d, const double* z, double rho, const Lane& L, int* base, double* eta) {
  const int l0 = L.id(), nl = L.count();
  if (K == 1) {
    *base = 0;
    *eta = rho * z[0] * z[0];
    return;
  }
  const bool last = j == K - 1;
  int b = j;
  double lo, hi, y;
  if (!last) {
    // which half: the sign at the midpoint, poles j and j + 1 set apart
    const double gap = d[j + 1] - d[j], mid = 0.5 * gap;
    double s = 0.0;
    for (int i = l0; i < K; i += nl)
      if (i != j && i != j + 1) s += z[i] * z[i] * dc_rcp((d[i] - d[j]) - mid);
    const double c = 1.0 + rho * L.sum(s);
    const double za = rho * z[j] * z[j], zb = rho * z[j + 1] * z[j + 1];
    const double g = c + za / (-mid) + zb / (gap - mid);
    // start: c + za / (0 - x) + zb / (gap - x) = 0 (x from pole j)
    const double a = c * gap + za + zb, q = za * gap, disc = sqrt(fabs(a * a - 4.0 * c * q));
    if (g >= 0.0) {
      lo = 0.0;
      hi = mid;
      y = a > 0.0 ? 2.0 * q / (a + disc) : (a - disc) / (2.0 * c);
    } else {
      b = j + 1;
      lo = -mid;
      hi = 0.0;
      // the same equation from pole j + 1: x' = x - gap
      const double a2 = -c * gap + za + zb, q2 = -zb * gap;
      const double d2 = sqrt(fabs(a2 * a2 - 4.0 * c * q2));
      y = a2 < 0.0 ? 2.0 * q2 / (a2 - d2) : (a2 + d2) / (2.0 * c);
    }
  } else {
    double s = 0.0;
    for (int i = l0; i < K; i += nl) s += z[i] * z[i];
    lo = 0.0;
    hi = rho * L.sum(s) * (1.0 + 4.0 * DC_EPS);
    y = rho * z[j] * z[j];
  }
  if (!(y > lo && y < hi)) y = 0.5 * (lo + hi);
  const double db = d[b];
  for (int it = 0; it < 80; ++it) {
    // psi: poles up to j (all terms negative), phi: the others (all positive)
    double ps = 0.0, dps = 0.0, ph = 0.0, dph = 0.0;
    for (int i = l0; i < K; i += nl) {
      const double iv = dc_rcp((d[i] - db) - y);
      const double t = z[i] * z[i] * iv;
      if (i <= j) {
        ps += t;
        dps = fma(t, iv, dps);
      } else {
        ph += t;
        dph = fma(t, iv, dph);
      }
    }
    L.sum4(ps, dps, ph, dph);
    ps *= rho;
    dps *= rho;
    ph *= rho;
    dph *= rho;
    const double w = 1.0 + ps + ph;
    if (fabs(w) <= 4.0 * DC_EPS * (1.0 + ph - ps)) break;
    if (w < 0.0) lo = y;
    else hi = y;
    double st;
    if (!last) {
      const double p1 = (d[j] - db) - y, p2 = (d[j + 1] - db) - y;
      const double c = w - p1 * dps - p2 * dph, a = (p1 + p2) * w - p1 * p2 * (dps + dph), q = p1 * p2 * w;
      const double disc = dc_sqrt(fabs(a * a - 4.0 * q * c));
      st = a <= 0.0 ? (a - disc) * dc_rcp(2.0 * c) : 2.0 * q * dc_rcp(a + disc);
    } else {
      // psi by r + s / (d_j - x): value and slope at y
      const double p1 = -y, r = 1.0 + ps - p1 * dps;
      // r + p1^2 dps / (p1 - st) = 0
      st = p1 + p1 * p1 * dps * dc_rcp(r);
    }
    if (!(w * st < 0.0)) st = -w * dc_rcp(dps + dph);
    double yn = y + st;
    if (!(yn > lo && yn < hi)) yn = 0.5 * (lo + hi);
    if (yn == y || yn == lo || yn == hi) break;
    y = yn;
  }
  *base = b;
  *eta = y;
}

// |z_i| for which the computed roots are exact (Gu and Eisenstat), up to the
// common factor that normalising the vectors removes.
template <typename Lane>
DC_HD double dc_zhat(int K, int i, const double* d, const int* base, const double* eta, double zi, const Lane& L) {
  double p = 1.0;
  for (int j = L.id(); j < K; j += L.count()) {
    const double num = (d[i] - d[base[j]]) - eta[j];
    p *= j == i ? num : num * dc_rcp(d[i] - d[j]);
  }
  p = sqrt(fabs(L.prod(p)));
  return zi < 0.0 ? -p : p;
}

}  // namespace dc
}  // namespace dsrg
