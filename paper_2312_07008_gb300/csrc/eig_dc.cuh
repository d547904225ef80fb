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
constexpr int DC_LEAF = 16;                        // largest leaf

// levels of the tree over n rows, leaves of at most DC_LEAF
DC_HD int dc_levels(int n) {
  int l = 0;
  while ((n + (1 << l) - 1) >> l > DC_LEAF) ++l;
  return l;
}
// first row of node t on level l (the nodes of level l + 1 halve them)
DC_HD int dc_bound(int n, int l, int t) { return (int)(((long)t * n) >> l); }

// The lanes that share one root or one node: a serial one (host) and a warp.
struct SerialLane {
  DC_HD int id() const { return 0; }
  DC_HD int count() const { return 1; }
  DC_HD double sum(double x) const { return x; }
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
DC_HD int dc_deflate(int m, const int* order, double* d, double* z, unsigned char* type, double rho, double tol, int* kcol,
                     double* kd, double* kz, unsigned char* ktype, int* dcol, double* dval, Rotation* rot, int* nrot) {
  int K = 0, nd = 0, nr = 0, prev = -1;
  double dp = 0.0, zp = 0.0;
  int tp = 0;
  for (int r = 0; r < m; ++r) {
    double dc = d[r], zc = z[r];
    int tc = type[r];
    if (!(rho * fabs(zc) > tol)) {
      dcol[nd] = order[r];
      dval[nd++] = dc;
      continue;
    }
    if (prev >= 0) {
      const double t = dc - dp, w2 = zp * zp + zc * zc;
      // the rotation leaves t zp zc / w2 off the diagonal
      if (fabs(t * zp * zc) <= tol * w2) {
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
      if (i != j && i != j + 1) s += z[i] * z[i] / ((d[i] - d[j]) - mid);
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
    double ps = 0.0, dps = 0.0, ph = 0.0, dph = 0.0, er = 0.0;
    for (int i = l0; i < K; i += nl) {
      const double iv = 1.0 / ((d[i] - db) - y);
      const double t = z[i] * z[i] * iv, t2 = t * iv;
      er += fabs(t);
      if (i <= j) {
        ps += t;
        dps += t2;
      } else {
        ph += t;
        dph += t2;
      }
    }
    ps = rho * L.sum(ps);
    dps = rho * L.sum(dps);
    er = 1.0 + rho * L.sum(er);
    if (!last) {
      ph = rho * L.sum(ph);
      dph = rho * L.sum(dph);
    }
    const double w = 1.0 + ps + ph;
    if (fabs(w) <= 4.0 * DC_EPS * er) break;
    if (w < 0.0) lo = y;
    else hi = y;
    double st;
    if (!last) {
      const double p1 = (d[j] - db) - y, p2 = (d[j + 1] - db) - y;
      const double c = w - p1 * dps - p2 * dph, a = (p1 + p2) * w - p1 * p2 * (dps + dph), q = p1 * p2 * w;
      const double disc = sqrt(fabs(a * a - 4.0 * q * c));
      st = a <= 0.0 ? (a - disc) / (2.0 * c) : 2.0 * q / (a + disc);
    } else {
      // psi by r + s / (d_j - x): value and slope at y
      const double p1 = -y, r = 1.0 + ps - p1 * dps;
      // r + p1^2 dps / (p1 - st) = 0
      st = p1 + p1 * p1 * dps / r;
    }
    if (!(w * st < 0.0)) st = -w / (dps + dph);
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
    p *= j == i ? num : num / (d[i] - d[j]);
  }
  p = sqrt(fabs(L.prod(p)));
  return zi < 0.0 ? -p : p;
}

}  // namespace dc
}  // namespace dsrg
