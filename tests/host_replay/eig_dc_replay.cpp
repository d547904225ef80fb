// Host replay of the divide-and-conquer stages (csrc/eig_dc.cuh): the same
// element functions as the kernels, called by plain loops with a serial lane.
// Input: tridiagonal d[n], e[n-1]; output: eigenvalues and vectors (columns),
// and the numbers of deflated columns and of rotations over all nodes.
#include <algorithm>
#include <cstring>
#include <vector>

#include "eig_dc.cuh"

using namespace dsrg::dc;
using std::vector;

static void leaf_jacobi(int m, vector<double>& A, vector<double>& Q) {
  for (int i = 0; i < m * m; ++i) Q[i] = i / m == i % m;
  for (int sweep = 0; sweep < 30; ++sweep) {
    double off = 0.0;
    for (int p = 0; p < m; ++p)
      for (int q = p + 1; q < m; ++q) {
        const double apq = A[p * m + q];
        off = std::max(off, fabs(apq));
        if (fabs(apq) < 1e-300) continue;
        const double th = (A[q * m + q] - A[p * m + p]) / (2 * apq);
        const double t = (th >= 0 ? 1 : -1) / (fabs(th) + sqrt(1 + th * th)), c = 1 / sqrt(1 + t * t), s = t * c;
        for (int k = 0; k < m; ++k) {
          const double a = A[p * m + k], b = A[q * m + k];
          A[p * m + k] = c * a - s * b;
          A[q * m + k] = s * a + c * b;
        }
        for (int k = 0; k < m; ++k) {
          double a = A[k * m + p], b = A[k * m + q];
          A[k * m + p] = c * a - s * b;
          A[k * m + q] = s * a + c * b;
          a = Q[k * m + p], b = Q[k * m + q];
          Q[k * m + p] = c * a - s * b;
          Q[k * m + q] = s * a + c * b;
        }
      }
    if (off < 1e-18) break;
  }
}

extern "C" void eig_dc_replay(int n, const double* d0, const double* e, double* lam, double* Qout, int* counts) {
  const int L = dc_levels(n);
  const size_t ld = n;
  vector<double> d(d0, d0 + n), Q(ld * n, 0.0), Q2(ld * n);
  double big = 0.0;
  for (int i = 0; i < n; ++i) big = std::max(big, std::max(fabs(d0[i]), i + 1 < n ? fabs(e[i]) : 0.0));
  const double tol = 4 * DC_EPS * big;
  counts[0] = counts[1] = 0;
  for (int t = 1; t < (1 << L); ++t) {
    const int k = dc_bound(n, L, t) - 1;
    d[k] -= fabs(e[k]);
    d[k + 1] -= fabs(e[k]);
  }
  for (int t = 0; t < (1 << L); ++t) {
    const int lo = dc_bound(n, L, t), m = dc_bound(n, L, t + 1) - lo;
    vector<double> A(m * m, 0.0), q(m * m);
    for (int i = 0; i < m; ++i) {
      A[i * m + i] = d[lo + i];
      if (i + 1 < m) A[i * m + i + 1] = A[(i + 1) * m + i] = e[lo + i];
    }
    leaf_jacobi(m, A, q);
    for (int i = 0; i < m; ++i) {
      d[lo + i] = A[i * m + i];
      for (int k = 0; k < m; ++k) Q[(lo + i) * ld + lo + k] = q[k * m + i];
    }
  }
  const SerialLane S;
  for (int l = L - 1; l >= 0; --l) {
    std::fill(Q2.begin(), Q2.end(), 0.0);
    for (int t = 0; t < (1 << l); ++t) {
      const int lo = dc_bound(n, l, t), hi = dc_bound(n, l, t + 1), mid = dc_bound(n, l + 1, 2 * t + 1), m = hi - lo;
      const double ec = e[mid - 1], rho = 2 * fabs(ec);
      vector<int> ord(m), kcol(m), dcol(m);
      vector<unsigned char> ty(m), kty(m);
      vector<double> sd(m), sz(m), kd(m), kz(m), dval(m);
      vector<Rotation> rot(m);
      for (int i = 0; i < m; ++i) ord[i] = i;
      std::stable_sort(ord.begin(), ord.end(), [&](int a, int b) { return d[lo + a] < d[lo + b]; });
      for (int r = 0; r < m; ++r) {
        const int c = lo + ord[r];
        sd[r] = d[c];
        ty[r] = c < mid ? 1 : 3;
        sz[r] = (c < mid ? Q[c * ld + mid - 1] : (ec < 0 ? -1 : 1) * Q[c * ld + mid]) * sqrt(0.5);
      }
      vector<unsigned char> fl(m);
      for (int r = 0; r < m; ++r) fl[r] = dc_flag(r, sd.data(), sz.data(), rho, tol);
      int nr = 0;
      const int K = dc_deflate(m, ord.data(), sd.data(), sz.data(), fl.data(), ty.data(), rho, tol, kcol.data(), kd.data(), kz.data(),
                               kty.data(), dcol.data(), dval.data(), rot.data(), &nr);
      counts[0] += m - K;
      counts[1] += nr;
      for (int r = 0; r < nr; ++r)
        for (int k = lo; k < hi; ++k) {
          double &a = Q[(lo + rot[r].p) * ld + k], &b = Q[(lo + rot[r].q) * ld + k];
          const double x = a, y = b;
          a = rot[r].c * x + rot[r].s * y;
          b = rot[r].c * y - rot[r].s * x;
        }
      vector<int> base(K);
      vector<double> eta(K), zh(K), u(K);
      for (int j = 0; j < K; ++j) dc_secular(K, j, kd.data(), kz.data(), rho, S, &base[j], &eta[j]);
      for (int i = 0; i < K; ++i) zh[i] = dc_zhat(K, i, kd.data(), base.data(), eta.data(), kz[i], S);
      for (int j = 0; j < K; ++j) {
        double s = 0.0;
        for (int i = 0; i < K; ++i) {
          u[i] = zh[i] / ((kd[i] - kd[base[j]]) - eta[j]);
          s += u[i] * u[i];
        }
        s = 1 / sqrt(s);
        for (int i = 0; i < K; ++i) {  // a kept column has rows of its own child only, type 2 of both
          const int a = kty[i] == 3 ? mid : lo, b = kty[i] == 1 ? mid : hi;
          for (int k = a; k < b; ++k) Q2[(lo + j) * ld + k] += u[i] * s * Q[(lo + kcol[i]) * ld + k];
        }
        d[lo + j] = kd[base[j]] + eta[j];
      }
      for (int r = 0; r < m - K; ++r) {
        d[lo + K + r] = dval[r];
        memcpy(&Q2[(lo + K + r) * ld + lo], &Q[(lo + dcol[r]) * ld + lo], sizeof(double) * m);
      }
    }
    std::swap(Q, Q2);
  }
  memcpy(lam, d.data(), sizeof(double) * n);
  memcpy(Qout, Q.data(), sizeof(double) * ld * n);
}
