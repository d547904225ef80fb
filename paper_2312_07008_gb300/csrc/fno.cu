// Truncation of the natural orbitals (Eqs. 9, 10 and the near-degeneracy
// widening of Sec. 2) and small helpers of the discarded-orbital correction.
#include "kernels.h"

namespace dsrg {

namespace {

// Decision of one block; the sums run in ascending order in one thread, the same
// arithmetic on every call.
//   mode 0: smallest N' with sum_{p<=N'} n_p >= (thr/100) sum_all n_p   (Eq. 10)
//   mode 1: N' = ceil(thr/100 * nv)                                       (Eq. 9)
//   mode 2: number of n_p >= thr                                          (n_kappa)
//   mode 3: N' = thr, rounded and clamped
// then while N' < nv and n_{N'} - n_{N'+1} < ratio * max(n_{N'}, n_{N'+1}): N'++.
// The ONs and their running sums pass through shared memory in pieces: one chain
// of additions instead of two over global loads (n = 1200: 89 us).
constexpr int CUT_PIECE = 2048;
__global__ void __launch_bounds__(256) truncate_kernel(int nv, const double* __restrict__ ons, int mode, double thr,
                                                       double ratio, int* nkept) {
  __shared__ double s[CUT_PIECE];
  __shared__ double s_sum;
  __shared__ int s_k;
  if (threadIdx.x == 0) {
    s_sum = 0.0;
    s_k = nv;
  }
  if (mode == 0) {
    // pass 0: the total; pass 1: the first running sum to reach the target (the
    // sums of a short list are still there)
    const int pieces = (nv + CUT_PIECE - 1) / CUT_PIECE;
    double target = 0.0;
    for (int pass = 0; pass < 2; ++pass) {
      for (int i = 0; i < pieces; ++i) {
        const int p0 = i * CUT_PIECE, m = min(CUT_PIECE, nv - p0);
        if (pass == 0 || pieces > 1) {
          __syncthreads();
          for (int p = threadIdx.x; p < m; p += 256) s[p] = ons[p0 + p];
          __syncthreads();
          if (threadIdx.x == 0) {
            double c = s_sum;
            for (int p = 0; p < m; ++p) {
              c += s[p];
              s[p] = c;
            }
            s_sum = c;
          }
          __syncthreads();
        }
        if (pass == 1) {
          int k = nv;
          for (int p = threadIdx.x; p < m; p += 256)
            if (s[p] >= target) {
              k = p0 + p + 1;
              break;
            }
          if (k < nv) atomicMin(&s_k, k);
        }
      }
      if (pass == 0) {
        target = thr / 100.0 * s_sum;
        __syncthreads();
        if (threadIdx.x == 0) s_sum = 0.0;
      }
    }
  } else if (mode == 2) {
    int c = 0;
    for (int p = threadIdx.x; p < nv; p += 256) c += (ons[p] >= thr) ? 1 : 0;
    __syncthreads();
    if (threadIdx.x == 0) s_k = 0;
    __syncthreads();
    atomicAdd(&s_k, c);
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  int k = s_k;
  if (mode == 1) k = (int)ceil(thr / 100.0 * nv - 1e-12);
  if (mode == 3) k = (int)rint(fmin(fmax(thr, 0.0), (double)nv));
  k = k < 0 ? 0 : (k > nv ? nv : k);
  while (k > 0 && k < nv && (ons[k - 1] - ons[k]) < ratio * fmax(ons[k - 1], ons[k])) ++k;
  *nkept = k;
}

__global__ void symmetrize_kernel(int n, double* D) {
  long idx = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (idx >= (long)n * n) return;
  int e = (int)(idx / n), f = (int)(idx % n);
  if (e >= f) return;
  double a = D[(long)e * n + f], b = D[(long)f * n + e];
  double s = 0.5 * (a + b);
  D[(long)e * n + f] = s;
  D[(long)f * n + e] = s;
}

// W[e][l] = eps_v[e] * V[e][l]  (first ncol columns, leading dimension ld)
__global__ void scale_rows_kernel(int nv, int ncol, long ld, const double* __restrict__ ev,
                                  const double* __restrict__ V, double* __restrict__ W) {
  long idx = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (idx >= (long)nv * ncol) return;
  int e = (int)(idx / ncol), l = (int)(idx % ncol);
  W[(long)e * ncol + l] = ev[e] * V[(long)e * ld + l];
}

// Bf[Q][h][x] = B[Q][h][x] for the active particle columns
__global__ void copy_active_kernel(long rows, int na, int np, int npf, const double* __restrict__ B,
                                   double* __restrict__ Bf) {
  long idx = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (idx >= rows * na) return;
  long r = idx / na;
  int x = (int)(idx % na);
  Bf[r * npf + x] = B[r * np + x];
}

__global__ void finite_kernel(const double* __restrict__ x, long n, int* flag) {
  long idx = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (idx < n && !isfinite(x[idx])) atomicExch(flag, 1);
}

}  // namespace

int truncate_ons(int nv, const double* ons, int mode, double thr, double ratio, int* nkept, cudaStream_t st) {
  truncate_kernel<<<1, 256, 0, st>>>(nv, ons, mode, thr, ratio, nkept);
  DSRG_LAUNCH_CHECK();
  return DSRG_FNO_OK;
}

int symmetrize(int n, double* D, cudaStream_t st) {
  long n2 = (long)n * n;
  if (n2 == 0) return DSRG_FNO_OK;
  symmetrize_kernel<<<ceil_div(n2, 256), 256, 0, st>>>(n, D);
  DSRG_LAUNCH_CHECK();
  return DSRG_FNO_OK;
}

int scale_rows(int nv, int ncol, long ld, const double* ev, const double* V, double* W, cudaStream_t st) {
  long n = (long)nv * ncol;
  if (n == 0) return DSRG_FNO_OK;
  scale_rows_kernel<<<ceil_div(n, 256), 256, 0, st>>>(nv, ncol, ld, ev, V, W);
  DSRG_LAUNCH_CHECK();
  return DSRG_FNO_OK;
}

int copy_active(long rows, int na, int np, int npf, const double* B, double* Bf, cudaStream_t st) {
  long n = rows * na;
  if (n == 0) return DSRG_FNO_OK;
  copy_active_kernel<<<ceil_div(n, 256), 256, 0, st>>>(rows, na, np, npf, B, Bf);
  DSRG_LAUNCH_CHECK();
  return DSRG_FNO_OK;
}

int check_finite(const double* x, long n, int* flag, cudaStream_t st) {
  if (n <= 0) return DSRG_FNO_OK;
  finite_kernel<<<ceil_div(n, 256), 256, 0, st>>>(x, n, flag);
  DSRG_LAUNCH_CHECK();
  return DSRG_FNO_OK;
}

}  // namespace dsrg
