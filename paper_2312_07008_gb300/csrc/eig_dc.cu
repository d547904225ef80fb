// Symmetric eigensolver of the larger matrices (Eq. 8), float64:
//   1. Householder reduction to tridiagonal form (Golub and Van Loan Sec. 8.3),
//      one cooperative launch;
//   2. divide and conquer on the tridiagonal matrix (eig_dc.cuh), a few
//      launches per level;
//   3. the reflectors applied to its vectors, one launch.
//
// What bounds it.  GB300 has two float64 lanes per SM, so the arithmetic (n^3
// FMAs each for 1 and 3, about n^3 / 2 for the last merge) is spread over all
// SMs: 5.7e6 clocks of the whole chip for n = 1200.  The rest are the n grid
// barriers of the reduction.  A Jacobi solve moves the whole matrix n - 1
// times per sweep with a barrier each time and needs 4 to 10 sweeps.  Measured
// (D_vv-like matrices): n = 1200 16.8 ms (column-pair Jacobi in double-float 97
// ms), n = 203 1.6 (9.1), n = 90 0.80 (2.7), n = 3600 0.37 s (4.8 s).  Against
// the first form of these kernels (27, 3.1, 1.5 ms): leaves of 8 rows instead of
// 16, deflation by all threads of a block, reciprocals and roots by iteration
// instead of the library's, scalar work by one warp beside the rows.
#include <algorithm>

#include "eig_dc.cuh"
#include "kernels.h"

namespace dsrg {

namespace {

using namespace dc;

constexpr int TNT = 256;                   // threads per block of the reduction
constexpr int TNW = TNT / 32;
constexpr size_t TRI_SMEM = 200 * 1024;
// the deflation of the largest matrix beside its 1040 bytes of static shared memory
constexpr int DC_DEFLATE_SMEM = DC_DEFLATE_ROW_BYTES * EIG_DC_MAX_N;
static_assert(DC_DEFLATE_SMEM + 1040 <= 232448, "shared memory per block");
constexpr double RSQRT2 = 0.70710678118654752440;

// ------------------------------------------------------------- reduction
struct TriArgs {
  int n, rows;      // rows held per block (cyclic: block b has rows b, b + G, ...)
  double* A;        // [n][n]; on return row j holds reflector v_j at k > j
  double *d, *e, *beta;
  double* pub;      // [2][2][n]: p and row j + 1 of even and odd steps
  unsigned* bar;    // arrivals, zero at launch
  int* status;      // [1] = 1: a barrier wait expired
  long long spin_limit;
};

// All blocks are co-resident (cooperative launch); arrivals only count up, so
// a barrier is one atomic and a poll.  Bounded; false once any wait expired.
__device__ bool tri_barrier(const TriArgs& P, unsigned target) {
  __shared__ int s_ok;
  __syncthreads();
  if (gridDim.x == 1) return true;
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(P.bar, 1u);
    volatile int* st = P.status + 1;
    long long it = 0;
    int ok = 1;
    unsigned cnt;
    while (true) {
      asm volatile("ld.acquire.gpu.u32 %0, [%1];" : "=r"(cnt) : "l"(P.bar) : "memory");
      if ((int)(cnt - target) >= 0) break;
      if (++it > P.spin_limit) {
        atomicExch(P.status + 1, 1);
        ok = 0;
        break;
      }
      if ((it & 255) == 0 && *st != 0) {
        ok = 0;
        break;
      }
    }
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

__device__ __forceinline__ double warp_sum(double x) { return WarpLane().sum(x); }

// Step j: every block knows row j of the reduced matrix (r), forms the same
// reflector from it, and in ONE pass over its own rows applies the rank-2
// update left from step j - 1 and multiplies by the new reflector:
//   A -= v w^T + w v^T with w = beta p - K v, K = beta^2 (p.v) / 2, so
//   A_ik -= (beta v_i) p_k + (beta p_i - 2 K v_i) v_k,   p'_i = sum_k A_ik v'_k.
// The products p' and row j + 1 are published, and every block forms p'.v' and
// row j + 1 of the next matrix by itself.  A is read and written once per step,
// from shared memory as long as a block's rows fit (SM).  A step is a chain of
// two block sums, the rows and one grid barrier: n = 203 1.95 -> 1.59 ms for the
// whole solve, n = 1200 18.5 -> 16.8, against a reflector formed before the rows.
// (Words tagged with the step's number and polled for in place of the barrier: n =
// 90 0.80 -> 0.75, n = 203 1.57, n = 300 2.30 -> 2.39, twice the bytes.)
template <bool SM>
__global__ void __launch_bounds__(TNT) tridiag_kernel(TriArgs P) {
  extern __shared__ double smem[];
  const int n = P.n, G = gridDim.x, b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  double* pv = smem;        // p of the previous step
  double* v0 = pv + n;      // v of the previous step
  double* v1 = v0 + n;      // v of this step
  double* rp = v1 + n;      // products of the own rows
  double* As = rp + P.rows; // own rows (SM)
  __shared__ double part[TNT], sc[5];
  auto row_ptr = [&](int li) { return SM ? As + (long)li * n : P.A + (long)(b + li * G) * n; };
  // sum of the threads' parts, by warp 0 (scalar work costs every warp that
  // repeats it 16 clocks an instruction of the SM's float64 lanes)
  auto total = [&]() {
    static_assert(TNW == 8, "a tree of eight");
    const double* x = part + lane;
    return warp_sum(((x[0] + x[32]) + (x[64] + x[96])) + ((x[128] + x[160]) + (x[192] + x[224])));
  };
  if (SM) {
    for (int li = warp; b + li * G < n; li += TNW) {
      const double* src = P.A + (long)(b + li * G) * n;
      double* dst = As + (long)li * n;
      for (int k = lane; k < n; k += 32) dst[k] = src[k];
    }
  }
  double dj = P.A[0], alpha = P.A[1], s2 = 0.0;  // dj, alpha: warp 0's
  for (int k = 1 + tid; k < n; k += TNT) {
    const double r = P.A[k];
    v1[k] = r;
    if (k > 1) s2 = fma(r, r, s2);
  }
  unsigned target = G;
  if (!tri_barrier(P, target)) return;  // every block has read its part of A
  double beta0 = 0.0, K2 = 0.0;         // of the previous step (none yet)
  for (int j = 0; j < n - 2; ++j) {
    // ---- reflector from row j (v1 holds A[j][k], k > j; s2 this thread's part of |r_{k > j + 1}|^2)
    // The rows need v_j only in their products, and there only element j + 1 is
    // not yet known: warp 0 forms the reflector while the others update the rows
    // and multiply by the elements beyond.
    part[tid] = s2;
    __syncthreads();
    double* pp = P.pub + (long)(j & 1) * 2 * n;
    double* pr = pp + n;
    const int li0 = b > j ? 0 : (j - b) / G + 1;  // first own row above j
    const int kbeg = (j + 1) & ~31;
    if (warp == 0) {
      const double sig = total();
      double ej = alpha, bt = 0.0, v = alpha;
      if (sig > 0.0) {
        // beta = 1 / (nrm (nrm + |alpha|))
        const double q = fma(alpha, alpha, sig), r = dc_rsqrt(q), nrm = q * r;
        ej = alpha > 0.0 ? -nrm : nrm;
        bt = r * r * dc_rcp(fma(fabs(alpha), r, 1.0));
        v = alpha - ej;
      }
      if (lane == 0) {
        sc[0] = bt;
        sc[1] = v;
        if (b == (j + 1) % G) {
          P.d[j] = dj;
          P.e[j] = ej;
          P.beta[j] = bt;
        }
      }
    }
    if (!SM || warp > 0) {  // rows in global memory: warp 0 takes its share of them as well
      for (int li = li0 + (SM ? warp - 1 : warp); b + li * G < n; li += SM ? TNW - 1 : TNW) {
        const int i = b + li * G;
        double* row = row_ptr(li);
        const double c1 = -beta0 * v0[i], c2 = fma(K2, v0[i], -beta0 * pv[i]);
        // four partial sums: a chain of float64 FMAs waits for each of them
        double acc[4] = {0.0, 0.0, 0.0, 0.0};
        const bool pub = i == j + 1;
        for (int k0 = kbeg + lane; k0 < n; k0 += 128) {
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int k = k0 + 32 * u;
            if (k > j && k < n) {
              double a = row[k];
              if (j > 0) {
                a = fma(c1, pv[k], fma(c2, v0[k], a));
                row[k] = a;
              }
              if (k > j + 1) acc[u] = fma(a, v1[k], acc[u]);
              if (pub) __stcg(pr + k, a);
            }
          }
        }
        const double ps = warp_sum((acc[0] + acc[1]) + (acc[2] + acc[3]));
        if (lane == 0) rp[li] = ps;
      }
    }
    __syncthreads();
    const double beta = sc[0];
    for (int li = li0 + tid; b + li * G < n; li += TNT) {
      const int i = b + li * G;
      const double p = fma(row_ptr(li)[j + 1], sc[1], rp[li]);
      __stcg(pp + i, p);
    }
    if (tid == TNT - 1) v1[j + 1] = sc[1];
    if (b == (j + 1) % G)
      for (int k = j + 1 + tid; k < n; k += TNT) P.A[(long)j * n + k] = k == j + 1 ? sc[1] : v1[k];
    // ---- p, p.v and row j + 1 of the next matrix
    const int i = j + 1;
    target += G;
    if (!tri_barrier(P, target)) return;
    double* vt = v0;
    v0 = v1;
    v1 = vt;
    double dot = 0.0;
    for (int k = i + tid; k < n; k += TNT) {
      pv[k] = __ldcg(pp + k);
      v1[k] = __ldcg(pr + k);
      dot = fma(pv[k], v0[k], dot);
    }
    part[tid] = dot;
    __syncthreads();
    beta0 = beta;
    if (warp == 0) {
      const double s = total();
      const double k2 = beta * (beta * s), vi = v0[i], pi = pv[i];  // beta^2 may overflow
      const double c1 = -beta * vi, c2 = fma(k2, vi, -beta * pi);
      dj = fma(c1, pi, fma(c2, vi, v1[i]));
      alpha = fma(c1, pv[i + 1], fma(c2, v0[i + 1], v1[i + 1]));
      if (lane == 0) {
        sc[2] = k2;
        sc[3] = c1;
        sc[4] = c2;
      }
      if (j == n - 3 && b == (n - 1) % G) {  // the last 2 x 2, by the owner of row n - 1
        const double pl = pv[n - 1], vl = v0[n - 1];
        if (lane == 0) {
          P.d[n - 2] = dj;
          P.e[n - 2] = alpha;
          P.d[n - 1] = fma(-beta * vl, pl, fma(fma(k2, vl, -beta * pl), vl, row_ptr((n - 1) / G)[n - 1]));
        }
      }
    }
    __syncthreads();
    K2 = sc[2];
    const double c1 = sc[3], c2 = sc[4];
    s2 = 0.0;
    for (int k = i + 1 + tid; k < n; k += TNT) {
      const double r = fma(c1, pv[k], fma(c2, v0[k], v1[k]));
      v1[k] = r;
      if (k > i + 1) s2 = fma(r, r, s2);
    }
  }
}

// -------------------------------------------------------- divide and conquer
struct DcArgs {
  int n, levels;
  const double *d, *e;
  double *lam;                       // eigenvalue of each column
  double *kd, *kz, *eta, *zhat, *dval;
  int *kcol, *kpos, *dcol, *base, *colpos;
  Rotation* rot;
  int4* node;                        // per node of the level: K, rotations, columns of types 1 + 2, of type 1
  double* U;                         // [n][n]: row (lo + j) = vector of root j in the node's kept columns
  double *Qin, *Qout;                // column-major
  double* anorm;
  int level;
};

// max |d|, |e| (one block)
__global__ void __launch_bounds__(256) dc_norm_kernel(DcArgs P) {
  __shared__ double red[256];
  double m = 0.0;
  for (int i = threadIdx.x; i < P.n; i += 256) {
    m = fmax(m, fabs(P.d[i]));
    if (i < P.n - 1) m = fmax(m, fabs(P.e[i]));
  }
  red[threadIdx.x] = m;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w) red[threadIdx.x] = fmax(red[threadIdx.x], red[threadIdx.x + w]);
    __syncthreads();
  }
  if (threadIdx.x == 0) *P.anorm = red[0];
}

// One warp per leaf: cyclic two-sided Jacobi (round-robin pairs) on the leaf's
// tridiagonal block with the couplings to its neighbours taken off.
__global__ void __launch_bounds__(32) dc_leaf_kernel(DcArgs P) {
  constexpr int M = DC_LEAF;
  __shared__ double A[M][M + 1], Q[M][M + 1], cs[M / 2], sn[M / 2];
  __shared__ int pp[M / 2], qq[M / 2];
  const int lane = threadIdx.x, leaf = blockIdx.x, n = P.n;
  const int lo = dc_bound(n, P.levels, leaf), hi = dc_bound(n, P.levels, leaf + 1), m = hi - lo;
  const int me = (m + 1) & ~1, half = me / 2;
  for (int t = lane; t < M * M; t += 32) {
    const int i = t / M, k = t % M;
    double a = 0.0;
    if (i < m && k < m) {
      if (i == k) {
        a = P.d[lo + i];
        if (i == 0 && lo > 0) a -= fabs(P.e[lo - 1]);
        if (i == m - 1 && hi < n) a -= fabs(P.e[hi - 1]);
      } else if (i - k == 1 || k - i == 1) {
        a = P.e[lo + min(i, k)];
      }
    }
    A[i][k] = a;
    Q[i][k] = i == k ? 1.0 : 0.0;
  }
  __syncwarp();
  const double anorm = *P.anorm, floor_ = 4.0 * DC_EPS * anorm;  // the deflation's tolerance
  const double unit = dc_rcp(anorm);                             // (unused when all entries are 0)
  for (int sweep = 0; sweep < 16 && m > 1; ++sweep) {
    bool any = false;
    for (int r = 0; r < me - 1; ++r) {
      if (lane < half) {
        const int i1 = lane == 0 ? 0 : (lane - 1 + r) % (me - 1) + 1;
        const int i2 = (me - 2 - lane + r) % (me - 1) + 1;
        const int p = min(i1, i2), q = max(i1, i2);
        double c = 1.0, s = 0.0;
        if (q < m) {
          const double apq = A[p][q];
          if (fabs(apq) > floor_) {
            // tan in float32: any t gives an orthogonal rotation, and the next
            // sweep takes off what this one leaves
            const float th = (float)((A[q][q] - A[p][p]) * unit) / (2.0f * (float)(apq * unit));
            const float t = copysignf(1.0f, th) / (fabsf(th) + sqrtf(fmaf(th, th, 1.0f)));
            c = dc_rsqrt(fma((double)t, (double)t, 1.0));
            s = (double)t * c;
            any = any || t != 0.0f;
          }
        }
        pp[lane] = p;
        qq[lane] = q;
        cs[lane] = c;
        sn[lane] = s;
      }
      __syncwarp();
      for (int t = lane; t < half * m; t += 32) {  // columns of A and Q
        const int h = t / m, k = t % m, p = pp[h], q = qq[h];
        const double c = cs[h], s = sn[h];
        if (q < m && s != 0.0) {
          const double a = A[k][p], bq = A[k][q];
          A[k][p] = c * a - s * bq;
          A[k][q] = s * a + c * bq;
          const double x = Q[k][p], y = Q[k][q];
          Q[k][p] = c * x - s * y;
          Q[k][q] = s * x + c * y;
        }
      }
      __syncwarp();
      for (int t = lane; t < half * m; t += 32) {  // rows of A
        const int h = t / m, k = t % m, p = pp[h], q = qq[h];
        const double c = cs[h], s = sn[h];
        if (q < m && s != 0.0) {
          const double a = A[p][k], bq = A[q][k];
          A[p][k] = c * a - s * bq;
          A[q][k] = s * a + c * bq;
        }
      }
      __syncwarp();
    }
    if (!__any_sync(0xffffffffu, any)) break;
  }
  for (int t = lane; t < m * m; t += 32) {
    const int c = t / m, k = t % m;
    P.Qout[(long)(lo + c) * n + lo + k] = Q[k][c];
  }
  if (lane < m) P.lam[lo + lane] = A[lane][lane];
}

// order-preserving integer key of a double (integer compares run at full rate)
__device__ __forceinline__ long long dc_key(double x) {
  const long long b = __double_as_longlong(x);
  return b < 0 ? (long long)(0x8000000000000000ULL) - b : b;
}

// One block per node: coupling vector, sort, deflation, grouping of the kept
// columns by the child whose rows they have.
__global__ void __launch_bounds__(256) dc_deflate_kernel(DcArgs P) {
  extern __shared__ double sm[];
  const int n = P.n, l = P.level, t = blockIdx.x;
  const int lo = dc_bound(n, l, t), hi = dc_bound(n, l, t + 1), mid = dc_bound(n, l + 1, 2 * t + 1), m = hi - lo;
  double* sd = sm;                                            // [m] sorted
  double* sz = sd + m;                                        // [m]
  long long* key = reinterpret_cast<long long*>(sz + m);      // [m] unsorted keys; then ci and kty
  int* ord = reinterpret_cast<int*>(key + m);                 // [m]
  unsigned char* ty = reinterpret_cast<unsigned char*>(ord + m);  // [m]
  unsigned char* fl = ty + m;                                     // [m]
  __shared__ int s_k, s_nr;
  const double ec = P.e[mid - 1], rho = 2.0 * fabs(ec);
  for (int i = threadIdx.x; i < m; i += 256) key[i] = dc_key(P.lam[lo + i]);
  __syncthreads();
  for (int i = threadIdx.x; i < m; i += 256) {
    const long long ki = key[i];
    int r = 0;
    for (int k = 0; k < m; ++k) r += key[k] < ki || (key[k] == ki && k < i);
    ord[r] = i;
    sd[r] = P.lam[lo + i];
    const bool top = lo + i < mid;
    const double q = P.Qin[(long)(lo + i) * n + (top ? mid - 1 : mid)];
    sz[r] = (!top && ec < 0.0 ? -RSQRT2 : RSQRT2) * q;
    ty[r] = top ? 1 : 3;
  }
  __syncthreads();
  const double tol = 4.0 * DC_EPS * *P.anorm;
  int* ci = reinterpret_cast<int*>(key);                          // [m] ranks of the columns with a z to speak of
  unsigned char* kty = reinterpret_cast<unsigned char*>(ci + m);  // [m]
  __shared__ int s_cnt[256];
  const int per = (m + 255) / 256, r0 = min(m, (int)threadIdx.x * per), r1 = min(m, r0 + per);
  int cnt = 0;
  for (int r = r0; r < r1; ++r) {
    fl[r] = dc_flag(r, sd, sz, rho, tol);
    cnt += !(fl[r] & 1);
  }
  s_cnt[threadIdx.x] = cnt;
  __syncthreads();
  for (int w = 1; w < 256; w <<= 1) {  // inclusive scan
    const int x = (int)threadIdx.x >= w ? s_cnt[threadIdx.x - w] : 0;
    __syncthreads();
    s_cnt[threadIdx.x] += x;
    __syncthreads();
  }
  int pos = s_cnt[threadIdx.x] - cnt;
  const int kept = s_cnt[255];
  for (int r = r0, q = pos; r < r1; ++r)
    if (!(fl[r] & 1)) ci[q++] = r;
  __syncthreads();
  bool close = false;
  for (int q = threadIdx.x + 1; q < kept; q += 256) close = close || dc_close(sd[ci[q - 1]], sz[ci[q - 1]], sd[ci[q]], sz[ci[q]], tol);
  if (!__syncthreads_or(close)) {
    // no pair to rotate (the usual case): the split by z is all of it
    for (int r = r0; r < r1; ++r) {
      if (!(fl[r] & 1)) {
        P.kcol[lo + pos] = ord[r];
        P.kd[lo + pos] = sd[r];
        P.kz[lo + pos] = sz[r];
        kty[pos++] = ty[r];
      } else {
        P.dcol[lo + r - pos] = ord[r];
        P.dval[lo + r - pos] = sd[r];
      }
    }
    if (threadIdx.x == 0) {
      s_k = kept;
      s_nr = 0;
    }
  } else if (threadIdx.x == 0) {
    int nr = 0;
    s_k = dc_deflate(m, ord, sd, sz, fl, ty, rho, tol, P.kcol + lo, P.kd + lo, P.kz + lo, kty, P.dcol + lo, P.dval + lo,
                     P.rot + lo, &nr);
    s_nr = nr;
  }
  __syncthreads();
  const int K = s_k;
  int c1 = 0, c2 = 0;
  for (int i = threadIdx.x; i < K; i += 256) {
    c1 += kty[i] == 1;
    c2 += kty[i] == 2;
  }
  __shared__ int s_c1, s_c2;
  if (threadIdx.x == 0) s_c1 = s_c2 = 0;
  __syncthreads();
  atomicAdd(&s_c1, c1);
  atomicAdd(&s_c2, c2);
  __syncthreads();
  c1 = s_c1;
  c2 = s_c2;
  for (int i = threadIdx.x; i < K; i += 256) {
    const int ti = kty[i];
    int r = ti == 1 ? 0 : (ti == 2 ? c1 : c1 + c2);
    for (int k = 0; k < i; ++k) r += kty[k] == ti;
    P.kpos[lo + i] = r;
    P.colpos[lo + r] = P.kcol[lo + i];
  }
  if (threadIdx.x == 0) P.node[t] = make_int4(K, s_nr, c1 + c2, c1);
}

__device__ __forceinline__ int dc_node_of(int n, int l, int i) {
  int t = (int)((((long)i + 1) << l) / n);
  while (t > 0 && dc_bound(n, l, t) > i) --t;
  while (dc_bound(n, l, t + 1) <= i) ++t;
  return t;
}

// The deflating rotations on the columns: a thread per row goes through the
// list (a column rotated as q may be the next rotation's p: kept in a register).
__device__ void dc_rotate_rows(const DcArgs& P, int row) {
  const int n = P.n, t = dc_node_of(n, P.level, row), lo = dc_bound(n, P.level, t);
  const int nr = P.node[t].y;
  const Rotation* R = P.rot + lo;
  double* Q = P.Qin + (long)lo * n + row;
  int cc = -1;
  double cv = 0.0;
  constexpr int B = 8;
  for (int k0 = 0; k0 < nr; k0 += B) {
    double x[B], y[B];
#pragma unroll
    for (int u = 0; u < B; ++u)
      if (k0 + u < nr) {  // no column is a q twice, nor a q after it was a p: the loads can run ahead
        x[u] = Q[(long)R[k0 + u].p * n];
        y[u] = Q[(long)R[k0 + u].q * n];
      }
#pragma unroll
    for (int u = 0; u < B; ++u)
      if (k0 + u < nr) {
        const Rotation r = R[k0 + u];
        const double a = r.p == cc ? cv : x[u];
        Q[(long)r.p * n] = r.c * a + r.s * y[u];
        cv = r.c * y[u] - r.s * a;
        cc = r.q;
        Q[(long)r.q * n] = cv;
      }
  }
}

// Blocks [0, rot_blocks): the rotations; the others: a warp per column, which
// solves the secular equation of a kept one and hands on a deflated one's value
// (one warp per block: the warps spread over all SMs' float64 lanes).
__global__ void __launch_bounds__(32) dc_secular_kernel(DcArgs P, int rot_blocks) {
  const int n = P.n;
  if ((int)blockIdx.x < rot_blocks) {
    const int row = blockIdx.x * 32 + threadIdx.x;
    if (row < n) dc_rotate_rows(P, row);
    return;
  }
  const int i = (int)blockIdx.x - rot_blocks;
  const int t = dc_node_of(n, P.level, i), lo = dc_bound(n, P.level, t), mid = dc_bound(n, P.level + 1, 2 * t + 1);
  const int K = P.node[t].x, j = i - lo;
  const WarpLane L;
  if (j >= K) {
    if (L.id() == 0) P.lam[i] = P.dval[lo + j - K];
    return;
  }
  const double rho = 2.0 * fabs(P.e[mid - 1]);
  int b;
  double eta;
  dc_secular(K, j, P.kd + lo, P.kz + lo, rho, L, &b, &eta);
  if (L.id() == 0) {
    P.base[i] = b;
    P.eta[i] = eta;
    P.lam[i] = P.kd[lo + b] + eta;
  }
}

__global__ void __launch_bounds__(32) dc_zhat_kernel(DcArgs P) {
  const int n = P.n, i = blockIdx.x;
  const int t = dc_node_of(n, P.level, i), lo = dc_bound(n, P.level, t), K = P.node[t].x, k = i - lo;
  if (k >= K) return;
  const WarpLane L;
  const double z = dc_zhat(K, k, P.kd + lo, P.base + lo, P.eta + lo, P.kz[i], L);
  if (L.id() == 0) P.zhat[i] = z;
}

// U row (lo + j): unit vector of root j over the node's kept columns, in the
// grouped order; a deflated column's vector is copied to its place in Qout.
__global__ void __launch_bounds__(32) dc_vectors_kernel(DcArgs P) {
  const int n = P.n, i = blockIdx.x, lane = threadIdx.x;
  const int l = P.level, t = dc_node_of(n, l, i), lo = dc_bound(n, l, t), hi = dc_bound(n, l, t + 1);
  const int K = P.node[t].x, j = i - lo;
  if (j >= K) {
    const double* src = P.Qin + (long)(lo + P.dcol[lo + j - K]) * n;
    double* dst = P.Qout + (long)i * n;
    for (int k = lo + lane; k < hi; k += 32) dst[k] = src[k];
    return;
  }
  const double db = P.kd[lo + P.base[i]], eta = P.eta[i];
  double* u = P.U + (long)i * n;
  double s = 0.0;
  for (int k = lane; k < K; k += 32) {
    const double x = P.zhat[lo + k] * dc_rcp((P.kd[lo + k] - db) - eta);
    u[P.kpos[lo + k]] = x;
    s = fma(x, x, s);
  }
  s = 1.0 / sqrt(warp_sum(s));
  for (int k = lane; k < K; k += 32) u[P.kpos[lo + k]] *= s;
}

// Qout[:, lo + j] = sum_k Qin[:, column k] U[j][k] over the rows of one child
// (blockIdx.z & 1), whose rows only the columns of its own type and type 2
// have.  T x T tiles of 256 threads: with two float64 lanes per SM a small tile
// already runs at the arithmetic's rate, and its many blocks fill the chip.
template <int T>
__global__ void __launch_bounds__(256) dc_gemm_kernel(DcArgs P) {
  constexpr int TK = 16, R = T / 16;
  __shared__ double As[TK][T + 1], Bs[TK][T + 1];
  __shared__ int s_col[TK];
  const int n = P.n, l = P.level, t = blockIdx.z >> 1, half = blockIdx.z & 1;
  const int lo = dc_bound(n, l, t), hi = dc_bound(n, l, t + 1), mid = dc_bound(n, l + 1, 2 * t + 1);
  const int4 nd = P.node[t];
  const int K = nd.x, r0 = half ? mid : lo, r1 = half ? hi : mid;
  const int kb = half ? nd.w : 0, ke = half ? K : nd.z;
  const int m0 = blockIdx.y * T, n0 = r0 + blockIdx.x * T;
  if (m0 >= K || n0 >= r1) return;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  double acc[R][R] = {};
  for (int k0 = kb; k0 < ke; k0 += TK) {
    if (threadIdx.x < TK) s_col[threadIdx.x] = k0 + threadIdx.x < ke ? P.colpos[lo + k0 + threadIdx.x] : -1;
    for (int x = threadIdx.x; x < T * TK; x += 256) {
      const int k = x % TK, mm = x / TK;
      As[k][mm] = (m0 + mm < K && k0 + k < ke) ? P.U[(long)(lo + m0 + mm) * n + k0 + k] : 0.0;
    }
    __syncthreads();
    for (int x = threadIdx.x; x < T * TK; x += 256) {
      const int nn = x % T, k = x / T, c = s_col[k];
      Bs[k][nn] = (c >= 0 && n0 + nn < r1) ? P.Qin[(long)(lo + c) * n + n0 + nn] : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < TK; ++k) {
      double a[R], q[R];
#pragma unroll
      for (int u = 0; u < R; ++u) {
        a[u] = As[k][ty + 16 * u];
        q[u] = Bs[k][tx + 16 * u];
      }
#pragma unroll
      for (int u = 0; u < R; ++u)
#pragma unroll
        for (int w = 0; w < R; ++w) acc[u][w] = fma(a[u], q[w], acc[u][w]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int u = 0; u < R; ++u)
#pragma unroll
    for (int w = 0; w < R; ++w) {
      const int j = m0 + ty + 16 * u, r = n0 + tx + 16 * w;
      if (j < K && r < r1) P.Qout[(long)(lo + j) * n + r] = acc[u][w];
    }
}

// A group of BK consecutive reflectors, applied from the highest row down, takes
// q to q + sum_t s_t v_t with s = W x, x_u = v_u . q and W lower triangular:
// s_t = -beta_t (x_t + sum_{u < t} s_u v_u . v_t).  wy[group]: the ten entries of
// W, row by row (one warp per group).
constexpr int BK = 4, WY = 10;
__device__ __forceinline__ int dc_group_row(int n, int g, int t) { return n - 3 - g * BK - t; }
__global__ void __launch_bounds__(32) dc_wy_kernel(int n, const double* __restrict__ Vh, const double* __restrict__ beta,
                                                   double* __restrict__ wy) {
  const int g = blockIdx.x, lane = threadIdx.x;
  double m[BK][BK] = {}, b[BK], w[BK][BK] = {};
#pragma unroll
  for (int t = 0; t < BK; ++t) {
    const int jt = dc_group_row(n, g, t);
    b[t] = jt < 0 ? 0.0 : beta[jt];
#pragma unroll
    for (int s = 0; s < t; ++s) {
      const int js = dc_group_row(n, g, s);
      double x = 0.0;
      if (jt >= 0)
        for (int k = js + 1 + lane; k < n; k += 32) x = fma(Vh[(long)js * n + k], Vh[(long)jt * n + k], x);
      m[s][t] = warp_sum(x);
    }
  }
#pragma unroll
  for (int t = 0; t < BK; ++t) {
    w[t][t] = -b[t];
#pragma unroll
    for (int u = 0; u < t; ++u) {
      double x = 0.0;
#pragma unroll
      for (int s = u; s < t; ++s) x = fma(w[s][u], m[s][t], x);
      w[t][u] = -b[t] * x;
    }
  }
  if (lane == 0) {
    int o = 0;
#pragma unroll
    for (int t = 0; t < BK; ++t)
#pragma unroll
      for (int u = 0; u <= t; ++u) wy[(long)g * WY + o++] = w[t][u];
  }
}

// V[:, c] = H_0 H_1 ... H_{n-3} Q[:, c]: a warp per column, the column in shared
// memory (each lane owns the rows equal to it modulo 32), no block barrier.
// BK reflectors at a time: independent chains.
__global__ void __launch_bounds__(256) dc_back_kernel(int n, const double* __restrict__ Vh, const double* __restrict__ wy,
                                                      const double* __restrict__ Q,
                                                      const double* __restrict__ lam, double* __restrict__ V, double* A,
                                                      int* status) {
  extern __shared__ double sq[];
  const int lane = threadIdx.x & 31, wpb = blockDim.x >> 5, c = blockIdx.x * wpb + (threadIdx.x >> 5);
  if (c >= n) return;
  double* q = sq + (long)(threadIdx.x >> 5) * n;
  const WarpLane L;
  for (int k = lane; k < n; k += 32) q[k] = Q[(long)c * n + k];
  for (int g = 0; g * BK < n - 2; ++g) {
    int j[BK];
    double x[BK] = {0.0, 0.0, 0.0, 0.0}, w[WY];
    const double* v[BK];
#pragma unroll
    for (int t = 0; t < BK; ++t) {
      const int jt = dc_group_row(n, g, t);
      j[t] = jt < 0 ? n : jt;                // beyond the last reflector: no rows
      v[t] = Vh + (long)(jt < 0 ? 0 : jt) * n;
    }
#pragma unroll
    for (int u = 0; u < WY; ++u) w[u] = wy[(long)g * WY + u];
    const int top = dc_group_row(n, g, 0), low = top - BK + 1 < 0 ? 0 : top - BK + 1;
    int k = ((low + 1) & ~31) + lane;
    // rows up to the highest reflector's first one: masked
    if (k <= top) {
#pragma unroll
      for (int t = 0; t < BK; ++t)
        if (k < n && k > j[t]) x[t] = v[t][k] * q[k];
      k += 32;
      if (k <= top) {
#pragma unroll
        for (int t = 0; t < BK; ++t)
          if (k < n && k > j[t]) x[t] = fma(v[t][k], q[k], x[t]);
        k += 32;
      }
    }
#pragma unroll 4
    for (int kk = k; kk < n; kk += 32) {
      const double y = q[kk];
#pragma unroll
      for (int t = 0; t < BK; ++t)
        x[t] = fma(v[t][kk], y, x[t]);
    }
    L.sum4(x[0], x[1], x[2], x[3]);
    const double s[BK] = {w[0] * x[0], fma(w[1], x[0], w[2] * x[1]), fma(w[3], x[0], w[4] * x[1]) + w[5] * x[2],
                          fma(w[6], x[0], w[7] * x[1]) + fma(w[8], x[2], w[9] * x[3])};
    for (int kk = ((low + 1) & ~31) + lane; kk < k && kk < n; kk += 32) {
      double y = q[kk];
#pragma unroll
      for (int t = 0; t < BK; ++t)
        if (kk > j[t]) y = fma(s[t], v[t][kk], y);
      q[kk] = y;
    }
#pragma unroll 4
    for (int kk = k; kk < n; kk += 32) {
      const double y0 = fma(s[1], v[1][kk], fma(s[0], v[0][kk], q[kk]));  // (a missing reflector's s is 0)
      q[kk] = y0 + fma(s[3], v[3][kk], s[2] * v[2][kk]);
    }
  }
  for (int k = lane; k < n; k += 32) V[(long)k * n + c] = q[k];
  if (lane == 0) {
    const double x = lam[c];
    A[(long)c * n + c] = x;  // the reflectors lie above the diagonal
    if (!isfinite(x)) atomicExch(status, 1);
  }
}

__global__ void dc_roots_test_kernel(int n, const double* x, double* rcp, double* rsqrt, double* root) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    rcp[i] = dc_rcp(x[i]);
    rsqrt[i] = dc_rsqrt(x[i]);
    root[i] = dc_sqrt(x[i]);
  }
}

}  // namespace

int eig_dc_roots_test(int n, const double* x, double* rcp, double* rsqrt, double* sqrt, cudaStream_t st) {
  dc_roots_test_kernel<<<ceil_div(n, 256), 256, 0, st>>>(n, x, rcp, rsqrt, sqrt);
  DSRG_LAUNCH_CHECK();
  return DSRG_FNO_OK;
}

// A (n x n, symmetric) is destroyed: on return its diagonal holds the
// eigenvalues (any order) and V's columns the eigenvectors.  work:
// eig_work_doubles(n) doubles; status_dev: four zeroed ints; bar: zeroed.
int eig_dc(int n, double* A, double* V, double* work, unsigned* bar, int* status_dev, long long spin_limit, bool shared,
           cudaStream_t st) {
  const long n2 = (long)n * n;
  double *Q0 = work, *Q1 = work + n2, *U = work + 2 * n2;
  double* red = work + 3 * n2;                           // 2 EIG_MAX_BLOCKS
  double* x = work + 3 * n2 + 2 * EIG_MAX_BLOCKS + 16;   // EIG_DC_VECTORS n
  auto take = [&](int k) {
    double* p = x;
    x += (long)k * n;
    return p;
  };
  DcArgs D{};
  TriArgs T{};
  T.n = n;
  T.A = A;
  T.d = take(1);
  T.e = take(1);
  T.beta = take(1);
  T.pub = take(4);
  T.bar = bar;
  T.status = status_dev;
  T.spin_limit = spin_limit;
  D.n = n;
  D.levels = dc_levels(n);
  D.d = T.d;
  D.e = T.e;
  D.lam = take(1);
  D.kd = take(1);
  D.kz = take(1);
  D.eta = take(1);
  D.zhat = take(1);
  D.dval = take(1);
  D.rot = reinterpret_cast<Rotation*>(take(3));
  D.node = reinterpret_cast<int4*>(((uintptr_t)take(2) + 15) & ~(uintptr_t)15);
  x += 2;
  D.kcol = reinterpret_cast<int*>(take(3));
  D.kpos = D.kcol + n;
  D.dcol = D.kpos + n;
  D.base = D.dcol + n;
  D.colpos = D.base + n;
  double* wy = take(3);  // WY per group of BK reflectors
  D.anorm = red;
  D.U = U;
  int dev = 0, sms = 0;
  DSRG_CUDA(cudaGetDevice(&dev));
  DSRG_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  // rows per block: enough to amortise a barrier, few enough to use every SM's
  // two float64 lanes (a shared device keeps half the SMs to the others)
  const int per = shared ? 8 : 4;
  const int G = std::max(1, std::min(std::min(shared ? sms / 2 : sms, EIG_MAX_BLOCKS), ceil_div(n, per)));
  T.rows = ceil_div(n, G);
  const size_t vec = sizeof(double) * (3 * (size_t)n + T.rows), own = sizeof(double) * (size_t)n * T.rows;
  const bool in_smem = vec + own <= TRI_SMEM;
  const size_t smem = vec + (in_smem ? own : 0);
  if (smem > TRI_SMEM) return DSRG_FNO_ERR_UNSUPPORTED;
  auto kern = in_smem ? tridiag_kernel<true> : tridiag_kernel<false>;
  DSRG_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TRI_SMEM));
  void* args[] = {&T};
  DSRG_CUDA(cudaLaunchCooperativeKernel((const void*)kern, dim3(G), dim3(TNT), args, smem, st));
  DSRG_LAUNCH_CHECK();
  // a node's columns are written in its own rows only: the others stay zero
  DSRG_CUDA(cudaMemsetAsync(work, 0, 2 * n2 * sizeof(double), st));
  dc_norm_kernel<<<1, 256, 0, st>>>(D);
  DSRG_LAUNCH_CHECK();
  D.Qout = Q0;
  dc_leaf_kernel<<<1 << D.levels, 32, 0, st>>>(D);
  DSRG_LAUNCH_CHECK();
  DSRG_CUDA(cudaFuncSetAttribute(dc_deflate_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, DC_DEFLATE_SMEM));
  for (int l = D.levels - 1; l >= 0; --l) {
    std::swap(Q0, Q1);
    D.level = l;
    D.Qin = Q1;
    D.Qout = Q0;
    const int nodes = 1 << l, mmax = dc_node_rows(n, l), hmax = dc_node_rows(n, l + 1);
    dc_deflate_kernel<<<nodes, 256, dc_deflate_bytes(n, l), st>>>(D);
    DSRG_LAUNCH_CHECK();
    const int rb = ceil_div(n, 32);
    dc_secular_kernel<<<rb + n, 32, 0, st>>>(D, rb);
    DSRG_LAUNCH_CHECK();
    dc_zhat_kernel<<<n, 32, 0, st>>>(D);
    DSRG_LAUNCH_CHECK();
    dc_vectors_kernel<<<n, 32, 0, st>>>(D);
    DSRG_LAUNCH_CHECK();
    if (mmax < 512) dc_gemm_kernel<16><<<dim3(ceil_div(hmax, 16), ceil_div(mmax, 16), 2 * nodes), 256, 0, st>>>(D);
    else dc_gemm_kernel<32><<<dim3(ceil_div(hmax, 32), ceil_div(mmax, 32), 2 * nodes), 256, 0, st>>>(D);
    DSRG_LAUNCH_CHECK();
  }
  // columns per block: all SMs first, at most eight warps each
  const int wfit = (int)(TRI_SMEM / (sizeof(double) * (size_t)n));
  const int wpb = std::max(1, std::min(std::min(8, wfit), ceil_div(n, sms)));
  DSRG_CUDA(cudaFuncSetAttribute(dc_back_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TRI_SMEM));
  dc_wy_kernel<<<ceil_div(n - 2, BK), 32, 0, st>>>(n, A, T.beta, wy);
  DSRG_LAUNCH_CHECK();
  dc_back_kernel<<<ceil_div(n, wpb), 32 * wpb, sizeof(double) * (size_t)n * wpb, st>>>(n, A, wy, Q0, D.lam, V, A, status_dev);
  DSRG_LAUNCH_CHECK();
  return DSRG_FNO_OK;
}

}  // namespace dsrg
