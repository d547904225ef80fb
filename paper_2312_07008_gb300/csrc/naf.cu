// Natural auxiliary functions (Sec. 4: the compression of the auxiliary
// basis the paper proposes for the PT2 step).
//
// W_PQ = sum_{ia} B^P_{ia} B^Q_{ia} over the hole-particle DF factors is
// diagonalised, W = U diag(w) U^T (w descending), and the factors are
// rotated to the eigenvectors with w > threshold:
//   B'^K_{ia} = sum_Q U_QK B^Q_{ia}.
// In the fast form both contractions run in the residue form: W with 10 moduli
// (its entries are sums of nh np products), B' with 12 (B' enters every
// integral, as the rotation to the frozen natural orbitals does);
// the eigensolve is that of the natural orbitals.
#include <math.h>

#include <vector>

#include "kernels.h"

namespace dsrg {

int impl_naf(Workspace& ws, int32_t nh, int32_t np, int32_t naux, const double* B, double threshold, int precision,
             double* B_out, double* w_out, int32_t* naux_out, cudaStream_t st) {
  if (nh <= 0 || np <= 0 || naux <= 0 || !B || !B_out || !naux_out || !isfinite(threshold)) return DSRG_FNO_ERR_ARG;
  if (precision != DSRG_FNO_FP64 && precision != DSRG_FNO_SLICED_BF16) return DSRG_FNO_ERR_UNSUPPORTED;
  if (!is_device_ptr(B) || !is_device_ptr(B_out) || (w_out && !is_device_ptr(w_out))) return DSRG_FNO_ERR_ARG;
  const long L = (long)nh * np;
  if (L * 2 > (1L << 31) || (long)naux * naux >= (1L << 31)) return DSRG_FNO_ERR_UNSUPPORTED;
  const size_t n2 = (size_t)naux * naux;
  const bool fast = precision == DSRG_FNO_SLICED_BF16;
  const int kw = RES_MOD, kb = RES_MOD_X;
  const int qpad = pad64(naux);
  const size_t fixed = 3 * ws_bytes(n2, sizeof(double)) + ws_bytes(eig_work_doubles(naux), sizeof(double)) +
                       ws_bytes(naux + 16, sizeof(double)) + ws_bytes(naux + 16, sizeof(int)) + ws_bytes(8, sizeof(int));
  // Fast form: pairs ia that pass through the metric (its contraction index) and the
  // rotation (rows) at a time, all of them unless the memory that calls plan with is
  // too small; the planes of the one, then (reusing the space) of the other.
  long lw = L, lb = L;
  int capw = RES_PLAIN_CAP, capb = RES_PLAIN_CAP;
  auto planes = [&] {
    const size_t p1 = ws_bytes((size_t)kw * naux * pad64((int)lw), 2) + residue_exps_bytes(naux) + ws_bytes(16, sizeof(int)) +
                      ws_bytes(residue_plain_bytes(kw, naux, naux, capw), 1);
    const size_t p2 = ws_bytes((size_t)kb * lb * qpad, 2) + ws_bytes((size_t)kb * naux * qpad, 2) + residue_exps_bytes(lb) +
                      residue_exps_bytes(naux) + ws_bytes(16, sizeof(int)) + ws_bytes(residue_plain_bytes(kb, naux, lb, capb), 1);
    return std::max(p1, p2);
  };
  if (fast && fixed + planes() > ws.cap) {
    const size_t budget = device_budget(ws.cap);
    lw = residue_rows_at_a_time(kw, L, qpad, budget);
    lb = residue_rows_at_a_time(kb, L, qpad, budget);
    capw = residue_cap(kw, budget);
    capb = residue_cap(kb, budget);
  }
  const int lpad = pad64((int)lw);
  DSRG_TRY(ws_reserve(ws, fixed + (fast ? planes() : 0)));
  {
    int* flag = ws_take<int>(ws, 8);
    int h = 0;
    DSRG_CUDA(cudaMemsetAsync(flag, 0, sizeof(int), st));
    DSRG_TRY(check_finite(B, (long)naux * L, flag, st));
    DSRG_CUDA(cudaMemcpyAsync(&h, flag, sizeof(int), cudaMemcpyDeviceToHost, st));
    DSRG_CUDA(cudaStreamSynchronize(st));
    if (h) return DSRG_FNO_ERR_NONFINITE;
  }
  double* W = ws_take<double>(ws, n2);
  double* V = ws_take<double>(ws, n2);
  double* U = ws_take<double>(ws, n2);
  double* work = ws_take<double>(ws, eig_work_doubles(naux));
  double* w = ws_take<double>(ws, naux + 16);
  int* ib = ws_take<int>(ws, naux + 16);
  if (!ib) return DSRG_FNO_ERR_NOMEM;
  const size_t base = ws.off;
  int* status = ib;
  int* rank = ib + 8;
  // ---- W = B2 B2^T, B2 = B as naux rows of length nh np
  {
    DSRG_PHASE("phase_naf_metric", st);
    if (fast) {
      ws.off = base;
      __nv_bfloat16* pl = ws_take<__nv_bfloat16>(ws, (size_t)kw * naux * lpad);
      int* ex = reinterpret_cast<int*>(ws_take<char>(ws, residue_exps_bytes(naux)));
      uint16_t* res = reinterpret_cast<uint16_t*>(ws_take<char>(ws, residue_plain_bytes(kw, naux, naux, capw)));
      int* err = ws_take<int>(ws, 16);
      if (!err) return DSRG_FNO_ERR_NOMEM;
      DSRG_CUDA(cudaMemsetAsync(err, 0, sizeof(int), st));
      for (long l0 = 0; l0 < L; l0 += lw) {
        const int n = (int)std::min(lw, L - l0), kp = pad64(n);
        DSRG_TRY(residue_stage(kw, B + l0, naux, n, L, 1, kp, pl, ex, st));
        DSRG_TRY(residue_plain(kw, naux, naux, pl, ex, naux, 0, pl, ex, kp, 1.0, l0 > 0, W, naux, 0, res, capw, err, st));
      }
      int h = 0;
      DSRG_CUDA(cudaMemcpyAsync(&h, err, sizeof(int), cudaMemcpyDeviceToHost, st));
      DSRG_CUDA(cudaStreamSynchronize(st));
      if (h) return DSRG_FNO_ERR_TIMEOUT;
    } else {
      DSRG_TRY(gemm_f64(naux, naux, (int)L, 1.0, B, L, true, B, L, true, 0.0, W, naux, 1, 0, 0, 0, st));
    }
  }
  // ---- W = U diag(w) U^T, w descending
  {
    DSRG_PHASE("phase_naf_eigen", st);
    DSRG_TRY(symmetrize(naux, W, st));
    DSRG_TRY(eig_sym_jacobi(naux, W, V, work, status, 60, st));
    DSRG_TRY(eig_sort(naux, W, V, w, U, rank, true, true, st));
  }
  std::vector<double> hw(naux);
  DSRG_CUDA(cudaMemcpyAsync(hw.data(), w, sizeof(double) * naux, cudaMemcpyDeviceToHost, st));
  DSRG_CUDA(cudaStreamSynchronize(st));
  int k = 0;
  while (k < naux && hw[k] > threshold) ++k;
  if (w_out) DSRG_CUDA(cudaMemcpyAsync(w_out, w, sizeof(double) * naux, cudaMemcpyDeviceToDevice, st));
  // ---- B'[K][ia] = sum_Q U[Q][K] B[Q][ia], K < k
  if (k > 0) {
    DSRG_PHASE("phase_naf_rotate", st);
    if (fast) {
      ws.off = base;
      __nv_bfloat16* pb = ws_take<__nv_bfloat16>(ws, (size_t)kb * lb * qpad);
      __nv_bfloat16* pu = ws_take<__nv_bfloat16>(ws, (size_t)kb * naux * qpad);
      int* eb = reinterpret_cast<int*>(ws_take<char>(ws, residue_exps_bytes(lb)));
      int* eu = reinterpret_cast<int*>(ws_take<char>(ws, residue_exps_bytes(naux)));
      uint16_t* res = reinterpret_cast<uint16_t*>(ws_take<char>(ws, residue_plain_bytes(kb, naux, lb, capb)));
      int* err = ws_take<int>(ws, 16);
      if (!err) return DSRG_FNO_ERR_NOMEM;
      DSRG_CUDA(cudaMemsetAsync(err, 0, sizeof(int), st));
      // rows of U^T (eigenvector K over Q: stride naux) and of B2^T (column ia over Q: stride L)
      DSRG_TRY(residue_stage(kb, U, k, naux, 1, naux, qpad, pu, eu, st));
      for (long l0 = 0; l0 < L; l0 += lb) {
        const int n = (int)std::min(lb, L - l0);
        DSRG_TRY(residue_stage(kb, B + l0, n, naux, 1, L, qpad, pb, eb, st));
        DSRG_TRY(residue_plain(kb, k, n, pu, eu, k, 0, pb, eb, qpad, 1.0, false, B_out + l0, L, 0, res, capb, err, st));
      }
      int h = 0;
      DSRG_CUDA(cudaMemcpyAsync(&h, err, sizeof(int), cudaMemcpyDeviceToHost, st));
      DSRG_CUDA(cudaStreamSynchronize(st));
      if (h) return DSRG_FNO_ERR_TIMEOUT;
    } else {
      DSRG_TRY(gemm_f64(k, (int)L, naux, 1.0, U, naux, false, B, L, false, 0.0, B_out, L, 1, 0, 0, 0, st));
    }
  }
  DSRG_CUDA(cudaStreamSynchronize(st));
  *naux_out = k;
  return DSRG_FNO_OK;
}

}  // namespace dsrg

using namespace dsrg;

extern "C" int dsrg_fno_naf(int32_t nh, int32_t np, int32_t naux, const double* B_hp, double threshold,
                            int32_t precision, double* B_out, double* w_out, int32_t* naux_out, void* stream) {
  std::lock_guard<std::mutex> lk(workspace_mutex());
  Workspace& ws = workspace_for_current_device();
  return impl_naf(ws, nh, np, naux, B_hp, threshold, precision, B_out, w_out, naux_out, (cudaStream_t)stream);
}
