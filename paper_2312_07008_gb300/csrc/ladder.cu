// Particle-particle ladder of Eq. 6 in the (truncated) virtual basis: the
// term of C2 = [O2, T2]_2 with four virtual indices, whose O(N_C^2 N_V^4)
// cost the FNO truncation cuts by (N_V'/N_V)^4:
//   C^{ij}_{ab} = sum_{cd} <ab|cd> T^{ij}_{cd},  <ab|cd> = sum_Q B^Q_{ac} B^Q_{bd}.
// Two contractions per block of A_BLK values of a:
//   1. I[(a c)][(b d)] = sum_Q B^Q_{ac} B^Q_{bd}          (M = A nv, N = nv^2, K = naux)
//      then the middle indices are swapped: I'[(a b)][(c d)]
//   2. C[p][(a b)] = sum_{(c d)} T[p][(c d)] I'[(a b)][(c d)]  (M = npairs, N = A nv, K = nv^2)
// Fast form: both in the residue form on the tensor cores, the first writing
// I' itself; float64 form: the float64 GEMM.  2 nv^4 (naux + npairs) flops.
#include <math.h>

#include <algorithm>

#include "kernels.h"

namespace dsrg {

namespace {

// out[a][b][c][d] = in[a][c][b][d] for a < A (rows of d copied whole)
__global__ void swap_middle_kernel(int A, int nv, const double* __restrict__ in, double* __restrict__ out) {
  const long row = blockIdx.x;  // (a, b, c) of out
  const int c = (int)(row % nv);
  const long t = row / nv;
  const int b = (int)(t % nv);
  const int a = (int)(t / nv);
  const double* src = in + (((long)a * nv + c) * nv + b) * nv;
  double* dst = out + row * nv;
  for (int d = threadIdx.x; d < nv; d += blockDim.x) dst[d] = src[d];
}

}  // namespace

static const int LADDER_A_BLK = 16;

// Fast form: values of a per block, hole pairs whose planes are held at a time, and
// output tiles whose residues are.
struct LadderPlan {
  int A, pairs, cap;
};

static size_t ladder_res_bytes(int nv, const LadderPlan& P) {
  const long nv2 = (long)nv * nv, blk = (long)P.A * nv;
  const size_t most = std::max(residue_plain_bytes(RES_MOD, blk, nv2), residue_plain_bytes(RES_MOD, P.pairs, blk));
  return std::min(most, P.cap * residue_tile_bytes(RES_MOD));
}

static size_t ladder_bytes(int nv, int naux, const LadderPlan& P) {
  const size_t nv2 = (size_t)nv * nv, blk = (size_t)P.A * nv, qpad = pad64(naux), vpad = pad64((int)nv2);
  return ws_bytes(blk * nv2, sizeof(double)) + ws_bytes(16, sizeof(int)) + ws_bytes(8, sizeof(int)) +
         ws_bytes(RES_MOD * nv2 * qpad, 2) + ws_bytes(RES_MOD * P.pairs * vpad, 2) + ws_bytes(RES_MOD * blk * vpad, 2) +
         residue_exps_bytes(nv2) + residue_exps_bytes(P.pairs) + residue_exps_bytes(blk) +
         ws_bytes(ladder_res_bytes(nv, P), 1);
}

// Up to 2^28 integrals per block (2 GB, and 5.4 GB of their planes), so that small
// bases run in one block and fill the chip, within the memory that calls plan with;
// down to 16 values of a.  Where even those take more than twice that, nine tenths of
// the free memory, fewer values and fewer pairs at a time: no call is refused for the
// sake of its blocks' size.  nv 119, naux 1500, 820 pairs: 9.0 ms in one block (7.3
// GB), 10.3 with 4 GB of the device free (held: 1.8 GB), 11.7 with 1.5, 18.8 with 1.0.
static LadderPlan ladder_plan(const Workspace& ws, int nv, int naux, int npairs) {
  const int least = std::min(LADDER_A_BLK, nv);
  LadderPlan P{(int)std::min<long>(nv, std::max<long>(least, (1L << 28) / ((long)nv * nv * nv))), npairs, RES_PLAIN_CAP};
  if (ladder_bytes(nv, naux, P) <= ws.cap) return P;
  const size_t budget = device_budget(ws.cap);
  if (ladder_bytes(nv, naux, P) <= budget) return P;
  P.cap = residue_cap(RES_MOD, budget);
  while (P.A > least && ladder_bytes(nv, naux, P) > budget) --P.A;
  while (P.A > 1 && ladder_bytes(nv, naux, P) > 2 * budget) --P.A;
  while (P.pairs > RES_TILE && ladder_bytes(nv, naux, P) > 2 * budget) P.pairs = std::max(RES_TILE, P.pairs / 2);
  return P;
}

int impl_ladder(Workspace& ws, int32_t nv, int32_t naux, const double* Bvv, int32_t npairs, const double* T,
                int32_t precision, double* C, cudaStream_t st) {
  if (nv <= 0 || naux <= 0 || npairs <= 0 || !Bvv || !T || !C) return DSRG_FNO_ERR_ARG;
  if (precision != DSRG_FNO_FP64 && precision != DSRG_FNO_SLICED_BF16) return DSRG_FNO_ERR_UNSUPPORTED;
  if (!is_device_ptr(Bvv) || !is_device_ptr(T) || !is_device_ptr(C)) return DSRG_FNO_ERR_ARG;
  const long nv2 = (long)nv * nv;
  if (nv2 * LADDER_A_BLK * nv >= (1L << 31) || (long)npairs * nv2 >= (1L << 31)) return DSRG_FNO_ERR_UNSUPPORTED;
  const bool fast = precision == DSRG_FNO_SLICED_BF16;
  const LadderPlan plan = fast ? ladder_plan(ws, nv, naux, npairs) : LadderPlan{std::min(LADDER_A_BLK, (int)nv), npairs, 0};
  const int A = plan.A;
  const long blk = (long)A * nv;  // rows (a c) or (a b) of one block
  const int nm = RES_MOD;
  const int qpad = pad64(naux), vpad = pad64((int)nv2);
  const size_t need = fast ? ladder_bytes(nv, naux, plan)
                           : 2 * ws_bytes((size_t)blk * nv2, sizeof(double)) + ws_bytes(16, sizeof(int)) + ws_bytes(8, sizeof(int));
  DSRG_TRY(ws_reserve(ws, need));
  {
    int* flag = ws_take<int>(ws, 8);
    int h = 0;
    DSRG_CUDA(cudaMemsetAsync(flag, 0, sizeof(int), st));
    DSRG_TRY(check_finite(Bvv, (long)naux * nv2, flag, st));
    DSRG_TRY(check_finite(T, (long)npairs * nv2, flag, st));
    DSRG_CUDA(cudaMemcpyAsync(&h, flag, sizeof(int), cudaMemcpyDeviceToHost, st));
    DSRG_CUDA(cudaStreamSynchronize(st));
    if (h) return DSRG_FNO_ERR_NONFINITE;
  }
  double* I2 = ws_take<double>(ws, (size_t)blk * nv2);
  int* err = ws_take<int>(ws, 16);
  if (!fast) {
    double* I1 = ws_take<double>(ws, (size_t)blk * nv2);
    if (!I1) return DSRG_FNO_ERR_NOMEM;
    for (int a0 = 0; a0 < nv; a0 += A) {
      const int na = std::min(A, nv - a0);
      const long rows = (long)na * nv;
      {
        DSRG_PHASE("phase_ladder_integrals", st);
        DSRG_TRY(gemm_f64((int)rows, (int)nv2, naux, 1.0, Bvv + (long)a0 * nv, nv2, false, Bvv, nv2, false, 0.0, I1, nv2,
                          1, 0, 0, 0, st));
        swap_middle_kernel<<<(unsigned)(rows * nv), 128, 0, st>>>(na, nv, I1, I2);
        DSRG_LAUNCH_CHECK();
      }
      DSRG_PHASE("phase_ladder_contract", st);
      DSRG_TRY(gemm_f64(npairs, (int)rows, (int)nv2, 1.0, T, nv2, true, I2, nv2, true, 0.0, C + (long)a0 * nv, nv2, 1, 0,
                        0, 0, st));
    }
    DSRG_CUDA(cudaStreamSynchronize(st));
    return DSRG_FNO_OK;
  }
  auto exps = [&ws](size_t rows) { return reinterpret_cast<int*>(ws_take<char>(ws, residue_exps_bytes(rows))); };
  __nv_bfloat16* pY = ws_take<__nv_bfloat16>(ws, (size_t)nm * nv2 * qpad);
  __nv_bfloat16* pT = ws_take<__nv_bfloat16>(ws, (size_t)nm * plan.pairs * vpad);
  __nv_bfloat16* pI = ws_take<__nv_bfloat16>(ws, (size_t)nm * blk * vpad);
  int *eY = exps(nv2), *eT = exps(plan.pairs), *eI = exps(blk);
  uint16_t* res = reinterpret_cast<uint16_t*>(ws_take<char>(ws, ladder_res_bytes(nv, plan)));
  if (!res) return DSRG_FNO_ERR_NOMEM;
  DSRG_CUDA(cudaMemsetAsync(err, 0, sizeof(int), st));
  {
    DSRG_PHASE("phase_ladder_integrals", st);
    // rows (b d) of the factors over Q (the rows (a c) are among them)
    DSRG_TRY(residue_stage(nm, Bvv, nv2, naux, 1, nv2, qpad, pY, eY, st));
  }
  for (int a0 = 0; a0 < nv; a0 += A) {
    const int na = std::min(A, nv - a0);
    const long rows = (long)na * nv;
    {
      DSRG_PHASE("phase_ladder_integrals", st);
      // written with the middle indices swapped
      DSRG_TRY(residue_plain(nm, (int)rows, (int)nv2, pY, eY, nv2, a0 * nv, pY, eY, qpad, 1.0, false, I2, nv2, nv, res,
                             plan.cap, err, st));
    }
    DSRG_PHASE("phase_ladder_contract", st);
    DSRG_TRY(residue_stage(nm, I2, rows, (int)nv2, nv2, 1, vpad, pI, eI, st));
    for (int p0 = 0; p0 < npairs; p0 += plan.pairs) {
      const int np = std::min(plan.pairs, npairs - p0);
      // rows p of the amplitudes over (c d): once for every block of a where all pairs are held
      if (a0 == 0 || plan.pairs < npairs)
        DSRG_TRY(residue_stage(nm, T + (long)p0 * nv2, np, (int)nv2, nv2, 1, vpad, pT, eT, st));
      DSRG_TRY(residue_plain(nm, np, (int)rows, pT, eT, np, 0, pI, eI, vpad, 1.0, false, C + (long)p0 * nv2 + (long)a0 * nv, nv2,
                             0, res, plan.cap, err, st));
    }
  }
  int h = 0;
  DSRG_CUDA(cudaMemcpyAsync(&h, err, sizeof(int), cudaMemcpyDeviceToHost, st));
  DSRG_CUDA(cudaStreamSynchronize(st));
  return h ? DSRG_FNO_ERR_TIMEOUT : DSRG_FNO_OK;
}

}  // namespace dsrg

using namespace dsrg;

extern "C" int dsrg_fno_ladder(int32_t nv, int32_t naux, const double* B_vv, int32_t npairs, const double* T,
                               int32_t precision, double* C_out, void* stream) {
  std::lock_guard<std::mutex> lk(workspace_mutex());
  Workspace& ws = workspace_for_current_device();
  return impl_ladder(ws, nv, naux, B_vv, npairs, T, precision, C_out, (cudaStream_t)stream);
}
