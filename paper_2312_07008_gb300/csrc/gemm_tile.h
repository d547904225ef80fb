// Tile edge of the generic float64 GEMM (gemm_f64.cu), host arithmetic only.
#pragma once

#include <initializer_list>

namespace dsrg {

constexpr long GEMM_F64_GRID_ROWS = 65535;  // row tiles of a launch (gridDim.y)

// The edge whose fullest SM does the least float64 work (blocks per SM times T^2;
// the larger on a tie, which reads less) among those whose row tiles fit one
// launch: 16 up to 1 048 560 rows, 32 up to twice that, 64 up to four times.
inline int gemm_f64_tile(long M, long N, int batch) {
  const long sms = 152;
  int best = 64;
  long best_cost = 0;
  for (int T : {64, 32, 16}) {
    const long rows = (M + T - 1) / T, blocks = rows * ((N + T - 1) / T) * batch;
    const long cost = (blocks + sms - 1) / sms * T * T;
    if (best_cost == 0 || (rows <= GEMM_F64_GRID_ROWS && cost * 10 < best_cost * 9)) {
      best_cost = cost;
      best = T;
    }
  }
  return best;
}

}  // namespace dsrg
