// Host replay of the float64 GEMM's tile rule (csrc/gemm_tile.h).
#include "gemm_tile.h"

extern "C" int replay_gemm_tile(long M, long N, int batch) { return dsrg::gemm_f64_tile(M, N, batch); }
