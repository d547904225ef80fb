// Host replay of the residue form's constant tables and row scales (csrc/residue.cuh).
#include "cuda_host_stub.h"

#include "residue.cuh"

using namespace dsrg::res;

extern "C" {
int replay_modulus(int i) { return modulus(i); }
void replay_modulus_table(int i, float* p, float* inv) {
  constexpr ModulusTable T;
  *p = T.p[i];
  *inv = T.inv[i];
}
double replay_norm_limit(int nm) { return nm == 10 ? norm_limit(10) : norm_limit(12); }
// integers of a row whose norm is formed over nsplit shares, as the staging kernels do
int replay_stage(int nm, int n, const double* v, int nsplit, long long* X) {
  const int per = (n + nsplit - 1) / nsplit;
  RowNorm r{0.0, 0};
  for (int q = 0; q < nsplit; ++q) {
    double s = 0.0;
    uint32_t hi = 0;
    for (int k = q * per; k < n && k < (q + 1) * per; ++k) {
      uint64_t b;
      __builtin_memcpy(&b, v + k, 8);
      const uint32_t h = (uint32_t)(b >> 32) & 0x7fffffffu;
      s += v[k] * v[k];
      hi = hi > h ? hi : h;
    }
    add_part(r, row_part(s, hi));
  }
  const int f = row_shift(r, n, replay_norm_limit(nm));
  if (f != SHIFT_INVALID)
    for (int k = 0; k < n; ++k) X[k] = scaled_integer(v[k], f);
  return f;
}
}
