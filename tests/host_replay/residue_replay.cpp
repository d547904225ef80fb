// Host replay of the residue form's arithmetic (csrc/residue.cuh): integers of
// a row, their centred residues, and the recombination of reduced products.
#include "cuda_host_stub.h"

#include "residue.cuh"

using namespace dsrg::res;

extern "C" {
int replay_modulus(int i) { return modulus(i); }
double replay_norm_limit(int nm) { return nm == 10 ? norm_limit(10) : norm_limit(12); }
int replay_row_shift(double sumsq, int K, int nm) { return row_shift(sumsq, K, replay_norm_limit(nm)); }
int replay_half_exponent(int nm) { return nm == 10 ? crt_half_exponent(10) : crt_half_exponent(12); }
double replay_half_mantissa(int nm) { return nm == 10 ? crt_half_mantissa(10) : crt_half_mantissa(12); }
// X[k] = round(v[k] 2^f) and its residues r[i][k]
void replay_residues(int nm, int n, const double* v, int f, long long* X, float* r) {
  for (int k = 0; k < n; ++k) {
    X[k] = scaled_integer(v[k], f);
    if (nm == 10) {
      const Pieces<3> a = pieces_of<3>(X[k]);
      for (int i = 0; i < nm; ++i) r[(long)i * n + k] = residue<10>(a, i);
    } else {
      const Pieces<4> a = pieces_of<4>(X[k]);
      for (int i = 0; i < nm; ++i) r[(long)i * n + k] = residue<12>(a, i);
    }
  }
}
// chunk sums of products (integers up to 2^24) reduced and added as the kernel does
float replay_reduce(const float* chunk, int n, int i) {
  const float p = (float)modulus(i), inv = 1.0f / p;
  float acc = 0.0f;
  for (int k = 0; k < n; ++k) acc += reduce(chunk[k], p, inv);
  acc = reduce(acc, p, inv);
  return acc < 0.0f ? acc + p : acc;
}
unsigned long long replay_crt(int nm, const float* r) {
  unsigned long long u = 0;
  for (int i = 0; i < nm; ++i)
    u = nm == 10 ? crt_add<10>(u, (uint32_t)r[i], i) : crt_add<12>(u, (uint32_t)r[i], i);
  return u;
}
}
