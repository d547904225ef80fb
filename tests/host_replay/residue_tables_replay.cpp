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
}
