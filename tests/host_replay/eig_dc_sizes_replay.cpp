// Host replay of the divide and conquer's launch sizes (csrc/eig_dc.cuh).
#include "cuda_host_stub.h"

#include "eig_dc.cuh"

extern "C" {
int replay_levels(int n) { return dsrg::dc::dc_levels(n); }
int replay_bound(int n, int l, int t) { return dsrg::dc::dc_bound(n, l, t); }
int replay_node_rows(int n, int l) { return dsrg::dc::dc_node_rows(n, l); }
int replay_deflate_bytes(int n, int l) { return dsrg::dc::dc_deflate_bytes(n, l); }
}
