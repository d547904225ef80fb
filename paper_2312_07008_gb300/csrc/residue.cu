// Residue form of the fast contractions (residue.cuh): staging of the
// operands, the tensor-core kernel and the kernels that put its residues
// together.
#include <cuda.h>

#include <algorithm>
#include <type_traits>

#include "dd.cuh"
#include "kernels.h"
#include "regularizer.cuh"
#include "residue.cuh"
#include "tc_ptx.cuh"

namespace dsrg {

namespace {

using namespace res;

// ---------------------------------------------------------------- staging
__device__ __forceinline__ double square_of(double v) { return v * v; }
__device__ __forceinline__ double zero_like(double) { return 0.0; }

__device__ __forceinline__ long long integer_of(double v, int f) { return scaled_integer(v, f); }

__device__ __forceinline__ uint32_t high_word(double v) { return (uint32_t)__double2hiint(v) & 0x7fffffffu; }

// Norms of the rows: part[split][row] (row_part) over the split's share of k.
// Source element (row, k) at src[row rs + k ks]; one of rs, ks is 1.
template <typename T>
__global__ void __launch_bounds__(256) row_norm_kernel(const T* __restrict__ src, long R, int K, long rs, long ks,
                                                       double* __restrict__ part) {
  const int per = (K + gridDim.y - 1) / gridDim.y;
  const int k0 = blockIdx.y * per, k1 = min(K, k0 + per);
  const long row0 = (long)blockIdx.x * 32;
  double s = 0.0;
  uint32_t hi = 0;
  auto take = [&](const T* p, int k, long step) {
    for (; k < k1; k += 8) {
      const T v = p[k * step];
      s += square_of(v);
      hi = max(hi, high_word(v));
    }
  };
  if (ks == 1) {  // 8 threads per row
    const long row = row0 + (threadIdx.x >> 3);
    if (row < R) take(src + row * rs, k0 + (threadIdx.x & 7), 1);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
      s += __shfl_xor_sync(0xffffffffu, s, o);
      hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    if (row < R && (threadIdx.x & 7) == 0) part[blockIdx.y * R + row] = row_part(s, hi);
    return;
  }
  // a lane per row, 8 warps over k
  __shared__ double red[8][32];
  __shared__ uint32_t red_hi[8][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const long row = row0 + lane;
  if (row < R) take(src + row * rs, k0 + w, ks);
  red[w][lane] = s;
  red_hi[w][lane] = hi;
  __syncthreads();
  if (w == 0 && row < R) {
#pragma unroll
    for (int q = 1; q < 8; ++q) {
      s += red[q][lane];
      hi = max(hi, red_hi[q][lane]);
    }
    part[blockIdx.y * R + row] = row_part(s, hi);
  }
}

// planes[i][row][k] = X mod p_i, centred (bf16, k padded to Kpad with zeros),
// exps[row] = -f.  A block takes 32 rows and `steps` blocks of 64 k, a thread
// 8 consecutive k of a row at a time (16-byte stores, 128 bytes per row).
// Bound by its stores (2 NM bytes per element; about 60 instructions each).
template <int NM, typename T>
__global__ void __launch_bounds__(256) residue_rows_kernel(const T* __restrict__ src, long R, int K, long rs, long ks,
                                                           int Kpad, int steps, const double* __restrict__ part,
                                                           int nsplit, __nv_bfloat16* __restrict__ planes,
                                                           int* __restrict__ exps) {
  __shared__ T tile[32][65];
  const long row0 = (long)blockIdx.x * 32;
  const int myrow = threadIdx.x >> 3, seg = threadIdx.x & 7;
  const long row = row0 + myrow;
  constexpr double LIMIT = norm_limit(NM);
  int f = 0;
  if (row < R) {
    RowNorm s{0.0, 0};
    for (int q = 0; q < nsplit; ++q) add_part(s, part[q * R + row]);
    f = row_shift(s, K, LIMIT);
    if (seg == 0 && blockIdx.y == 0) exps[row] = -f;
    if (f == SHIFT_INVALID) f = 0;
  }
  for (int st = 0; st < steps; ++st) {
    const int k0 = (blockIdx.y * steps + st) * 64;
    if (k0 >= Kpad) break;
    T v[8];
    if (ks == 1) {
      const T* p = src + row * rs + k0 + seg * 8;
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] = (row < R && k0 + seg * 8 + j < K) ? p[j] : zero_like(T());
    } else {
      const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
      __syncthreads();
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int k = w + 8 * q;
        tile[lane][k] = (row0 + lane < R && k0 + k < K) ? src[(row0 + lane) * rs + (long)(k0 + k) * ks] : zero_like(T());
      }
      __syncthreads();
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] = tile[myrow][seg * 8 + j];
    }
    if (row >= R) continue;
    Pieces<pieces_for(NM)> x[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) x[j] = pieces_of<pieces_for(NM)>(integer_of(v[j], f));
#pragma unroll
    for (int i = 0; i < NM; ++i) {
      __nv_bfloat162 h[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) h[j] = __floats2bfloat162_rn(residue<NM>(x[2 * j], i), residue<NM>(x[2 * j + 1], i));
      *reinterpret_cast<uint4*>(planes + ((long)i * R + row) * Kpad + k0 + seg * 8) = *reinterpret_cast<uint4*>(h);
    }
  }
}

// ------------------------------------------------------------- GEMM kernel
// A pair of CTAs (a cluster of 2) multiplies a 256 x 256 tile modulo one p:
// each CTA loads 128 rows of A and 128 of B per 64-wide k block, the leader
// issues cta_group::2 MMAs (M = 256, N = 256), and each CTA's 128 accumulator
// rows lie in its own TMEM, two sets of 256 columns.  A set holds the sum over
// 256 k, an integer of magnitude <= 256 2^16 = 2^24 that the float32
// accumulator has exactly; 8 warps per CTA take it modulo p (exact in float32)
// while the other set fills, and add it up in registers (16 warps of 64 columns
// were slower: 195 against 177 ms per opdm pass of nvir 1200).  Residues in [0, p)
// go to res[unit][column group of 8][256 rows][8 columns] (16-bit).
// Bound by the tensor pipe under the power cap: the pair contraction of an opdm
// pass of nvir 1200 / naux 3600 takes 154 ms, 1.74 PFLOP/s executed (five digit
// planes, 15 products on a 128 x 48 tile: 319 ms at 1.25).  The 256 x 256 tile
// moves 64 bytes per clock and SM from L2 at the pipe's full rate, and the
// reduction takes 4 packed float32 instructions per pair of sums and 256 k.
constexpr int GT_M = 256;             // rows and columns of a tile
constexpr int G_STAGES = 6;
constexpr int G_HALF = 128 * 128;     // bytes of 128 rows of a k block
constexpr int G_STAGE_BYTES = 2 * G_HALF;
constexpr int G_SMEM = G_STAGES * G_STAGE_BYTES + 1024 + 256;
constexpr int G_CHUNK = 4;            // k blocks per exact sum
constexpr int G_COLS = 128;           // columns of a reduction warp
constexpr int G_WARPS = 4 * (256 / G_COLS);
constexpr int G_THREADS = 128 + 32 * G_WARPS;  // warps 0, 1: TMA, MMA; from 4 on: reduction
constexpr long long G_WAIT = 4000000000LL;  // ~2 s of clock cycles
static_assert(G_SMEM <= 232448, "dynamic shared memory per block");

enum { RG_PAIR = 0, RG_PLAIN = 1, RG_SYRK = 2 };
constexpr int RG_BAND = 8;  // row tiles per band of the plain order

struct ResGemm {
  int mode, nm;
  int nkb;            // k blocks of one matrix
  int ntiles;         // tiles per segment
  int tile0;          // plain mode: first tile of the launch
  int arow0;          // plain mode: A's first row in its planes
  int nseg, nr;       // syrk: segments, matrices (1 segment, 1 matrix otherwise)
  int ntm, ntn;
  long nunits;        // nseg x nm x ntiles
  const int2* tiles;  // pair mode
  ResSegment seg[RES_MAX_SEGMENTS];
  const double* sign; // syrk: sign of each matrix
  uint16_t* res;
  int* err;
};

__constant__ ModulusTable c_moduli = ModulusTable();

// unit -> tile, modulus and matrices [r0, r1); the moduli of a segment run one
// after another over all its tiles, so that a modulus's planes stay in L2
struct ResUnit {
  int mt, nt, mod, r0, r1, want;
  long out;
};
__device__ __forceinline__ void rg_tile(const ResGemm& P, int t, int* mt, int* nt) {
  if (P.mode == RG_PAIR) {
    const int2 q = P.tiles[t];
    *mt = q.x;
    *nt = q.y;
  } else if (P.mode == RG_PLAIN) {
    t += P.tile0;
    const int per_band = RG_BAND * P.ntn, b = t / per_band;
    const int rows = min(RG_BAND, P.ntm - b * RG_BAND), r = t - b * per_band;
    *nt = r / rows;
    *mt = b * RG_BAND + r % rows;
  } else {  // upper tiles, row by row
    int m = 0, r = t;
    while (r >= P.ntn - m) {
      r -= P.ntn - m;
      ++m;
    }
    *mt = m;
    *nt = m + r;
  }
}
__device__ __forceinline__ ResUnit rg_decode(const ResGemm& P, long u) {
  ResUnit x;
  const long per = (long)P.ntiles * P.nm;
  const int seg = (int)(u / per), rem = (int)(u - seg * per);
  x.mod = rem / P.ntiles;
  const int t = rem - x.mod * P.ntiles;
  x.out = ((long)seg * P.ntiles + t) * P.nm + x.mod;
  x.r0 = P.seg[seg].r0;
  x.r1 = P.seg[seg].r1;
  x.want = P.seg[seg].sign;
  rg_tile(P, t, &x.mt, &x.nt);
  return x;
}
// whether matrix r belongs to the unit's segment (sign 0: all of its range)
__device__ __forceinline__ bool rg_takes(const ResGemm& P, const ResUnit& x, int r) {
  return x.want == 0 || (P.sign[r] < 0.0) == (x.want < 0);
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(G_THREADS, 1)
    residue_gemm_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB, ResGemm P) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + G_STAGES * G_STAGE_BYTES);
  uint64_t* empty = full + G_STAGES;
  uint64_t* tfull = empty + G_STAGES;
  uint64_t* tempty = tfull + 2;
  uint64_t* done_bar = tempty + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done_bar + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = tc::cluster_rank();
  const long cluster = blockIdx.x >> 1, nclusters = gridDim.x >> 1;
  if (threadIdx.x == 0) {
    for (int s = 0; s < G_STAGES; ++s) {
      tc::mbar_init(&full[s], 1);
      tc::mbar_init(&empty[s], 1);
    }
    for (int q = 0; q < 2; ++q) {
      tc::mbar_init(&tfull[q], 1);
      tc::mbar_init(&tempty[q], 2 * G_WARPS);  // of both CTAs
    }
    tc::mbar_init(done_bar, 1);
    *abort_flag = 0;
    tc::fence_barrier_init();
  }
  if (warp == 0 && lane == 0) {
    tc::prefetch_tmap(&mapA);
    tc::prefetch_tmap(&mapB);
  }
  if (warp == 1) tc::tmem_alloc2(tmem_slot, 512);
  tc::tc_fence_before();
  __syncthreads();
  tc::cluster_sync();  // both CTAs' barriers are initialised
  tc::tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  // The two issuing warps run their loops whole, and one elected thread issues:
  // in a one-thread branch the operands of every instruction pass through
  // registers first, and the MMA thread, at 870 clocks per k block against the
  // tensor cores' 512, was what the kernel waited for (1.50 PFLOP/s executed;
  // neither more stages, L2 prefetches nor a contiguous operand layout changed it).
  const bool elected = tc::elect_one();
  if (warp == 0) {
    // -------------------------------------------------------- TMA producer
    uint32_t it = 0;
    for (long u = cluster; u < P.nunits && !*abort_flag; u += nclusters) {
      const ResUnit x = rg_decode(P, u);
      const int arow = P.arow0 + x.mt * GT_M + rank * 128, brow = x.nt * GT_M + rank * 128;
      for (int r = x.r0; r < x.r1 && !*abort_flag; ++r) {
        if (!rg_takes(P, x, r)) continue;
        for (int kb = 0; kb < P.nkb; ++kb, ++it) {
          const int s = it % G_STAGES;
          if (!__all_sync(0xffffffffu, tc::mbar_wait(&empty[s], ((it / G_STAGES) & 1) ^ 1, G_WAIT))) {
            *abort_flag = 1;
            if (elected) atomicExch(P.err, 1);
            break;
          }
          uint8_t* sa = smem + s * G_STAGE_BYTES;
          const uint32_t bar = tc::map_to_cta(&full[s], 0);
          if (elected) {
            // both CTAs' loads are counted by the leader's barrier
            if (rank == 0) tc::mbar_arrive_expect_tx(&full[s], 2 * G_STAGE_BYTES);
            tc::tma_load_4d_pair(sa, &mapA, kb * 64, arow, r, x.mod, bar);
            tc::tma_load_4d_pair(sa + G_HALF, &mapB, kb * 64, brow, r, x.mod, bar);
          }
          __syncwarp();
        }
      }
    }
    // no CTA leaves before its last loads and the commits on its barriers
    // have landed (bounded)
    for (uint32_t k = it > (uint32_t)G_STAGES ? it - G_STAGES : 0; k < it; ++k)
      tc::mbar_wait(&empty[k % G_STAGES], (k / G_STAGES) & 1, G_WAIT);
    __syncwarp();
  } else if (warp == 1) {
    // ---------------------------------------------- MMA issuer (leader only)
    if (rank == 0) {
      uint32_t it = 0, chunk = 0;
      const uint32_t idesc = tc::make_idesc_bf16(256, 256);
      const uint64_t desc0 = tc::make_sdesc_sw128(tc::smem_u32(smem));
      for (long u = cluster; u < P.nunits && !*abort_flag; u += nclusters) {
        const ResUnit x = rg_decode(P, u);
        int nk = (x.r1 - x.r0) * P.nkb;
        if (x.want != 0)
          for (int r = x.r0; r < x.r1; ++r) nk -= rg_takes(P, x, r) ? 0 : P.nkb;
        for (int kb = 0; kb < nk; ++kb, ++it) {
          const int kc = kb % G_CHUNK, s = it % G_STAGES;
          const uint32_t set = chunk & 1;
          bool ok = kc != 0 || tc::mbar_wait(&tempty[set], ((chunk >> 1) & 1) ^ 1, G_WAIT);
          ok = ok && tc::mbar_wait(&full[s], (it / G_STAGES) & 1, G_WAIT);
          if (!__all_sync(0xffffffffu, ok)) {
            *abort_flag = 1;
            if (elected) atomicExch(P.err, 2);
            break;
          }
          tc::tc_fence_after();
          const bool last = kc == G_CHUNK - 1 || kb == nk - 1;
          if (elected) {
            // start-address field += bytes / 16 (no carry: shared addresses < 2^18)
            const uint64_t ad = desc0 + (uint64_t)((s * G_STAGE_BYTES) >> 4), bd = ad + (uint64_t)(G_HALF >> 4);
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
              tc::mma2_bf16(tmem + set * 256, ad + kk * 2, bd + kk * 2, idesc, (kc | kk) ? 1u : 0u);
            tc::mma2_commit_both(&empty[s]);
            if (last) tc::mma2_commit_both(&tfull[set]);
          }
          __syncwarp();
          if (last) ++chunk;
        }
      }
      if (elected) tc::mma2_commit(done_bar);
      __syncwarp();
      tc::mbar_wait(done_bar, 0, G_WAIT);
    }
    __syncwarp();
  } else if (warp >= 4) {
    // ------------------------------------------------------------ reduction
    const int q = warp & 3, cg = (warp - 4) >> 2;  // lanes of TMEM, column group
    const int row = rank * 128 + q * 32 + lane;
    const uint32_t taddr = tmem + ((uint32_t)(q * 32) << 16) + cg * G_COLS;
    const uint32_t t_empty0 = tc::map_to_cta(&tempty[0], 0), t_empty1 = tc::map_to_cta(&tempty[1], 0);
    uint32_t chunk = 0;
    bool failed = false;
    for (long u = cluster; u < P.nunits && !failed; u += nclusters) {
      const ResUnit x = rg_decode(P, u);
      const float p = c_moduli.p[x.mod], inv = c_moduli.inv[x.mod];
      int nk = 0;
      for (int r = x.r0 + lane; r < x.r1; r += 32) nk += rg_takes(P, x, r) ? P.nkb : 0;
      nk = __reduce_add_sync(0xffffffffu, nk);
      const int nchunks = (nk + G_CHUNK - 1) / G_CHUNK;
      const tc::f32x2 inv2 = tc::f2_set(inv, inv), neg2 = tc::f2_set(-p, -p), mag2 = tc::f2_set(ROUND_MAGIC, ROUND_MAGIC),
                      nmag2 = tc::f2_set(-ROUND_MAGIC, -ROUND_MAGIC);
      tc::f32x2 acc[G_COLS / 2];
#pragma unroll
      for (int c = 0; c < G_COLS / 2; ++c) acc[c] = tc::f2_set(0.f, 0.f);
      for (int k = 0; k < nchunks; ++k) {
        const uint32_t set = chunk & 1;
        if (!__all_sync(0xffffffffu, tc::mbar_wait(&tfull[set], (chunk >> 1) & 1, G_WAIT))) {
          *abort_flag = 1;
          atomicExch(P.err, 4);
          failed = true;
          break;
        }
        tc::tc_fence_after();
#pragma unroll
        for (int c0 = 0; c0 < G_COLS; c0 += 16) {
          float v[16];
          tc::tmem_ld16(taddr + set * 256 + c0, v);
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const tc::f32x2 y = tc::f2_set(v[2 * j], v[2 * j + 1]);
            const tc::f32x2 t = tc::f2_add(tc::f2_fma(y, inv2, mag2), nmag2);
            acc[c0 / 2 + j] = tc::f2_add(acc[c0 / 2 + j], tc::f2_fma(t, neg2, y));
          }
        }
        tc::tc_fence_before();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive_remote(set ? t_empty1 : t_empty0);
        ++chunk;
        if ((k & 0x3fff) == 0x3fff) {  // sums of 2^14 reduced chunks stay below 2^22
#pragma unroll
          for (int c = 0; c < G_COLS / 2; ++c) {
            const tc::f32x2 t = tc::f2_add(tc::f2_fma(acc[c], inv2, mag2), nmag2);
            acc[c] = tc::f2_fma(t, neg2, acc[c]);
          }
        }
      }
      if (failed) break;
      uint16_t* dst = P.res + x.out * (GT_M * GT_M) + ((long)cg * (G_COLS / 8) * GT_M + row) * 8;
#pragma unroll
      for (int g = 0; g < G_COLS / 8; ++g) {
        uint32_t w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          float a, b;
          tc::f2_get(acc[g * 4 + j], &a, &b);
          a = reduce(a, p, inv);
          b = reduce(b, p, inv);
          if (a < 0.f) a += p;
          if (b < 0.f) b += p;
          // the low mantissa bits of 2^23 + x are the integer x
          w[j] = __byte_perm(__float_as_uint(a + 8388608.0f), __float_as_uint(b + 8388608.0f), 0x5410);
        }
        *reinterpret_cast<uint4*>(dst + (long)g * GT_M * 8) = make_uint4(w[0], w[1], w[2], w[3]);
      }
    }
  }
  __syncwarp();
  tc::tc_fence_before();
  __syncthreads();
  tc::cluster_sync();
  tc::tc_fence_after();
  if (warp == 1) tc::tmem_dealloc2(tmem, 512);
}

// -------------------------------------------------- Eq. A7 on the residues
__device__ __forceinline__ float pow2_float(int e) {  // 2^e, 0 and infinity beyond float32
  return e < -126 ? 0.0f : (e > 127 ? __int_as_float(0x7f800000) : __int_as_float((e + 127) << 23));
}

// 2^45 times the signed fraction u 2^-63, double-float
__device__ __forceinline__ dd fraction_dd(uint64_t u) {
  const float top = __int_as_float(0x4B400000 + ((int)(u >> 32) >> 9)) - 12582912.0f;
  const float mid = __int_as_float(0x4B000000 | ((int)(u >> 18) & 0x7FFFFF)) - 8388608.0f;
  const float low = __int_as_float(0x4B000000 | ((int)u & 0x3FFFF)) - 8388608.0f;
  dd x = two_sum(top * 8388608.0f, mid);
  x.lo = __fmaf_rn(low, 1.0f / 262144.0f, x.lo);
  return quick_two_sum(x.hi, x.lo);
}

// tau / kappa (vv, double-float) and t^{ij}_{ex} (va / av, float64) of the
// tiles [0, gridDim.y) of a launch of the contraction: residues put together,
// Eq. A7 applied.  A block takes 32 rows of a tile, 64 columns at a time.  First
// a warp reads a column group of 8 (512 contiguous bytes of every residue plane)
// and each thread puts 8 elements of a row together, into shared memory; then
// the lanes run along the rows, so that the results leave as contiguous rows and
// the regulariser's code is there once.  (Written from the 8-element threads, 8
// bytes to 32 rows at once, an opdm pass of nvir 1200 spent 96 ms here; with the
// regulariser unrolled for 8 elements 57 ms, waiting for instructions.)
// Delta = hp[row] + hp[column].  Bound by the float32 pipe (72 %) and instruction
// issue (68 %): about 100 instructions for the residues of an element beside some
// 100 for its regulariser, two rows packed (250 one by one; nvir 443 with 5 active
// orbitals 2.13 -> 1.74 ms).
struct PairResidues {
  const int2* tiles;
  const uint16_t* res;
  const int* exps;
  const float2* hp;
  const int* slot_of;
  float2 *tau, *kap;
  double* ts;
  const RegTables* reg;
  int nh, na, np, nv;
  double s;
};
constexpr int EPI_GROUPS = 8;  // column groups per step

__global__ void __launch_bounds__(256, 4) pair_epilogue_residue_kernel(PairResidues P) {
  constexpr int NM = RES_MOD, W = 8 * EPI_GROUPS;
  __shared__ RegTables R;
  __shared__ float2 sN[32][W + 1];
  __shared__ float s_fr[32];
  __shared__ float2 s_hp[32];
  __shared__ int s_i[32], s_a[32];
  for (int k = threadIdx.x; k < (int)(sizeof(RegTables) / sizeof(float)); k += 256)
    reinterpret_cast<float*>(&R)[k] = reinterpret_cast<const float*>(P.reg)[k];
  const int2 t = P.tiles[blockIdx.y];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, np = P.np, na = P.na, nv = P.nv, total = P.nh * np;
  const int row0 = t.x * GT_M + blockIdx.x * 32;
  if (row0 >= total) return;
  constexpr double MU = crt_half_mantissa(NM);
  constexpr int EX = crt_half_exponent(NM) - 45;
  if (threadIdx.x < 32) {
    const int row = min(row0 + lane, total - 1), i = row / np;
    s_i[lane] = i;
    s_a[lane] = row0 + lane < total ? row - i * np : -1;
    s_hp[lane] = P.hp[row];
    s_fr[lane] = pow2_float(P.exps[row] + EX / 2);
  }
  const dd s = dd_from_double(P.s), mu = {(float)MU, (float)(MU - (double)(float)MU)};
  const uint16_t* res = P.res + (long)blockIdx.y * NM * GT_M * GT_M + (blockIdx.x * 32 + lane) * 8;
  for (int g0 = 0; g0 < 32; g0 += EPI_GROUPS) {
    const int cs = t.y * GT_M + g0 * 8;  // first column of the step
    if (cs >= total) break;
    __syncthreads();                     // row data and tables; the last step's elements are read
    {
      uint32_t w[NM][4];
      const int g = g0 + warp;
#pragma unroll
      for (int m = 0; m < NM; ++m) {
        const uint4 q = __ldcs(reinterpret_cast<const uint4*>(res + ((long)m * 32 + g) * GT_M * 8));
        w[m][0] = q.x;
        w[m][1] = q.y;
        w[m][2] = q.z;
        w[m][3] = q.w;
      }
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        uint64_t u = 0;
#pragma unroll
        for (int m = 0; m < NM; ++m) u = crt_add<NM>(u, (w[m][c >> 1] >> (16 * (c & 1))) & 0xffffu, m);
        const dd x = fraction_dd(u);
        sN[lane][warp * 8 + c] = make_float2(x.hi, x.lo);
      }
    }
    __syncthreads();
#pragma unroll 1
    for (int q = 0; q < W / 32; ++q) {
      const int C = cs + q * 32 + lane;
      if (C >= total) continue;
      const int j = C / np, b = C - j * np;
      const bool bv = b >= na;
      const float2 hc = P.hp[C];
      const float fc = pow2_float(P.exps[C] + EX - EX / 2);
#pragma unroll 1
      for (int u = 0; u < 4; u += 2) {  // two rows at a time, packed
        const int rr = warp * 4 + u;
        int slot[2], a[2], i[2];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          a[k] = s_a[rr + k];
          i[k] = s_i[rr + k];
          const bool av = a[k] >= na;
          // vv -> tau, kappa; va -> ts[i][j]; av -> ts[j][i], written by the va element of (i, i) itself
          const bool use = a[k] >= 0 && ((av && bv) || (P.ts != nullptr && (av || (bv && i[k] != j))));
          slot[k] = use ? P.slot_of[(long)i[k] * P.nh + j] : -1;
        }
        if (slot[0] < 0 && slot[1] < 0) continue;
        const float2 f0 = sN[rr][q * 32 + lane], f1 = sN[rr + 1][q * 32 + lane], h0 = s_hp[rr], h1 = s_hp[rr + 1];
        const f32x2 fr = f2_set(s_fr[rr], s_fr[rr + 1]), fc2 = f2_set(fc, fc);
        dd2 n = dd_mul(dd2{f2_set(f0.x, f1.x), f2_set(f0.y, f1.y)}, dd_splat<f32x2>(mu));
        n = {f2_mul(f2_mul(n.hi, fr), fc2), f2_mul(f2_mul(n.lo, fr), fc2)};
        dd2 r1, y;
        regularize(dd_add(dd2{f2_set(h0.x, h1.x), f2_set(h0.y, h1.y)}, dd_splat<f32x2>(dd{hc.x, hc.y})), s, R, &r1, &y);
        const dd2 x = dd_mul(n, r1);
        const dd2 k2 = dd_mul(n, dd_add_ordered(dd_splat<f32x2>(dd_make(1.0f)), y));
        float xh[2], xl[2], kh[2], kl[2];
        fl_get(x.hi, xh);
        fl_get(x.lo, xl);
        fl_get(k2.hi, kh);
        fl_get(k2.lo, kl);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          if (slot[k] < 0) continue;
          const bool av = a[k] >= na;
          if (av && bv) {
            const long o = ((long)slot[k] * nv + (a[k] - na)) * nv + (b - na);
            P.tau[o] = make_float2(xh[k], xl[k]);
            P.kap[o] = make_float2(kh[k], kl[k]);
          } else if (av) {
            P.ts[(((long)i[k] * P.nh + j) * nv + (a[k] - na)) * na + b] = dd_to_double(dd{xh[k], xl[k]});
          } else {
            P.ts[(((long)j * P.nh + i[k]) * nv + (b - na)) * na + a[k]] = dd_to_double(dd{xh[k], xl[k]});
          }
        }
      }
    }
  }
}

// ------------------------------------- products in float64 from the residues
// (signed fraction u 2^-63) (M / 2) 2^e as float64, by integer arithmetic: the
// two float64 lanes of an SM would make these kernels five times slower.
template <int NM>
__device__ __forceinline__ double fraction_f64(uint64_t u, int e) {
  constexpr uint64_t MANT = (uint64_t)(crt_half_mantissa(NM) * 9223372036854775808.0);  // [2^63, 2^64)
  if (e > 50000) return __longlong_as_double((long long)2047 << 52);  // a row whose norm overflows
  const bool neg = (long long)u < 0;
  const uint64_t t = __umul64hi(neg ? 0 - u : u, MANT);  // mag mantissa / 2
  if (t == 0) return 0.0;
  const int lz = __clzll((long long)t);
  const uint64_t m = (((t << lz) >> 1) + 512) >> 10;       // 53 bits, or 2^53 after rounding up
  const int ex = 1023 + 63 - lz - 62 + crt_half_exponent(NM) + e;
  if (ex <= 0) return 0.0;
  const uint64_t b = ((uint64_t)ex << 52) + (m - ((uint64_t)1 << 52));
  return __longlong_as_double((long long)(ex >= 2047 ? (uint64_t)2047 << 52 : b) | (neg ? (long long)1 << 63 : 0));
}

template <int NM>
__device__ __forceinline__ void load_residues(const uint16_t* res, int g, uint32_t (&w)[NM][4]) {
#pragma unroll
  for (int m = 0; m < NM; ++m) {
    const uint4 q = __ldcs(reinterpret_cast<const uint4*>(res + ((long)m * 32 + g) * GT_M * 8));
    w[m][0] = q.x;
    w[m][1] = q.y;
    w[m][2] = q.z;
    w[m][3] = q.w;
  }
}
template <int NM>
__device__ __forceinline__ uint64_t recombine(const uint32_t (&w)[NM][4], int c) {
  uint64_t u = 0;
#pragma unroll
  for (int m = 0; m < NM; ++m) u = crt_add<NM>(u, (w[m][c >> 1] >> (16 * (c & 1))) & 0xffffu, m);
  return u;
}

// Plain products (opdm's small terms, the rotation of B, the ladder, natural
// auxiliary functions, the full energy's integrals): at nvir 1200 the small terms
// of an opdm pass take 12.3 ms instead of 17.4, the rotation of B to 203 orbitals
// 1.3 instead of 3.6 ms (12 moduli against the 21 products of six digit planes).
// C[m][n] = (add ? C[m][n] : 0) + alpha A[m] . B[n], or with swap = v > 0 and
// rows (a, c), columns (b, d) of v values each: C[((a v + b) v + c) v + d].
struct PlainOut {
  const int *ea, *eb;
  int M, N;
  double* C;
  long ldc;
  double alpha;
  int add, swap;
};
// As in the pair epilogue a block takes 32 rows of a tile, 64 columns at a time:
// column groups from the residues into shared memory, rows out of it (stored
// from the threads of a column group, 8 bytes to a row at a time, the integrals
// of the ladder, nv 119, took 6.55 ms instead of 5.16).
template <int NM>
__global__ void __launch_bounds__(256) plain_residue_kernel(ResGemm P, PlainOut O) {
  constexpr int W = 8 * EPI_GROUPS;
  __shared__ double sV[32][W + 1];
  __shared__ long s_off[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int mt, nt;
  rg_tile(P, blockIdx.y, &mt, &nt);
  const int m0 = mt * GT_M + blockIdx.x * 32, rows = min(32, O.M - m0), v = O.swap;
  if (rows <= 0) return;
  if (threadIdx.x < 32) {
    const int m = m0 + lane;
    s_off[lane] = v ? ((long)(m / v) * v * v + m % v) * v : (long)m * O.ldc;
  }
  const int e = O.ea[m0 + min(lane, rows - 1)];
  const uint16_t* res = P.res + (long)blockIdx.y * NM * GT_M * GT_M + (blockIdx.x * 32 + lane) * 8;
  for (int g0 = 0; g0 < 32; g0 += EPI_GROUPS) {
    const int cs = nt * GT_M + g0 * 8, n0 = cs + warp * 8;
    if (cs >= O.N) break;
    __syncthreads();  // the last step's elements are read
    if (n0 < O.N) {
      uint32_t w[NM][4];
      load_residues<NM>(res, g0 + warp, w);
#pragma unroll
      for (int c = 0; c < 8; ++c)
        sV[lane][warp * 8 + c] = fraction_f64<NM>(recombine<NM>(w, c), e + O.eb[min(n0 + c, O.N - 1)]);
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < W / 32; ++q) {
      const int n = cs + q * 32 + lane;
      if (n >= O.N) break;
      double* dst = O.C + (v ? (long)(n / v) * v * v + n % v : (long)n);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int r = warp + 8 * u;
        if (r >= rows) break;
        double x = sV[r][q * 32 + lane];
        if (O.alpha != 1.0) x *= O.alpha;
        dst[s_off[r]] = O.add ? dst[s_off[r]] + x : x;
      }
    }
  }
}

// Rank-K update of D_vv, sums over all rows of all dressed matrices: bound by the
// tensor cores.  opdm pass of nvir 1200 (10 active, K = 5.9e6): the products take
// 72 to 77 ms (1.5 to 1.6 PFLOP/s at the power cap) instead of the digit planes'
// 120; the staging 33 ms instead of 28, for ten planes instead of five.  D[e][f] +=
// the sum over the segments, in a fixed order, of sign A_s[e] . A_s[f] (upper tiles,
// mirrored).
__global__ void __launch_bounds__(256) syrk_residue_kernel(const __grid_constant__ ResGemm P, const int* __restrict__ exps,
                                                           int nv, double* D) {
  constexpr int NM = RES_MOD_S;
  __shared__ double part[8][32][9];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int mt, nt;
  rg_tile(P, blockIdx.y, &mt, &nt);
  const int g = blockIdx.x, e0 = mt * GT_M + blockIdx.z * 32, f0 = nt * GT_M + g * 8, e = e0 + lane;
  if (e0 >= nv || f0 >= nv || f0 + 7 < e0) return;
  double acc[8] = {};
  for (int s = warp; s < P.nseg; s += 8) {  // a warp per segment, eight columns of 32 rows
    const int* ex = exps + (long)P.seg[s].scale * nv;
    uint32_t w[NM][4];
    load_residues<NM>(P.res + (((long)s * P.ntiles + blockIdx.y) * NM) * GT_M * GT_M + (blockIdx.z * 32 + lane) * 8, g, w);
    const int ee = ex[min(e, nv - 1)];
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const double v = fraction_f64<NM>(recombine<NM>(w, c), ee + ex[min(f0 + c, nv - 1)]);
      acc[c] += P.seg[s].sign < 0 ? -v : v;
    }
  }
#pragma unroll
  for (int c = 0; c < 8; ++c) part[warp][lane][c] = acc[c];
  __syncthreads();
  const int r = threadIdx.x >> 3, c = threadIdx.x & 7, er = e0 + r, f = f0 + c;
  if (er >= nv || f >= nv || f < er) return;
  double v = part[0][r][c];
#pragma unroll
  for (int q = 1; q < 8; ++q) v += part[q][r][c];
  D[(long)er * nv + f] += v;
  if (f != er) D[(long)f * nv + er] += v;
}

// -f of row e of scale group s, from its norm over the group's matrices: the
// bounds of the tiles' rows (32 columns for the first n_core matrices, 16 for the
// others).  Eight threads per row, each its share of the matrices in a fixed order.
__global__ void __launch_bounds__(256) segment_shift_kernel(int nv, int n_core, ResGemm P, const float* __restrict__ rowpart,
                                                            int* __restrict__ exps) {
  __shared__ double red[8][32];
  const int lane = threadIdx.x & 31, part = threadIdx.x >> 5, e = blockIdx.x * 32 + lane, s = blockIdx.y;
  if (P.seg[s].sign < 0) return;  // the two signs of a range share its scales
  constexpr double LIMIT = norm_limit(RES_MOD_S);
  double x = 0.0;
  const int stride = (nv + 15) / 16;
  if (e < nv)
    for (int r = P.seg[s].r0 + part; r < P.seg[s].r1; r += 8) {
      const int w = r < n_core ? 32 : 16, nt = (nv + w - 1) / w;
      const float* p = rowpart + (long)r * stride * nv + e;
      double y = 0.0;
      for (int t = 0; t < nt; ++t) {
        const double m = p[(long)t * nv];
        y = fma(m, m, y);
      }
      x += y;
    }
  red[part][lane] = x;
  __syncthreads();
  if (part != 0 || e >= nv) return;
#pragma unroll
  for (int q = 1; q < 8; ++q) x += red[q][lane];
  // |hi + lo| <= |hi| (1 + 2^-23); float32 sums of up to 32 squares and their root
  const int f = row_shift(x * (1.0 + 1e-5), (P.seg[s].r1 - P.seg[s].r0) * nv, LIMIT);
  exps[(long)P.seg[s].scale * nv + e] = -f;
}

// Two dressed elements times 2^(fa + fb), rounded, in the pieces of pieces_of<3>:
// X < 2^44.4, so hi leaves pieces of 2^30 (below 2^14.4) and 2^15, lo (below 2^21)
// of 2^15, and what is left of both (below 2^15, rounded to 2^-9 and then to an
// integer): every partial sum of a residue stays below 2^24.
struct Pieces2 {
  f32x2 x[3];
};
__device__ __forceinline__ f32x2 f2_rint(f32x2 v) {
  return f2_sub(f2_add(v, f2_set(ROUND_MAGIC, ROUND_MAGIC)), f2_set(ROUND_MAGIC, ROUND_MAGIC));
}
__device__ __forceinline__ Pieces2 pieces2_of(float4 v, float fa, float fb) {
  const f32x2 sa = f2_set(fa, fa), sb = f2_set(fb, fb);
  f32x2 h = f2_mul(f2_mul(f2_set(v.x, v.z), sa), sb), l = f2_mul(f2_mul(f2_set(v.y, v.w), sa), sb);
  const f32x2 up15 = f2_set(-32768.0f, -32768.0f), dn15 = f2_set(1.0f / 32768.0f, 1.0f / 32768.0f);
  Pieces2 p;
  p.x[2] = f2_rint(f2_mul(h, f2_set(1.0f / 1073741824.0f, 1.0f / 1073741824.0f)));
  h = f2_fma(p.x[2], f2_set(-1073741824.0f, -1073741824.0f), h);
  const f32x2 h1 = f2_rint(f2_mul(h, dn15)), l1 = f2_rint(f2_mul(l, dn15));
  p.x[1] = f2_add(h1, l1);
  p.x[0] = f2_rint(f2_add(f2_fma(h1, up15, h), f2_fma(l1, up15, l)));
  return p;
}

// Residue planes [RES_MOD_S][nr][nv][Kpad] of the dressed matrices (double-float
// rows, contiguous), scaled by their segment's row exponents.  Bound by memory: 8
// bytes read and 20 written per element; float32 arithmetic in packed pairs, about
// 50 instructions per element (165 with 64-bit integers; nvir 600 with 40 core and
// 10 active orbitals 4.99 -> 3.96 ms, 6.5 TB/s).  Exponents beyond +-126 need two
// factors.
__global__ void __launch_bounds__(256, 3) residue_dressed_kernel(const float2* __restrict__ src, int nv, int nr, int Kpad,
                                                              const int* __restrict__ exps, const int* __restrict__ scale_of,
                                                              __nv_bfloat16* __restrict__ planes) {
  constexpr Tables<RES_MOD_S> T{};
  const long R = (long)nr * nv, row = (long)blockIdx.x * 32 + (threadIdx.x >> 3);
  if (row >= R) return;
  const int r = (int)(row / nv), e = (int)(row - (long)r * nv);
  const int ex = exps[(long)scale_of[r] * nv + e];
  const int f = ex == -SHIFT_INVALID ? 0 : min(max(-ex, -252), 252);
  const float fa = pow2_float(f / 2), fb = pow2_float(f - f / 2);
  const bool wide = nv % 2 == 0;  // rows start on 16 bytes
  for (int k0 = (threadIdx.x & 7) * 8; k0 < Kpad; k0 += 64) {
    const float2* p = src + row * nv + k0;
    Pieces2 x[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (wide) {
        if (k0 + 2 * j < nv) v = reinterpret_cast<const float4*>(p)[j];
      } else {
        if (k0 + 2 * j < nv) {
          const float2 q = p[2 * j];
          v.x = q.x;
          v.y = q.y;
        }
        if (k0 + 2 * j + 1 < nv) {
          const float2 q = p[2 * j + 1];
          v.z = q.x;
          v.w = q.y;
        }
      }
      x[j] = pieces2_of(v, fa, fb);
    }
#pragma unroll
    for (int i = 0; i < RES_MOD_S; ++i) {
      const f32x2 c15 = f2_set(T.c15[i], T.c15[i]), c30 = f2_set(T.c30[i], T.c30[i]), inv = f2_set(T.inv[i], T.inv[i]),
                  np = f2_set(-T.p[i], -T.p[i]), magic = f2_set(ROUND_MAGIC, ROUND_MAGIC);
      __nv_bfloat162 h[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        f32x2 t = f2_fma(x[j].x[2], c30, f2_fma(x[j].x[1], c15, x[j].x[0]));
        t = f2_fma(f2_sub(f2_fma(t, inv, magic), magic), np, t);
        float a, b;
        f2_get(t, &a, &b);
        h[j] = __floats2bfloat162_rn(a, b);
      }
      *reinterpret_cast<uint4*>(planes + ((long)i * R + row) * Kpad + k0) = *reinterpret_cast<uint4*>(h);
    }
  }
}

// ------------------------------------------------------- host side helpers
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// 4-D map over planes [nm][nr][rows][Kpad] (bf16), box {64 k, 128 rows, 1, 1}, 128-byte swizzle
int plane_map(CUtensorMap* map, const void* planes, int nm, long nr, long rows, int Kpad) {
  EncodeTiledFn fn = reinterpret_cast<EncodeTiledFn>(tensor_map_encoder());
  if (!fn) return DSRG_FNO_ERR_CUDA;
  cuuint64_t dims[4] = {(cuuint64_t)Kpad, (cuuint64_t)rows, (cuuint64_t)nr, (cuuint64_t)nm};
  cuuint64_t strides[3] = {(cuuint64_t)Kpad * 2, (cuuint64_t)rows * Kpad * 2, (cuuint64_t)nr * rows * Kpad * 2};
  cuuint32_t box[4] = {64, 128, 1, 1}, estr[4] = {1, 1, 1, 1};
  const CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(planes), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? DSRG_FNO_OK : DSRG_FNO_ERR_CUDA;
}

int launch_gemm(const void* pa, long rows_a, const void* pb, long rows_b, int Kpad, ResGemm P, cudaStream_t st) {
  if (P.nunits <= 0) return DSRG_FNO_OK;
  if (Kpad % 64 != 0) return DSRG_FNO_ERR_ARG;
  P.nkb = Kpad / 64;
  CUtensorMap ma, mb;
  DSRG_TRY(plane_map(&ma, pa, P.nm, P.nr, rows_a, Kpad));
  DSRG_TRY(plane_map(&mb, pb, P.nm, P.nr, rows_b, Kpad));
  int dev = 0, sms = 0;
  DSRG_CUDA(cudaGetDevice(&dev));
  DSRG_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  DSRG_CUDA(cudaFuncSetAttribute(residue_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, G_SMEM));
  const int clusters = (int)std::min<long>(sms / 2, P.nunits);
  void* tok = nullptr;
  if (profiling()) {
    // executed tensor-core flops: whole tiles, every modulus
    const double fl = 2.0 * GT_M * GT_M * (double)Kpad * P.nr * P.nm * (double)P.ntiles;
    prof_begin(P.mode == RG_PAIR ? "residue_gemm_pair" : (P.mode == RG_SYRK ? "residue_gemm_syrk" : "residue_gemm_plain"),
               fl, st, &tok);
  }
  residue_gemm_kernel<<<2 * clusters, G_THREADS, G_SMEM, st>>>(ma, mb, P);
  DSRG_LAUNCH_CHECK();
  prof_end(tok, st);
  return DSRG_FNO_OK;
}

template <int NM, typename T>
int stage_rows(const T* src, long R, int K, long rs, long ks, int Kpad, __nv_bfloat16* planes, int* exps, double* part,
               cudaStream_t st) {
  if (R <= 0) return DSRG_FNO_OK;
  if (Kpad % 64 != 0 || Kpad < K) return DSRG_FNO_ERR_ARG;
  // enough blocks for two waves: few rows share their k
  const int rb = (int)((R + 31) / 32), want = std::max(1, ceil_div(RES_STAGE_BLOCKS, rb));
  const int nsplit = std::max(1, std::min(want, ceil_div(K, 256)));
  row_norm_kernel<T><<<dim3(rb, nsplit), 256, 0, st>>>(src, R, K, rs, ks, part);
  DSRG_LAUNCH_CHECK();
  const int nb = Kpad / 64, steps = std::max(1, ceil_div(nb, want));
  residue_rows_kernel<NM, T><<<dim3(rb, ceil_div(nb, steps)), 256, 0, st>>>(src, R, K, rs, ks, Kpad, steps, part, nsplit,
                                                                             planes, exps);
  DSRG_LAUNCH_CHECK();
  return DSRG_FNO_OK;
}

}  // namespace

size_t residue_exps_bytes(size_t R) {
  return ws_bytes(R, sizeof(int)) + ws_bytes(R + 32 * (RES_STAGE_BLOCKS + 1), sizeof(double));
}

int residue_stage(int nm, const double* src, long R, int K, long rs, long ks, int Kpad, __nv_bfloat16* planes, int* exps,
                  cudaStream_t st) {
  double* part = reinterpret_cast<double*>(reinterpret_cast<char*>(exps) + ws_bytes(R, sizeof(int)));
  if (nm == RES_MOD) return stage_rows<RES_MOD>(src, R, K, rs, ks, Kpad, planes, exps, part, st);
  if (nm == RES_MOD_X) return stage_rows<RES_MOD_X>(src, R, K, rs, ks, Kpad, planes, exps, part, st);
  return DSRG_FNO_ERR_ARG;
}

size_t residue_plain_bytes(int nm, long M, long N, int cap) {
  const long tiles = (long)ceil_div(M, GT_M) * ceil_div(N, GT_M);
  return (size_t)std::min<long>(tiles, cap) * residue_tile_bytes(nm);
}

size_t residue_tile_bytes(int nm) { return (size_t)nm * GT_M * GT_M * sizeof(uint16_t); }

// tau, kappa and ts of a batch of pairs, `cap` tiles of residues at a time.
int residue_pair(const Geometry& g, const __nv_bfloat16* planes, const int* exps, int Kpad, const int2* tiles, int ntiles,
                 const int* slot_of, const float2* hp, uint16_t* res, int cap, float2* tau, float2* kap, double* ts,
                 int* err, cudaStream_t st) {
  const long rows = (long)g.nh * g.np;
  PairResidues E{};
  DSRG_TRY(reg_tables_device(&E.reg));
  E.exps = exps;
  E.hp = hp;
  E.slot_of = slot_of;
  E.tau = tau;
  E.kap = kap;
  E.ts = ts;
  E.nh = g.nh;
  E.na = g.na;
  E.np = g.np;
  E.nv = g.nv;
  E.s = g.s;
  E.res = res;
  for (int t0 = 0; t0 < ntiles; t0 += cap) {
    const int nt = std::min(cap, ntiles - t0);
    ResGemm P{};
    P.mode = RG_PAIR;
    P.nm = RES_MOD;
    P.ntiles = nt;
    P.nseg = 1;
    P.nr = 1;
    P.seg[0] = ResSegment{0, 1, 0, 0};
    P.nunits = (long)nt * RES_MOD;
    P.tiles = tiles + t0;
    P.res = res;
    P.err = err;
    DSRG_TRY(launch_gemm(planes, rows, planes, rows, Kpad, P, st));
    DSRG_PHASE("phase_pair_epilogue", st);
    E.tiles = tiles + t0;
    pair_epilogue_residue_kernel<<<dim3(GT_M / 32, nt), 256, 0, st>>>(E);
    DSRG_LAUNCH_CHECK();
  }
  return DSRG_FNO_OK;
}

// C = alpha A B^T, or with add C += alpha A B^T, for M rows of A from row a0 of
// its planes [nm][rows_a][Kpad] and all N of B's [nm][N][Kpad].  With swap = v,
// rows (a, c) and columns (b, d) of v values each, element (a, c), (b, d) goes
// to C[((a v + b) v + c) v + d].  res: cap tiles of residues.
int residue_plain(int nm, int M, int N, const __nv_bfloat16* pa, const int* ea, long rows_a, int a0,
                  const __nv_bfloat16* pb, const int* eb, int Kpad, double alpha, bool add, double* C, long ldc, int swap,
                  uint16_t* res, int cap, int* err, cudaStream_t st) {
  if (M <= 0 || N <= 0) return DSRG_FNO_OK;
  ResGemm P{};
  P.arow0 = a0;
  P.mode = RG_PLAIN;
  P.nm = nm;
  P.ntm = ceil_div(M, GT_M);
  P.ntn = ceil_div(N, GT_M);
  P.nseg = 1;
  P.nr = 1;
  P.seg[0] = ResSegment{0, 1, 0, 0};
  P.res = res;
  P.err = err;
  const PlainOut O{ea + a0, eb, M, N, C, ldc, alpha, add ? 1 : 0, swap};
  const int total = P.ntm * P.ntn;
  for (P.tile0 = 0; P.tile0 < total; P.tile0 += cap) {
    P.ntiles = std::min(cap, total - P.tile0);
    P.nunits = (long)P.ntiles * nm;
    DSRG_TRY(launch_gemm(pa, rows_a, pb, N, Kpad, P, st));
    const dim3 grid(GT_M / 32, P.ntiles);
    if (nm == RES_MOD) plain_residue_kernel<RES_MOD><<<grid, 256, 0, st>>>(P, O);
    else plain_residue_kernel<RES_MOD_X><<<grid, 256, 0, st>>>(P, O);
    DSRG_LAUNCH_CHECK();
  }
  return DSRG_FNO_OK;
}

// Segments of the rank-K update over nr matrices of which those from n_signed
// on may carry a minus sign: every range of scales is one segment, or two (one
// per sign).  A range's rows share one scale; eight or more keep what that costs
// below a bit.  Segments differ in length (signs), so the smaller D is, the more
// are taken, down to 20 rounds of units on the pairs of SMs (nvir 300: 0.43 ms with
// 32 to 64, 0.61 with 8 to 16; nvir 1200: 69 and 65 ms, for starting the units and
// their residues).  Of the counts from that to twice it the one whose units leave
// the least of the last round idle.
static int residue_least_segments(int nv) {
  const int nt = ceil_div(nv, GT_M), units = nt * (nt + 1) / 2 * RES_MOD_S;
  return std::min(RES_MAX_SEGMENTS / 2, std::max(8, 20 * 76 / units));
}
int residue_segments(int nv, int nr, int n_signed, ResSegment* seg) {
  const int nt = ceil_div(nv, GT_M), units = nt * (nt + 1) / 2 * RES_MOD_S, pairs = 76, least = residue_least_segments(nv);
  int best = least;
  double best_eff = 0.0;
  for (int k = least; k <= 2 * least; ++k) {
    const long u = (long)units * k;
    const double eff = (double)u / ((double)ceil_div(u, pairs) * pairs);
    if (eff > best_eff + 0.005) {
      best_eff = eff;
      best = k;
    }
  }
  int n = 0, scale = 0;
  auto add = [&](int b, int e, int count, bool both) {
    count = std::max(1, std::min(count, e - b));
    for (int k = 0; k < count; ++k) {
      const int r0 = b + (int)((long)(e - b) * k / count), r1 = b + (int)((long)(e - b) * (k + 1) / count);
      seg[n++] = ResSegment{r0, r1, both ? 1 : 0, scale};
      if (both) seg[n++] = ResSegment{r0, r1, -1, scale};
      ++scale;
    }
  };
  // shares of the segments in proportion to the matrices, at least one range each
  const int plain = std::min(n_signed, nr), sg = nr - plain;
  const int np = plain > 0 ? std::max(1, (int)((long)best * plain / nr)) : 0;
  if (plain > 0) add(0, plain, sg > 0 ? std::min(np, best - 2) : np, false);
  if (sg > 0) add(plain, nr, std::max(1, (best - np) / 2), true);
  return n;
}

size_t residue_syrk_res_bytes(int nv) {
  const int nt = ceil_div(nv, GT_M);
  return (size_t)2 * residue_least_segments(nv) * (nt * (nt + 1) / 2) * residue_tile_bytes(RES_MOD_S);
}

// D += sum_r sign_r Sig_r Sig_r^T.  rowpart: as dress_dd writes it; exps: RES_MAX_SEGMENTS nv ints; scale_of: nr ints (host list, copied).
int residue_syrk(int nv, int nr, int n_signed, const float2* sig, const float* rowpart, const double* sign,
                 __nv_bfloat16* planes, int* exps, int* scale_of, int Kpad, uint16_t* res, double* D, int* err,
                 cudaStream_t st) {
  if (nr <= 0 || nv <= 0) return DSRG_FNO_OK;
  ResGemm P{};
  P.mode = RG_SYRK;
  P.nm = RES_MOD_S;
  P.ntm = P.ntn = ceil_div(nv, GT_M);
  P.ntiles = P.ntm * (P.ntm + 1) / 2;
  P.nseg = residue_segments(nv, nr, n_signed, P.seg);
  P.nr = nr;
  P.nunits = (long)P.nseg * P.nm * P.ntiles;
  P.sign = sign;
  P.res = res;
  P.err = err;
  std::vector<int> so(nr);
  for (int s = 0; s < P.nseg; ++s)
    for (int r = P.seg[s].r0; r < P.seg[s].r1; ++r) so[r] = P.seg[s].scale;
  DSRG_CUDA(cudaMemcpyAsync(scale_of, so.data(), sizeof(int) * nr, cudaMemcpyHostToDevice, st));
  {
    DSRG_PHASE("phase_stage_sig", st);
    segment_shift_kernel<<<dim3(ceil_div(nv, 32), P.nseg), 256, 0, st>>>(nv, n_signed, P, rowpart, exps);
    DSRG_LAUNCH_CHECK();
    residue_dressed_kernel<<<(unsigned)ceil_div((long)nr * nv, 32), 256, 0, st>>>(sig, nv, nr, Kpad, exps, scale_of,
                                                                                  planes);
    DSRG_LAUNCH_CHECK();
  }
  DSRG_TRY(launch_gemm(planes, nv, planes, nv, Kpad, P, st));
  syrk_residue_kernel<<<dim3(GT_M / 8, P.ntiles, GT_M / 32), 256, 0, st>>>(P, exps, nv, D);
  DSRG_LAUNCH_CHECK();
  return DSRG_FNO_OK;
}

}  // namespace dsrg
