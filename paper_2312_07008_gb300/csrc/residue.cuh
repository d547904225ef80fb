// Residue form of the fast contractions: arithmetic shared by its kernels.
//
// A row v of length K becomes integers X = round(v 2^f) with |X| <= S in the
// 2-norm, so that by Cauchy-Schwarz every product |X_a . Y_b| <= S^2 < M / 2,
// M the product of NM pairwise coprime moduli p <= 512.  The product is formed
// modulo each p from centred residues (|r| <= 256, exact in bfloat16) and put
// together by the Chinese remainder theorem.  What errs is the rounding of X and, in
// the fraction of M that the residues are put together as, that of the theorem's
// weights to 2^-64: below 2^-49 |v| |w|, typically 2^-51; far less than the first
// with NM = 10, as much or more with 12.  (Ozaki, Uchino and Imamura, "Ozaki scheme II", 2025, for the idea of a GEMM
// modulo small coprimes.)
//
// NM = 10 (M = 2^89.7, S = 2^44.3) against five base-256 digit planes: 10
// tensor-core products instead of 15, an error of about 2^-45 |v| |w| instead
// of 2^-40 K^1/2 max|v| max|w| (no product is dropped).  NM = 12 (S = 2^53.2)
// takes the place of six digit planes (21 products).
#pragma once
#include <math.h>
#include <stdint.h>

namespace dsrg {
namespace res {

constexpr int NMAX = 12;
constexpr int modulus(int i) {
  constexpr int p[NMAX] = {512, 511, 509, 507, 505, 503, 499, 493, 491, 487, 479, 473};
  return p[i];
}
// 2^e mod p, centred
constexpr int pow2_mod(int e, int i) {
  long r = 1;
  for (int k = 0; k < e; ++k) r = r * 2 % modulus(i);
  return (int)(2 * r > modulus(i) ? r - modulus(i) : r);
}
// (M / p_i)^-1 mod p_i
constexpr int crt_inverse(int nm, int i) {
  const int p = modulus(i);
  long m = 1;
  for (int k = 0; k < nm; ++k)
    if (k != i) m = m * (modulus(k) % p) % p;
  for (int x = 1; x < p; ++x)
    if (m * x % p == 1) return x;
  return 0;
}
// round(2^64 inv_i / p_i): sum_i r_i C_i mod 2^64 is 2^64 (X / M mod 1) up to NM 2^8
constexpr uint64_t crt_weight(int nm, int i) {
  const unsigned __int128 num = ((unsigned __int128)crt_inverse(nm, i) << 64) + modulus(i) / 2;
  return (uint64_t)(num / modulus(i));
}
// The tables as values: indexed by unrolled loops they become immediates (the
// functions above would run on the device).
template <int NM>
struct Tables {
  uint64_t weight[NM];
  float p[NM], inv[NM], c15[NM], c30[NM], c45[NM];
  constexpr Tables() : weight{}, p{}, inv{}, c15{}, c30{}, c45{} {
    for (int i = 0; i < NM; ++i) {
      weight[i] = crt_weight(NM, i);
      p[i] = (float)modulus(i);
      inv[i] = 1.0f / (float)modulus(i);
      c15[i] = (float)pow2_mod(15, i);
      c30[i] = (float)pow2_mod(30, i);
      c45[i] = (float)pow2_mod(45, i);
    }
  }
};

// p and 1 / p of every modulus: the contraction kernel's constant memory, initialised
// with the module, so that no launch on any stream can precede it.
struct ModulusTable {
  float p[NMAX], inv[NMAX];
  constexpr ModulusTable() : p{}, inv{} {
    for (int i = 0; i < NMAX; ++i) {
      p[i] = (float)modulus(i);
      inv[i] = 1.0f / (float)modulus(i);
    }
  }
};

// M / 2 = mantissa 2^exponent, mantissa in [1, 2)
constexpr double crt_half_mantissa(int nm) {
  double m = 0.5;
  for (int i = 0; i < nm; ++i) m *= modulus(i);
  while (m >= 2.0) m *= 0.5;
  return m;
}
constexpr int crt_half_exponent(int nm) {
  double m = 0.5;
  int e = 0;
  for (int i = 0; i < nm; ++i) m *= modulus(i);
  while (m >= 2.0) {
    m *= 0.5;
    ++e;
  }
  return e;
}
// S: largest 2-norm of a row of integers (a little below sqrt(M / 2))
constexpr double norm_limit(int nm) {
  double s = crt_half_mantissa(nm);
  const int e = crt_half_exponent(nm);
  if (e & 1) s *= 2.0;
  double r = s;
  for (int k = 0; k < 60; ++k) r = 0.5 * (r + s / r);
  for (int k = 0; k < e / 2; ++k) r *= 2.0;
  return r * (1.0 - 1e-9);
}

constexpr float ROUND_MAGIC = 12582912.0f;  // 1.5 2^23: adding it rounds |x| < 2^22 to an integer

// t - p round(t / p) for an integer |t| < 2^24 + 2^12: exact, |result| <= p / 2 + 1
__host__ __device__ __forceinline__ float reduce(float t, float p, float inv) {
#ifdef __CUDA_ARCH__
  const float q = __fadd_rn(__fmaf_rn(t, inv, ROUND_MAGIC), -ROUND_MAGIC);
  return __fmaf_rn(q, -p, t);
#else
  const float q = __builtin_fmaf(t, inv, ROUND_MAGIC) - ROUND_MAGIC;
  return __builtin_fmaf(q, -p, t);
#endif
}

// An integer |X| < 2^54 in pieces of 15 bits, X = x0 + 2^15 x1 + 2^30 x2 + 2^45
// x3 with |x0|, |x1|, |x2| <= 2^14 (NP = 3: x2 takes the rest, |X| <= 2^44.4).
template <int NP>
struct Pieces {
  float x[NP];
};
template <int NP>
__host__ __device__ __forceinline__ Pieces<NP> pieces_of(long long X) {
  Pieces<NP> r;
#pragma unroll
  for (int k = 0; k < NP - 1; ++k) {
    const int x = (((int)X + 0x4000) & 0x7fff) - 0x4000;
    r.x[k] = (float)x;
    X = (X - x) >> 15;
  }
  r.x[NP - 1] = (float)(int)X;
  return r;
}
constexpr int pieces_for(int nm) { return nm > 10 ? 4 : 3; }

// centred residue of the pieced integer modulo p_i: every partial sum is an
// integer below 2^24, so the float32 arithmetic is exact
__host__ __device__ __forceinline__ float fma32(float a, float b, float c) {
#ifdef __CUDA_ARCH__
  return __fmaf_rn(a, b, c);
#else
  return __builtin_fmaf(a, b, c);
#endif
}
template <int NM>
__host__ __device__ __forceinline__ float residue(const Pieces<pieces_for(NM)>& a, int i) {
  constexpr Tables<NM> T{};
  float t = fma32(a.x[2], T.c30[i], fma32(a.x[1], T.c15[i], a.x[0]));
  if constexpr (pieces_for(NM) == 4) t = fma32(a.x[3], T.c45[i], t);
  return reduce(t, T.p[i], T.inv[i]);
}

// round(v 2^f) (half away from zero), |v 2^f| < 2^54
__host__ __device__ __forceinline__ long long scaled_integer(double v, int f) {
  long long b;
#ifdef __CUDA_ARCH__
  b = __double_as_longlong(v);
#else
  __builtin_memcpy(&b, &v, 8);
#endif
  const int E = (int)((b >> 52) & 0x7FF);
  if (E == 0) return 0;
  const long long m = (b & 0xFFFFFFFFFFFFFLL) | (1LL << 52);
  const int sh = 1075 - E - f;
  long long X = 0;
  if (sh <= 0) X = sh > -10 ? m << -sh : 0;
  else if (sh < 63) X = (m + (1LL << (sh - 1))) >> sh;
  return b < 0 ? -X : X;
}

// Largest f with |v| 2^f + K^1/2 / 2 (the roundings) within S; 0 for a zero
// row, SHIFT_INVALID where |v|^2 is not finite.
constexpr int SHIFT_INVALID = -100000;
__host__ __device__ __forceinline__ int row_shift(double sumsq, int K, double limit) {
  if (!(sumsq > 0.0)) return sumsq == 0.0 ? 0 : SHIFT_INVALID;
  if (sumsq > 1.7e308) return SHIFT_INVALID;
  const double room = (limit - 0.5 * sqrt((double)K) - 1.0) / sqrt(sumsq);
  int e;
  frexp(room, &e);  // room = m 2^e, m in [1/2, 1): 2^(e - 1) <= room
  return e - 1 < 1000 ? e - 1 : 1000;
}

// A row's norm from its parts.  A part is the sum of its elements' squares or, where the
// largest element lies beyond 2^+-480 and its square near the ends of float64's range,
// that element's biased exponent E as the negative number of E units of 2^-1074: it
// adds nothing to a sum, and a look at the sign finds it (a comparison and a conversion
// in float64, 16 parts a row, cost 12 us in every staging of the small terms).  hi: the
// largest high word of |v|.
__host__ __device__ __forceinline__ double row_part(double sumsq, uint32_t hi) {
  const uint32_t E = hi >> 20;
  if (E == 0) return 0.0;  // elements below 2^-1022 are staged as zeros
  if ((E >= 543 && E <= 1503) || E == 2047) return sumsq;
  const uint64_t b = ((uint64_t)1 << 63) | E;
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double d;
  __builtin_memcpy(&d, &b, 8);
  return d;
#endif
}
struct RowNorm {
  double sumsq;
  int e;  // largest exponent of the parts that are one, 0: none
};
__host__ __device__ __forceinline__ void add_part(RowNorm& r, double part) {
#ifdef __CUDA_ARCH__
  const int hi = __double2hiint(part), lo = __double2loint(part);
#else
  uint64_t b;
  __builtin_memcpy(&b, &part, 8);
  const int hi = (int)(b >> 32), lo = (int)b;
#endif
  const int e = hi < 0 ? lo : 0;
  r.e = r.e > e ? r.e : e;
  r.sumsq += part;
}
// As above; a part by exponent counts as K elements of 2^(e - 1022), above all of its
// own: the row keeps half of log2 K bits less than by its norm, as many as by its
// largest element.
__host__ __device__ __forceinline__ int row_shift(const RowNorm& r, int K, double limit) {
  if (r.e == 0 || !(r.sumsq <= 1.7e308)) return row_shift(r.sumsq, K, limit);
  if (r.e < 1023 && r.sumsq > 0.0) return row_shift(r.sumsq + K * ldexp(1.0, 2 * (r.e - 1022)), K, limit);
  int e;
  frexp((limit - 0.5 * sqrt((double)K) - 1.0) / sqrt((double)K), &e);
  return e - 1 - (r.e - 1022);
}

// The contraction: u = sum_i r_i C_i mod 2^64 as a signed fraction of M, i.e.
// value = u 2^-63 (M / 2) 2^(e_a + e_b) for row exponents e = -f.
template <int NM>
__host__ __device__ __forceinline__ uint64_t crt_add(uint64_t u, uint32_t r, int i) {
  constexpr Tables<NM> T{};
  return u + (uint64_t)r * T.weight[i];
}

}  // namespace res
}  // namespace dsrg
