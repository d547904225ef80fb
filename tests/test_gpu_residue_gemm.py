"""The residue form's contraction by itself (test hook of the library) against
float64 products of the same rows, at the edges of its 256 x 256 tiles, of its
64-wide k blocks and of the 256 k that one exact sum takes, with the row shapes
that set the scale of a row or the size of its sums."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2312_07008_gb300 as pkg  # noqa: E402

dp = ctypes.POINTER(ctypes.c_double)
LIMIT = {10: 2.0 ** 44.3, 12: 2.0 ** 53.2}     # largest norm of a row of integers


def gemm(nmod, A, B):
    (M, K), N = A.shape, B.shape[0]
    C = np.full((M, N), np.nan)
    A, B = np.ascontiguousarray(A), np.ascontiguousarray(B)
    st = pkg.load().dsrg_fno_debug_residue_gemm(nmod, M, N, K, A.ctypes.data_as(dp), B.ctypes.data_as(dp), C.ctypes.data_as(dp))
    assert st == 0, st
    return C


def check(nmod, A, B, wide=True):
    exact = A.astype(np.longdouble) @ B.T.astype(np.longdouble) if wide else A @ B.T
    na, nb = np.sqrt((A * A).sum(1)), np.sqrt((B * B).sum(1))
    # X = a 2^f + d, |d| <= 1/2, |X| >= LIMIT / 2 (less the roundings): each product is
    # off by K^1/2 (|X| + |Y|) / 2 + K / 4 units; the weights of the recombination are
    # rounded to 2^-64 of M = 2 LIMIT^2, nmod residues below 2^9; float64 output
    K = A.shape[1]
    tol = 2.2 * np.sqrt(K) / LIMIT[nmod] + nmod * 2.0 ** 8 * 8 * 2.0 ** -64 + 2.0 ** -52 + (0.0 if wide else K * 2.0 ** -53)
    assert np.all(np.abs(gemm(nmod, A, B) - exact) <= tol * na[:, None] * nb[None, :])


@pytest.mark.parametrize("nmod", [10, 12])
@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (256, 256, 64), (257, 255, 65), (128, 129, 256), (300, 157, 257), (40, 600, 1100)])
def test_product_at_tile_edges(nmod, M, N, K):
    rng = np.random.default_rng(M + N + K)
    check(nmod, rng.standard_normal((M, K)) * np.exp(rng.uniform(-20, 5, (M, 1))), 1e-3 * rng.standard_normal((N, K)))


@pytest.mark.parametrize("nmod", [10, 12])
def test_rows_that_stress_scale_and_sums(nmod):
    rng = np.random.default_rng(nmod)
    K = 1000
    rows = np.stack([np.full(K, 0.7), -np.full(K, 0.7), np.where(np.arange(K) == 3, 1.0, 1e-12), np.zeros(K),
                     rng.standard_normal(K) * np.exp(-0.05 * np.arange(K)), np.where(np.arange(K) % 2, 1.0, -1.0),
                     1e-20 * rng.standard_normal(K), 1e15 * rng.standard_normal(K)])
    check(nmod, rows, rows)


def test_more_tiles_than_the_residues_held_at_a_time():
    rng = np.random.default_rng(5)
    check(10, rng.standard_normal((17000, 70)), rng.standard_normal((4200, 70)), wide=False)   # 67 x 17 tiles of 256
