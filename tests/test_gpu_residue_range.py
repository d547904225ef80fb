"""Rows of any size in float64's range through the residue form: the contraction by
itself, and the ladder, whose result scales with its amplitudes.  (Their squares leave
the range below 1e-154 and above 1e154.)"""
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


@pytest.mark.parametrize("nmod", [10, 12])
@pytest.mark.parametrize("K", [7, 300, 1100])
@pytest.mark.parametrize("sa,sb", [(1e-200, 1e200), (1e-290, 1e160), (1e250, 1e-170), (1e-160, 1.0), (1.0, 1e160), (1e-140, 1e-140)])
def test_contraction(nmod, K, sa, sb):
    rng = np.random.default_rng(K)
    a, b = rng.standard_normal((40, K)), rng.standard_normal((33, K))
    a[3, K // 2:] *= 1e-30                       # its second half far below its first
    A, B = np.ascontiguousarray(sa * a), np.ascontiguousarray(sb * b)
    C = np.full((40, 33), np.nan)
    assert pkg.load().dsrg_fno_debug_residue_gemm(nmod, 40, 33, K, A.ctypes.data_as(dp), B.ctypes.data_as(dp), C.ctypes.data_as(dp)) == 0
    exact = (a.astype(np.longdouble) @ b.T.astype(np.longdouble)) * np.longdouble(sa) * np.longdouble(sb)
    na, nb = np.sqrt((a * a).sum(1)), np.sqrt((b * b).sum(1))
    # the tolerance of the rows in the middle of the range (test_gpu_residue_gemm.py) with a norm
    # of at least LIMIT / (4 K^1/2) instead of LIMIT / 2: scaled by the largest element
    tol = 2.2 * np.sqrt(K) / LIMIT[nmod] * 2.0 * np.sqrt(K) + nmod * 2.0 ** 8 * 8 * 2.0 ** -64 * 4.0 * K + 2.0 ** -52
    assert np.all(np.abs(C - exact) <= tol * na[:, None] * nb[None, :] * sa * sb)


@pytest.mark.parametrize("scale", [1e-250, 1e-165, 1e170, 1e250])
def test_ladder_scales_with_its_amplitudes(scale):
    gen = torch.Generator(device="cuda").manual_seed(4)
    b = torch.randn((40, 13, 13), dtype=torch.float64, device="cuda", generator=gen)
    b = (0.5 * (b + b.transpose(1, 2))).contiguous()
    t = torch.randn((21, 13, 13), dtype=torch.float64, device="cuda", generator=gen)
    want, got = torch.empty_like(t), torch.empty_like(t)
    pkg.dsrg_fno_ladder(b, t, want, precision=pkg.FP64)
    pkg.dsrg_fno_ladder(b, scale * t, got)
    # the test_gpu_ladder.py bound of the fast form
    assert float((got / scale - want).abs().max()) <= 1e-10 * float(want.abs().max())
