"""The divide-and-conquer eigensolver on the GPU (dsrg_fno_truncate's solver
above 32 rows) at the edges of its leaves, its two GEMM tiles, its blocks'
rows in shared memory (up to about 1700) and in global memory, against LAPACK."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2312_07008_gb300 as pkg  # noqa: E402


def solve(D):
    n = D.shape[0]
    d = torch.tensor(D, dtype=torch.float64, device="cuda")
    on = torch.empty(n, dtype=torch.float64, device="cuda")
    no = torch.empty((n, n), dtype=torch.float64, device="cuda")
    pkg.dsrg_fno_truncate(n, d, pkg.MODE_PO, 99.0, 0.01, on, no)
    return on.cpu().numpy(), no.cpu().numpy()


def matrix(rng, n, kind):
    if kind == "full":
        X = rng.standard_normal((n, n))
        return X + X.T
    if kind == "diagonal":
        return np.diag(rng.standard_normal(n))
    if kind == "zero":
        return np.zeros((n, n))
    if kind == "low rank":
        X = rng.standard_normal((n, 3))
        return X @ X.T
    X = rng.standard_normal((n, 2 * n)) * np.exp(-0.05 * np.arange(n))[:, None]   # graded, like D_vv
    return X @ X.T


@pytest.mark.parametrize("n,kind", [(n, k) for n in (33, 34, 48, 63, 65, 128, 129, 511, 513)
                                    for k in ("full", "diagonal", "zero", "low rank", "graded")]
                         + [(n, k) for n in (1023, 1747) for k in ("full", "graded")])
def test_against_lapack(n, kind):
    rng = np.random.default_rng(n)
    D = matrix(rng, n, kind)
    w = np.linalg.eigvalsh(D)[::-1]
    scale = max(np.abs(w).max(), 1e-300)
    on, no = solve(D)
    # Householder reduction: of the order of n roundings (2^-53) in norm, times a small factor
    tol = 8 * n * 2.0 ** -53
    assert np.all(np.diff(on) <= 0.0)
    assert np.abs(on - w).max() <= tol * scale
    assert np.abs(no.T @ no - np.eye(n)).max() <= tol
    assert np.abs((no * on) @ no.T - D).max() <= tol * scale


def test_not_a_number_is_reported():
    D = np.eye(100)
    D[40, 41] = D[41, 40] = np.nan
    with pytest.raises(pkg.DsrgFnoError) as ei:
        solve(D)
    assert ei.value.status == -4
