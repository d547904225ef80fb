"""The divide-and-conquer eigensolver beyond the sizes whose rows fit shared
memory, up to the largest that the dispatch lets in, by the residual and the orthogonality of its vectors."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2312_07008_gb300 as pkg  # noqa: E402


@pytest.mark.parametrize("n", [2500, 7700])
def test_residual_and_orthogonality(n):
    gen = torch.Generator(device="cuda").manual_seed(n)
    z = torch.randn((n, 2 * n), dtype=torch.float64, device="cuda", generator=gen)
    z *= torch.exp(-0.01 * torch.arange(n, device="cuda").double())[:, None]
    d = z @ z.T
    d = 0.5 * (d + d.T)
    del z
    on = torch.empty(n, dtype=torch.float64, device="cuda")
    no = torch.empty((n, n), dtype=torch.float64, device="cuda")
    pkg.dsrg_fno_truncate(n, d, pkg.MODE_PO, 99.0, 0.01, on, no)
    scale = float(on.abs().max())
    # of the order of n roundings (2^-53) in norm, times a small factor, as for the smaller matrices
    tol = 8 * n * 2.0 ** -53
    assert bool((on[1:] <= on[:-1]).all())
    assert abs(float(on.sum() - d.trace())) <= tol * n * scale
    assert float((no.T @ no - torch.eye(n, dtype=torch.float64, device="cuda")).abs().max()) <= tol
    assert float(((no * on) @ no.T - d).abs().max()) <= tol * scale
    pkg.load().dsrg_fno_release()
