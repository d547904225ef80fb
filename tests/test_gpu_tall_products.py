"""Float64 products with more rows than 16-row tiles fit one launch: the ladder's
contraction of a small basis with many hole pairs, in the float64 form."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2312_07008_gb300 as pkg  # noqa: E402


@pytest.mark.parametrize("npairs", [16 * 65535, 16 * 65535 + 1, 32 * 65535 + 1])
def test_ladder_with_many_pairs(npairs):
    nv, naux = 3, 5
    gen = torch.Generator(device="cuda").manual_seed(1)
    b = torch.randn((naux, nv, nv), dtype=torch.float64, device="cuda", generator=gen)
    b = (0.5 * (b + b.transpose(1, 2))).contiguous()
    t = torch.randn((npairs, nv, nv), dtype=torch.float64, device="cuda", generator=gen)
    c = torch.full_like(t, float("nan"))
    pkg.dsrg_fno_ladder(b, t, c, precision=pkg.FP64)
    ints = torch.einsum("qac,qbd->abcd", b, b)
    want = torch.einsum("abcd,pcd->pab", ints, t)
    # 5 and 9 products per sum, in float64
    assert float((c - want).abs().max()) <= 32 * 2.0 ** -53 * 9 * float(ints.abs().max() * t.abs().max())
