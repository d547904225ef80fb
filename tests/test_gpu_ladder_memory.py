"""The ladder's fast form on a nearly full device: the blocks follow the memory that
is free, down to a few values of a and a part of the hole pairs at a time, and the
result is that of one block."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2312_07008_gb300 as pkg  # noqa: E402

MB = 1 << 20


def leave_free(megabytes):
    """Device memory taken until that much is left."""
    pkg.dsrg_fno_release()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    return torch.empty(free - megabytes * MB, dtype=torch.uint8, device="cuda")


def run(nv, naux, npairs, megabytes=None):
    gen = torch.Generator(device="cuda").manual_seed(nv)
    b = 0.05 * torch.randn((naux, nv, nv), dtype=torch.float64, device="cuda", generator=gen)
    b = (0.5 * (b + b.transpose(1, 2))).contiguous()
    t = 0.05 * torch.randn((npairs, nv, nv), dtype=torch.float64, device="cuda", generator=gen)
    c = torch.full_like(t, float("nan"))
    hold = leave_free(megabytes) if megabytes else None
    try:
        pkg.dsrg_fno_ladder(b, t, c)
        torch.cuda.synchronize()
    finally:
        held = pkg.dsrg_fno_debug_workspace_bytes()
        del hold
        torch.cuda.empty_cache()
        pkg.dsrg_fno_release()
    return c.cpu(), held


# bytes of the planes that every plan holds: 20 nv^2 naux of B; all pairs' 20 nv^2 npairs
@pytest.mark.parametrize("nv,naux,npairs,megabytes", [
    (119, 1500, 820, 4000),     # one block of all a takes 7.6 GB
    (119, 1500, 820, 1500),
    (119, 1500, 820, 1000),     # fewer than 16 values of a
    (61, 300, 3001, 400),       # a part of the pairs at a time (all: 230 MB beside 25 MB of B)
])
def test_blocks_follow_the_free_memory(nv, naux, npairs, megabytes):
    want, _ = run(nv, naux, npairs)
    got, held = run(nv, naux, npairs, megabytes)
    assert held <= megabytes * MB
    # the same integers and products; a row's scale may differ by one bit where its
    # norm, summed in another order, lies next to a power of two: errors of 2^-43 of the norms
    assert float((got - want).abs().max()) <= 1e-11 * float(want.abs().max())
