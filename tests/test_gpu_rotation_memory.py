"""The rotation of B, the full energy's integrals and the natural auxiliary functions
of the fast form on a nearly full device: their operands go through in parts, and the
results are those of one part."""
import pytest

from synth import make_problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2312_07008_gb300 as pkg  # noqa: E402

MB = 1 << 20


def both(call, megabytes):
    """The call with the whole device and with that much of it left."""
    out = []
    for mb in (None, megabytes):
        pkg.dsrg_fno_release()
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        hold = torch.empty(torch.cuda.mem_get_info()[0] - mb * MB, dtype=torch.uint8, device="cuda") if mb else None
        try:
            out.append(call())
            held = pkg.dsrg_fno_debug_workspace_bytes()
        finally:
            del hold
            torch.cuda.empty_cache()
            pkg.dsrg_fno_release()
    assert held <= megabytes * MB
    return out


def problem(nvir, naux):
    return pkg.problem_from_synth(make_problem(18, 2, nvir, naux, seed=6, nstates=2), "cuda", pkg.SLICED_BF16)


def test_correction():
    # the rotated operand's planes: 24 bytes an element, 460 MB
    prob = problem(300, 3000)
    no = torch.linalg.qr(torch.randn((300, 300), dtype=torch.float64, device="cuda", generator=torch.Generator(device="cuda").manual_seed(1)))[0]
    no = no.contiguous()
    (de, ef), (de2, ef2) = both(lambda: pkg.dsrg_fno_discarded_correction(prob, 100, no, e2_mo=-1.0), 400)
    assert abs(ef2 - ef) <= 1e-7 and abs(de2 - de) <= 1e-7


def test_full_energy():
    # 20 bytes an element of B: 360 MB
    prob = problem(300, 3000)
    (e, evv), (e2, evv2) = both(lambda: pkg.dsrg_fno_pt2_energy_mr(prob), 380)
    assert abs(e2 - e) <= 1e-7 and abs(evv2 - evv) <= 1e-7


def test_natural_auxiliary_functions():
    nh, np_, naux = 20, 300, 1500
    gen = torch.Generator(device="cuda").manual_seed(2)
    b = torch.randn((naux, nh, np_), dtype=torch.float64, device="cuda", generator=gen)
    b *= 0.05 * torch.exp(-1.5 * torch.arange(naux, device="cuda").double() / naux)[:, None, None]
    thr = float(torch.sort((b * b).sum((1, 2)), descending=True).values[1000])

    def call():
        out, w = torch.zeros_like(b), torch.empty(naux, dtype=torch.float64, device="cuda")
        k = pkg.dsrg_fno_naf(nh, np_, naux, b, thr, pkg.SLICED_BF16, out, w)
        w, out = w.cpu(), out.cpu()
        return k, w, out
    # planes and residues of the rotation 450 MB beside 150 MB of matrices
    (k, w, out), (k2, w2, out2) = both(call, 340)
    assert k2 == k
    # W rounds to 2^-43 of its rows' norms in one part as in several
    assert float((w2 - w).abs().max()) <= 1e-11 * float(w.max())
    # the vectors are fixed as well as their eigenvalues are apart: W and B' give the same Gram matrix
    flat = out.reshape(naux, -1)[:k]
    flat2 = out2.reshape(naux, -1)[:k]
    g, g2 = flat.T[:200] @ flat[:, :200], flat2.T[:200] @ flat2[:, :200]
    assert float((g2 - g).abs().max()) <= 1e-9 * float(g.abs().max())
