"""Passes of the fast form on a nearly full device: where the ten residue planes of B
do not fit, the pair contraction takes five digit planes, and the energy and the
density are those of the residue form within the fast form's targets."""
import pytest

from synth import make_problem

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


def launches(name):
    return pkg.dsrg_fno_profile_query(name)[1]


def run(call, megabytes):
    hold = leave_free(megabytes) if megabytes else None
    pkg.dsrg_fno_profile_enable(True)
    try:
        out = call()
        kinds = launches("residue_gemm_pair"), launches("sliced_gemm_pair")
    finally:
        pkg.dsrg_fno_profile_enable(False)
        held = pkg.dsrg_fno_debug_workspace_bytes()
        del hold
        torch.cuda.empty_cache()
        pkg.dsrg_fno_release()
    return out, kinds, held


# planes of B: 20 bytes an element in the residue form, 10 as digit planes
@pytest.mark.parametrize("density,nvir,naux,megabytes", [(False, 300, 3000, 270), (True, 120, 6000, 440)])
def test_digit_planes_where_the_residue_planes_do_not_fit(density, nvir, naux, megabytes):
    p = make_problem(12 if nvir == 300 else 18, 2, nvir, naux, seed=4, nstates=2)
    prob = pkg.problem_from_synth(p, "cuda", pkg.SLICED_BF16)
    d = torch.zeros((nvir, nvir), dtype=torch.float64, device="cuda")

    def call():
        return pkg.dsrg_fno_vv_opdm(prob, d) if density else pkg.dsrg_fno_pt2_energy(prob)

    e_want, kinds, _ = run(call, None)
    d_want = d.clone()
    assert kinds[0] > 0 and kinds[1] == 0
    d.zero_()
    e, kinds, held = run(call, megabytes)
    assert kinds[0] == 0 and kinds[1] > 0 and held <= megabytes * MB
    assert abs(e - e_want) <= 1e-7
    assert float((d - d_want).abs().max()) <= 1e-8 * float(d_want.abs().max())
