"""The regulariser in the contraction kernel's output stage (3 and 4 digit planes, the
forms that have it) against the separate kernel over the stored contraction tiles."""
import numpy as np
import pytest

from synth import make_problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2312_07008_gb300 as pkg  # noqa: E402


@pytest.mark.parametrize("planes", [3, 4])
@pytest.mark.parametrize("ncore,nact,nvir,naux", [(4, 3, 150, 300), (6, 0, 97, 250), (2, 1, 64, 65)])
def test_fused_equals_separate(planes, ncore, nact, nvir, naux):
    p = make_problem(seed=47, s=0.5, ncore=ncore, nact=nact, nvir=nvir, naux=naux, nstates=2)
    gp = pkg.problem_from_synth(p, "cuda", pkg.SLICED_BF16, planes)
    out = []
    try:
        for fused in (False, True):
            pkg.dsrg_fno_debug_set_fused_epilogue(fused)
            pkg.dsrg_fno_profile_enable(True)
            d = torch.empty((nvir, nvir), dtype=torch.float64, device="cuda")
            e2 = pkg.dsrg_fno_vv_opdm(gp, d)
            separate = pkg.dsrg_fno_profile_query("phase_pair_epilogue")[1]
            assert (separate == 0) == fused
            out.append((e2, d.cpu().numpy(), pkg.dsrg_fno_pt2_energy(gp)))
    finally:
        pkg.dsrg_fno_profile_enable(False)
        pkg.dsrg_fno_debug_set_fused_epilogue(False)
    (e0, d0, ee0), (e1, d1, ee1) = out
    # Delta is formed with different double-float roundings: each element to about 1e-13
    assert abs(e1 - e0) <= 1e-12 * abs(e0) and abs(ee1 - ee0) <= 1e-12 * abs(e0)
    assert np.max(np.abs(d1 - d0)) <= 1e-12 * np.max(np.abs(d0))
