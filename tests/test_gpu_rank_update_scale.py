"""D_vv of the fast form at the edges of its rank-K update, with the bound that the ten
moduli and the rows' own norms give (a scale one modulus or a few bits short fails)."""
import numpy as np
import pytest

import oracle as O
from synth import make_problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2312_07008_gb300 as pkg  # noqa: E402

# Integers of a row over its range have a norm of LIMIT / 2 = 2^43.3 = 1.1e13 at least (ten
# moduli; a power of two).  Rounding them (uniform, 0.29 rms) moves X . Y by 0.29 2^1/2 |X|
# rms: 3.8e-14 of |x| |y|, six times that for the largest element 2.3e-13.  The same of the
# pair contraction on its rows of 70: an element nu, about |v| |w| / 70^1/2, is off by 3.2e-13
# of itself, sums of 31 and more products of two of them by 2 / 31^1/2 of that rms, six times
# 1.2e-13.  Regulariser and dressing: 1e-13 on each factor.  (Nine moduli: the first term
# times 2^4.5, 5e-12.)
TOL = 2.3e-13 + 6 * 1.2e-13 + 2e-13


@pytest.mark.parametrize("ncore,nact,nvir", [
    (1, 0, 31), (2, 0, 33), (8, 0, 65), (4, 0, 255), (4, 0, 257), (12, 0, 200), (0, 2, 31), (3, 2, 64), (2, 3, 129), (6, 4, 257)])
def test_density_within_the_bound_of_its_scale(ncore, nact, nvir):
    p = make_problem(seed=7 + nvir, s=0.5, ncore=ncore, nact=nact, nvir=nvir, naux=70, nstates=2)
    ref = O.solve(p, cuts=())
    d = torch.full((nvir, nvir), float("nan"), dtype=torch.float64, device="cuda")
    pkg.dsrg_fno_vv_opdm(pkg.problem_from_synth(p, "cuda", pkg.SLICED_BF16, 0), d)
    err = np.max(np.abs(d.cpu().numpy() - ref["dvv"])) / np.max(np.abs(ref["dvv"]))
    print(f"ncore {ncore} nact {nact} nvir {nvir}: {err:.1e} of the largest element")
    assert err <= TOL
