"""D_vv of the fast form at the edges of its rank-K update (256 x 256 tiles of D,
64-wide k blocks, ranges of matrices that share a row scale, one or both signs)
and of the core pairs' dressing (32 x 32 tiles), against the FP64 oracle."""
import numpy as np
import pytest

import oracle as O
from synth import make_problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2312_07008_gb300 as pkg  # noqa: E402

# A range's row is scaled to a norm bound 2^39.8 = LIMIT of 9 moduli (10: 2^44.3); the bound from
# tiles' largest elements is at most 32^1/2 times the norm and the scale a power of
# two, so |X| >= LIMIT / 11.4 = 8.4e10.  Rounding to integers (uniform, 0.29 rms) moves
# X . Y by 0.29 2^1/2 |X| rms, or 4.9e-12 of |x| |y|; six times that for the largest
# of the elements.  Sums over the ranges stay below the largest diagonal element of
# sum lambda+ sigma sigma^T, which the positive part dominates.
TOL = 3e-11


@pytest.mark.parametrize("ncore,nact,nvir", [
    (1, 0, 31), (2, 0, 32), (3, 0, 33), (8, 0, 65), (4, 0, 255), (4, 0, 257),
    (0, 2, 31), (2, 1, 33), (3, 2, 64), (2, 3, 129), (1, 2, 257)])
def test_density_at_the_edges(ncore, nact, nvir):
    p = make_problem(seed=7 + nvir, s=0.5, ncore=ncore, nact=nact, nvir=nvir, naux=70, nstates=2)
    ref = O.solve(p, cuts=())
    d = torch.full((nvir, nvir), float("nan"), dtype=torch.float64, device="cuda")
    e2 = pkg.dsrg_fno_vv_opdm(pkg.problem_from_synth(p, "cuda", pkg.SLICED_BF16, 0), d)
    got = d.cpu().numpy()
    scale = np.max(np.abs(ref["dvv"]))
    assert np.max(np.abs(got - ref["dvv"])) <= TOL * scale
    assert np.array_equal(got, got.T)
    assert abs(e2 - ref["e2"]) <= 1e-10 * abs(ref["e2"]) + 1e-12
