"""The workspace of a density pass holds what the pass uses: in the residue form no
partial sums of the rank-K update."""
import pytest

from synth import make_problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2312_07008_gb300 as pkg  # noqa: E402


def pad64(k):
    return -(-k // 64) * 64


def test_workspace_of_a_closed_shell_density():
    nh, nv, nq = 6, 700, 200
    p = make_problem(nh, 0, nv, nq, seed=2, nstates=1)
    d = torch.empty((nv, nv), dtype=torch.float64, device="cuda")
    pkg.dsrg_fno_release()
    pkg.dsrg_fno_vv_opdm(pkg.problem_from_synth(p, "cuda", pkg.SLICED_BF16), d)
    held = pkg.dsrg_fno_debug_workspace_bytes()
    pairs, outs = nh * (nh + 1) // 2, nh * nh                       # one dressed matrix of (m, m), two of (m, n)
    tile = 10 * 256 * 256 * 2                                       # residues of an output tile
    rows = -(-nv // 256)
    least = 8                                                       # ranges of the update: 20 * 76 / (10 * 6 tiles) is 25
    least = max(least, 20 * 76 // (10 * rows * (rows + 1) // 2))
    need = 8 * nv * nv * (2 * pairs + outs)                         # tau, kappa, dressed matrices
    need += 20 * nh * nv * pad64(nq) + 20 * outs * nv * pad64(nv)   # planes of B and of the dressed matrices
    need += 4 * outs * nv * -(-nv // 16)                            # norms of their rows' tiles
    need += 2 * least * (rows * (rows + 1) // 2) * tile             # residues of the update
    need += pairs * (-(-nv // 256) + 1) ** 2 * tile                 # residues of the contraction, at most
    assert held <= need + (8 << 20)
    pkg.dsrg_fno_release()
