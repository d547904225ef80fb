"""The batch workers' workspaces are kept between calls with different numbers of
workers as long as they fit the share that each worker has."""
import pytest

from synth import make_problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2312_07008_gb300 as pkg  # noqa: E402


@pytest.mark.parametrize("precision", [pkg.FP64, pkg.SLICED_BF16])
def test_calls_with_few_and_many_workers_in_turn(precision):
    p = make_problem(3, 2, 40, 130, seed=9, nstates=2)
    probs = [pkg.problem_from_synth(p, "cuda", precision) for _ in range(24)]
    lib = pkg.load()
    pkg.dsrg_fno_release()
    start = lib.dsrg_fno_debug_workspace_allocations()
    energies = []
    for _ in range(4):
        for workers in (2, 8):
            res = pkg.dsrg_fno_batch_run(probs, nworkers=workers)
            assert all(r["status"] == 0 for r in res)
            energies += [r["e2"] for r in res]
    # every item needs the same few megabytes: one allocation for each worker that took one
    assert lib.dsrg_fno_debug_workspace_allocations() - start <= 8
    assert len(set(energies)) == 1
    pkg.dsrg_fno_release()
