"""The first fast-form call of a process on a stream that does not order itself
against the default stream (as the batch workers' streams and torch's side
streams do not): it gives what the next call gives, bit for bit."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = """
import torch
import paper_2312_07008_gb300 as pkg
from synth import make_problem
p = make_problem(seed=3, s=0.5, ncore=3, nact=2, nvir=40, naux=300, nstates=2)
prob = pkg.problem_from_synth(p, "cuda", pkg.SLICED_BF16)
st = torch.cuda.Stream()
torch.cuda.synchronize()
out = []
for _ in range(3):
    d = torch.full((40, 40), float("nan"), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    e = pkg.dsrg_fno_vv_opdm(prob, d, stream=st.cuda_stream)
    st.synchronize()
    out.append((e, d.cpu()))
assert all(e == out[0][0] and torch.equal(d, out[0][1]) for e, d in out), [e for e, _ in out]
"""


def test_first_call_on_a_side_stream():
    subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, check=True, timeout=300)
