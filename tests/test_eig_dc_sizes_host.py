"""Launch sizes of the divide-and-conquer eigensolver on the CPU: on every level
every node fits the rows and the shared memory that its launch is given, up to
the largest matrix that the dispatch lets in."""
import ctypes
import os
import re
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2312_07008_gb300", "csrc")
MIN_N, MAX_N = map(int, re.search(r"EIG_DC_MIN_N = (\d+), EIG_DC_MAX_N = (\d+)", open(os.path.join(CSRC, "kernels.h")).read()).groups())


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("dc") / "replay.so")
    host = os.path.join(ROOT, "tests", "host_replay")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", host, "-I", CSRC,
                    os.path.join(host, "eig_dc_sizes_replay.cpp"), "-o", so], check=True)
    return ctypes.CDLL(so)


@pytest.mark.parametrize("n", [MIN_N, 34, 63, 64, 65, 511, 512, 513, 1747, 4095, 4096, 4097, MAX_N - 1, MAX_N])
def test_nodes_fit_their_launch(lib, n):
    per_row = 30                       # three words of 8 bytes, one of 4, two of 1
    for level in range(lib.replay_levels(n) + 1):
        bounds = [lib.replay_bound(n, level, t) for t in range((1 << level) + 1)]
        assert bounds[0] == 0 and bounds[-1] == n
        largest = max(b - a for a, b in zip(bounds, bounds[1:]))
        assert largest == lib.replay_node_rows(n, level)
        assert per_row * largest == lib.replay_deflate_bytes(n, level) <= per_row * MAX_N
    assert per_row * MAX_N + 1040 <= 232448     # beside the kernel's static shared memory
