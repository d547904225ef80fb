"""The divide-and-conquer eigensolver's element functions on the CPU: its
deflation, secular roots and vectors, replayed by plain loops, against LAPACK
on tridiagonal matrices at the edges of its leaves and of its deflation (no
coupling, tight clusters, repeated and graded eigenvalues)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def replay(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("dc") / "replay.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_2312_07008_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "host_replay", "eig_dc_replay.cpp"), "-o", so], check=True)
    lib = ctypes.CDLL(so)
    dp = ctypes.POINTER(ctypes.c_double)

    def solve(d, e):
        n = len(d)
        d = np.ascontiguousarray(d, dtype=np.float64)
        e = np.ascontiguousarray(np.append(e, 0.0), dtype=np.float64)
        lam, q, cnt = np.zeros(n), np.zeros((n, n)), np.zeros(2, dtype=np.int32)
        lib.eig_dc_replay(n, d.ctypes.data_as(dp), e.ctypes.data_as(dp), lam.ctypes.data_as(dp), q.ctypes.data_as(dp),
                          cnt.ctypes.data_as(ctypes.POINTER(ctypes.c_int)))
        return lam, q.T, cnt
    return solve


def tridiagonals(n):
    rng = np.random.default_rng(n)
    yield "random", rng.standard_normal(n), rng.standard_normal(n - 1), False
    yield "uncoupled", rng.standard_normal(n), np.zeros(n - 1), True
    yield "zero", np.zeros(n), np.zeros(n - 1), True
    yield "wilkinson", np.abs(np.arange(n) - n // 2).astype(float), np.ones(n - 1), False
    yield "glued", rng.standard_normal(n), 10.0 ** rng.uniform(-18, 0, n - 1), False
    yield "negative coupling", np.full(n, 2.0), -np.ones(n - 1), False
    yield "graded", 10.0 ** -np.linspace(0, 30, n), 0.5 * 10.0 ** -np.linspace(0, 30, n)[:-1], False
    yield "two values", np.where(np.arange(n) % 3 == 0, 2.5, 1e-3), 1e-13 * rng.standard_normal(n - 1), False


@pytest.mark.parametrize("n", [33, 48, 49, 64, 65, 129, 257])
def test_stages_against_lapack(replay, n):
    for name, d, e, all_deflated in tridiagonals(n):
        lam, q, cnt = replay(d, e)
        T = np.diag(d) + np.diag(e, 1) + np.diag(e, -1)
        scale = max(np.abs(T).max(), 1e-300)
        # n roundings of 2^-53 per entry, with a factor 4 for the levels
        tol = 4 * n * 2.0 ** -53
        assert np.abs(np.sort(lam) - np.linalg.eigvalsh(T)).max() <= tol * scale, name
        assert np.abs(q.T @ q - np.eye(n)).max() <= tol, name
        assert np.abs((q * lam) @ q.T - T).max() <= tol * scale, name
        if all_deflated:
            assert cnt[0] > 0 and cnt[1] == 0
