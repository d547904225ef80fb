"""The residue form's constant tables and the scales of its rows, over the whole range
of float64, on the CPU (csrc/residue.cuh)."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2312_07008_gb300", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("res") / "replay.so")
    host = os.path.join(ROOT, "tests", "host_replay")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", host, "-I", CSRC,
                    os.path.join(host, "residue_tables_replay.cpp"), "-o", so], check=True)
    L = ctypes.CDLL(so)
    L.replay_norm_limit.restype = ctypes.c_double
    return L


def test_every_constant_of_the_device_has_its_value_in_the_source():
    """A table copied to the device at run time is ordered before a kernel only on
    the stream of the copy; one initialised with the module always is."""
    for f in sorted(os.listdir(CSRC)):
        for line in open(os.path.join(CSRC, f)):
            if line.startswith("__constant__"):
                assert "=" in line, (f, line)


def test_table_of_moduli(lib):
    p, inv = ctypes.c_float(), ctypes.c_float()
    for i in range(12):
        lib.replay_modulus_table(i, ctypes.byref(p), ctypes.byref(inv))
        assert p.value == lib.replay_modulus(i)
        assert inv.value == np.float32(1.0) / np.float32(lib.replay_modulus(i))


def rows(n):
    rng = np.random.default_rng(n)
    z = rng.standard_normal(n)
    first = np.arange(n) < n // 2
    yield z
    for scale in (1e-300, 1e-290, 1e-200, 1e-160, 1e-150, 1e-144, 1e144, 1e150, 1e160, 1e200, 1e290):
        yield scale * z
        yield np.where(first, scale * z, z)                 # one share in range, one not
        yield np.where(first, scale * z, 1e-170 * z)        # neither, by different exponents
        yield np.where(np.arange(n) == n - 1, scale, 0.0)


@pytest.mark.parametrize("nm", [10, 12])
@pytest.mark.parametrize("n", [1, 2, 300, 1024])
def test_scale_of_rows_of_any_size(lib, nm, n):
    limit = lib.replay_norm_limit(nm)
    for v in rows(n):
        for nsplit in (1, 2, 4):
            X = np.zeros(n, dtype=np.int64)
            w = np.ascontiguousarray(v)
            f = lib.replay_stage(nm, n, w.ctypes.data_as(ctypes.POINTER(ctypes.c_double)), nsplit,
                                 X.ctypes.data_as(ctypes.POINTER(ctypes.c_longlong)))
            assert sum(int(x) ** 2 for x in X) ** 0.5 <= limit
            if not v.any():
                continue
            # at most the bits that a bound by the largest element costs (n^1/2), and the two of
            # the power of two below and of that element's exponent
            assert max(abs(int(x)) for x in X) * 4.1 * n ** 0.5 >= limit
            two_f = Fraction(2) ** f
            for k in np.unique(np.linspace(0, n - 1, 7).astype(int)):
                assert abs(Fraction(float(v[k])) * two_f - int(X[k])) <= Fraction(1, 2) or abs(v[k]) < 2.3e-308
            assert f != -100000
    for bad in (np.inf, np.nan):
        v = np.ones(n)
        v[n // 2] = bad
        assert lib.replay_stage(nm, n, v.ctypes.data_as(ctypes.POINTER(ctypes.c_double)), 1,
                                np.zeros(n, dtype=np.int64).ctypes.data_as(ctypes.POINTER(ctypes.c_longlong))) == -100000
