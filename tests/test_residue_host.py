"""Arithmetic of the residue form on the CPU (csrc/residue.cuh): the residues
represent the integers of a row, and reduced chunk sums of their products give
back the product of the rows, for rows of every shape the form accepts (equal
entries, one large entry, tiny and huge scales, the largest norm)."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
dp = ctypes.POINTER(ctypes.c_double)
fp = ctypes.POINTER(ctypes.c_float)


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("res") / "replay.so")
    host = os.path.join(ROOT, "tests", "host_replay")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", host, "-I",
                    os.path.join(ROOT, "paper_2312_07008_gb300", "csrc"), os.path.join(host, "residue_replay.cpp"), "-o", so],
                   check=True)
    L = ctypes.CDLL(so)
    L.replay_norm_limit.restype = L.replay_half_mantissa.restype = ctypes.c_double
    L.replay_row_shift.argtypes = [ctypes.c_double, ctypes.c_int, ctypes.c_int]
    L.replay_reduce.restype = ctypes.c_float
    L.replay_crt.restype = ctypes.c_ulonglong
    return L


def stage(lib, nm, v):
    n = len(v)
    f = lib.replay_row_shift(float(v @ v), n, nm)
    X, r = np.zeros(n, dtype=np.int64), np.zeros((nm, n), dtype=np.float32)
    v = np.ascontiguousarray(v)
    lib.replay_residues(nm, n, v.ctypes.data_as(dp), f, X.ctypes.data_as(ctypes.POINTER(ctypes.c_longlong)),
                        r.ctypes.data_as(fp))
    return f, X, r


def rows(n):
    rng = np.random.default_rng(n)
    yield rng.standard_normal(n)
    yield rng.standard_normal(n) * np.exp(-0.05 * np.arange(n))
    yield np.full(n, 0.7)
    yield np.where(np.arange(n) == n // 2, 1.0, 1e-9)
    yield 1e-25 * rng.standard_normal(n)
    yield 1e20 * rng.standard_normal(n)
    yield np.zeros(n)


@pytest.mark.parametrize("nm", [10, 12])
def test_moduli_are_coprime_and_their_product_is_what_the_scale_assumes(lib, nm):
    p = [lib.replay_modulus(i) for i in range(nm)]
    assert all(np.gcd(a, b) == 1 for i, a in enumerate(p) for b in p[:i]) and max(p) <= 512
    M = 1
    for q in p:
        M *= q
    half = Fraction(lib.replay_half_mantissa(nm)) * 2 ** lib.replay_half_exponent(nm)
    assert abs(half / Fraction(M, 2) - 1) < Fraction(1, 2 ** 50)
    assert Fraction(lib.replay_norm_limit(nm)) ** 2 < Fraction(M, 2)


@pytest.mark.parametrize("nm,n", [(10, 1), (10, 256), (10, 700), (12, 300)])
def test_product_of_rows(lib, nm, n):
    M = 1
    for i in range(nm):
        M *= lib.replay_modulus(i)
    staged = [(v, *stage(lib, nm, v)) for v in rows(n)]
    for v, f, X, r in staged:
        assert np.all(np.abs(r) <= 256)
        for i in range(nm):
            p = lib.replay_modulus(i)
            assert np.all((X - r[i].astype(np.int64)) % p == 0)
        norm = sum(int(x) ** 2 for x in X)
        assert 2 * norm < M
        if v.any():
            assert norm ** 0.5 > 0.45 * lib.replay_norm_limit(nm) or n == 1      # no precision given away
    for a, (v, fa, X, r) in enumerate(staged):
        for w, fb, Y, s in staged[a:]:
            Z = sum(int(x) * int(y) for x, y in zip(X, Y))
            red = np.zeros(nm, dtype=np.float32)
            for i in range(nm):
                prod = r[i].astype(np.float64) * s[i]
                chunks = np.add.reduceat(prod, np.arange(0, n, 256)).astype(np.float32)
                assert np.all(np.abs(chunks) <= 2.0 ** 24)
                red[i] = lib.replay_reduce(np.ascontiguousarray(chunks).ctypes.data_as(fp), len(chunks), i)
                assert int(red[i]) % lib.replay_modulus(i) == Z % lib.replay_modulus(i)
            u = int(lib.replay_crt(nm, red.ctypes.data_as(fp)))
            u -= (u >> 63) << 64
            # weights rounded to 2^-64: nm residues of at most 2^9, half a unit each
            assert abs(u - Fraction(Z * 2 ** 64, M)) <= nm * 2 ** 8


@pytest.mark.parametrize("nm", [10, 12])
def test_reduction_is_exact_next_to_every_half_period(lib, nm):
    """Sums up to 2^24 next to odd multiples of p / 2, where the rounded
    quotient may go either way: the residue stays right and within p / 2 + 1."""
    rng = np.random.default_rng(nm)
    for i in range(nm):
        p = lib.replay_modulus(i)
        k = np.unique(np.concatenate([np.arange(0, 2 ** 24 // p, 97), [2 ** 24 // p - 1]]))
        for t in np.concatenate([k * p + p // 2 + o for o in (-1, 0, 1)] + [rng.integers(-2 ** 24, 2 ** 24, 200)]):
            x = np.array([t], dtype=np.float32)
            assert int(lib.replay_reduce(x.ctypes.data_as(fp), 1, i)) % p == int(t) % p
