"""The residue form's constant tables on the CPU (csrc/residue.cuh)."""
import ctypes
import os
import subprocess

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
    return ctypes.CDLL(so)


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
