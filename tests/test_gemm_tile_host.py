"""The float64 GEMM's tile rule on the CPU: whatever tile it takes, the launch has
no more row tiles than a grid may have whenever 64-row tiles fit one."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
GRID = 65535


@pytest.fixture(scope="module")
def tile(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("tile") / "replay.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_2312_07008_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "host_replay", "gemm_tile_replay.cpp"), "-o", so], check=True)
    lib = ctypes.CDLL(so)
    lib.replay_gemm_tile.argtypes = [ctypes.c_long, ctypes.c_long, ctypes.c_int]
    return lib.replay_gemm_tile


@pytest.mark.parametrize("N", [1, 10, 16, 17, 32, 33, 64, 144, 400])
@pytest.mark.parametrize("M", [1, 300, 16 * GRID - 1, 16 * GRID, 16 * GRID + 1, 1_100_000, 32 * GRID, 32 * GRID + 1, 64 * GRID])
def test_row_tiles_fit_a_launch(tile, M, N):
    T = tile(M, N, 1)
    assert T in (16, 32, 64) and -(-M // T) <= GRID


def test_small_products_fill_the_chip(tile):
    assert tile(300, 300, 1) == 16 and tile(1200, 1200, 1) in (32, 64) and tile(3600 * 70, 203, 1) in (32, 64)
