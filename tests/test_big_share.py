"""Blocks for placements of more than 32 instances beside smaller ones (csrc/route.cuh): enough to hold them at once, no fewer than their
share of the work, never more than there are blocks or placements."""
import ctypes
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def big_share(tmp_path_factory):
    lib = str(tmp_path_factory.mktemp("share") / "libshare.so")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-Wall", "-Werror", "-shared", "-fPIC", "-o", lib, os.path.join(HERE, "share_host.cpp")])
    f = ctypes.CDLL(lib).big_share
    f.restype, f.argtypes = ctypes.c_uint32, [ctypes.c_uint64, ctypes.c_uint64, ctypes.c_uint32, ctypes.c_uint32]
    return f


@pytest.mark.parametrize("grid", [1, 2, 148])
@pytest.mark.parametrize("warps", [1, 3, 16])
def test_bounds(big_share, warps, grid):
    for big in (1, 2, 15, 16, 17, 148, 149, 10_000, 1 << 40):
        last = None
        for small in (0, 1, 100, 2499, 30_000, 1 << 40):
            got = big_share(big, small, warps, grid)
            assert 1 <= got <= min(grid, big)
            assert got >= min(grid, big, -(-big // warps)) and got * (8 * big + small) >= min(8 * big * grid, min(grid, big) * (8 * big + small))
            assert last is None or got <= last  # more smaller placements, no more blocks for the larger ones
            last = got


def test_what_was_measured(big_share):
    """2,500 placements of which 100 are larger, 5,000 of which 12 are: counted by parts (two and three models) they got fewer blocks."""
    assert big_share(100, 2400, 6, 148) > big_share(100, 2400 * 2, 6, 148) > big_share(100, 2400 * 3, 6, 148)
    assert big_share(12, 4988, 6, 148) > big_share(12, 4988 * 3, 6, 148)
