"""The step counts of the walking and packed kernels (csrc/steps.cuh, compiled here without CUDA): ceil(dt / s) from a high product,
over the steps and times the kernels take and at their edges."""
import ctypes
import os
import random
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    lib = str(tmp_path_factory.mktemp("steps") / "libsteps.so")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-Wall", "-Werror", "-shared", "-fPIC", "-o", lib, os.path.join(HERE, "steps_host.cpp")])
    lib = ctypes.CDLL(lib)
    for f in (lib.exact_steps, lib.corrected_steps, lib.corrected_steps64):
        f.restype, f.argtypes = ctypes.c_uint32, [ctypes.c_int64, ctypes.c_uint32]
    return lib


@pytest.mark.parametrize("steps, largest, s_most", [("exact_steps", (1 << 31) - (1 << 24) - 1, 1 << 24), ("corrected_steps", (1 << 31) - 1, 1 << 30),
                                                    ("corrected_steps64", (1 << 50) - 1, 1 << 30)])
def test_step_counts(host, steps, largest, s_most):
    rng, f = random.Random(1), getattr(host, steps)
    sizes = [1, 2, 3, 5, 7, 40, 641, 9150, 65535, 65536, 65537, s_most - 1, s_most] + [rng.randrange(1, 1 << rng.randrange(1, s_most.bit_length())) for _ in range(400)]
    for s in sizes:
        for dt in [0, 1, s - 1, s, s + 1, 7 * s - 1, 7 * s, 7 * s + 1, largest - 1, largest, largest // s * s] + [rng.randrange(largest + 1) for _ in range(60)]:
            if 0 <= dt <= largest:
                want = -(-dt // s)
                if want < 1 << 32:
                    assert f(dt, s) == want, (dt, s)
