"""The step counts of the walking and packed kernels (csrc/walk_kernel.cuh: walk_steps, csrc/walk_dynamic.cuh: walk_exact_entry),
in whole numbers: ceil(dt / s) from a high product, over the steps and times the kernels take and at their edges."""
import random

import pytest

M32 = 0xFFFFFFFF


def _exact(dt, s):
    sh = (s - 1).bit_length() if s > 1 else 0
    m = ((1 << (31 + sh)) + s - 1) // s
    assert m <= M32 and (s << 5 | sh) <= M32
    d = 2 * (dt + s - 1)
    assert d <= M32
    return (d * m >> 32) >> sh


def _corrected(dt, s):
    rs, d = M32 // s, dt + s - 1
    assert d <= M32
    q = d * rs >> 32
    return q + (1 if d - q * s >= s else 0)


@pytest.mark.parametrize("steps, largest, s_most", [(_exact, (1 << 31) - (1 << 24) - 1, 1 << 24), (_corrected, (1 << 31) - 1, 1 << 30)])
def test_step_counts(steps, largest, s_most):
    rng = random.Random(1)
    sizes = [1, 2, 3, 5, 7, 40, 641, 9150, 65535, 65536, 65537, s_most - 1, s_most] + [rng.randrange(1, 1 << rng.randrange(1, s_most.bit_length())) for _ in range(400)]
    for s in sizes:
        for dt in [0, 1, s - 1, s, s + 1, 7 * s - 1, 7 * s, 7 * s + 1, largest - 1, largest, largest // s * s] + [rng.randrange(largest + 1) for _ in range(60)]:
            if 0 <= dt <= largest:
                assert steps(dt, s) == -(-dt // s), (dt, s)
