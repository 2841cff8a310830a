"""Placements that share the steps of a warp (csrc/eval_pack.cu): a large, lightly loaded batch.  Sizes around the widths of
a group, the last groups of a bucket empty, waits and rejections in some groups only, epochs moved, one-token requests,
placements that leave the 32-bit horizon while their neighbours do not."""
import numpy as np
import pytest

import gen
from test_gpu_walk import _check, _lists

pytestmark = pytest.mark.gpu


def _trace(n, rate, seed, models, far):
    tr = gen.make_trace(n, rate, seed, model_mix=models)
    rng = np.random.default_rng(seed)
    tr["out_tokens"][rng.random(n) < 0.1] = 1
    if far:  # pauses beyond the reach of an epoch, and decodes beyond the horizon
        tr["arrival_us"][n // 3:] += 200_000_000
        tr["arrival_us"][n // 2:] += 7_000_000_000
        tr["out_tokens"][rng.random(n) < 0.02] = 65535
    return tr


@pytest.mark.parametrize("flags", [0, 1])
@pytest.mark.parametrize("far", [False, True])
def test_one_model(oracle_mod, flags, far):
    import paper_2509_06362_b200 as m
    prof, rng = gen.profile_node(1), np.random.default_rng(5)
    lists = _lists(prof, rng, (1, 2, 3, 4, 5, 8), (2, 16, 32, 64), 1060)
    lists += _lists(prof, rng, (1, 2, 4, 7, 8, 9, 17), (1, 2), 5)
    classes = gen.make_classes([(None, None, None)] * 3 if far else [(500_000, 50_000, None), (2_000_000, 150_000, None), (None, None, 180_000_000)])
    off, inst = gen.candidates_from_lists(lists)
    mask = None if far else rng.integers(0, 8, size=len(lists)).astype(np.uint32)
    want = _check(oracle_mod, m, prof, _trace(150, 3.0, 7, (1.0,), far), classes, off, inst, flags, mask)
    assert (want["attempts"] > want["n_counted"]).any() and (want["n_served"] > 0).mean() > 0.5


@pytest.mark.parametrize("flags", [0, 1])
def test_three_models(oracle_mod, flags):
    import paper_2509_06362_b200 as m
    prof, rng = gen.profile_multimodel(1), np.random.default_rng(6)
    lists = _lists(prof, rng, (3, 5, 6, 8), (4, 32, 64), 4610) + _lists(prof, rng, (1, 2, 10), (1, 64), 33)
    classes = gen.make_classes([(500_000, 50_000, None), (2_000_000, 150_000, None), (None, None, 180_000_000)])
    off, inst = gen.candidates_from_lists(lists)
    _check(oracle_mod, m, prof, _trace(60, 2.0, 8, (0.6, 0.3, 0.1), False), classes, off, inst, flags)
