"""Placements of more than 32 instances side by side with smaller ones that need one, two and more parts of a warp's shared memory, and
with smaller ones that queues have replayed in parts."""
import numpy as np
import pytest

import gen
from gpu_common import assert_records_equal

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flags", [0, 1, 2, 8, 9])
@pytest.mark.parametrize("n_small, n_big", [(60, 5), (2400, 100)])
def test_rooms(oracle_mod, n_small, n_big, flags):
    import paper_2509_06362_b200 as m
    rng = np.random.default_rng(n_small)
    prof = gen.profile_multimodel(1)
    ok = [(k, s) for k in range(3) for s in range(prof["n_strategies"]) if prof["devices"][s] >= prof["min_devices"][k]]
    # a slot takes some 12 bytes: 32 instances of 64 slots each need several times what one of 16 warps has
    caps = [(1, 2), (16,), (32, 64), (64,)]
    lists = []
    for i in range(n_small + n_big):
        n = int(rng.integers(1, 33)) if i < n_small else int(rng.integers(33, 129))
        lists.append([ok[j] + (int(rng.choice(caps[i % 4])),) for j in rng.integers(0, len(ok), size=n)])
    rng.shuffle(lists)
    off, inst = gen.candidates_from_lists(lists)
    tr = gen.make_trace(150, 80.0, 3, model_mix=(0.6, 0.3, 0.1))
    classes = gen.make_classes([(500_000, 50_000, None), (2_000_000, 150_000, None), (None, None, 180_000_000)])
    c = m.Context(0)
    c.load_profile(prof)
    got = c.results_to_numpy(c.eval_placements(c.load_trace(tr, classes), c.to_device(off), c.to_device(inst), 1024, flags=flags))
    assert_records_equal(got, oracle_mod.eval_placements(prof, tr, classes, off, inst, 1024, None, flags), f"flags {flags}")
    c.close()
