"""End indexes of the packed kernel's keys (csrc/eval_pack.cu) when instances are never idle: the step counters go past what a key
holds and are moved back between chunks of requests."""
import numpy as np
import pytest

import gen
from test_gpu_pack import _mostly_not_loaded
from test_gpu_walk import _check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flags", [0, 1])
def test_counters_moved_back(oracle_mod, flags):
    import paper_2509_06362_b200 as m
    rng = np.random.default_rng(2)
    W, n = gen.WMAX, 1100
    step = np.ones((1, 2, W), dtype=np.int32)
    step[0, 1] = 2  # steps of 1 and 2 us
    prof = {"n_models": 1, "n_strategies": 2, "wmax": W, "devices": np.ones(2, dtype=np.int32), "min_devices": np.ones(1, dtype=np.int32),
            "prefill_base_us": np.zeros((1, 2), dtype=np.int32), "prefill_q16": np.zeros((1, 2), dtype=np.int32), "step_us": step}
    tr = np.zeros(n, dtype=gen.REQUEST_DTYPE)
    tr["arrival_us"] = np.cumsum(rng.integers(30_000, 40_000, size=n))  # every request overlaps the next: 38 million steps without a pause
    tr["out_tokens"] = rng.integers(60_000, 65_536, size=n)
    lists = [[(0, int(rng.integers(2)), int(rng.choice([4, 9, 16, 64]))) for _ in range(k)] for k in [1, 2, 3, 4, 5, 8] * 700]
    lists[:40] = [[(0, 0, 8)], [(0, 1, 4)]] * 20
    assert _mostly_not_loaded(prof, lists, [tr])
    off, inst = gen.candidates_from_lists(lists)
    want = _check(oracle_mod, m, prof, tr, gen.make_classes([(None, None, None)]), off, inst, flags)
    assert (want["n_served"] == n).all() and want["makespan_us"].max() > 1 << 25
