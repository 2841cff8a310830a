"""Requests with much time looked at by themselves (csrc/walk_dynamic.cuh): traces that end in and between chunks, with the patient
requests spread, in one piece, at either end, none or all of them; placements that fall behind by more than the others' limits and
catch up again; masks that leave one kind out; traces with and without such requests in one call."""
import numpy as np
import pytest

import gen
from gpu_common import assert_records_equal

pytestmark = pytest.mark.gpu

CLASSES = [(500_000, 50_000, None), (2_000_000, None, 60_000_000), (None, None, 120_000_000), (100_000_000, None, None)]


def _trace(n, kind, rng):
    tr = gen.make_trace(max(n, 1), 40.0, 5, model_mix=(0.5, 0.3, 0.2), cv=3.0)[:n]
    patient = {"spread": rng.random(n) < 0.2, "block": np.arange(n) // 100 % 3 == 1, "first": np.arange(n) < 5,
               "last": np.arange(n) >= n - 5, "none": np.zeros(n, bool), "all": np.ones(n, bool)}[kind]
    tr["cls"] = np.where(patient, rng.integers(2, 4, size=n), rng.integers(0, 2, size=n))
    tr["out_tokens"] = np.where(patient, rng.integers(1, 3000, size=n), rng.integers(1, 300, size=n))
    # quiet stretches in which a placement that has fallen behind catches up
    tr["arrival_us"] += np.cumsum(np.where(np.arange(n) % 211 == 210, 90_000_000, 0))
    return tr


def _placements(prof, rng):
    ok = [(m, s) for m in range(3) for s in range(prof["n_strategies"]) if prof["devices"][s] >= prof["min_devices"][m]]
    return gen.candidates_from_lists([[ok[i] + (int(rng.choice([1, 4, 16, 64])),) for i in rng.integers(0, len(ok), size=k)]
                                      for k in [0, 1, 1, 2, 2, 3, 3, 4, 6, 8, 16, 32] * 3])


@pytest.mark.parametrize("flags", [0, 1])
@pytest.mark.parametrize("kind, n", [("spread", 31), ("spread", 32), ("spread", 1000), ("spread", 1313), ("block", 1201), ("first", 800),
                                     ("last", 831), ("none", 500), ("all", 500)])
def test_records(oracle_mod, kind, n, flags):
    import paper_2509_06362_b200 as m
    rng = np.random.default_rng(n)
    prof = gen.profile_multimodel(1)
    off, inst = _placements(prof, rng)
    classes = gen.make_classes(CLASSES)
    tr = _trace(n, kind, rng)
    c = m.Context(0)
    c.load_profile(prof)
    t = c.load_trace(tr, classes)
    d_off, d_inst = c.to_device(off), c.to_device(inst)
    for mask in (None, 3, 12, 4, 2, 9):
        mk = None if mask is None else np.full(len(off) - 1, mask, dtype=np.uint32)
        got = c.results_to_numpy(c.eval_placements(t, d_off, d_inst, 1024, None if mk is None else c.to_device(mk), flags))
        assert_records_equal(got, oracle_mod.eval_placements(prof, tr, classes, off, inst, 1024, mk, flags), f"mask {mask}")
    c.close()


def test_several_traces(oracle_mod):
    import paper_2509_06362_b200 as m
    rng = np.random.default_rng(3)
    prof = gen.profile_multimodel(1)
    off, inst = _placements(prof, rng)
    classes = gen.make_classes(CLASSES)
    traces = [_trace(n, k, rng) for n, k in ((700, "spread"), (333, "none"), (0, "none"), (640, "block"))]
    c = m.Context(0)
    c.load_profile(prof)
    out = c.eval_placements_multi([c.load_trace(t, classes) for t in traces], c.to_device(off), c.to_device(inst), 1024)
    got = c.results_to_numpy(out).reshape(len(traces), len(off) - 1)
    for g, t in zip(got, traces):
        assert_records_equal(g, oracle_mod.eval_placements(prof, t, classes, off, inst, 1024, None, 0), len(t))
    c.close()


@pytest.mark.parametrize("rows", [[(0, None, None), (1, None, None), (None, None, None)], [(7, None, None), (None, None, 56)],
                                  [(1_000_000, None, None), (None, None, (1 << 30) - 1)], [(1_000_000, None, None), (1 << 31, None, None)]])
def test_limits(oracle_mod, rows):
    """No time at all, limits whose ratio is just enough, the largest that 32-bit times hold and beyond."""
    import paper_2509_06362_b200 as m
    rng = np.random.default_rng(8)
    prof = gen.profile_multimodel(1)
    off, inst = _placements(prof, rng)
    classes = gen.make_classes(rows)
    tr = _trace(900, "spread", rng)
    tr["cls"] = np.where(rng.random(900) < 0.3, len(rows) - 1, rng.integers(0, len(rows) - 1, size=900))
    c = m.Context(0)
    c.load_profile(prof)
    got = c.results_to_numpy(c.eval_placements(c.load_trace(tr, classes), c.to_device(off), c.to_device(inst), 1024))
    assert_records_equal(got, oracle_mod.eval_placements(prof, tr, classes, off, inst, 1024, None, 0), "records")
    c.close()
