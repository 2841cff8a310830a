"""When the scan turns to the list of patient requests (csrc/walk_dynamic.cuh): lists that end early or become sparse, epochs that move while
the list is read, more classes than a mask has bits.  The same trace with further classes in between, which no request has, is loaded
without a list: the list must not cost what it cannot give."""
import numpy as np
import pytest

import gen
from gpu_common import assert_records_equal
from test_gpu_patient import _placements, _trace

pytestmark = pytest.mark.gpu

SHORT = [(500_000, 50_000, None), (2_000_000, 150_000, None)]
BETWEEN = [(14_000_000, None, None), (90_000_000, None, None), (600_000_000, None, None)]  # no ratio of eight


def _early(n, kind, rng):
    """Patient requests (class 2) at the beginning, after that none or few."""
    tr = gen.make_trace(n, 64.0, 5, model_mix=(0.6, 0.3, 0.1))
    r = np.arange(n)
    patient = r < n // 20
    if kind == "few":
        patient |= r % 700 == 0
    if kind == "thinner":
        patient |= (r % 50 == 0) & (r < n // 2) | (r % 333 == 0)
    tr["cls"] = np.where(patient, 2, rng.integers(0, 2, size=n))
    tr["out_tokens"] = np.where(patient, rng.integers(2000, 8000, size=n), rng.integers(1, 300, size=n))
    return tr


def _time(c, t, d_off, d_inst, mask):
    import torch
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    a.record()
    c.eval_placements(t, d_off, d_inst, 1024, mask)
    b.record()
    torch.cuda.synchronize()
    return a.elapsed_time(b)


@pytest.mark.parametrize("mask", [None, 4])
def test_cost(mask):
    import paper_2509_06362_b200 as m
    rng = np.random.default_rng(4)
    prof = gen.profile_multimodel(1)
    lists = [[(int(k), int(rng.choice((3, 6))), 8) for k in np.sort(rng.integers(0, 3, size=3))] for _ in range(6000)]
    off, inst = gen.candidates_from_lists(lists)
    tr = _early(40_000, "none", rng)
    c = m.Context(0)
    c.load_profile(prof)
    last = (None, None, 1_050_000_000)
    with_list, without = (c.load_trace(tr, gen.make_classes(SHORT + [last] + x)) for x in ([], BETWEEN))
    d_off, d_inst = c.to_device(off), c.to_device(inst)
    mk = None if mask is None else c.to_device(np.full(len(lists), mask, dtype=np.uint32))
    times = np.array([[_time(c, t, d_off, d_inst, mk) for t in (with_list, without)] for _ in range(12)])[2:]
    c.close()
    assert times[:, 0].min() < 1.05 * times[:, 1].min(), times


@pytest.mark.parametrize("limit", [60_000_000, 1_050_000_000, None])
@pytest.mark.parametrize("kind", ["none", "few", "thinner"])
def test_records(oracle_mod, kind, limit):
    import paper_2509_06362_b200 as m
    rng = np.random.default_rng(7)
    prof = gen.profile_multimodel(1)
    off, inst = _placements(prof, rng)
    classes = gen.make_classes(SHORT + [(None, None, limit)])
    tr = _early(6017, kind, rng)
    c = m.Context(0)
    c.load_profile(prof)
    t = c.load_trace(tr, classes)
    for mask in (None, 4, 6):
        mk = None if mask is None else np.full(len(off) - 1, mask, dtype=np.uint32)
        got = c.results_to_numpy(c.eval_placements(t, c.to_device(off), c.to_device(inst), 1024, None if mk is None else c.to_device(mk)))
        want = oracle_mod.eval_placements(prof, tr, classes, off, inst, 1024, mk, 0)
        assert_records_equal(got, want, f"mask {mask}")
        # clocks ahead of arrivals by more than an epoch's reach
        assert limit == 60_000_000 or (want["max_ttft_us"] > 1 << 27).any()
    c.close()


def test_more_classes_than_a_mask_has_bits(oracle_mod):
    import paper_2509_06362_b200 as m
    rng = np.random.default_rng(9)
    prof = gen.profile_multimodel(1)
    off, inst = _placements(prof, rng)
    tr = _trace(1313, "spread", rng)
    tr["cls"] = np.where(tr["cls"] >= 2, rng.integers(30, 40, size=1313), rng.integers(0, 30, size=1313))
    classes = gen.make_classes([(500_000 + 10_000 * k, 50_000, None) for k in range(30)] + [(None, None, 100_000_000 + 10_000_000 * k) for k in range(10)])
    c = m.Context(0)
    c.load_profile(prof)
    got = c.results_to_numpy(c.eval_placements(c.load_trace(tr, classes), c.to_device(off), c.to_device(inst), 1024))
    assert_records_equal(got, oracle_mod.eval_placements(prof, tr, classes, off, inst, 1024, None, 0), "40 classes")
    c.close()
