"""Placements that share the steps of a warp (csrc/eval_pack.cu): a large, lightly loaded batch.  Sizes around the widths of
a group, the last groups of a bucket empty, waits and rejections in some groups only, epochs moved, one-token requests,
placements that leave the 32-bit horizon while their neighbours do not."""
import numpy as np
import pytest

import gen
from gpu_common import assert_records_equal
from test_gpu_walk import _check, _lists, _past_the_horizon

pytestmark = pytest.mark.gpu


def _trace(n, rate, seed, models, far):
    tr = gen.make_trace(n, rate, seed, model_mix=models)
    rng = np.random.default_rng(seed)
    tr["out_tokens"][rng.random(n) < 0.1] = 1
    if far:  # pauses beyond the reach of an epoch, and decodes beyond the horizon
        tr["arrival_us"][n // 3:] += 200_000_000
        tr["arrival_us"][n // 2:] += 7_000_000_000
        tr["out_tokens"][rng.random(n) < 0.2] = 65535
    return tr


def _leave(want):
    """Do some placements leave the 32-bit horizon, and most not?  (Times count from an epoch that is no later than a request's
    arrival, and less than 2^27 us earlier.)"""
    e2e = want["max_e2e_us"]
    return (e2e > 0x60000000).any() and (e2e < 0x60000000 - (1 << 27)).mean() > 0.5


def _mostly_not_loaded(prof, lists, traces):
    """Do the traces together (harmonic mean of their output tokens a second) leave most placements unloaded?  That and the
    size of the batch decide that it is packed."""
    rates = []
    for t in traces:
        span = (t["arrival_us"][-1] - t["arrival_us"][0]) * 1e-6 if len(t) > 1 else 0.0
        rates.append(t["out_tokens"].astype(np.int64).sum() / span if span else 1.0)
    demand = len(traces) / sum(1.0 / r for r in rates)
    supply = [sum(b * 1_000_000 // int(prof["step_us"][m, s, b - 1]) for m, s, b in lst) for lst in lists if 0 < len(lst) <= 8]
    return 2 * sum(demand >= 2 * x for x in supply) < len(supply)


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
    assert not far or _leave(want)


@pytest.mark.parametrize("flags", [0, 1])
def test_steps_behind_one_that_left_the_horizon(oracle_mod, flags):
    import paper_2509_06362_b200 as m
    prof, tr, lists = _past_the_horizon(3, 4300, heavy=0.1)
    off, inst = gen.candidates_from_lists(lists)
    assert _mostly_not_loaded(prof, lists, [tr])
    want = _check(oracle_mod, m, prof, tr, gen.make_classes([(None, None, None)]), off, inst, flags)
    gone = want["max_e2e_us"] > 0x60000000
    assert gone.mean() > 0.3 and (~gone).mean() > 0.05


@pytest.mark.parametrize("flags", [0, 1])
def test_three_models(oracle_mod, flags):
    import paper_2509_06362_b200 as m
    prof, rng = gen.profile_multimodel(1), np.random.default_rng(6)
    lists = _lists(prof, rng, (3, 5, 6, 8), (4, 32, 64), 4610) + _lists(prof, rng, (1, 2, 10), (1, 64), 33)
    classes = gen.make_classes([(500_000, 50_000, None), (2_000_000, 150_000, None), (None, None, 180_000_000)])
    off, inst = gen.candidates_from_lists(lists)
    _check(oracle_mod, m, prof, _trace(60, 2.0, 8, (0.6, 0.3, 0.1), False), classes, off, inst, flags)


@pytest.mark.parametrize("flags", [0, 1])
@pytest.mark.parametrize("far", [False, True])
@pytest.mark.parametrize("copies", [1, 3])  # 4,464 items: 12 warps per SM hold them at once; 13,392: 14 take several each
def test_several_traces(oracle_mod, copies, far, flags):
    """Every item of the packed kernel exists once per trace: records, unserved requests and histograms go to the trace's own
    block, traces of other lengths (an empty one among them) end at other times, and a placement that leaves the horizon under
    one trace is replayed under all of them."""
    import torch
    import paper_2509_06362_b200 as m
    prof, rng = gen.profile_node(1), np.random.default_rng(15)
    lists = _lists(prof, rng, (1, 2, 3, 4, 5, 8), (2, 16, 32, 64), 183) + _lists(prof, rng, (1, 3, 7, 9, 17, 33), (1, 2), 3)
    classes = gen.make_classes([(None, None, None)] * 3 if far else [(500_000, 50_000, None), (2_000_000, 150_000, None), (None, None, 180_000_000)])
    off, inst = gen.candidates_from_lists(lists)
    traces = [_trace(150, 3.0, 7, (1.0,), False), _trace(97, 2.0, 8, (1.0,), far), _trace(1, 2.0, 9, (1.0,), False)[:0],
              _trace(131, 1.0, 10, (1.0,), False)] * copies
    mask = None if far else rng.integers(0, 8, size=len(lists)).astype(np.uint32)
    n, n_tr = len(lists), len(traces)
    assert n * n_tr > 4096 and _mostly_not_loaded(prof, lists, traces)
    c = m.Context(0)
    c.load_profile(prof)
    handles = [c.load_trace(t, classes) for t in traces]
    rej = torch.full((n_tr * n, 16), 77, dtype=torch.int32, device="cuda")
    hist = torch.full((n_tr * n, 64), 77, dtype=torch.int32, device="cuda")
    out = c.eval_placements_multi(handles, c.to_device(off), c.to_device(inst), 10 ** 6, None if mask is None else c.to_device(mask),
                                  flags, rejected_by_model=rej, ttft_hist=hist)
    torch.cuda.synchronize()
    got = c.results_to_numpy(out).reshape(n_tr, n)
    rej, hist = (x.cpu().numpy().view(np.uint32).reshape(n_tr, n, -1) for x in (rej, hist))
    c.close()
    wanted = []
    for k, t in enumerate(traces[:4]):
        want = oracle_mod.eval_placements(prof, t, classes, off, inst, 10 ** 6, mask, flags)
        want_rej = oracle_mod.rejected_by_model(prof, t, classes, off, inst, 10 ** 6, mask, flags)
        want_hist = oracle_mod.ttft_hist(prof, t, classes, off, inst, 10 ** 6, mask, flags)
        for j in range(k, n_tr, 4):
            assert_records_equal(got[j], want, f"trace {j}, flags {flags}")
            assert (rej[j] == want_rej).all() and (hist[j] == want_hist).all(), j
        wanted.append(want)
    assert [_leave(w) for w in wanted] == [False, far, False, False]
