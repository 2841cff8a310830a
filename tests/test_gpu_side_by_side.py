"""Batches of placements of up to 32 instances and of more: the two kernels run side by side, on blocks that are shared out by how many of
each there are."""
import numpy as np
import pytest

import gen
from gpu_common import assert_records_equal

pytestmark = pytest.mark.gpu


def _batch(n_small, n_big, seed):
    rng = np.random.default_rng(seed)
    cfg = gen.make_config("multimodel", n_cand=1, n_req=10)
    prof = cfg["profile"]
    ok = [(m, s) for m in range(prof["n_models"]) for s in range(prof["n_strategies"]) if prof["devices"][s] >= prof["min_devices"][m]]
    sizes = np.concatenate([rng.integers(0, 33, size=n_small), rng.integers(33, 129, size=n_big)])
    rng.shuffle(sizes)
    lists = [[ok[i] + (int(rng.choice([1, 2, 8, 16, 64])),) for i in rng.integers(0, len(ok), size=n)] for n in sizes]
    off, inst = gen.candidates_from_lists(lists)
    return prof, cfg["classes"], off, inst


def _want(oracle_mod, prof, tr, classes, off, inst, flags):
    want = oracle_mod.eval_placements(prof, tr, classes, off, inst, 1024, None, flags)
    assert (want["status"] == 0).all() and want["n_served"].max() > 0
    return want


@pytest.mark.parametrize("flags", [0, 1, 2, 8])
@pytest.mark.parametrize("n_small, n_big", [(300, 1), (150, 40), (3, 200), (0, 150), (40, 0)])
def test_every_share(oracle_mod, n_small, n_big, flags):
    import paper_2509_06362_b200 as m
    prof, classes, off, inst = _batch(n_small, n_big, n_small + n_big)
    traces = [gen.make_trace(250 - 100 * i, 60.0 + 100 * i, 3 + i, model_mix=(0.6, 0.3, 0.1)) for i in range(2)]
    c = m.Context(0)
    c.load_profile(prof)
    handles = [c.load_trace(t, classes) for t in traces]
    d_off, d_inst = c.to_device(off), c.to_device(inst)
    one = c.results_to_numpy(c.eval_placements(handles[0], d_off, d_inst, 1024, flags=flags))
    both = c.results_to_numpy(c.eval_placements_multi(handles, d_off, d_inst, 1024, flags=flags)).reshape(2, len(off) - 1)
    for t, tr in enumerate(traces):
        want = _want(oracle_mod, prof, tr, classes, off, inst, flags)
        assert_records_equal(both[t], want, f"trace {t}")
        if t == 0:
            assert_records_equal(one, want, "one trace")
    c.close()


def test_in_a_graph(oracle_mod):
    """Captured, and replayed twice over cleared records."""
    import torch
    import paper_2509_06362_b200 as m
    prof, classes, off, inst = _batch(100, 30, 5)
    tr = gen.make_trace(200, 80.0, 9, model_mix=(0.6, 0.3, 0.1))
    c = m.Context(0)
    c.load_profile(prof)
    h = c.load_trace(tr, classes)
    d_off, d_inst = c.to_device(off), c.to_device(inst)
    out = c.eval_placements(h, d_off, d_inst, 1024)  # (buffers)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out = c.eval_placements(h, d_off, d_inst, 1024)
    want = _want(oracle_mod, prof, tr, classes, off, inst, 0)
    for _ in range(2):
        out.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert_records_equal(c.results_to_numpy(out), want, "replayed")
    del graph
    c.close()
