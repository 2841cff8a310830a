"""Rounds of the walking kernel's usual body (csrc/walk_dynamic.cuh) where they can go wrong: many completions at one boundary
(more than the ring holds, and at the boundary a request waits for), choices more than a minute ahead, where keys are cut off,
requests of one token that find everything full, waits that move the epoch, batch caps at the edges of a block of slots."""
import numpy as np
import pytest

import gen
from test_gpu_walk import _check

pytestmark = pytest.mark.gpu


def _profile(steps, prefill_base, q16=0):
    s, W = len(steps), gen.WMAX
    step = np.zeros((2, s, W), dtype=np.int32)
    for k, (base, slope) in enumerate(steps):
        step[:, k] = base + slope * np.arange(W)
    return {"n_models": 2, "n_strategies": s, "wmax": W, "devices": np.ones(s, dtype=np.int32), "min_devices": np.ones(2, dtype=np.int32),
            "prefill_base_us": np.full((2, s), prefill_base, dtype=np.int32), "prefill_q16": np.full((2, s), q16, dtype=np.int32),
            "step_us": step}


def _requests(n, gaps, outs, rng, two_models=True):
    tr = np.zeros(n, dtype=gen.REQUEST_DTYPE)
    tr["arrival_us"] = np.cumsum(rng.choice(gaps, size=n))
    tr["in_tokens"] = rng.choice([0, 7, 500], size=n)
    tr["out_tokens"] = rng.choice(outs, size=n)
    tr["cls"] = rng.integers(0, 3, size=n)
    tr["model"] = rng.integers(0, 2, size=n) if two_models else 0
    return tr


@pytest.mark.parametrize("flags", [0, 1])
@pytest.mark.parametrize("case", ["together", "far ahead", "one token", "epochs"])
def test_rounds(oracle_mod, case, flags):
    import paper_2509_06362_b200 as m
    rng = np.random.default_rng(77)
    n, q16 = 1200, 0
    caps = [1, 2, 7, 8, 9, 16, 63, 64]
    classes = gen.make_classes([(None, None, None), (None, None, None), (None, None, (1 << 30) - 1)])
    if case == "together":  # no prefill, steps and lengths that divide one another: whole batches end at one boundary
        prof, tr = _profile([(1000, 0), (2000, 0), (500, 500)], 0), _requests(n, [0, 0, 0, 0, 1000, 30_000], [2, 3, 5, 5, 9], rng)
    elif case == "far ahead":  # waits and prefills of minutes
        prof, tr = _profile([(1 << 20, 0), (1 << 22, 7), (3000, 1)], 40_000_000), _requests(n, [0, 1000, 10 ** 6], [1, 2, 30], rng)
        n, q16 = 300, 65536
        tr = tr[:n]
    elif case == "one token":
        prof, tr = _profile([(30_000, 100), (9000, 0), (17, 1)], 2000, 3000), _requests(n, [0, 10, 4000], [1, 1, 1, 40], rng)
        classes = gen.make_classes([(200_000, 5000, None), (50_000, None, 900_000), (None, 40_000, None)])
    else:  # an epoch's reach is 2^27 us: pauses around it, and waits that get there
        prof, tr = _profile([(50_000, 11), (1 << 21, 0), (70_001, 3)], 1000, 100), _requests(n, [0, 1000, 10 ** 6, (1 << 27) - 1, 1 << 27], [2, 40, 200], rng)
    lists = []
    for k in (1, 2, 3, 8, 31, 32):
        for _ in range(6):
            lists.append([(int(rng.integers(2)), int(rng.integers(3)), int(rng.choice(caps))) for _ in range(k)])
    lists += [[(0, 0, 64), (0, 0, 64), (1, 1, 64), (1, 2, 64)], [(0, 0, 64)] * 16 + [(1, 0, 64)] * 16]
    off, inst = gen.candidates_from_lists(lists)
    mask = np.array([(1 + i) % 8 or 7 for i in range(len(lists))], dtype=np.uint32)
    for mk in (None, mask):
        want = _check(oracle_mod, m, prof, tr, classes, off, inst, flags, mk)
    assert want["n_served"].max() > 100 and (want["attempts"] > want["n_counted"]).any()


@pytest.mark.parametrize("flags", [8, 9])
@pytest.mark.parametrize("n_models", [1, 2, 5])
def test_queues_by_model(oracle_mod, n_models, flags):
    """With queues the models of a placement are replayed side by side: placements of no, some and all models, requests of models
    that a placement has no instance of (reported by one part only), several traces in one pass."""
    import torch
    import paper_2509_06362_b200 as m
    from gpu_common import assert_records_equal
    rng = np.random.default_rng(5)
    W = gen.WMAX
    prof = {"n_models": n_models, "n_strategies": 2, "wmax": W, "devices": np.ones(2, dtype=np.int32), "min_devices": np.ones(n_models, dtype=np.int32),
            "prefill_base_us": rng.integers(0, 3000, size=(n_models, 2)).astype(np.int32), "prefill_q16": np.full((n_models, 2), 9000, dtype=np.int32),
            "step_us": rng.integers(5000, 30_000, size=(n_models, 2, W)).astype(np.int32)}
    lists = [[]] + [[(int(rng.integers(n_models)), int(rng.integers(2)), int(rng.choice([1, 3, 8, 64]))) for _ in range(int(rng.integers(1, 33)))] for _ in range(60)]
    lists += [[(n_models - 1, 1, 2)], [(0, 0, 1)] * 33]
    off, inst = gen.candidates_from_lists(lists)
    tr = _requests(700, [0, 1000, 60_000], [1, 2, 100, 400], rng)
    tr["model"] = rng.integers(0, n_models, size=len(tr))
    classes = gen.make_classes([(None, None, None), (600_000, 20_000, None), (None, None, 9_000_000)])
    mask = rng.integers(0, 8, size=len(lists)).astype(np.uint32)
    for mk in (None, mask):
        want = _check(oracle_mod, m, prof, tr, classes, off, inst, flags, mk)
    assert want["n_served"].max() > 100 and (want["n_rejected"] > 0).any()
    c = m.Context(0)
    c.load_profile(prof)
    traces = [tr, tr[:333], tr[:0], tr[100:]]
    out = c.eval_placements_multi([c.load_trace(t, classes) for t in traces], c.to_device(off), c.to_device(inst), 10 ** 6, c.to_device(mask), flags)
    torch.cuda.synchronize()
    got = c.results_to_numpy(out).reshape(len(traces), len(lists))
    for k, t in enumerate(traces):
        assert_records_equal(got[k], oracle_mod.eval_placements(prof, t, classes, off, inst, 10 ** 6, mask, flags), f"trace {k}")
    c.close()


@pytest.mark.parametrize("n", [1332, 1333])  # as many parts as there may be, and one placement more: all of them whole
def test_queues_of_many_models(oracle_mod, n):
    import paper_2509_06362_b200 as m
    rng = np.random.default_rng(n)
    W = gen.WMAX
    prof = {"n_models": 16, "n_strategies": 1, "wmax": W, "devices": np.ones(1, dtype=np.int32), "min_devices": np.ones(16, dtype=np.int32),
            "prefill_base_us": rng.integers(0, 3000, size=(16, 1)).astype(np.int32), "prefill_q16": np.full((16, 1), 9000, dtype=np.int32),
            "step_us": rng.integers(5000, 30_000, size=(16, 1, W)).astype(np.int32)}
    off, inst = gen.candidates_from_lists([[(int(k), 0, int(rng.choice([1, 3, 8]))) for k in rng.integers(0, 16, size=16)] for _ in range(n)])
    tr = _requests(200, [0, 1000, 60_000], [1, 2, 100, 400], rng)
    tr["model"] = rng.integers(0, 16, size=len(tr))
    classes = gen.make_classes([(None, None, None), (600_000, 20_000, None), (None, None, 9_000_000)])
    want = _check(oracle_mod, m, prof, tr, classes, off, inst, 8)
    assert want["n_served"].max() > 50 and (want["n_rejected"] > 0).any()
