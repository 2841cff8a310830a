"""The walking kernel (csrc/walk_kernel.cuh) at its edges: placements of 0 to 128 instances, whose state is at and
beyond one and several warps' parts of the pool, and the 32-bit times: arrivals far beyond the
epoch, long waits, and placements that leave the horizon and are handed over in mid-trace."""
import numpy as np
import pytest

import gen
from gpu_common import assert_records_equal

pytestmark = pytest.mark.gpu


def _run(m, prof, tr, classes, off, inst, flags, mask=None):
    import torch
    c = m.Context(0)
    c.load_profile(prof)
    t = c.load_trace(tr, classes)
    n = len(off) - 1
    idx = np.arange(0, n, 3, dtype=np.uint32)
    rej = torch.empty((n, 16), dtype=torch.int32, device="cuda")
    hist = torch.empty((n, 64), dtype=torch.int32, device="cuda")
    d_mask = None if mask is None else c.to_device(mask)
    out, dumps = c.eval_placements(t, c.to_device(off), c.to_device(inst), 10 ** 6, d_mask, flags, dump_idx=idx,
                                   rejected_by_model=rej, ttft_hist=hist)
    torch.cuda.synchronize()
    got = c.results_to_numpy(out)
    res = got, {k: v.cpu().numpy() for k, v in dumps.items()}, rej.cpu().numpy(), hist.cpu().numpy(), idx
    c.close()
    return res


def _check(oracle_mod, m, prof, tr, classes, off, inst, flags, mask=None):
    got, gd, rej, hist, idx = _run(m, prof, tr, classes, off, inst, flags, mask)
    want, wd = oracle_mod.eval_placements(prof, tr, classes, off, inst, 10 ** 6, mask, flags, dump_idx=idx)
    assert_records_equal(got, want, f"flags {flags}")
    for k in wd:
        assert (gd[k] == wd[k]).all(), k
    assert (hist.sum(axis=1) == want["n_served"]).all()
    assert (rej.sum(axis=1) == want["n_rejected"]).all()
    return want


def _lists(prof, rng, sizes, caps, per_size):
    dev, mind = np.asarray(prof["devices"]), np.asarray(prof["min_devices"])
    lists = []
    for n in sizes:
        for _ in range(per_size):
            lst = []
            for _ in range(n):
                mod = int(rng.integers(prof["n_models"]))
                lst.append((mod, int(rng.choice(np.nonzero(dev >= mind[mod])[0])), int(rng.choice(caps))))
            lists.append(lst)
    return lists


@pytest.mark.parametrize("flags", [0, 1])
@pytest.mark.parametrize("seed", [0, 1, 2])
def test_placement_sizes_and_pool_parts(oracle_mod, seed, flags):
    import paper_2509_06362_b200 as m
    prof = gen.profile_multimodel(1)
    rng = np.random.default_rng(40 + seed)
    # 32 x 64 slots need several warps' parts
    lists = _lists(prof, rng, [0, 1, 3, 4, 5, 8, 9, 16, 17, 31, 32], [1, 2, 7, 8, 9], 4)
    lists += _lists(prof, rng, [1, 2, 4, 8, 16, 32], [63, 64], 3)
    lists += _lists(prof, rng, [33, 128], [1, 64], 2)
    order = rng.permutation(len(lists))
    off, inst = gen.candidates_from_lists([lists[i] for i in order])
    tr = gen.make_trace(900, 60.0, 5, model_mix=(0.5, 0.3, 0.2), cv=2.0)
    tr["out_tokens"][rng.random(len(tr)) < 0.1] = 1
    classes = gen.make_classes([(500_000, 50_000, None), (20_000_000, None, None), (None, None, 180_000_000)])
    want = _check(oracle_mod, m, prof, tr, classes, off, inst, flags)
    assert want["n_served"].max() > 300


@pytest.mark.parametrize("flags", [0, 1])
def test_times_at_and_beyond_the_horizon(oracle_mod, flags):
    import paper_2509_06362_b200 as m
    W = gen.WMAX
    rng = np.random.default_rng(9)
    step = np.zeros((2, 3, W), dtype=np.int32)
    step[:, 0] = 40 + np.arange(W)
    step[:, 1] = (1 << 24) - 1 - np.arange(W)   # the largest steps the kernel takes: most of these leave the horizon
    step[:, 2] = rng.integers(10_000, 30_000, size=(2, W))
    prof = {"n_models": 2, "n_strategies": 3, "wmax": W, "devices": np.array([1, 1, 2], dtype=np.int32),
            "min_devices": np.array([1, 1], dtype=np.int32),
            "prefill_base_us": np.array([[0, 1 << 20, 7], [3, 0, 1 << 24]], dtype=np.int32),
            "prefill_q16": np.array([[0, 65536, 65536], [1, 0, 12345]], dtype=np.int32), "step_us": step}
    n = 1500
    tr = np.zeros(n, dtype=gen.REQUEST_DTYPE)
    gaps = rng.choice([0, 1000, 10 ** 6, 10 ** 8, 5 * 10 ** 9, 3 * 10 ** 11], size=n, p=[0.2, 0.4, 0.25, 0.11, 0.03, 0.01])
    tr["arrival_us"] = np.minimum(np.cumsum(gaps), (1 << 50) - 1)
    tr["in_tokens"] = rng.choice([0, 1, 4096, 1 << 27], size=n, p=[0.3, 0.3, 0.35, 0.05])
    tr["out_tokens"] = rng.choice([1, 2, 300, 4000, 65535], size=n, p=[0.1, 0.2, 0.4, 0.25, 0.05])
    tr["cls"] = rng.integers(0, 3, size=n)
    tr["model"] = rng.integers(0, 2, size=n)
    classes = gen.make_classes([(None, None, None), ((1 << 30) - 1, None, (1 << 30) - 1), (10 ** 8, 10 ** 6, None)])
    lists = [[(0, 0, 64), (1, 0, 64)], [(0, 2, 4), (1, 2, 2)], [(0, 1, 1), (1, 1, 2)], [(0, 2, 64), (1, 2, 3), (0, 0, 1)],
             [(0, 0, 1)], [(1, 2, 64)] * 20, [(0, 2, 1), (1, 2, 1)], [(0, 0, 8), (0, 1, 8), (1, 0, 8), (1, 2, 1)]]
    off, inst = gen.candidates_from_lists(lists)
    want = _check(oracle_mod, m, prof, tr, classes, off, inst, flags)
    assert want["n_served"].max() > 500


def test_overloaded_without_limits(oracle_mod):
    """Requests that nothing turns away queue for hours at the dispatcher: arrivals far before the epoch."""
    import paper_2509_06362_b200 as m
    prof = gen.profile_decay()
    tr = gen.make_trace(2000, 4.0, 3, model_mix=(1, 1, 1), doc_class=None)
    tr["out_tokens"] = np.random.default_rng(4).integers(300, 1001, size=len(tr))
    classes = gen.make_classes([(None, None, None), (None, 60_000, None), (None, 100_000, None)])
    off, inst = gen.candidates_from_lists([[(0, 0, 1), (1, 0, 1), (2, 3, 1)], [(0, 0, 2), (1, 1, 4), (2, 6, 2)], [(2, 3, 1)]])
    mask = np.array([7, 7, 1], dtype=np.uint32)
    want = _check(oracle_mod, m, prof, tr, classes, off, inst, 0, mask)
    assert (want["max_ttft_us"] > 1 << 31).any()


def _past_the_horizon(seed, n_lists, n=96, heavy=0.2):
    """Placements of one model that get beyond the horizon in the middle of a chunk of 32 requests, with more requests behind:
    decodes of hours, prefills of minutes in a row, one-token requests, nothing has a limit."""
    rng = np.random.default_rng(seed)
    W = gen.WMAX
    step = np.empty((1, 6, W), dtype=np.int32)
    step[0, :4] = np.array([[1], [40], [33_500], [(1 << 24) - 1]])
    step[0, 4:] = rng.choice([1, 7, 1000, 33_500, 1 << 20, (1 << 24) - 1], size=(2, W))
    prof = {"n_models": 1, "n_strategies": 6, "wmax": W, "devices": np.ones(6, dtype=np.int32),
            "min_devices": np.ones(1, dtype=np.int32), "prefill_base_us": np.array([[0, 1, 2000, 0, 0, 5]], dtype=np.int32),
            "prefill_q16": np.full((1, 6), 65536, dtype=np.int32), "step_us": step}
    tr = np.zeros(n, dtype=gen.REQUEST_DTYPE)
    gaps = rng.choice([0, 1000, 10 ** 6, 10 ** 7], size=n)
    gaps[n - 1] = 2 * 10 ** 11  # and a long pause, so that little is asked of a placement on average
    tr["arrival_us"] = np.cumsum(gaps)
    tr["in_tokens"] = rng.choice([0, 1, 1000, 1 << 24, (1 << 28) - 4096], size=n, p=[0.2, 0.2, 0.4 - heavy, 0.2, heavy])
    tr["out_tokens"] = rng.choice([1, 2, 301, 65535], size=n, p=[0.4, 0.2, 0.4 - heavy, heavy])
    lists = [[(0, int(rng.choice(6, p=[0.3, 0.2, 0.2, 0.1, 0.1, 0.1])), int(rng.choice([1, 1, 2, 3, 8, 9, 64])))
              for _ in range(int(rng.choice([1, 1, 2, 3, 5, 8])))] for _ in range(n_lists)]
    lists[:2] = [[(0, 2, 1)], [(0, 0, 2)] * 40]
    return prof, tr, lists


@pytest.mark.parametrize("flags", [0, 1, 2, 3])
@pytest.mark.parametrize("seed", [0, 1, 2])
def test_rounds_behind_one_that_left_the_horizon(oracle_mod, seed, flags):
    import paper_2509_06362_b200 as m
    prof, tr, lists = _past_the_horizon(seed, 300)
    off, inst = gen.candidates_from_lists(lists)
    want = _check(oracle_mod, m, prof, tr, gen.make_classes([(None, None, None)]), off, inst, flags)
    assert (want["max_e2e_us"] > 0x60000000).mean() > 0.3


@pytest.mark.parametrize("flags", [0, 1, 2, 3, 8, 9])
def test_tables_and_limits_beyond_32_bit_times(oracle_mod, flags):
    """A batch that 32-bit times cannot hold runs with 64-bit ones from its start: decode steps and prefill bases of 2^30 us,
    inputs of four billion tokens, limits of 2^40 us, arrivals up to 2^50; placements of 1 to 128 instances."""
    import paper_2509_06362_b200 as m
    W = gen.WMAX
    rng = np.random.default_rng(23)
    step = np.zeros((2, 3, W), dtype=np.int32)
    step[:, 0] = 1 + np.arange(W)
    step[:, 1] = (1 << 30) - np.arange(W)
    step[:, 2] = rng.integers(1, 1 << 20, size=(2, W))
    prof = {"n_models": 2, "n_strategies": 3, "wmax": W, "devices": np.ones(3, dtype=np.int32), "min_devices": np.ones(2, dtype=np.int32),
            "prefill_base_us": np.array([[0, 1 << 30, 7], [3, 0, 1 << 20]], dtype=np.int32),
            "prefill_q16": np.array([[0, (1 << 31) - 1, 65536], [1, 0, 123456]], dtype=np.int32), "step_us": step}
    n = 500
    tr = np.zeros(n, dtype=gen.REQUEST_DTYPE)
    gaps = rng.choice([0, 1, 1000, 10 ** 7, 5 * 10 ** 9, 3 * 10 ** 12], size=n, p=[0.2, 0.2, 0.3, 0.2, 0.07, 0.03])
    tr["arrival_us"] = np.minimum(np.cumsum(gaps) * 20, (1 << 50) - 1)
    tr["in_tokens"] = rng.choice([0, 1, 4096, 2 ** 32 - 1], size=n, p=[0.4, 0.3, 0.25, 0.05])
    tr["out_tokens"] = rng.choice([1, 2, 300, 40000, 65535], size=n)
    tr["cls"] = rng.integers(0, 3, size=n)
    tr["model"] = rng.integers(0, 2, size=n)
    classes = gen.make_classes([(None, None, None), (1 << 40, 1 << 40, 1 << 40), (10 ** 9, 10 ** 6, None)])
    lists = _lists(prof, rng, (1, 2, 5, 8, 17, 32), (1, 2, 7, 64), 6) + _lists(prof, rng, (33, 64, 128), (1, 9, 64), 3)
    off, inst = gen.candidates_from_lists(lists)
    want = _check(oracle_mod, m, prof, tr, classes, off, inst, flags)
    assert (want["makespan_us"] > 1 << 40).all() and (want["status"] == 0).mean() > 0.5
