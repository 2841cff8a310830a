"""Placements whose room is at the edge of what the kernels have (csrc/route.cuh), scored on the GPU: tables of many rows together
with many classes and full batch caps, in batches that walk, that may pack, and with the thread mapping's smallest pools."""
import numpy as np
import pytest

import gen
from gpu_common import assert_records_equal, gpu_eval
from test_gpu_walk import _check

pytestmark = pytest.mark.gpu


def _tables(n_models, n_strategies, rng):
    W = gen.WMAX
    return {"n_models": n_models, "n_strategies": n_strategies, "wmax": W, "devices": np.ones(n_strategies, dtype=np.int32),
            "min_devices": np.ones(n_models, dtype=np.int32),
            "prefill_base_us": rng.integers(0, 3000, size=(n_models, n_strategies)).astype(np.int32),
            "prefill_q16": np.full((n_models, n_strategies), 9000, dtype=np.int32),
            "step_us": (rng.integers(5000, 20_000, size=(n_models, n_strategies, 1)) + 150 * np.arange(W)).astype(np.int32)}


def _placement(prof, n, cap, rng):
    return [(int(rng.integers(prof["n_models"])), int(rng.integers(prof["n_strategies"])), cap) for _ in range(n)]


def _workload(n, rate, n_models, n_classes, rng):
    tr = gen.make_trace(n, rate, 5, model_mix=(1.0,) * n_models)
    tr["cls"] = rng.integers(0, n_classes, size=n)
    tr["out_tokens"][rng.random(n) < 0.1] = 1
    limits = [(None, None, None), (500_000, 50_000, None), (None, None, 30_000_000), (3_000_000, 20_000, 90_000_000)]
    return tr, gen.make_classes([limits[i % 4] for i in range(n_classes)])


@pytest.mark.parametrize("flags", [0, 1, 2, 8])
@pytest.mark.parametrize("n_models", [1, 16])
@pytest.mark.parametrize("rows, n_classes", [(256, 256), (160, 71)])
def test_large_tables_and_full_caps(oracle_mod, rows, n_classes, n_models, flags):
    import paper_2509_06362_b200 as m
    rng = np.random.default_rng(rows + n_models)
    prof = _tables(n_models, rows // n_models, rng)
    sizes = [(n, cap) for n in (1, 7, 8, 31, 32, 33, 128) for cap in (8, 9, 64)]
    off, inst = gen.candidates_from_lists([_placement(prof, n, cap, rng) for n, cap in sizes])
    tr, classes = _workload(400, 100.0, n_models, n_classes, rng)
    want = _check(oracle_mod, m, prof, tr, classes, off, inst, flags)
    assert (want["status"] == 0).all() and want["n_served"].max() > 200


@pytest.mark.parametrize("flags", [0, 1])
@pytest.mark.parametrize("rows", [80, 81, 256])
def test_large_tables_and_64_bit_times(oracle_mod, rows, flags):
    import paper_2509_06362_b200 as m
    rng = np.random.default_rng(rows)
    prof = _tables(1, rows, rng)
    off, inst = gen.candidates_from_lists([_placement(prof, n, cap, rng) for n in (1, 8, 32, 33, 128) for cap in (1, 64)])
    tr, classes = _workload(400, 100.0, 1, 71, rng)
    classes["e2e_us"] = np.where(classes["e2e_us"] < 0, 1 << 39, classes["e2e_us"])
    want = _check(oracle_mod, m, prof, tr, classes, off, inst, flags)
    assert (want["status"] == 0).all() and want["n_served"].max() > 200


@pytest.mark.parametrize("flags", [0, 1])
@pytest.mark.parametrize("rows", [52, 53, 128, 129])
def test_rows_with_and_without_reciprocals(oracle_mod, rows, flags):
    """Either side of the lines from which on the rows carry no reciprocals: whatever a round divides by, steps of 1 us and of 2^24 - 1
    and an idle instance's among them."""
    import paper_2509_06362_b200 as m
    rng = np.random.default_rng(rows)
    prof = _tables(1, rows, rng)
    prof["step_us"][0, 0], prof["step_us"][0, 1] = 1, (1 << 24) - 1
    lists = [_placement(prof, n, cap, rng) for n in (1, 5, 32, 33, 70, 128) for cap in (1, 2, 9, 64)]
    off, inst = gen.candidates_from_lists(lists + [[(0, 0, 64)], [(0, 1, 3), (0, 0, 2)], [(0, 1, 1)] * 40 + [(0, 0, 64)] * 40])
    tr, classes = _workload(600, 60.0, 1, 4, rng)
    want = _check(oracle_mod, m, prof, tr, classes, off, inst, flags)
    assert (want["status"] == 0).all() and want["n_served"].max() > 300


@pytest.mark.parametrize("flags", [0, 1])
def test_full_caps_in_a_batch_that_packs(oracle_mod, flags):
    import paper_2509_06362_b200 as m
    rng = np.random.default_rng(9)
    prof = _tables(1, 100, rng)
    lists = [_placement(prof, 1 + k % 3, 32, rng) for k in range(4200)]
    for at, (n, cap) in enumerate([(128, 64), (128, 63), (128, 32), (33, 64), (32, 64), (9, 64)]):
        lists[700 * at] = _placement(prof, n, cap, rng)
    off, inst = gen.candidates_from_lists(lists)
    tr, classes = _workload(60, 1.0, 1, 4, rng)
    want = _check(oracle_mod, m, prof, tr, classes, off, inst, flags)
    assert (want["status"] == 0).all()


def test_full_caps_with_the_smallest_thread_pools(oracle_mod, monkeypatch):
    import paper_2509_06362_b200 as m
    monkeypatch.setenv("MAASO_THREAD_ARENA_KB", "0")
    rng = np.random.default_rng(3)
    prof = _tables(2, 10, rng)
    tr, classes = _workload(300, 20.0, 2, 4, rng)
    for blocks in range(16, 0, -1):  # the most blocks per SM, so the smallest pools, that the call accepts
        monkeypatch.setenv("MAASO_THREAD_BLOCKS", str(blocks))
        c = m.Context(0)
        try:
            for n in (16, 24, 32, 64, 128):  # (a batch each: what is launched goes by the instances in all)
                off, inst = gen.candidates_from_lists([_placement(prof, n, 64, rng)])
                got, _ = gpu_eval(c, prof, tr, classes, off, inst, 10 ** 6, None, 0, 3)
                want = oracle_mod.eval_placements(prof, tr, classes, off, inst, 10 ** 6, None, 0)
                assert_records_equal(got, want, f"{n} instances, {blocks} blocks")
            return
        except m.MaasoError as e:
            assert "no shared memory" in str(e)
        finally:
            c.close()
    assert False, "no pool size was accepted"
