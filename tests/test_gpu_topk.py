"""Selection at the sizes and ties where its passes go different ways: few records (all of them ranked), one
chunk, one record more than a chunk, several passes; equal words in masses, means beyond the word's 30 bits,
fewer scored records than asked for."""
import numpy as np
import pytest

import gen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2509_06362_b200 as m
    c = m.Context(0)
    yield c
    c.close()


def _records(n, kind, rng):
    rec = np.zeros(n, dtype=gen.RESULT_DTYPE)
    rec["n_hit"] = rng.integers(0, 100_000, n)
    rec["n_served"] = rng.integers(0, 100_000, n)
    rec["sum_ttft_us"] = rng.integers(0, 1 << 40, n)
    if kind == "equal":
        rec["n_hit"], rec["n_served"], rec["sum_ttft_us"] = 5, 9, 1234
    elif kind == "unserved":
        rec["n_hit"] = rec["n_served"] = rec["sum_ttft_us"] = 0
        rec["n_hit"][:: 97] = 1
    elif kind == "fractions":   # the same whole microseconds, other fractions, some of them equal
        rec["n_hit"] = 7
        rec["n_served"] = rng.integers(4_000_000_000, 4_294_967_295, n)
        rec["sum_ttft_us"] = 3 * rec["n_served"].astype(np.int64) + rng.integers(0, 3, n)
    elif kind == "clamped":     # means beyond 2^30 microseconds
        rec["n_hit"] = 7
        rec["n_served"] = rng.integers(1, 4, n)
        rec["sum_ttft_us"] = (1 << 62) - rng.integers(0, 5, n)
    elif kind == "invalid":
        rec["status"] = 2
        rec["status"][rng.integers(0, n, max(1, n // 1000))] = 0
    return rec


@pytest.mark.parametrize("kind", ["spread", "equal", "unserved", "fractions", "clamped", "invalid"])
@pytest.mark.parametrize("n", [1, 64, 1409, 8193, 16384, 16385, 70_001])
def test_topk_sizes_and_ties(ctx, oracle_mod, n, kind):
    import torch
    rng = np.random.default_rng(n)
    rec = _records(n, kind, rng)
    dev = torch.from_numpy(rec.view(np.uint8).reshape(n, 128)).cuda()
    scores = np.round(rng.normal(size=n), 1 if kind == "equal" else 12) + 0.0  # no negative zeros
    for k in (1, 64, 1000):
        idx, out = ctx.topk(dev, k)
        idx_s, _ = ctx.topk_scores(dev, torch.from_numpy(scores).cuda(), k)
        got, got_s = idx.cpu().numpy().view(np.uint32), idx_s.cpu().numpy().view(np.uint32)
        want, want_s = oracle_mod.topk(rec, k), oracle_mod.topk_scores(scores, k)
        m = min(n, k)
        assert got[:m].tolist() == want[:m].tolist() and (got[m:] == 0xFFFFFFFF).all()
        assert got_s[:m].tolist() == want_s[:m].tolist()
        assert ctx.results_to_numpy(out)[:m].tobytes() == rec[want[:m]].tobytes()


@pytest.mark.parametrize("most", [3, 5_000, 2 ** 32 - 1])   # the last one needs 64-bit sums
@pytest.mark.parametrize("n", [1, 5, 33, 1000])
def test_percentiles_of_partial_warps_and_large_counts(ctx, oracle_mod, n, most):
    import torch
    rng = np.random.default_rng(n)
    hist = rng.integers(0, most, (n, 64), endpoint=True).astype(np.uint32)
    hist[rng.random((n, 64)) < 0.6] = 0
    hist[::7] = 0
    permille = rng.integers(1, 1001, {3: 1, 5_000: 3}.get(most, 16)).astype(np.uint32)
    got = ctx.ttft_percentiles(torch.from_numpy(hist.view(np.int32)).cuda(), permille).cpu().numpy()
    assert (got == oracle_mod.ttft_percentiles(hist, permille)).all()


@pytest.mark.parametrize("offset", [1, 2, 3, 4])
def test_percentiles_of_histograms_at_any_word(ctx, oracle_mod, offset):
    """The histograms are an array of words and may start at any of them (a slice of a larger buffer)."""
    import torch
    n = 37
    rng = np.random.default_rng(offset)
    hist = rng.integers(0, 5_000, (n, 64)).astype(np.uint32)
    hist[::5] = 0
    buffer = torch.full((n * 64 + 8,), -1, dtype=torch.int32, device="cuda")
    view = buffer[offset:offset + n * 64].view(n, 64)
    view.copy_(torch.from_numpy(hist.view(np.int32)))
    permille = np.array((1, 500, 900, 990, 1000), dtype=np.uint32)
    assert view.is_contiguous() and (view.data_ptr() % 16 != 0) == (offset != 4)
    assert (ctx.ttft_percentiles(view, permille).cpu().numpy() == oracle_mod.ttft_percentiles(hist, permille)).all()
