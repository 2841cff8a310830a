"""Which packed kernel replays a batch (csrc/eval_pack.cu): 12 or 14 warps per SM, by the number of items and not of placements, as
between four and eight of them share an item; and the kernel with 14 on one model, whose admissions move step counters back."""
import re

import numpy as np
import pytest

import gen
from gpu_common import assert_records_equal
from test_gpu_pack import _mostly_not_loaded, _trace

pytestmark = pytest.mark.gpu


def _sms():
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count


def _warps(call):
    """Warps per block of the packed kernel that ran longest during `call`."""
    import torch
    from torch.profiler import ProfilerActivity, profile
    torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA]) as p:
        call()
        torch.cuda.synchronize()
    ran = [(e.time_range.elapsed_us(), e.name) for e in p.events()
           if e.device_type == torch.autograd.DeviceType.CUDA and "eval_pack_kernel" in e.name]
    return int(re.search(r"(\d+)>", max(ran)[1]).group(1))


def _items(lists, n_traces):
    four, eight = sum(1 <= len(x) <= 4 for x in lists), sum(5 <= len(x) <= 8 for x in lists)
    return (-(-four // 8) + -(-eight // 4)) * n_traces


@pytest.mark.parametrize("flags", [0, 1])
@pytest.mark.parametrize("n_traces", [1, 2])
@pytest.mark.parametrize("per_sm, more, warps", [(12, 0, 12), (12, 1, 14), (16, 0, 14), (16, 1, 12), (24, 0, 12), (24, 1, 14)])
@pytest.mark.parametrize("fours", [25, 75])  # per cent of the items that are eight placements of up to 4 instances
def test_kernel_by_items(oracle_mod, fours, per_sm, more, warps, n_traces, flags):
    import paper_2509_06362_b200 as m
    prof, rng = gen.profile_node(1), np.random.default_rng(fours)
    hold = per_sm * _sms()
    four = hold // n_traces * fours // 100
    sizes = [4] * (8 * four) + [7] * (4 * (hold // n_traces - four)) + [3] * more
    ok = np.nonzero(np.asarray(prof["devices"]) >= prof["min_devices"][0])[0]
    kinds = [[(0, int(rng.choice(ok)), int(rng.choice((2, 16, 64)))) for _ in range(8)] for _ in range(40)]
    lists = [kinds[i % 40][:k] for i, k in enumerate(sizes)]
    assert _items(lists, n_traces) == hold + more * n_traces
    traces = [_trace(90 - 30 * k, 3.0, 7 + k, (1.0,), False) for k in range(n_traces)]
    assert _mostly_not_loaded(prof, lists, traces)
    classes = gen.make_classes([(500_000, 50_000, None), (2_000_000, 150_000, None), (None, None, 180_000_000)])
    off, inst = gen.candidates_from_lists(lists)
    c = m.Context(0)
    c.load_profile(prof)
    handles, d_off, d_inst, out = [c.load_trace(t, classes) for t in traces], c.to_device(off), c.to_device(inst), []
    call = lambda: out.append(c.eval_placements_multi(handles, d_off, d_inst, 10 ** 6, flags=flags))
    call()
    assert _warps(call) == warps
    got = c.results_to_numpy(out[-1]).reshape(n_traces, len(lists))
    c.close()
    for g, t in zip(got, traces):
        assert_records_equal(g, oracle_mod.eval_placements(prof, t, classes, off, inst, 10 ** 6, None, flags), f"{per_sm} items per SM and {more}")


@pytest.mark.parametrize("flags", [0, 1])
def test_counters_moved_back(oracle_mod, flags):
    """Step counters that go past what a key holds, one model under several traces, more items than 12 warps hold."""
    import torch
    import paper_2509_06362_b200 as m
    rng = np.random.default_rng(4)
    W, n = gen.WMAX, 1100
    step = np.ones((1, 2, W), dtype=np.int32)
    step[0, 1] = 2
    prof = {"n_models": 1, "n_strategies": 2, "wmax": W, "devices": np.ones(2, dtype=np.int32), "min_devices": np.ones(1, dtype=np.int32),
            "prefill_base_us": np.zeros((1, 2), dtype=np.int32), "prefill_q16": np.zeros((1, 2), dtype=np.int32), "step_us": step}
    classes = gen.make_classes([(None, None, None)])
    traces = []
    for k in range(3):
        tr = np.zeros(n - 50 * k, dtype=gen.REQUEST_DTYPE)
        tr["arrival_us"] = np.cumsum(rng.integers(30_000, 40_000, size=len(tr)))  # every request overlaps the next
        tr["out_tokens"] = rng.integers(60_000, 65_536, size=len(tr))
        traces.append(tr)
    lists = [[(0, int(rng.integers(2)), int(rng.choice([4, 9, 16, 64]))) for _ in range(k)] for k in [1, 2, 3, 4, 5, 8] * 720]
    assert _mostly_not_loaded(prof, lists, traces) and 12 * _sms() < _items(lists, 3) <= 16 * _sms()
    off, inst = gen.candidates_from_lists(lists)
    c = m.Context(0)
    c.load_profile(prof)
    handles, d_off, d_inst, out = [c.load_trace(t, classes) for t in traces], c.to_device(off), c.to_device(inst), []
    hist = torch.zeros((3 * len(lists), 64), dtype=torch.int32, device="cuda")
    call = lambda: out.append(c.eval_placements_multi(handles, d_off, d_inst, 10 ** 6, flags=flags, ttft_hist=hist))
    assert _warps(call) == 14
    got = c.results_to_numpy(out[-1]).reshape(3, len(lists))
    hist = hist.cpu().numpy().view(np.uint32).reshape(3, len(lists), 64)
    c.close()
    for k, t in enumerate(traces):
        want = oracle_mod.eval_placements(prof, t, classes, off, inst, 10 ** 6, None, flags)
        assert_records_equal(got[k], want, f"trace {k}")
        assert (want["n_served"] == len(t)).all() and want["makespan_us"].max() > 1 << 25
        assert (hist[k] == oracle_mod.ttft_hist(prof, t, classes, off, inst, 10 ** 6, None, flags)).all()
