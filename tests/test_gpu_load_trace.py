"""Loading a trace whose classes differ in patience (csrc/prep.cu): the list of its patient requests takes no copy and no launch of its
own, and is right at the edges of the tiles that it is made in and over more tiles than a block has threads."""
import numpy as np
import pytest

import gen
from gpu_common import assert_records_equal
from test_gpu_patient import CLASSES, _placements, _trace

pytestmark = pytest.mark.gpu


def _device_work(load):
    """Copies and kernels on the device while `load` runs."""
    import torch
    from torch.profiler import ProfilerActivity, profile
    torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA]) as p:
        load()
        torch.cuda.synchronize()
    on_device = [e.name for e in p.events() if e.device_type == torch.autograd.DeviceType.CUDA]
    return sorted("copy" if "Memcpy" in x else "kernel" for x in on_device if "Memset" not in x)


def test_no_copy_and_no_launch_more():
    import torch
    import paper_2509_06362_b200 as m
    tr = _trace(5000, "spread", np.random.default_rng(1))
    c = m.Context(0)
    c.load_profile(gen.profile_multimodel(1))
    apart, alike = gen.make_classes(CLASSES), gen.make_classes([(500_000, 50_000, None)] * 4)
    for classes in (apart, alike):  # (the kernels are loaded)
        c.free_trace(c.load_trace(tr, classes))
    with_list, without = (_device_work(lambda: c.free_trace(c.load_trace(tr, x))) for x in (apart, alike))
    assert without.count("kernel") >= 1 and without.count("copy") >= 1
    assert with_list == without
    c.close()


@pytest.mark.parametrize("n", [255, 256, 257, 511, 512, 513, 70_001])
def test_edges_of_tiles(oracle_mod, n):
    import paper_2509_06362_b200 as m
    rng = np.random.default_rng(n)
    prof = gen.profile_multimodel(1)
    off, inst = _placements(prof, rng)
    classes = gen.make_classes(CLASSES)
    tr = _trace(n, "spread", rng)
    c = m.Context(0)
    c.load_profile(prof)
    t = c.load_trace(tr, classes)
    for mask in (None, 12):  # (the second: the list alone)
        mk = None if mask is None else np.full(len(off) - 1, mask, dtype=np.uint32)
        got = c.results_to_numpy(c.eval_placements(t, c.to_device(off), c.to_device(inst), 1024, None if mk is None else c.to_device(mk)))
        assert_records_equal(got, oracle_mod.eval_placements(prof, tr, classes, off, inst, 1024, mk, 0), f"mask {mask}")
    c.close()
