"""Placements of 32 and 33 instances where the budget allows 32 and 33 devices: the kernel for more than 32 instances is launched
only if a valid placement can have so many (csrc/maaso_api.cu), and what is over the budget is refused either way."""
import numpy as np
import pytest

import gen
from gpu_common import assert_records_equal

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flags", [0, 1, 2, 4, 8])
@pytest.mark.parametrize("budget", [31, 32, 33, 34])
def test_budget(oracle_mod, budget, flags):
    import paper_2509_06362_b200 as m
    prof = gen.profile_node(1)
    one = int(np.nonzero(np.asarray(prof["devices"]) == 1)[0][0])
    off, inst = gen.candidates_from_lists([[(0, one, 4)] * k for k in (1, 31, 32, 33, 34)])
    classes = gen.make_classes([(500_000, 50_000, None), (None, None, 180_000_000)])
    tr = gen.make_trace(200, 80.0, 3)
    tr["cls"] = np.arange(200) % 2
    c = m.Context(0)
    c.load_profile(prof)
    got = c.results_to_numpy(c.eval_placements(c.load_trace(tr, classes), c.to_device(off), c.to_device(inst), budget, flags=flags))
    want = oracle_mod.eval_placements(prof, tr, classes, off, inst, budget, None, flags)
    assert (want["status"] != 0).tolist() == [k > budget for k in (1, 31, 32, 33, 34)]
    assert_records_equal(got, want, f"budget {budget}")
    c.close()
