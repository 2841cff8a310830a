"""Final ranks of the selection (csrc/topk.cu) where the number of threads that share one survivor changes: 128, 256 and 512 of them."""
import numpy as np
import pytest

from test_gpu_topk import _records, ctx  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["spread", "equal", "fractions"])
@pytest.mark.parametrize("n", [127, 128, 129, 255, 256, 257, 511, 512, 513, 1024])
def test_ranks(ctx, oracle_mod, n, kind):  # noqa: F811
    import torch
    rec = _records(n, kind, np.random.default_rng(n))
    dev = torch.from_numpy(rec.view(np.uint8).reshape(n, 128)).cuda()
    for k in (1, 31, n):
        idx, sel = ctx.topk(dev, k)
        want = oracle_mod.topk(rec, k)
        assert idx.cpu().numpy().view(np.uint32).tolist() == want.tolist(), k
        assert ctx.results_to_numpy(sel).tobytes() == rec[want].tobytes(), k
