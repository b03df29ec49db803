"""The batched strip launch's unit size: every size gives the same decompositions, and it is
what the launch uses (two small tensors in one unit each take longer than in many)."""
import numpy as np
import pytest
import torch

import ttinputs as ti
from oracle import tt as OT
from paper_2111_10448_gb300 import TTSketch
from tests.gpu_util import to_dev

pytestmark = pytest.mark.gpu
SHAPES = [([22, 20, 12, 20], 3), ([10] * 5, 4), ([9, 31, 7], 5), ([32, 3, 5, 31], 6), ([8, 3, 4, 3, 2, 9], 3)]


def _batch(prec, shapes=SHAPES):
    probs, xs = [], []
    for i, (dims, r) in enumerate(shapes):
        N = np.cumprod([1] + dims)
        ranks = [min(r, int(N[k]), int(N[-1] // N[k])) for k in range(len(dims) + 1)]
        xs.append(ti.random_tt(dims, ranks, seed=i).astype(np.float32))
        probs.append(dict(dims=dims, ranks=ranks, p=5, seed=50 + i))
    return TTSketch(None, batch=probs, prec=prec), xs


# bars as in test_gpu_batched_widths
@pytest.mark.parametrize("prec,bar", [("bf16", 8e-5), ("tf32", 3e-6)])
@pytest.mark.parametrize("shape", [(32, 4, 4), (64, 1, 1), (1, 1, 1), (2, 1, 1), (1, 4, 1), (1, 8, 1), (8, 8, 1),
                                   (8, 2 ** 31 - 1, 1)])
def test_every_unit_size(shape, prec, bar):
    t, xs = _batch(prec)
    X = [to_dev(x) for x in xs]
    t.batch_config(*shape)
    for _ in range(2):
        t.batched(X)
        assert t.status()[0] == 0
        for i, x in enumerate(xs):
            assert np.linalg.norm(OT.tt_full(t.core_list(i)) - x) <= bar * np.linalg.norm(x), i


def test_unit_size_is_used():
    t, xs = _batch("bf16", SHAPES[:2])
    X = [to_dev(x) for x in xs]
    ms = {}
    for shape in ((8, 8, 1), (1, 1, 1), (32, 4, 4)):
        t.batch_config(*shape)
        for _ in range(3):
            t.batched(X)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(20):
            t.batched(X)
        e1.record()
        torch.cuda.synchronize()
        ms[shape] = e0.elapsed_time(e1)
    # 0.51, 0.15 and 0.15 ms a call
    assert ms[8, 8, 1] > 1.5 * ms[1, 1, 1] and ms[8, 8, 1] > 1.5 * ms[32, 4, 4], ms
