"""Batches whose tensors need different padded sketch widths (16 and 32 columns)
run on the small-plane kernel, each tensor at its own width: every tensor is
recovered as the single-tensor call recovers it.  Bars: the split of X resolves
2^-17 (BF16) or 2^-22 (TF32, FP16); the least-squares core and the bases of
well-conditioned random TT tensors amplify that by less than 10."""
import numpy as np
import pytest
import torch

import ttinputs as ti
from oracle import tt as OT
from paper_2111_10448_gb300 import TTSketch
from tests.gpu_util import to_dev

pytestmark = pytest.mark.gpu

SHAPES = [([8, 9, 8], 2), ([20, 21, 20], 12), ([9, 8, 10, 9], 3), ([12, 6, 7, 12], 11), ([32, 4, 31], 16),
          ([9] * 5, 4), ([10, 3, 3, 3, 3, 10], 3), ([24, 5, 24], 13)]


@pytest.mark.parametrize("prec,bar", [("bf16", 8e-5), ("tf32", 3e-6), ("fp16", 3e-6)])
def test_mixed_widths(prec, bar):
    probs, xs = [], []
    for i, (dims, r) in enumerate(SHAPES * 5):
        N = np.cumprod([1] + dims)
        ranks = [min(r, int(N[k]), int(N[-1] // N[k])) for k in range(len(dims) + 1)]
        x = ti.random_tt(dims, ranks, seed=i).astype(np.float32)
        m = float(np.max(np.abs(x)))
        probs.append(dict(dims=dims, ranks=ranks, p=5, seed=50 + i,
                          x_scale_log2=15 - int(np.frexp(m)[1]) if prec == "fp16" else 0))
        xs.append(x)
    assert {16, 32} == {16 if max(p["ranks"]) + 5 <= 16 else 32 for p in probs}
    t = TTSketch(None, batch=probs, prec=prec)
    X = [to_dev(x) for x in xs]
    for _ in range(2):   # a second call on the same workspace
        t.batched(X)
        assert t.status()[0] == 0
        for i, x in enumerate(xs):
            got = OT.tt_full(t.core_list(i))
            assert np.linalg.norm(got - x) <= bar * np.linalg.norm(x), (i, probs[i]["dims"])
