"""The sketch kernels beside the strip kernel, on shapes that are theirs: the small-plane and
tile kernels of single problems against the oracle's sketches, those of batches (both padded
widths at once, several kL blocks, tensors of d = 7 beside smaller ones) by recovery.  Bars as in
test_gpu_strip and test_gpu_batched_widths; a Khatri-Rao entry of six factors, whose FP32 errors
add up, lands on the other side of a rounding boundary twice as often as one of three:
sqrt(2) times the Frobenius bar."""
import numpy as np
import pytest
import torch

import ttinputs as ti
from oracle import philox, pstt2 as OP
from oracle import tt as OT
from paper_2111_10448_gb300 import TTSketch
from tests.gpu_util import sketch_dict, to_dev

pytestmark = pytest.mark.gpu


def _scale_of(x):
    return 15 - int(np.frexp(float(np.max(np.abs(x))))[1])


def _split(x, prec, s):
    xs = np.asarray(x, dtype=np.float64) * 2.0 ** s
    hi = philox.round_to(xs, prec)
    return (hi + philox.round_to(xs - hi, prec)) * 2.0 ** -s


@pytest.mark.parametrize("prec", ["bf16", "tf32", "fp16"])
@pytest.mark.parametrize("name,dims,r,p,slabs,drm", [
    ("small-plane", [9, 4, 5, 3, 4, 3, 10], 4, 5, [10], "gauss"),
    ("small-plane", [20, 3, 4, 3, 3, 2, 31], 10, 9, [11, 20], "gauss"),
    ("small-plane", [20, 5, 6, 31], 8, 9, [31], "kr"),
    ("tile", [130, 3, 2, 3, 2, 3, 70], 3, 5, [70], "gauss"),      # several 64 x 32 tiles a plane
    ("tile", [65, 2, 3, 2, 2, 2, 3, 33], 6, 12, [20, 13], "gauss"),
    ("tile", [40, 3, 2, 3, 2, 3, 70], 3, 5, [70], "kr"),
])
def test_single(name, dims, r, p, slabs, drm, prec):
    x = np.random.default_rng(3).standard_normal(int(np.prod(dims))).astype(np.float32)
    s = _scale_of(x) if prec == "fp16" else 0
    ranks = [1] + [r] * (len(dims) - 1) + [1]
    t = TTSketch(dims, ranks=ranks, p=p, seed=4, x_dtype=torch.float32, prec=prec, drm=drm, x_scale_log2=s)
    n = int(np.prod(dims[:-1]))
    X = to_dev(x)
    t.begin()
    a = 0
    for c in slabs:
        assert t.kernel_name(c) == name
        t.accumulate(X[a * n:(a + c) * n], a, c)
        a += c
    sk = {k: v * 2.0 ** -s for k, v in sketch_dict(t).items()}
    t.finalize()
    o = OP.pstt2(_split(x, prec, s), dims, ranks=ranks, p=p, seed=4, passes=1, test_fmt=prec, drm=drm)
    for key, ty in (("S", 0), ("R", 1)):
        for k, S in o["sketch"][key].items():
            G = sk[(ty, k)]
            assert G.shape == S.shape
            fro = np.linalg.norm(G - S) / np.linalg.norm(S)
            mx = np.max(np.abs(G - S)) / np.max(np.abs(S))
            bar = 1e-4 * (2 ** 0.5 if drm == "kr" and len(dims) == 7 else 1)
            assert fro <= bar and mx <= 2e-3, (key, k, fro, mx)


SMALL = [([8, 9, 8], 2), ([20, 21, 20], 12), ([5, 4, 3, 5, 4, 3, 5], 3), ([12, 6, 7, 12], 11), ([32, 4, 31], 16),
         ([3, 2, 3, 2, 2, 3, 2, 3], 2), ([10, 3, 3, 3, 3, 10], 3), ([31, 2, 3, 2, 3, 2, 30], 12)]


@pytest.mark.parametrize("prec,bar", [("bf16", 8e-5), ("tf32", 3e-6), ("fp16", 3e-6)])
@pytest.mark.parametrize("name,shapes", [
    ("small-plane", SMALL),                                              # padded widths 16 and 32
    ("small-plane", [s for s in SMALL if s[1] <= 11]),                   # 16 alone
    ("small-plane", [([20, 21, 20], 12), ([31, 2, 3, 2, 3, 2, 30], 12)]),   # 32 alone
    ("tile", [([40, 6, 35], 5), ([8, 9, 8], 2), ([20, 21, 20], 12), ([70, 50], 20), ([9] * 4, 3)]),
    ("tile", [([32, 40, 32], 30), ([30, 4, 50, 3], 8)]),                 # small planes, 35 columns
])
def test_batch(name, shapes, prec, bar):
    probs, xs = [], []
    for i, (dims, r) in enumerate(shapes * 3):
        N = np.cumprod([1] + dims)
        ranks = [min(r, int(N[k]), int(N[-1] // N[k])) for k in range(len(dims) + 1)]
        x = ti.random_tt(dims, ranks, seed=i).astype(np.float32)
        probs.append(dict(dims=dims, ranks=ranks, p=5, seed=50 + i, x_scale_log2=_scale_of(x) if prec == "fp16" else 0))
        xs.append(x)
    t = TTSketch(None, batch=probs, prec=prec)
    assert t.kernel_name() == name
    X = [to_dev(x) for x in xs]
    for shape in ((64, 4, 4), (1, 1, 1), (8, 4, 1)):
        t.batch_config(*shape)
        for _ in range(2):   # a second call on the same workspace
            t.batched(X)
            assert t.status()[0] == 0
            for i, x in enumerate(xs):
                got = OT.tt_full(t.core_list(i))
                assert np.linalg.norm(got - x) <= bar * np.linalg.norm(x), (shape, i, probs[i]["dims"])
