"""GPU parity of the strip kernel (shapes outside the tcgen05 and small-plane
kernels): every entry of every sketch against the oracle's FP64 products of the
split X with its rounded test matrices, at the edges of the kernel's split
(strips of 128 rows of i_1, tiles of 64 or 32 columns, unit and flush
boundaries, every padded width, unaligned rows and slabs, both test-matrix
kinds).  Bars as in test_gpu_mixed: test-matrix flips to the neighbouring value
bound the relative Frobenius difference by 1e-4 and the largest by 2e-3 of
max |S|."""
import numpy as np
import pytest
import torch

import ttinputs as ti
from oracle import philox, pstt2 as OP
from paper_2111_10448_gb300 import TTSketch
from tests.gpu_util import sketch_dict, to_dev

pytestmark = pytest.mark.gpu


def _scale_of(x):
    m = float(np.max(np.abs(x)))
    return 0 if m == 0.0 else 15 - int(np.frexp(m)[1])


def _split(x, prec, s):
    xs = np.asarray(x, dtype=np.float64) * 2.0 ** s
    hi = philox.round_to(xs, prec)
    return (hi + philox.round_to(xs - hi, prec)) * 2.0 ** -s


CASES = [
    # dims, width rank r, oversampling p, slab sizes of the last mode
    ([129, 40], 3, 5, [40]),                      # two strips, d = 2
    ([16, 3, 65], 3, 5, [65]),                    # one m-tile, a second column tile of one column
    ([33, 5, 4, 36], 4, 5, [36]),                 # unaligned rows
    ([36, 21, 3, 35], 6, 12, [35]),               # kL past the row sums' flush, 3 octets
    ([257, 2, 130], 20, 6, [64, 1, 65]),          # odd slabs: unaligned slab starts, 4 octets
    ([34, 5, 4, 3, 33], 9, 28, [33]),             # three column sketches, 5 octets
    ([40, 3, 5, 2, 2, 37], 8, 36, [37]),          # d = 6, 6 octets
    ([64, 4, 64], 30, 34, [64]),                  # 8 octets
    ([144, 3, 2, 200], 5, 6, [100, 100]),         # several column tiles a unit
    ([1, 50, 70], 2, 5, [70]),                    # a single row of i_1
    ([129, 40, 40, 65], 6, 5, [65]),              # staged test-matrix rows on both sides
    ([129, 40, 40, 65], 6, 5, [33, 32]),          # on the row side alone
]


@pytest.mark.parametrize("drm", ["gauss", "kr"])
@pytest.mark.parametrize("prec", ["tf32", "bf16", "fp16"])
@pytest.mark.parametrize("dims,r,p,slabs", CASES)
def test_strip_sketches_match_oracle(dims, r, p, slabs, prec, drm):
    x = np.random.default_rng(3).standard_normal(int(np.prod(dims))).astype(np.float32)
    s = _scale_of(x) if prec == "fp16" else 0
    ranks = [1] + [r] * (len(dims) - 1) + [1]
    t = TTSketch(dims, ranks=ranks, p=p, seed=4, x_dtype=torch.float32, prec=prec, drm=drm, x_scale_log2=s)
    assert t.kernel_kind() == 1
    n = int(np.prod(dims[:-1]))
    # the slabs lie one entry past a 16-byte boundary of their buffer
    buf = torch.empty(x.size + 1, dtype=torch.float32, device="cuda")
    buf[1:] = to_dev(x)
    t.begin()
    a = 0
    for c in slabs:
        t.accumulate(buf[1 + a * n:1 + (a + c) * n], a, c)
        a += c
    sk = {k: v * 2.0 ** -s for k, v in sketch_dict(t).items()}
    t.finalize()
    o = OP.pstt2(_split(x, prec, s), dims, ranks=ranks, p=p, seed=4, passes=1, test_fmt=prec, drm=drm)
    for name, ty in (("S", 0), ("R", 1)):
        for k, S in o["sketch"][name].items():
            G = sk[(ty, k)]
            assert G.shape == S.shape
            fro = np.linalg.norm(G - S) / np.linalg.norm(S)
            mx = np.max(np.abs(G - S)) / np.max(np.abs(S))
            assert fro <= 1e-4 and mx <= 2e-3, (name, k, fro, mx)


@pytest.mark.parametrize("prec", ["bf16", "tf32"])
def test_strip_aligned_equals_unaligned(prec):
    """The 16-byte copies and the copies of unaligned rows give the same sketches
    up to summation order (FP64 sums of FP32 partials: 1e-6)."""
    dims = [132, 6, 5, 68]
    x = np.random.default_rng(5).standard_normal(int(np.prod(dims))).astype(np.float32)
    buf = torch.empty(x.size + 8, dtype=torch.float32, device="cuda")
    got = []
    for off in (0, 1, 2, 3):
        buf[off:off + x.size] = to_dev(x)
        t = TTSketch(dims, ranks=[1, 5, 5, 5, 1], p=6, seed=4, x_dtype=torch.float32, prec=prec)
        t.begin()
        t.accumulate(buf[off:off + x.size], 0, dims[-1])
        got.append(sketch_dict(t))
        t.finalize()
    for g in got[1:]:
        for k in g:
            assert np.linalg.norm(g[k] - got[0][k]) <= 1e-6 * np.linalg.norm(got[0][k])


GROUPED = [
    # small planes: tiles of several kL (i_2) and kR (i_{d-1}) values, ragged at both ends
    ([8, 3, 5, 9], 3, 5, [9]),
    ([24, 5, 3, 24], 6, 5, [24]),
    ([24, 7, 2, 5, 3, 23], 10, 10, [23]),         # d = 6, three sketches a side
    ([9, 7, 5, 8, 6, 9], 4, 5, [4, 5]),           # slabs
    ([16, 9, 3, 17, 32], 8, 9, [32]),
    ([31, 4, 3, 30], 5, 6, [30]),                 # unaligned rows
    ([32, 3, 32], 20, 10, [32]),                  # one kR value
    ([12, 1, 9, 11], 4, 4, [11]),
    ([1, 6, 5, 3], 2, 2, [3]),
    ([20, 18], 6, 6, [18]),
    ([10, 40, 12, 8], 5, 6, [1, 7]),
    ([24, 24, 24, 24, 24], 10, 10, [24]),         # with staged test-matrix rows
    ([40, 5, 6, 7, 20], 9, 6, [20]),              # grouped along i_{d-1} and i_2, past the small-plane limit
]


@pytest.mark.parametrize("prec", ["tf32", "bf16", "fp16"])
@pytest.mark.parametrize("dims,r,p,slabs", GROUPED)
def test_strip_grouped_planes_match_oracle(dims, r, p, slabs, prec):
    x = np.random.default_rng(6).standard_normal(int(np.prod(dims))).astype(np.float32)
    s = _scale_of(x) if prec == "fp16" else 0
    ranks = [1] + [r] * (len(dims) - 1) + [1]
    t = TTSketch(dims, ranks=ranks, p=p, seed=4, x_dtype=torch.float32, prec=prec, x_scale_log2=s)
    n = int(np.prod(dims[:-1]))
    buf = to_dev(x)
    t.begin()
    a = 0
    for c in slabs:
        t.accumulate(buf[a * n:(a + c) * n], a, c)
        a += c
    sk = {k: v * 2.0 ** -s for k, v in sketch_dict(t).items()}
    t.finalize()
    o = OP.pstt2(_split(x, prec, s), dims, ranks=ranks, p=p, seed=4, passes=1, test_fmt=prec)
    for name, ty in (("S", 0), ("R", 1)):
        for k, S in o["sketch"][name].items():
            G = sk[(ty, k)]
            assert G.shape == S.shape
            fro = np.linalg.norm(G - S) / np.linalg.norm(S)
            mx = np.max(np.abs(G - S)) / np.max(np.abs(S))
            assert fro <= 1e-4 and mx <= 2e-3, (name, k, fro, mx)
