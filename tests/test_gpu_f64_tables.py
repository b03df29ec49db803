"""FP64 sketch kernel with staged test-matrix rows and 64-column tiles: every entry of
every sketch against the oracle, at the edges of both rules (rows staged for one side,
both or none, slabs whose tables differ, ragged tiles, both test-matrix kinds).  Bar:
sums of K <= 1e6 terms whose rounding errors add at random, sqrt(K) 2^-53 ~ 1.1e-13 of
the norm, and normals one or two units in the last place apart: 1e-12."""
import numpy as np
import pytest
import torch

from oracle import pstt2 as OP
from paper_2111_10448_gb300 import TTSketch
from tests.gpu_util import sketch_dict, to_dev

pytestmark = pytest.mark.gpu

CASES = [
    ([70, 20, 20, 65], 10, 8, [65]),          # both sides staged, ragged 64 x 64 tiles
    ([70, 20, 20, 65], 10, 8, [33, 32]),      # a wide slab, a narrow one at an offset
    ([130, 24, 24, 20], 13, 8, [20]),         # 32-column tiles, three strips
    ([64, 64, 3, 64], 30, 34, [64]),          # widest sketch
    ([600, 40, 90], 5, 4, [1, 89]),           # d = 3: a slab of one column
    ([9, 8, 7, 6], 4, 4, [6]),                # too little to stage
    ([40, 7, 6, 5, 4, 33], 6, 6, [33]),       # three sketches a side
]


@pytest.mark.parametrize("drm", ["gauss", "kr"])
@pytest.mark.parametrize("xf64", [True, False])
@pytest.mark.parametrize("dims,r,p,slabs", CASES)
def test_f64_sketches_match_oracle(dims, r, p, slabs, xf64, drm):
    x = np.random.default_rng(7).standard_normal(int(np.prod(dims)))
    if not xf64:
        x = x.astype(np.float32)
    ranks = [1] + [r] * (len(dims) - 1) + [1]
    t = TTSketch(dims, ranks=ranks, p=p, seed=6, prec="fp64", drm=drm,
                 x_dtype=torch.float64 if xf64 else torch.float32)
    n = int(np.prod(dims[:-1]))
    X = to_dev(x, torch.float64 if xf64 else torch.float32)
    assert X.numel() == n * dims[-1]
    t.begin()
    a = 0
    for c in slabs:
        t.accumulate(X[a * n:(a + c) * n], a, c)
        a += c
    sk = sketch_dict(t)
    t.finalize()
    o = OP.pstt2(x.astype(np.float64), dims, ranks=ranks, p=p, seed=6, passes=1, drm=drm)
    for name, ty in (("S", 0), ("R", 1)):
        for k, S in o["sketch"][name].items():
            G = sk[(ty, k)]
            assert G.shape == S.shape
            assert np.linalg.norm(G - S) <= 1e-12 * np.linalg.norm(S), (name, k)
