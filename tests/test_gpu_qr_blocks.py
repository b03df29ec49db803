"""Basis QRs at the edges of their splits: fewer rows than columns, one block, roots small
enough to be pivoted as they stand (up to six times the width, or 8192 entries in up to 256
rows: width 32 at its 8 l rows) and larger ones, several levels, widths from one to eight octets of columns.  A tensor of exact rank is recovered
to rounding (a Gaussian sketch of width rank + 6 or more is conditioned below 1e3:
1e-11), and the right core's rows are orthonormal to 1e-12."""
import numpy as np
import pytest
import torch

from paper_2111_10448_gb300 import TTSketch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r,p", [(1, 6), (5, 6), (10, 7), (20, 12), (26, 9), (50, 14)])
@pytest.mark.parametrize("blocks,extra", [(1, -1), (1, 0), (1, 1), (6, 0), (6, 1), (8, 0), (8, 1), (0, 256), (0, 257), (0, 900), (0, 20011)])
def test_exact_rank_is_recovered(blocks, extra, r, p):
    n2 = blocks * (r + p) + extra
    g = torch.Generator(device="cuda")
    g.manual_seed(n2 + r)
    A = torch.randn(80, r, dtype=torch.float64, device="cuda", generator=g)
    B = torch.randn(n2, r, dtype=torch.float64, device="cuda", generator=g)
    X = (B @ A.T).reshape(-1).contiguous()   # first mode fastest
    t = TTSketch([80, n2], ranks=[1, r, 1], p=p, seed=2, prec="fp64", x_dtype=torch.float64)
    t.pstt2(X)
    assert t.status()[0] == 0
    err = float(torch.linalg.norm(t.reconstruct(torch.float64) - X) / torch.linalg.norm(X))
    assert err <= 1e-11
    M = t.core_list()[1].reshape(r, n2)
    assert np.abs(M @ M.T - np.eye(r)).max() <= 1e-12
