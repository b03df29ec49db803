"""A NaN or an infinity in X: the call ends, the cores hold NaNs, ranks and status are those of
the rank rule (a column with a NaN is left as it is by the QR and counts as zero), never "B is
singular", which would blame the test matrix."""
import numpy as np
import pytest
import torch

from paper_2111_10448_gb300 import TTSketch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("kw,status", [("ranks", 0), ("eps", 7)])
@pytest.mark.parametrize("prec", ["fp64", "bf16", "tf32"])
@pytest.mark.parametrize("dims", [[20, 21, 22], [40, 30, 50, 20], [9] * 5])
def test_nonfinite_entry(dims, prec, kw, status, bad):
    d = len(dims)
    dt = torch.float64 if prec == "fp64" else torch.float32
    X = torch.randn(int(np.prod(dims)), dtype=dt, device="cuda")
    X[777] = bad
    args = dict(ranks=[1] + [4] * (d - 1) + [1], p=4) if kw == "ranks" else dict(eps=1e-3, rmax=6, p=4)
    t = TTSketch(dims, seed=1, prec=prec, x_dtype=dt, **args).pstt2(X)
    st, ranks = t.status()
    assert st == status
    assert ranks == [1] + [4 if kw == "ranks" else 6] * (d - 1) + [1]
    assert bool(torch.isnan(t.cores).any())
