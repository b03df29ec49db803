"""How far the strip kernel's column sums are from the exact sums over the very test-matrix
rows that it draws (read back through one-hot tensors).  X is the sum of its two parts, so
that the FP32 additions are all that is measured.

Bar, relative Frobenius: the 64 x 32 tile kernel's errors, whose sums went to FP64 after 32
terms each (a chain of four tensor-core additions in 16 bits, eight in TF32, not rounded to
nearest): 1.05e-7, 1.34e-7 and 2.00e-7 in BF16, FP16 and TF32, the same for 32 to 100
last-mode indices and any number of planes."""
import numpy as np
import pytest
import torch

from paper_2111_10448_gb300 import TTSketch

pytestmark = pytest.mark.gpu
FMT = {"bf16": torch.bfloat16, "fp16": torch.float16}


def _round(x, prec):
    if prec != "tf32":
        return x.to(FMT[prec]).float()
    b = x.view(torch.int32)
    return ((b + 0xFFF + ((b >> 13) & 1)) & ~0x1FFF).view(torch.float32)


def column_errors(dims, r, p, prec):
    n1, n2, n3, nd = dims
    W = n2 * n3
    t = TTSketch(dims, ranks=[1, r, r, r, 1], p=p, seed=4, x_dtype=torch.float32, prec=prec)
    dev = "cuda"

    def sketch(x, k):
        t.begin()
        t.accumulate(x, 0, nd)
        s = [s for ty, kk, s in t.sketches() if ty == 0 and kk == k][0].clone()
        t.finalize()
        return s

    # X(:, w, b) with X[w, i_1] per b: entry i_1 + n_1 (w + W b)
    hot = torch.zeros(nd * W, n1, device=dev)
    O1 = torch.empty(W * nd, r + p, dtype=torch.float64, device=dev)   # row w + W b
    i = torch.arange(n1, device=dev)
    for r0 in range(0, W * nd, n1):
        rows = torch.clamp(r0 + i, max=W * nd - 1)
        hot[rows, i] = 1.0
        O1[rows] = sketch(hot.reshape(-1), 1)
        hot[rows, i] = 0.0
    # Omega_2, rows kR + n_3 b: one row for every (i_1, kL)
    H = torch.zeros(nd, n3, n2, n1, device=dev)
    q = torch.arange(n1 * n2, device=dev)
    O2 = torch.empty(n3 * nd, r + p, dtype=torch.float64, device=dev)
    for r0 in range(0, n3 * nd, n1 * n2):
        rows = torch.clamp(r0 + q, max=n3 * nd - 1)
        H[rows // n3, rows % n3, q // n1, q % n1] = 1.0
        O2[rows] = sketch(H.reshape(-1), 2)
        H.zero_()
    g = torch.Generator(device=dev)
    g.manual_seed(1)
    x = torch.randn(nd * n3 * n2 * n1, device=dev, generator=g)
    hi = _round(x, prec)
    x = hi + _round(x - hi, prec)
    X = x.double()
    S1 = X.reshape(nd * W, n1).T @ O1
    S2 = X.reshape(nd * n3, n2 * n1).T @ O2
    return [float(torch.linalg.norm(sketch(x, k) - S) / torch.linalg.norm(S)) for k, S in ((1, S1), (2, S2))]


BARS = {"bf16": 1.06e-7, "fp16": 1.35e-7, "tf32": 2.02e-7}


@pytest.mark.parametrize("prec", ["bf16", "fp16", "tf32"])
@pytest.mark.parametrize("dims,r,p", [([128, 40, 40, 64], 6, 5), ([112, 24, 36, 96], 18, 10), ([300, 24, 20, 100], 25, 10)])
def test_column_sums(dims, r, p, prec):
    e1, e2 = column_errors(dims, r, p, prec)
    assert max(e1, e2) <= BARS[prec], (e1, e2)


def test_column_sums_of_long_units():
    """Register chains as long as they get (the tile kernel: 1.01e-7)."""
    e1, e2 = column_errors([112, 100, 100, 112], 6, 5, "bf16")
    assert max(e1, e2) <= 1.01e-7, (e1, e2)
