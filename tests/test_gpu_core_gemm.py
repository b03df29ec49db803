"""Cores large enough for the digit-arithmetic core product (2^25 FMAs): the middle
core as (Q^T S) M, the other left cores and the right cores.  FP64 plans recover
exact-rank tensors to 1e-11, every core equals its defining product of the
neighbouring cores' orthonormal bases, and the gradient (which forms H when it runs)
passes a directional central difference."""
import numpy as np
import pytest
import torch

from paper_2111_10448_gb300 import PSTT2Fn, TTReconstructFn, TTSketch

pytestmark = pytest.mark.gpu

CASES = [([200, 300, 40], [1, 20, 20, 1], 10), ([260, 250, 2, 6, 8], [1, 24, 24, 24, 8, 1], 8),
         ([4, 5, 320, 280], [1, 4, 20, 20, 1], 9), ([150, 31, 301], [1, 50, 40, 1], 14),
         ([130, 131, 63], [1, 33, 63, 1], 1)]


def _tensor(dims, r, dev="cuda", seed=5):
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    L = torch.ones(1, 1, dtype=torch.float64, device=dev)
    for k, n in enumerate(dims):   # L: rows (i_k .. i_1 slowest first), column-major flat
        G = torch.randn(r[k], n, r[k + 1], dtype=torch.float64, device=dev, generator=g)
        L = torch.einsum("ua,anc->nuc", L, G).reshape(-1, r[k + 1])
    return L[:, 0].contiguous()


@pytest.mark.parametrize("dims,r,p", CASES)
@pytest.mark.parametrize("drm", ["gauss", "kr"])
def test_recovery(dims, r, p, drm):
    X = _tensor(dims, r)
    t = TTSketch(dims, ranks=r, p=p, seed=1, prec="fp64", x_dtype=torch.float64, drm=drm)
    for _ in range(2):
        t.pstt2(X)
    assert t.status()[0] == 0
    err = float(torch.linalg.norm(t.reconstruct(torch.float64) - X) / torch.linalg.norm(X))
    assert err <= 1e-11
    # left cores before the middle one are orthonormal, right ones after it row-orthonormal
    ds = (len(dims) + 1) // 2
    for k, G in enumerate(t.core_list(), start=1):
        a, n, c = G.shape
        if k < ds:
            M = G.reshape(a * n, c)
            assert np.abs(M.T @ M - np.eye(c)).max() <= 1e-12
        elif k > ds:
            M = G.reshape(a, n * c)
            assert np.abs(M @ M.T - np.eye(a)).max() <= 1e-12


def test_scaled_and_nonfinite():
    dims, r, p = CASES[0]
    X = _tensor(dims, r)
    t = TTSketch(dims, ranks=r, p=p, seed=1, prec="fp64", x_dtype=torch.float64)
    for s in (2.0 ** -400, 2.0 ** 400):
        t.pstt2(X * s)
        err = float(torch.linalg.norm((t.reconstruct(torch.float64) / s - X)) / torch.linalg.norm(X))
        assert err <= 1e-11
    Y = X.clone()
    Y[777] = float("nan")
    t.pstt2(Y)
    assert bool(torch.isnan(t.cores).any())


def test_gradient():
    dims, r, p = CASES[0]
    X = _tensor(dims, r)
    X = X / torch.linalg.norm(X)
    g = torch.Generator(device="cuda")
    g.manual_seed(9)
    X = X + 1e-3 * torch.randn(X.numel(), dtype=torch.float64, device="cuda", generator=g) / np.sqrt(X.numel())
    D = torch.randn(X.numel(), dtype=torch.float64, device="cuda", generator=g) / np.sqrt(X.numel())
    C = torch.randn(X.numel(), dtype=torch.float64, device="cuda", generator=g)
    t = TTSketch(dims, ranks=r, p=p, seed=1, prec="fp64", x_dtype=torch.float64, diff=True)

    def loss(x):
        return torch.sum(C * TTReconstructFn.apply(PSTT2Fn.apply(x, t), t, torch.float64))

    x = X.clone().requires_grad_(True)
    loss(x).backward()
    h = 1e-6
    fd = (float(loss(X + h * D)) - float(loss(X - h * D))) / (2 * h)
    assert abs(fd - float(torch.sum(x.grad * D))) <= 1e-6 * float(torch.linalg.norm(x.grad) * torch.linalg.norm(D))
