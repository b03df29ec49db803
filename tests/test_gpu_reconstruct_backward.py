"""The adjoint of the reconstruction (two products at the middle, cores absorbing
one mode at a time) against torch autograd of the contraction in FP64, over
orders, ragged shapes and every rank instance.  Bar: FP64 rounding of sums of at
most a few 10^5 terms, 1e-12 of the gradient's norm per core."""
import numpy as np
import pytest
import torch

from paper_2111_10448_gb300 import TTSketch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,r", [([37, 53], 5), ([3, 200], 2), ([21, 33, 40], 9), ([40, 5, 41], 17),
                                    ([70, 9, 66], 40), ([12, 13, 11, 14], 8), ([33, 1, 7, 34], 6),
                                    ([6, 7, 8, 5, 9], 4), ([5, 4, 3, 6, 5, 4], 3)])
@pytest.mark.parametrize("dt", [torch.float32, torch.float64])
def test_matches_autograd(dims, r, dt):
    d = len(dims)
    t = TTSketch(dims, ranks=[1] + [r] * (d - 1) + [1], p=3, seed=1, prec="fp64", x_dtype=torch.float64, diff=True)
    it = t.items[0]
    rp = it["rpad"]
    rng = np.random.default_rng(4)
    cores = [torch.tensor(rng.standard_normal((rp[k], dims[k], rp[k + 1])), requires_grad=True) for k in range(d)]
    dX = torch.tensor(rng.standard_normal(int(np.prod(dims)))).to(dt)
    X = cores[0].reshape(dims[0], rp[1])
    for G in cores[1:]:
        X = (X @ G.reshape(G.shape[0], -1)).reshape(-1, G.shape[2])
    # row-major tensor; dX is column-major flat
    ref_dX = dX.double().reshape(dims[::-1]).permute(*range(d - 1, -1, -1)).reshape(-1)
    torch.sum(X.reshape(-1) * ref_dX).backward()
    flat = torch.zeros(t.core_entries, dtype=torch.float64)
    for k, G in enumerate(cores):
        flat[it["core_off"][k + 1]:it["core_off"][k + 1] + G.numel()] = G.detach().permute(2, 1, 0).reshape(-1)
    got = t.reconstruct_backward(dX.cuda(), cores=flat.cuda()).cpu()
    for k, G in enumerate(cores):
        g = got[it["core_off"][k + 1]:it["core_off"][k + 1] + G.numel()].reshape(rp[k + 1], dims[k], rp[k])
        ref = G.grad.permute(2, 1, 0)
        assert float(torch.linalg.norm(g - ref)) <= 1e-12 * float(torch.linalg.norm(ref)), k


@pytest.mark.parametrize("dims,r", [([515, 517], 5), ([520, 640], 12), ([70, 30, 130], 17), ([90, 40, 100], 40),
                                    ([30, 20, 21, 30], 8), ([4096, 64], 63), ([64, 5000], 33)])
@pytest.mark.parametrize("kind", ["normal", "range", "nan"])
def test_digit_products_match_autograd(dims, r, kind):
    """FP32 data large enough for the digit products, at ragged 64 x 64 tiles and every
    column-octet instance: rows and columns of very different magnitudes, and a NaN that
    reaches the entries it reaches in FP64 and no others."""
    d = len(dims)
    t = TTSketch(dims, ranks=[1] + [r] * (d - 1) + [1], p=1, seed=1, prec="fp64", x_dtype=torch.float64, diff=True)
    it = t.items[0]
    rp = it["rpad"]
    rng = np.random.default_rng(4)
    cores = [torch.tensor(rng.standard_normal((rp[k], dims[k], rp[k + 1])), requires_grad=True) for k in range(d)]
    dX = rng.standard_normal(dims).astype(np.float32)
    if kind == "range":
        dX *= np.exp2(-(np.arange(dims[0]) % 90)).astype(np.float32).reshape([-1] + [1] * (d - 1))
        dX *= np.exp2((np.arange(dims[-1]) % 31)).astype(np.float32)
    if kind == "nan":
        dX[3, ..., 5] = np.nan
    X = cores[0].reshape(dims[0], rp[1])
    for G in cores[1:]:
        X = (X @ G.reshape(G.shape[0], -1)).reshape(-1, G.shape[2])
    torch.sum(X.reshape(-1) * torch.tensor(dX).double().reshape(-1)).backward()
    flat = torch.zeros(t.core_entries, dtype=torch.float64)
    for k, G in enumerate(cores):
        flat[it["core_off"][k + 1]:it["core_off"][k + 1] + G.numel()] = G.detach().permute(2, 1, 0).reshape(-1)
    dev = torch.tensor(dX).permute(*range(d - 1, -1, -1)).reshape(-1).contiguous().cuda()
    got = t.reconstruct_backward(dev, cores=flat.cuda()).cpu()
    for k, G in enumerate(cores):
        g = got[it["core_off"][k + 1]:it["core_off"][k + 1] + G.numel()].reshape(rp[k + 1], dims[k], rp[k])
        ref = G.grad.permute(2, 1, 0)
        if kind == "nan":
            assert torch.equal(torch.isnan(g), torch.isnan(ref))
            g, ref = torch.nan_to_num(g), torch.nan_to_num(ref)
        # per slice of the mode: rows of small magnitude keep their own relative error
        if k == 0 and kind == "range":
            err = torch.linalg.norm(g - ref, dim=(0, 2)) / torch.linalg.norm(ref, dim=(0, 2))
            assert float(err.max()) <= 1e-12
        assert float(torch.linalg.norm(g - ref)) <= 1e-12 * float(torch.linalg.norm(ref)), k
