"""Digit products where the large factors of a sum do not meet: every entry is held to
Σ |terms|, as in FP64, not to the largest factors of its row and column.

Bar: the kernels accept a chunk's digits while they are within K 2^-57 (K terms, 32 or 64) of
factors whose products' magnitudes add up to 1/256 (32) or 1/128 (64) of the largest, 2^-44 of
Σ |terms|; the rest are FP64 sums over at most a few thousand terms, 2^-42."""
import numpy as np
import pytest
import torch

from paper_2111_10448_gb300 import TTSketch

pytestmark = pytest.mark.gpu
BAR = 2.0 ** -41


def _flat(t, cores):
    it = t.items[0]
    f = np.zeros(t.core_entries)
    for k, G in enumerate(cores, start=1):
        f[it["core_off"][k]:it["core_off"][k] + G.size] = G.reshape(-1, order="F")
    return torch.tensor(f, device="cuda")


@pytest.mark.parametrize("e", [0, 10, 30, 60, 100])
@pytest.mark.parametrize("r", [5, 13, 20, 50])
def test_adjoint_entrywise(r, e):
    """dX is 2^-e where the interfaces are 1 and 1 where they are 2^-e (rows and columns by
    their parity, neighbours in one chunk)."""
    n, m = 300, 517
    t = TTSketch([n, m], ranks=[1, r, 1], p=1, seed=1, prec="fp64", x_dtype=torch.float64, diff=True)
    rp = t.items[0]["rpad"][1]
    rng = np.random.default_rng(r)
    L, R = rng.uniform(1, 2, (n, rp)), rng.uniform(1, 2, (rp, m))
    L[0::2, 0::2] *= 2.0 ** -e
    L[1::2, 1::2] *= 2.0 ** -e
    R[0::2, 0::2] *= 2.0 ** -e
    R[1::2, 1::2] *= 2.0 ** -e
    for cols in (0, 1):   # against the rows, against the columns
        dX = rng.uniform(-2, 2, (n, m)).astype(np.float32)
        if cols:
            dX[:, 1::2] *= np.float32(2.0 ** -e)
        else:
            dX[1::2] *= np.float32(2.0 ** -e)
        got = t.reconstruct_backward(torch.tensor(dX.reshape(-1, order="F"), device="cuda"),
                                     cores=_flat(t, [L[None], R[:, :, None]])).cpu().numpy()
        off = t.items[0]["core_off"]
        g1 = got[off[1]:off[1] + n * rp].reshape((n, rp), order="F")
        g2 = got[off[2]:off[2] + rp * m].reshape((rp, m), order="F")
        D = dX.astype(np.float64)
        assert np.all(np.abs(g1 - D @ R.T) <= BAR * (np.abs(D) @ np.abs(R.T)))
        assert np.all(np.abs(g2 - L.T @ D) <= BAR * (np.abs(L.T) @ np.abs(D)))


@pytest.mark.parametrize("e", [0, 30, 60, 100])
def test_core_entrywise(e):
    """The middle core (Q^T S) M from a stream's state whose S_1 has exact orthonormal columns of
    disjoint support (Q = S_1 without rounding) and whose S_2 = w z^T is 2^-e on the support
    of every other column: core(a, i, :) = t(a, i) (z^T M) for all a, the small ones too."""
    dims, r, p = [256, 256, 40], 20, 10
    w = r + p
    t = TTSketch(dims, ranks=[1, r, r, 1], p=p, seed=1, prec="fp64", x_dtype=torch.float64)
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    X = torch.randn(int(np.prod(dims)), dtype=torch.float64, device="cuda", generator=g)
    t.begin()
    t.accumulate(X, 0, dims[2])
    sk = [(ty, k, S.shape) for ty, k, S in t.sketches()]
    state = t.export_state()
    n = sum(a * b for _, _, (a, b) in sk)
    flat = state[state.size - 8 * n:].view(np.float64)
    rng = np.random.default_rng(4)
    S1 = np.zeros((256, w))
    for a in range(w):   # heads (rows below w) zero: reflectors I - v v^T without rounding
        S1[32 + a:160:32, a] = 0.5
    W = rng.uniform(1, 2, (256, 256))
    W[33:160:2] *= 2.0 ** -e
    z = rng.standard_normal(w)
    at = 0
    for ty, k, (a, b) in sk:
        if ty == 0 and k == 1:
            assert (a, b) == S1.shape
            flat[at:at + a * b] = S1.reshape(-1, order="F")
        elif ty == 0 and k == 2:
            flat[at:at + a * b] = np.outer(W.reshape(-1, order="F"), z).reshape(-1, order="F")
        at += a * b
    t.import_state(state)
    t.finalize()
    G = t.core_list()[1]
    T = S1[:, :r].T @ W
    q = G[0, 0] / T[0, 0]
    # z^T M cancels to about 1/10 of its terms; 1e-11 for their sums
    assert np.all(np.abs(G - T[:, :, None] * q) <= 1e-11 * T[:, :, None] * np.abs(q).max())
