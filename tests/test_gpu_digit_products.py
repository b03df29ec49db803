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
