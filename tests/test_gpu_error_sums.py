"""Error sums of FP32 data against quadruple precision: residuals down to the rounding of
an FP64 product, sums without a bias, trains beyond FP32's range.

Bars.  A residual is known as from an FP64 sum of rank terms: rank 2^-53 of the rms term where
it is all that is left, (rank + 2) 2^-53 of the largest term at worst.  Sums of squares
are compensated within a chunk and FP64 above it: 2^-51.  Out of FP32's range they are
plain FP64 sums, a few hundred addends a thread: 2^-46."""
import numpy as np
import pytest
import torch

from paper_2111_10448_gb300 import TTSketch

pytestmark = pytest.mark.gpu


def _plan(n, m, r):
    return TTSketch([n, m], ranks=[1, r, 1], p=2, seed=1, prec="fp64", x_dtype=torch.float32)


def _error(t, L, R, X):
    it = t.items[0]
    rp = it["rpad"][1]
    r = L.shape[1]
    f = np.zeros(t.core_entries)
    G1, G2 = np.zeros((1, L.shape[0], rp)), np.zeros((rp, R.shape[1], 1))
    G1[0, :, :r], G2[:r, :, 0] = L, R
    for k, G in ((1, G1), (2, G2)):
        f[it["core_off"][k]:it["core_off"][k] + G.size] = G.reshape(-1, order="F")
    return t.error(torch.tensor(X.reshape(-1, order="F"), device="cuda"), cores=torch.tensor(f, device="cuda")).tolist()


def _exact(L, R, X):
    """(sum (X - L R)^2, sum X^2, largest |term|) in quadruple precision."""
    q = np.longdouble
    ref = np.zeros(X.shape, dtype=q)
    for c in range(L.shape[1]):
        ref += L[:, c:c + 1].astype(q) * R[c:c + 1].astype(q)
    d = X.astype(q) - ref
    return np.sum(d * d), np.sum(X.astype(q) ** 2), np.max(np.abs(L), axis=0) @ np.max(np.abs(R), axis=1)


@pytest.mark.parametrize("r", [4, 8, 10, 24, 40, 60])
@pytest.mark.parametrize("noise", [1.0, 1e-4, 0.0])
def test_sums(r, noise):
    n, m = 1009, 803
    rng = np.random.default_rng(r)
    L, R = rng.standard_normal((n, r)), rng.standard_normal((r, m))
    X = (L @ R + noise * rng.standard_normal((n, m))).astype(np.float32)
    e2, x2, big = _exact(L, R, X)
    g2, h2 = _error(_plan(n, m, r), L, R, X)
    d = float(np.sqrt(e2)) + np.sqrt(n * m) * (r + 2) * 2.0 ** -53 * big
    assert abs(h2 - x2) <= 2.0 ** -51 * x2
    assert abs(g2 - e2) <= 2.0 ** -51 * e2 + (d * d - float(e2))


@pytest.mark.parametrize("r", [4, 8, 12, 30])
def test_tensor_met_to_rounding(r):
    """X is an FP32 tensor that the cores' exact product equals but for FP64 roundings of
    the cores: what is left is the size of FP64 rounding errors."""
    n, m = 1009, 803
    rng = np.random.default_rng(r)
    A, B = rng.integers(-40, 41, (n, r)).astype(np.float64), rng.integers(-40, 41, (r, m)).astype(np.float64)
    s = rng.uniform(1, 2, r)
    X = (A @ B).astype(np.float32)
    assert np.array_equal(X.astype(np.float64), A @ B)
    L, R = A * s, B / s[:, None]
    e2, x2, _ = _exact(L, R, X)
    g2, h2 = _error(_plan(n, m, r), L, R, X)
    assert h2 == float(x2)   # integers
    rms = np.sqrt(np.mean(A * A) * np.mean(B * B))
    assert g2 <= 2 * float(e2) + n * m * (r * 2.0 ** -53 * rms) ** 2


@pytest.mark.parametrize("e,xe", [(200, 0), (60, 100), (-200, -200), (-180, -140), (-90, -60), (130, 126)])
def test_range(e, xe):
    """X~ of magnitude 2^e, X of magnitude 2^xe (zero below FP32's range)."""
    n, m, r = 1009, 803, 5
    rng = np.random.default_rng(abs(e))
    L, R = rng.standard_normal((n, r)) * 2.0 ** (e // 2), rng.standard_normal((r, m)) * 2.0 ** (e - e // 2)
    X = (rng.uniform(-1, 1, (n, m)) * 2.0 ** xe).astype(np.float32)
    e2, x2, big = _exact(L, R, X)
    g2, h2 = _error(_plan(n, m, r), L, R, X)
    assert abs(h2 - float(x2)) <= 2.0 ** -46 * float(x2)
    assert abs(g2 - float(e2)) <= 2.0 ** -46 * float(e2)
