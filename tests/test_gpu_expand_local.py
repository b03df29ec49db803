"""FP32 reconstruction and error sums where the interfaces' large entries do not meet:
localised components, cancellation, values at and past the ends of FP32's range.

Bar of an FP32 entry: it comes from an FP64 sum (relative error rank 2^-53 of the terms'
magnitudes, as is the reference's) and is rounded to FP32; the kernel's own bound for what
it keeps is 1/8 of the half-ulp step 2^-24 more: |got - ref| <= 2^-24 (1 + 1/4) |ref| +
2 rank 2^-53 sum |terms| + 2^-149.  Error sums: the residual of an entry is known to rank
2^-52 of the column's largest term, sums of squares to 2^-50."""
import numpy as np
import pytest
import torch

from paper_2111_10448_gb300 import TTSketch

pytestmark = pytest.mark.gpu


def _plan(n, m, r):
    return TTSketch([n, m], ranks=[1, r, 1], p=2, seed=1, prec="fp64", x_dtype=torch.float32)


def _cores(t, L, R):
    """The flat cores of L R (two modes: L is core 1, R core 2)."""
    it = t.items[0]
    rp = it["rpad"][1]
    n, r = L.shape
    f = np.zeros(t.core_entries)
    G1, G2 = np.zeros((1, n, rp)), np.zeros((rp, R.shape[1], 1))
    G1[0, :, :r], G2[:r, :, 0] = L, R
    for k, G in ((1, G1), (2, G2)):
        f[it["core_off"][k]:it["core_off"][k] + G.size] = G.reshape(-1, order="F")
    return torch.tensor(f, device="cuda")


def _localised(rng, n, m, r, e):
    """Component c lives on the rows = c mod r and the columns = c mod r, at 2^-e elsewhere."""
    u, v, c = np.arange(n)[:, None] % r, np.arange(m)[None, :] % r, np.arange(r)
    L = np.where(u == c, 1.0, 2.0 ** -e) * rng.uniform(1, 2, (n, r))
    R = np.where(v == c[:, None], 1.0, 2.0 ** -e) * rng.uniform(1, 2, (r, m))
    return L, R


def _check(t, L, R):
    with np.errstate(over="ignore"):
        ref = L @ R
        terms = np.abs(L) @ np.abs(R)
        got = t.reconstruct(torch.float32, cores=_cores(t, L, R)).cpu().numpy().reshape(ref.shape, order="F")
        fin = np.isfinite(ref.astype(np.float32))
        assert np.array_equal(np.isfinite(got), fin)
        g, w = got[fin].astype(np.float64), ref[fin]
        bar = 2.0 ** -24 * 1.25 * np.abs(w) + 2 * L.shape[1] * 2.0 ** -53 * terms[fin] + 2.0 ** -149
    assert np.all(np.abs(g - w) <= bar)
    return ref


@pytest.mark.parametrize("r", [2, 5, 8, 9, 16, 30, 47, 60])
@pytest.mark.parametrize("e", [12, 30, 45, 60])
def test_fp32_output_localised(r, e):
    n, m = (1030, 801) if r >= 8 else (2102, 1605)   # small ranks are FP64 below 3 2^21 / rank entries
    rng = np.random.default_rng(r)
    t = _plan(n, m, r)
    _check(t, *_localised(rng, n, m, r, e))


@pytest.mark.parametrize("r", [3, 12, 50])
def test_fp32_output_cancellation(r):
    """Terms that cancel to 2^-20 and less of their magnitude, exact zeros among them."""
    n, m = 1501, 1410
    rng = np.random.default_rng(r + 100)
    L, R = rng.standard_normal((n, r)), rng.standard_normal((r, m))
    L[:, -1], R[-1] = L[:, 0], -R[0] * (1 + 2.0 ** -rng.integers(18, 52, m))
    L[:, 1:-1] = 0
    t = _plan(n, m, r)
    ref = _check(t, L, R)
    assert np.median(np.abs(ref)) < 2.0 ** -18


@pytest.mark.parametrize("r", [8, 16, 40, 60])
@pytest.mark.parametrize("e", [6, 14, 22])
def test_fp32_output_coherent_digits(r, e):
    """Every digit of half the factors +127 (what is dropped adds up), cancelled down to 2^-e by factors
    whose digits end after the third."""
    n, m = 1030, 801
    rng = np.random.default_rng(e)
    a = sum(127.0 * 256.0 ** -i for i in range(1, 7))
    L = np.full((n, r), a) * 2.0 ** rng.integers(0, 2, (n, 1))
    R = np.full((r, m), a)
    b = np.round(a * a * 2 ** 20) / 2 ** 20
    L[:, r // 2:] = np.sign(L[:, r // 2:]) * 0.5 * L[:, :1] / a
    R[r // 2:] = -2.0 * b * (1 - 2.0 ** -e * rng.integers(1, 4, (1, m)))
    _check(_plan(n, m, r), L, R)


@pytest.mark.parametrize("scale", [-140, -120, 120])
def test_fp32_output_ends_of_the_range(scale):
    n, m, r = 1100, 1000, 6
    rng = np.random.default_rng(3)
    t = _plan(n, m, r)
    L, R = rng.standard_normal((n, r)), rng.standard_normal((r, m))
    L *= 2.0 ** rng.integers(-12, 12, (n, 1)).astype(np.float64)
    _check(t, L * 2.0 ** (scale // 2), R * 2.0 ** (scale - scale // 2))
    # FP64 subnormal factors against huge ones
    L2, R2 = L.copy(), R.copy()
    L2[:, 2] *= 2.0 ** -1060
    R2[2] *= 2.0 ** 1000
    _check(t, L2, R2)
