"""The digit-arithmetic reconstruction (FP32 output) and error sums against
NumPy FP64.

Bars: an FP32 entry is the FP64 one rounded to nearest (2^-24 of its magnitude,
a little more because the last Horner step rounds a value that is itself off by
2^-32 of it) plus the dropped digits, at most rank 2^-34 of the largest term
|L(u, c) Rt(c, v)| of its row and column; the error sums are off by at most 2^-40
relative plus what the dropped digits (rank 2^-42 of the largest term) change
in the residual."""
import numpy as np
import pytest
import torch

from paper_2111_10448_gb300 import TTSketch

pytestmark = pytest.mark.gpu


def _plan(dims, r):
    ranks = [1] + [r] * (len(dims) - 1) + [1]
    return TTSketch(dims, ranks=ranks, p=2, seed=1, prec="fp64", x_dtype=torch.float32)


def _cores(t, rng, scale=1.0):
    it = t.items[0]
    out = []
    for k in range(1, it["d"] + 1):
        out.append(scale * rng.standard_normal((it["rpad"][k - 1], it["dims"][k - 1], it["rpad"][k])))
    return out


def _flat(t, cores):
    it = t.items[0]
    f = np.zeros(t.core_entries)
    for k, G in enumerate(cores, start=1):
        f[it["core_off"][k]:it["core_off"][k] + G.size] = G.reshape(-1, order="F")
    return torch.tensor(f, device="cuda")


def _interfaces(cores):
    d = len(cores)
    ds = (d + 1) // 2
    L = np.ones((1, 1))
    for G in cores[:ds]:
        a, n, b = G.shape
        L = (L @ G.reshape((a, n * b), order="F")).reshape((L.shape[0] * n, b), order="F")
    R = np.ones((1, 1))
    for G in cores[ds:][::-1]:
        a, n, b = G.shape
        R = (G.reshape((a * n, b), order="F") @ R).reshape((a, n * R.shape[1]), order="F")
    return L, R


CASES = [
    ([1200, 700], 1), ([1017, 1001], 3), ([64, 12289], 5), ([33, 40, 600], 16), ([40, 39, 520], 17),
    ([31, 9, 29, 100], 33), ([99, 91, 92], 60), ([12288, 65], 7), ([30, 31, 30, 31], 10), ([90, 100, 89], 8),
    ([1000, 800], 9),
]


def _check(t, cores):
    L, R = _interfaces(cores)
    ref = L @ R
    term = np.max(np.abs(L)[:, :, None].max(axis=0) * np.abs(R)[:, :].max(axis=1)[:, None]) if L.size else 0.0
    got = t.reconstruct(torch.float32, cores=_flat(t, cores)).cpu().numpy().reshape(ref.shape, order="F")
    bar = 2.0 ** -24 * 1.01 * np.abs(ref) + L.shape[1] * 2.0 ** -34 * term
    assert np.all(np.abs(got - ref) <= bar)
    return ref, term


@pytest.mark.parametrize("dims,r", CASES)
def test_fp32_output(dims, r):
    t = _plan(dims, r)
    ref, _ = _check(t, _cores(t, np.random.default_rng(7)))
    assert ref.size >= 3 << 18


@pytest.mark.parametrize("e", [-60, 30])
def test_fp32_output_scales_and_gauge(e):
    """Powers of two between the two interfaces and per rank index, zero rows and
    columns, and entries from 2^-300 of the largest up."""
    dims, r = [300, 8, 900], 12
    t = _plan(dims, r)
    rng = np.random.default_rng(8)
    cores = _cores(t, rng)
    k = 2.0 ** rng.integers(-200, 200, cores[1].shape[2]).astype(np.float64)
    cores[1] = cores[1] * k
    cores[2] = cores[2] / k[:, None, None] * 2.0 ** e
    cores[0][:, 5, :] = 0.0
    cores[2][:, 7, :] = 0.0
    cores[2][3, :, :] = 0.0
    cores[0][:, 9, :] *= 2.0 ** -300
    L, R = _interfaces(cores)
    ref = L @ R
    got = t.reconstruct(torch.float32, cores=_flat(t, cores)).cpu().numpy().reshape(ref.shape, order="F")
    term = np.max([np.max(np.abs(L[:, c])) * np.max(np.abs(R[c])) for c in range(L.shape[1])])
    bar = 2.0 ** -24 * 1.01 * np.abs(ref) + L.shape[1] * 2.0 ** -34 * term + 2.0 ** -149
    assert np.all(np.abs(got - ref) <= bar)
    assert np.all(got[5::300] == 0.0)


@pytest.mark.parametrize("dims,r", CASES)
@pytest.mark.parametrize("noise", [1.0, 1e-4])
@pytest.mark.parametrize("off", [0, 1])
def test_error_sums(dims, r, noise, off):
    t = _plan(dims, r)
    rng = np.random.default_rng(9)
    cores = _cores(t, rng)
    L, R = _interfaces(cores)
    ref = (L @ R).reshape(-1, order="F")
    x = (ref + noise * np.sqrt(np.mean(ref ** 2)) * rng.standard_normal(ref.size)).astype(np.float32)
    buf = torch.empty(x.size + 1, dtype=torch.float32, device="cuda")
    buf[off:off + x.size] = torch.tensor(x)
    e2, x2 = t.error(buf[off:off + x.size], cores=_flat(t, cores)).cpu().numpy()
    x = x.astype(np.float64)
    assert abs(x2 - np.sum(x * x)) <= 2.0 ** -40 * np.sum(x * x)
    res = np.sum((x - ref) ** 2)
    assert abs(e2 - res) <= (2.0 ** -40 + 2 * L.shape[1] * 2.0 ** -42 * 16 / noise) * res


def test_error_sums_extremes():
    """Entries near the ends of FP32's range, an exact tensor and a zero one."""
    dims, r = [128, 23, 300], 4
    t = _plan(dims, r)
    rng = np.random.default_rng(10)
    for scale, xs in ((1e-12, 1e-30), (1e9, 1e30), (1.0, 1e-38)):
        cores = _cores(t, rng, scale)
        x = (xs * rng.standard_normal(int(np.prod(dims)))).astype(np.float32)
        L, R = _interfaces(cores)
        ref = (L @ R).reshape(-1, order="F")
        e2, x2 = t.error(torch.tensor(x, device="cuda"), cores=_flat(t, cores)).cpu().numpy()
        x = x.astype(np.float64)
        big = max(np.max(np.abs(ref)), np.max(np.abs(x)))
        assert abs(x2 - np.sum(x * x)) <= 1e-9 * np.sum(x * x) + x.size * (2.0 ** -60 * big) ** 2
        assert abs(e2 - np.sum((x - ref) ** 2)) <= 1e-9 * np.sum((x - ref) ** 2)
    cores = [np.round(4 * c) for c in _cores(t, rng)]   # integers: X is exact in FP32
    L, R = _interfaces(cores)
    ref = (L @ R).reshape(-1, order="F")
    assert np.all(ref == ref.astype(np.float32))
    e2, x2 = t.error(torch.tensor(ref.astype(np.float32), device="cuda"), cores=_flat(t, cores)).cpu().numpy()
    assert e2 <= (2.0 ** -38) ** 2 * x2 and abs(x2 - np.sum(ref * ref)) <= 1e-12 * x2
    z = [0 * c for c in cores]
    e2, x2 = t.error(torch.tensor(ref.astype(np.float32), device="cuda"), cores=_flat(t, z)).cpu().numpy()
    assert e2 == x2 > 0
    assert float(t.reconstruct(torch.float32, cores=_flat(t, z)).abs().max()) == 0.0


@pytest.mark.parametrize("bad", [float("inf"), float("nan")])
def test_nonfinite(bad):
    """Non-finite cores and tensors spread as in plain FP64 arithmetic."""
    dims, r = [300, 8, 600], 5
    t = _plan(dims, r)
    rng = np.random.default_rng(11)
    cores = _cores(t, rng)
    x = rng.standard_normal(int(np.prod(dims))).astype(np.float32)
    xb = x.copy()
    xb[12345] = bad
    e2, x2 = t.error(torch.tensor(xb, device="cuda"), cores=_flat(t, cores)).cpu().numpy()
    same = (lambda v: np.isinf(v)) if np.isinf(bad) else (lambda v: np.isnan(v))
    assert same(e2) and same(x2)
    cores[0][0, 17, 2] = bad
    cores[2][1, 333, 0] = bad
    with np.errstate(invalid="ignore"):
        L, R = _interfaces(cores)
        ref = (L @ R).astype(np.float32)
    got = t.reconstruct(torch.float32, cores=_flat(t, cores)).cpu().numpy().reshape(ref.shape, order="F")
    fin = np.isfinite(ref)
    assert np.array_equal(np.isfinite(got), fin)
    assert np.allclose(got[fin], ref[fin], rtol=1e-6, atol=1e-5)
