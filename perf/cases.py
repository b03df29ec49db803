"""The workloads the library is timed on: what a program that compresses tensors
does with it, through the public entry points of paper_2111_10448_gb300.

Every case is one call (or one stream of calls) on data that is on the GPU and a
plan that such a program keeps.  Five kinds of work:

  compress    TTSketch.pstt2, or begin / accumulate / finalize over slabs of the
              last mode: a dense tensor becomes TT cores.  Cores of FP32 tensors
              are handed on in FP32, the way a compressed FP32 tensor is stored.
              With round_trip the dense X~ comes back as well (compress,
              transmit, expand), and then it is what is returned: X~ is the
              result that does not depend on a choice of basis between cores.
  expand      TTSketch.reconstruct on stored cores.
  verify      TTSketch.error: is a stored train still within tolerance of X?
  gradient    PSTT2Fn and TTReconstructFn under autograd, forward and backward.
  batch       TTSketch.batched: many small uneven tensors in one call.
  tucker      tucker2tt and back with tt2tucker.

Tensors are random TT tensors (N(0,1) cores, the precision, batched and
differentiation workloads) or sums of plane waves on a grid (a function tensor of
known ranks that is well conditioned, for the large shapes).  Both have exact low
TT rank, so X~ in exact arithmetic is X up to the added noise.
"""
import math

import torch

from paper_2111_10448_gb300 import (PSTT2Fn, TTReconstructFn, TTSketch, tt2tucker, tucker2tt, x_scale_log2)

_KEYS = dict(work="compress", dims="", data="tt", rank=0, ranks="", noise=0.0, eps=0.0, rmax=0, p=5, prec="fp64",
             x="f32", drm="gauss", slab=0, passes=1, one_sided=False, round_trip=False, count=0, n_outer=0, trank=0)


def _case(name=None, **kw):
    c = dict(name=name) if name else {}
    c.update({k: kw.get(k, v) for k, v in _KEYS.items() if k in kw or k in ("work", "dims", "prec", "p")})
    return c


def _get(case, key):
    return case.get(key, _KEYS[key])


def _dims(case):
    return [int(v) for v in case["dims"].split("x")]


def listed():
    return [
        # The smallest call: 16^4 doubles, ranks asked for slightly above the tensor's own.  Launch latency.
        _case("fp64_16p4", dims="16x16x16x16", data="tt", ranks="3,4,3", rank=4, p=5, prec="fp64", x="f64",
              round_trip=True),
        # Tolerance mode on a noisy six-way tensor with small modes, out and back.
        _case("bf16_24p6_eps", dims="24x24x24x24x24x24", data="tt", ranks="10,10,10,10,10", noise=1e-6, eps=1e-5,
              rmax=16, p=10, prec="bf16", round_trip=True),
        # The streaming workload: 17 GB in slabs of 1 GiB, Khatri-Rao test matrices, FP16 split, tolerance mode.
        _case("fp16_256p4_slabs", dims="256x256x256x256", data="wave", ranks="4,4,4", eps=1e-6, rmax=6, p=10,
              prec="fp16", drm="kr", slab=16),
        # A resident 1 GiB tensor in one call, dense Gaussian test matrices.
        _case("bf16_128p4", dims="128x128x128x128", data="wave", ranks="6,6,6", rank=6, p=10, prec="bf16"),
        # The large three-way function tensor (few modes, long ones, higher rank).
        _case("bf16_960p3", dims="960x960x960", data="wave", ranks="25,25", rank=25, p=10, prec="bf16"),
        # The large five-way function tensor, 33 GB.
        _case("bf16_96p5", dims="96x96x96x96x96", data="wave", ranks="18,18,18,18", rank=18, p=10, prec="bf16"),
        # Uneven odd modes, as measured data comes; TF32.
        _case("tf32_ragged4", dims="61x53x67x47", data="tt", ranks="7,9,6", rank=9, p=6, prec="tf32",
              round_trip=True),
        # Many small tensors of uneven shape in one call.
        _case("bf16_batch512", work="batch", count=512, p=5, prec="bf16"),
        # A training step: the gradient of || TT(X) - T ||^2 with respect to X.
        _case("bf16_grad_32p5", work="gradient", dims="32x32x32x32x32", data="tt", ranks="8,8,8,8", rank=8, p=5,
              prec="bf16"),
        # Expanding a stored train to the dense 17 GB tensor.
        _case("expand_256p4", work="expand", dims="256x256x256x256", rank=6, x="f32"),
        # Checking a stored train against its tensor.
        _case("verify_24p6", work="verify", dims="24x24x24x24x24x24", rank=10, noise=1e-4, x="f32"),
        # A Tucker tensor to TT and back: the core tensor is 64^4 doubles, the full one 256^4 and never formed.
        _case("fp64_tucker_64p4", work="tucker", dims="64x64x64x64", data="tt", ranks="8,8,8", rank=8, p=10,
              prec="fp64", x="f64", n_outer=256, trank=40),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_dims(rng, d, entries, lo, hi):
    """d mode sizes around entries^(1/d), uneven, each in [lo, hi]."""
    n = entries ** (1.0 / d)
    return [max(lo, min(hi, int(round(n * math.exp(rng.uniform(-0.3, 0.3)))))) for _ in range(d)]


def draw(rng):
    kind = rng.choice(["small", "compress", "compress", "compress", "planes", "slabs", "batch", "gradient", "expand",
                       "verify", "tucker"])
    if kind == "small":
        d = rng.choice([2, 3, 4])
        dims = _draw_dims(rng, d, _log_int(rng, 4e3, 2e6), 9, 1000)
        r = rng.randint(2, 6)
        return _case(dims="x".join(map(str, dims)), data="tt", ranks=",".join([str(r)] * (d - 1)), rank=r,
                     p=rng.randint(5, 10), prec="fp64", x="f64", round_trip=True, drm=rng.choice(["gauss", "kr"]))
    if kind == "compress":
        d = rng.choice([3, 4, 5, 6])
        dims = _draw_dims(rng, d, _log_int(rng, 2e6, 1e9), 9, 1100)
        r = rng.randint(2, min(25, min(dims) - 2))
        return _case(dims="x".join(map(str, dims)), data="tt" if min(dims) < 64 else "wave",
                     ranks=",".join([str(r)] * (d - 1)), rank=r, p=rng.randint(6, 10),
                     prec=rng.choice(["bf16", "tf32", "fp16"]), drm=rng.choice(["gauss", "gauss", "kr"]),
                     round_trip=rng.random() < 0.5)
    if kind == "planes":  # whole tensors of 128- and 256-wide outer modes
        d = rng.choice([3, 4])
        mid = [_log_int(rng, 17, 150) for _ in range(d - 2)]
        dims = [rng.choice([128, 256])] + mid + [rng.choice([128, 256])]
        r = rng.randint(2, 6)
        return _case(dims="x".join(map(str, dims)), data="tt", ranks=",".join([str(r)] * (d - 1)), rank=6, p=10,
                     prec=rng.choice(["bf16", "fp16"]), round_trip=True)
    if kind == "slabs":
        n1, mid = rng.choice([128, 256, 200]), [_log_int(rng, 40, 256) for _ in range(2)]
        nd = 16 * rng.randint(3, 16) + rng.choice([0, 0, 5])
        return _case(dims="x".join(map(str, [n1] + mid + [nd])), data="wave", ranks="4,4,4", eps=1e-6, rmax=6, p=10,
                     prec=rng.choice(["fp16", "fp16", "bf16"]), drm=rng.choice(["kr", "gauss"]),
                     slab=rng.choice([16, 32, 64]), round_trip=True)
    if kind == "batch":
        return _case(work="batch", count=_log_int(rng, 8, 400), p=rng.randint(5, 8),
                     prec=rng.choice(["bf16", "fp16", "tf32"]))
    if kind == "gradient":
        d = rng.choice([3, 4, 5])
        dims = _draw_dims(rng, d, _log_int(rng, 1e5, 3e7), 9, 300)
        r = rng.randint(2, 8)
        return _case(work="gradient", dims="x".join(map(str, dims)), data="tt", ranks=",".join([str(r)] * (d - 1)),
                     rank=r, p=rng.randint(5, 8), prec=rng.choice(["bf16", "tf32", "fp64"]))
    if kind in ("expand", "verify"):
        d = rng.choice([2, 3, 4, 5, 6])
        dims = _draw_dims(rng, d, _log_int(rng, 1e5, 2e9 if kind == "expand" else 5e8), 3, 40000)
        return _case(work=kind, dims="x".join(map(str, dims)), rank=rng.randint(2, 24),
                     x=rng.choice(["f32", "f32", "f64"]), **({"noise": 1e-4} if kind == "verify" else {}))
    s = [_log_int(rng, 24, 72) for _ in range(rng.choice([3, 4]))]
    r = rng.randint(4, 9)
    return _case(work="tucker", dims="x".join(map(str, s)), data="tt", ranks=",".join([str(r)] * (len(s) - 1)), rank=r,
                 p=rng.randint(5, 10), prec="fp64", x="f64", n_outer=rng.randint(80, 300), trank=rng.randint(4, 20))


# ------------------------------------------------------------------- tensors
def _gen(seed, k=0):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 64 + k)
    return g


def _rank_list(case, d):
    if _get(case, "ranks"):
        r = [int(v) for v in case["ranks"].split(",")]
    else:
        r = [int(case["rank"])] * (d - 1)
    return _clamp(_dims(case), [1] + r + [1])


def _clamp(dims, r):
    """Ranks no larger than the tensor's unfoldings allow."""
    d, r = len(dims), list(r)
    for k in range(1, d):
        r[k] = min(r[k], r[k - 1] * dims[k - 1])
    for k in range(d - 1, 0, -1):
        r[k] = min(r[k], r[k + 1] * dims[k])
    return r


def _tt_cores(dims, r, seed):
    g = _gen(seed)
    return [torch.randn(r[k], dims[k], r[k + 1], dtype=torch.float64, device="cuda", generator=g)
            for k in range(len(dims))]


def _wave_cores(dims, rank, seed):
    """Cores of sum_m a_m cos(phi_m + sum_k w_{m,k} i_k) (+ a constant when the
    rank is odd): 2 x 2 rotations along the diagonal, TT rank `rank`."""
    g = _gen(seed)
    d, m = len(dims), rank // 2
    # frequencies in distinct bands, so that the waves stay apart along every mode
    w = torch.rand(m, d, dtype=torch.float64, device="cuda", generator=g)
    perm = torch.stack([torch.randperm(m, device="cuda", generator=g) for _ in range(d)], 1).to(torch.float64) \
        if m else w
    w = math.pi * (0.08 + 0.84 * (perm + 0.2 + 0.6 * w) / max(m, 1))
    ph = 2 * math.pi * torch.rand(m, dtype=torch.float64, device="cuda", generator=g)
    amp = 0.6 + 0.8 * torch.rand(m + 1, dtype=torch.float64, device="cuda", generator=g)
    cores = []
    for k, n in enumerate(dims):
        G = torch.zeros(rank, n, rank, dtype=torch.float64, device="cuda")
        i = torch.arange(n, dtype=torch.float64, device="cuda")
        for j in range(m):
            t = w[j, k] * i + (ph[j] if k == 0 else 0.0)
            G[2 * j, :, 2 * j] = G[2 * j + 1, :, 2 * j + 1] = torch.cos(t)
            G[2 * j, :, 2 * j + 1] = -torch.sin(t)
            G[2 * j + 1, :, 2 * j] = torch.sin(t)
        if rank % 2:
            G[rank - 1, :, rank - 1] = 1.0
        cores.append(G)
    left = torch.zeros(1, rank, dtype=torch.float64, device="cuda")
    left[0, 0:2 * m:2] = amp[:m]
    if rank % 2:
        left[0, rank - 1] = amp[m]
    right = torch.zeros(rank, 1, dtype=torch.float64, device="cuda")
    right[0:2 * m:2, 0] = 1.0
    if rank % 2:
        right[rank - 1, 0] = 1.0
    cores[0] = torch.einsum("ab,bnc->anc", left, cores[0])
    cores[-1] = torch.einsum("anb,bc->anc", cores[-1], right)
    return cores


def _data_cores(case, seed):
    dims = _dims(case)
    if _get(case, "data") == "wave":
        return _wave_cores(dims, _rank_list(case, len(dims))[1], seed)
    return _tt_cores(dims, _rank_list(case, len(dims)), seed)


def _dense(cores, dtype):
    """The dense column-major (i_1 fastest) tensor of a list of cores, formed in
    FP64 and stored as dtype."""
    d = len(cores)
    L = cores[0][0].t()                                   # r x n_1, transposed left interface
    for G in cores[1:(d + 1) // 2]:
        L = torch.einsum("au,anc->cnu", L, G).reshape(G.shape[2], -1)
    R = cores[-1][:, :, 0].t()                            # M x r
    for G in cores[(d + 1) // 2:-1][::-1]:
        R = torch.einsum("anc,vc->vna", G, R).reshape(-1, G.shape[0])
    n, m = L.shape[1], R.shape[0]
    out = torch.empty(m, n, dtype=dtype, device=L.device)
    step = max(1, (1 << 28) // n)
    for a in range(0, m, step):
        out[a:a + step] = R[a:a + step] @ L
    return out.reshape(-1)


def _dtype(case):
    return torch.float64 if _get(case, "x") == "f64" else torch.float32


def _add_noise(x, rel, seed):
    if rel:
        norm = torch.linalg.vector_norm(x, dtype=torch.float64)
        step = 1 << 26
        g = _gen(seed, 1)
        for a in range(0, x.numel(), step):
            y = x[a:a + step]
            y += torch.randn(y.numel(), dtype=x.dtype, device=x.device, generator=g) * \
                (rel * norm / math.sqrt(x.numel())).to(x.dtype)
    return x


def _tensor(case, seed):
    return _add_noise(_dense(_data_cores(case, seed), _dtype(case)), _get(case, "noise"), seed)


def _batch_specs(case):
    """Uneven shapes, d in 3..6 and n in 8..32 (at most 2e6 entries), ranks 2..16."""
    import random
    rng = random.Random(int(case["count"]))
    specs = []
    for _ in range(int(case["count"])):
        d, n = rng.randint(3, 6), rng.randint(8, 32)
        n = min(n, int(math.floor(2e6 ** (1.0 / d) + 1e-9)))
        specs.append(([n] * d, _clamp([n] * d, [1] + [rng.randint(2, 16) for _ in range(d - 1)] + [1])))
    return specs


def _flat_cores(sk, cores):
    """Cores in the flat layout of TTSketch.cores."""
    flat = torch.zeros_like(sk.cores)
    it = sk.items[0]
    for k, G in enumerate(cores, start=1):
        r0, n, r1 = G.shape
        flat[it["core_off"][k]:it["core_off"][k] + r0 * n * r1] = G.permute(2, 1, 0).reshape(-1)
    return flat


# --------------------------------------------------------------------- cases
def _plan(case, X, **kw):
    dims = _dims(case)
    if _get(case, "eps"):
        kw.update(eps=case["eps"], rmax=case["rmax"])
    else:
        kw.update(ranks=_clamp(dims, [1] + [int(case["rank"])] * (len(dims) - 1) + [1]))
    prec = case["prec"]
    return TTSketch(dims, p=case["p"], seed=1, prec=prec, drm=_get(case, "drm"), passes=_get(case, "passes"),
                    one_sided=_get(case, "one_sided"), x_dtype=_dtype(case),
                    x_scale_log2=x_scale_log2(X) if prec == "fp16" else 0, **kw)


def prepare(case, seed):
    work = _get(case, "work")
    if work == "batch":
        specs = _batch_specs(case)
        Xs, probs = [], []
        for b, (dims, r) in enumerate(specs):
            Xs.append(_dense(_tt_cores(dims, r, 1009 * seed + b), torch.float32))
            probs.append(dict(dims=dims, ranks=r, p=case["p"], seed=1000 + b))
        if case["prec"] == "fp16":
            for pr, x in zip(probs, Xs):
                pr["x_scale_log2"] = x_scale_log2(x)
        sk = TTSketch(None, batch=probs, p=case["p"], prec=case["prec"])
        return dict(work=work, sk=sk, Xs=Xs)
    if work == "tucker":
        G = _tensor(case, seed)
        g = _gen(seed, 2)
        A = [torch.linalg.qr(torch.randn(case["n_outer"], s, dtype=torch.float64, device="cuda", generator=g))[0]
             for s in _dims(case)]
        r = _clamp(_dims(case), [1] + [case["rank"]] * (len(A) - 1) + [1])
        return dict(work=work, G=G, A=A, p=case["p"], ranks=r, trank=case["trank"])
    if work in ("expand", "verify"):
        dims = _dims(case)
        r = _clamp(dims, [1] + [int(case["rank"])] * (len(dims) - 1) + [1])
        sk = TTSketch(dims, ranks=r, p=case["p"], seed=1, prec="fp64", x_dtype=_dtype(case))
        cores = _tt_cores(dims, r, seed)
        s = dict(work=work, sk=sk, cores=_flat_cores(sk, cores), dtype=_dtype(case))
        if work == "verify":
            s["X"] = _add_noise(_dense(cores, _dtype(case)), case["noise"], seed)
        return s
    X = _tensor(case, seed)
    s = dict(work=work, X=X, dtype=_dtype(case), round_trip=_get(case, "round_trip"))
    if work == "gradient":
        s["sk"] = _plan(case, X, diff=True)
        s["T"] = torch.randn(X.numel(), dtype=X.dtype, device="cuda", generator=_gen(seed, 3))
        return s
    s["sk"] = _plan(case, X)
    if _get(case, "slab"):
        n, nd1 = _dims(case)[-1], X.numel() // _dims(case)[-1]
        s["slabs"] = [(X[a * nd1:min(n, a + case["slab"]) * nd1], a, min(n, a + case["slab"]) - a)
                      for a in range(0, n, case["slab"])]
    return s


def run(s):
    work = s["work"]
    if work == "batch":
        s["sk"].batched(s["Xs"])
        return {"cores": s["sk"].cores.to(torch.float32), "ranks": s["sk"].ranks}
    if work == "tucker":
        cores, _ = tucker2tt(s["G"], s["A"], ranks=s["ranks"], p=s["p"], seed=1)
        H, A = tt2tucker(cores, [s["trank"]] * len(cores), p=s["p"], seed=3)
        return {"cores": cores, "H": H, "A": A}
    if work == "expand":
        return s["sk"].reconstruct(s["dtype"], cores=s["cores"])
    if work == "verify":
        return s["sk"].error(s["X"], cores=s["cores"])
    sk = s["sk"]
    if work == "gradient":
        x = s["X"].detach().requires_grad_(True)
        xt = TTReconstructFn.apply(PSTT2Fn.apply(x, sk), sk, s["dtype"])
        loss = torch.sum((xt - s["T"]) ** 2)
        loss.backward()
        return {"xt": xt.detach(), "loss": loss.detach(), "grad": x.grad}
    if "slabs" in s:
        sk.begin()
        for slab, first, count in s["slabs"]:
            sk.accumulate(slab, first, count)
        sk.finalize()
    else:
        sk.pstt2(s["X"])
    if s["round_trip"]:
        return {"xt": sk.reconstruct(s["dtype"])}
    return {"cores": sk.cores.to(s["dtype"]), "ranks": sk.ranks}


def work(case):
    kind = _get(case, "work")
    if kind == "batch":
        by = fl = 0.0
        for dims, r in _batch_specs(case):
            n = math.prod(dims)
            by += 4 * n + 4 * sum(r[k] * dims[k] * r[k + 1] for k in range(len(dims)))
            fl += 2.0 * n * sum(v + case["p"] for v in r[1:-1] + [max(r)])
        return {"bytes": by, "flops": fl}
    dims = _dims(case)
    n, d = math.prod(dims), len(dims)
    xb = 8 if _get(case, "x") == "f64" else 4
    r = case["rmax"] if _get(case, "eps") else int(case["rank"])
    rs = _clamp(dims, [1] + [r] * (d - 1) + [1])
    cores = sum(rs[k] * dims[k] * rs[k + 1] for k in range(d))
    mid = rs[(d + 1) // 2]
    if kind == "expand":
        return {"bytes": xb * n + 8 * cores, "flops": 2.0 * n * mid}
    if kind == "verify":
        return {"bytes": xb * n + 8 * cores, "flops": 2.0 * n * mid}
    sketch = 2.0 * n * d * (r + case["p"])                     # d sketches of width r + p
    if kind == "tucker":
        m = case["n_outer"]
        out = sum(rs[k] * m * rs[k + 1] for k in range(d))
        return {"bytes": xb * n + 8 * out * 3, "flops": sketch + 2.0 * sum(rs[k] * m * rs[k + 1] * dims[k]
                                                                          for k in range(d))}
    if kind == "gradient":
        return {"bytes": 5 * xb * n, "flops": 2 * sketch + 3 * 2.0 * n * mid}   # X, T read; X~, dX~, dX written
    if _get(case, "round_trip"):
        return {"bytes": 2 * xb * n, "flops": sketch + 2.0 * n * mid}
    return {"bytes": xb * n + xb * cores, "flops": sketch}


def exact(case, seed):
    """X~ of a tensor of exact low rank is that tensor (its noise and the rounding
    of its storage aside); cores have no such value (they follow the test
    matrices), and neither has a gradient."""
    kind = _get(case, "work")
    if kind in ("expand", "verify"):
        dims = _dims(case)
        r = _clamp(dims, [1] + [int(case["rank"])] * (len(dims) - 1) + [1])
        xt = _dense(_tt_cores(dims, r, seed), torch.float64)
        if kind == "expand":
            return xt
        x = _add_noise(_dense(_tt_cores(dims, r, seed), _dtype(case)), case["noise"], seed)
        e = n2 = torch.zeros((), dtype=torch.float64, device="cuda")
        for a in range(0, xt.numel(), 1 << 26):
            y = x[a:a + (1 << 26)].double()
            e = e + torch.sum((y - xt[a:a + (1 << 26)]) ** 2)
            n2 = n2 + torch.sum(y * y)
        return torch.stack([e, n2])
    if kind == "compress" and _get(case, "round_trip"):
        return {"xt": _dense(_data_cores(case, seed), torch.float64)}
    if kind == "gradient":
        return {"xt": _dense(_data_cores(case, seed), torch.float64), "loss": None, "grad": None}
    return None
