"""Benchmark of the PSTT2-onepass hot path on GB300 (one JSON line on stdout).

Workload (the large streaming configuration): X is the Hilbert-type tensor
1/(x_{i1}+x_{i2}+x_{i3}+x_{i4}), x on a uniform grid of [1, 2], d = 4,
n = 256 (4.29e9 FP32 entries, 17.18 GB), eps = 1e-6, p = 10, rmax = 6.
One step = the whole hot path on one tensor: zero the sketches, sketch every
unfolding in one pass over X (the fused multi-sketch kernel), and form the
TT cores (FP64 TSQR/CPQR, rank rule, least-squares middle core, core
products).  `value` = entries/s with X resident in HBM; `e2e` = the same
through the C ABI with X in pinned HOST memory, copied to the device in 1 GiB
slabs inside the timed region, and the cores copied back.

Arms: default = this library (mixed BF16 tensor-core sketch; the FP64 GPU path
is timed beside it); --impl reference = the FP64 CPU oracle on a bounded
sample of the same workload (there is no other implementation of the method).
"""
import argparse
import json
import os
import statistics
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "PSTT2 tensor entries/s and HBM roofline fraction, mixed vs FP64 GPU at eps=1e-6"
WORKLOAD = dict(dims=[256, 256, 256, 256], eps=1e-6, p=10, rmax=6, seed=1)
SLAB = 16  # last-mode slices per 1 GiB slab (256^3 * 4 B * 16 = 1 GiB)
HEADLINE_DRM = "kr"  # the paper's test matrices for its streaming implementation (Sec. 4.2)
# FP16 hi + lo of X 2^s: 2^-22 relative, below the rank threshold eps / sqrt(d - 1)
# that the BF16 split (2^-17) cannot resolve, at BF16's cost
HEADLINE_PREC = "fp16"
FP64_PEAK_TFLOPS = 1.25  # nominal GB300 FP64 (no measured figure on this machine)


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=50)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="gb300", choices=["gb300", "reference"])
    ap.add_argument("--prec", default=HEADLINE_PREC, choices=["fp16", "bf16", "tf32"],
                    help="sketch precision of the headline (fp16: X 2^s split into FP16 hi + lo)")
    ap.add_argument("--drm", default=HEADLINE_DRM, choices=["gauss", "kr"],
                    help="test matrices of the headline: dense Gaussian or Khatri-Rao")
    ap.add_argument("--slab", type=int, default=SLAB, help="last-mode slices per accumulate (16 = 1 GiB at n=256)")
    ap.add_argument("--n", type=int, default=256, help="mode size (default: the 17 GB workload)")
    ap.add_argument("--nlast", type=int, default=0,
                    help="size of the last mode (default n); with --slab it keeps the slab shape of a launch "
                         "on a smaller tensor (profiling)")
    ap.add_argument("--mid", type=int, default=0,
                    help="size of the two middle modes (default n); a smaller value keeps the kernel's "
                         "tile shape on a smaller tensor (profiling)")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-fp64", action="store_true")
    ap.add_argument("--no-cpu", action="store_true")
    ap.add_argument("--no-batched", action="store_true")
    ap.add_argument("--no-forms", action="store_true", help="skip the precision and differentiation forms")
    ap.add_argument("--no-second", action="store_true", help="skip the paper's second workloads (Table 1 shapes)")
    ap.add_argument("--second-only", default="",
                    help="run only these second workloads (comma list of hilbert3,hilbert5,hilbert9,bumps3)")
    ap.add_argument("--no-onesided", action="store_true", help="skip the one-sided PSTT-onepass sub-line")
    ap.add_argument("--onesided-only", action="store_true", help="run only the one-sided PSTT-onepass sub-line")
    ap.add_argument("--no-tucker", action="store_true", help="skip the Tucker2TT sub-line")
    ap.add_argument("--tucker-only", action="store_true", help="run only the Tucker2TT sub-line")
    ap.add_argument("--batch", type=int, default=512, help="tensors in the batched workload")
    ap.add_argument("--batched-only", action="store_true",
                    help="run only the batched workload (profiling); prints its own JSON line")
    ap.add_argument("--batch-prec", default="bf16,fp64", help="precisions of the batched workload")
    ap.add_argument("--diff-only", action="store_true",
                    help="run only the differentiation form (profiling); prints its own JSON line")
    ap.add_argument("--precision-only", default="",
                    help="run only the precision form in these precisions, e.g. 'bf16' or 'fp64,tf32,bf16' "
                         "(profiling); prints its own JSON line")
    ap.add_argument("--batch-shape", default="",
                    help="fixed launch shape 'ta,chunk,ctas_per_sm' instead of the autotuner")
    return ap.parse_args()


# ------------------------------------------------------------------ clocks
class ClockSampler:
    """nvidia-smi sampling of SM clocks and throttle reasons during a region."""
    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index):
        self.index = index
        self.proc = None
        self.lines = []

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--id={self.index}", f"--query-gpu={self.Q}",
                                          "--format=csv,noheader,nounits", "-lms", "50"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
        except OSError:
            self.proc = None

    def _read(self):
        for ln in self.proc.stdout:
            self.lines.append(ln.strip())

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        self.t.join(timeout=2)
        sm, mx, reasons, power = [], [], set(), []
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            f = [v.strip() for v in ln.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                mx.append(float(f[2]))
                power.append(float(f[3]))
            except ValueError:
                continue
            for nm, v in zip(names, f[5:9]):
                if v.lower() == "active":
                    reasons.add(nm)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": sorted(reasons), "samples": len(sm),
                "power_w_max": max(power) if power else None}


# ------------------------------------------------------------------- peaks
def measured_peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        with open(p) as f:
            d = json.load(f)
        return d.get("hbm_gbs"), "measured"
    return 6800.0, "fallback"


def measured_tensor_peak(prec):
    """Dense tensor peak (TFLOP/s) for the sketch's MMA type: the measured BF16
    burst figure, or for TF32 that figure times the nominal TF32/BF16 ratio
    (1.1 / 2.25)."""
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    bf16, kind = 1900.0, "fallback"
    if os.path.exists(p):
        with open(p) as f:
            d = json.load(f)
        if d.get("bf16_tflops"):
            bf16, kind = d["bf16_tflops"], "measured"
    if prec in ("bf16", "fp16"):  # kind::f16: the same MMA rate for both operand types
        return bf16, f"{kind} bf16_tflops"
    return bf16 * 1.1 / 2.25, f"{kind} bf16_tflops x 1.1/2.25"


def traffic_record(kernel_tag):
    """DRAM bytes per launch from the committed ncu summary, when it was taken
    on the current source of that kernel (else None)."""
    p = os.path.join(ROOT, "profiles", "traffic.json")
    if not os.path.exists(p):
        return None
    with open(p) as f:
        rec = json.load(f)
    r = rec.get(kernel_tag)
    if not r:
        return None
    try:
        import hashlib
        src = open(os.path.join(ROOT, r["source"]), "rb").read()
        if "region" in r:  # the kernel's own code: from the first marker to the end of the second
            a = src.index(r["region"][0].encode())
            b = src.index(r["region"][1].encode(), a) + len(r["region"][1])
            src = src[a:b]
        if hashlib.sha256(src).hexdigest()[:16] != r["source_sha"]:
            return None
    except (OSError, ValueError):
        return None
    return r["dram_bytes_per_launch"]


# -------------------------------------------------------------- CPU oracle
def cpu_sample(steps=1, n=128, drm=HEADLINE_DRM):
    """The FP64 oracle as it stands, on a bounded sample of the workload: the
    same Hilbert-type function at d = 4 with a smaller n (n = 128: 268M
    entries), same eps, p, rmax, test matrices, one-pass.  Returns entries/s,
    the threads used, the sample description and the per-step times."""
    import numpy as np
    import ttinputs as ti
    from oracle import pstt2 as OP
    dims = [n] * 4
    x = ti.hilbert_type(dims, np.float32).astype(np.float64)
    times = []
    for _ in range(steps):
        t0 = time.perf_counter()
        OP.pstt2(x, dims, eps=WORKLOAD["eps"], rmax=WORKLOAD["rmax"], p=WORKLOAD["p"], seed=WORKLOAD["seed"],
                 passes=1, drm=drm)
        times.append(time.perf_counter() - t0)
    try:
        from threadpoolctl import threadpool_info
        cores = max([i.get("num_threads", 1) for i in threadpool_info()] + [1])
    except Exception:
        cores = os.cpu_count()
    return n ** 4 / statistics.median(times), cores, (
        f"oracle.pstt2 one-pass on the Hilbert-type tensor at d=4, n={n} ({n ** 4} entries), eps=1e-6, "
        f"p=10, rmax=6, {'Khatri-Rao' if drm == 'kr' else 'dense Gaussian'} test matrices; "
        f"entries/s = entries / wall time"), times


def cpu_sample_one_core(n=64, drm=HEADLINE_DRM):
    """The same oracle sample on one host core: a child process with every
    BLAS / OpenMP pool limited to one thread (n = 64, 16.8M entries)."""
    env = dict(os.environ, OMP_NUM_THREADS="1", OPENBLAS_NUM_THREADS="1", MKL_NUM_THREADS="1",
               BLIS_NUM_THREADS="1", NUMEXPR_NUM_THREADS="1")
    code = f"import json, bench; v, _, s, _ = bench.cpu_sample(1, {n}, {drm!r}); print(json.dumps([v, s]))"
    try:
        r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, env=env, capture_output=True, text=True,
                           timeout=300)
        v, sample = json.loads(r.stdout.strip().splitlines()[-1])
        return {"value": v, "unit": "entries/s", "cores": 1, "sample": sample}
    except Exception as ex:  # a baseline figure only; the line goes on without it
        return {"error": f"{type(ex).__name__}: {ex}"}


def reference_sample_n(steps, drm, budget_s=150.0):
    """Largest sample size n in {32, 48, 64, 96, 128} whose `steps` oracle
    runs fit the time budget (cost scales with n^4; measured at n = 32)."""
    t32 = cpu_sample(1, 32, drm)[3][0]
    best = 32
    for n in (48, 64, 96, 128):
        if t32 * (n / 32) ** 4 * steps <= budget_s:
            best = n
    return best


def run_reference(a):
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    steps = max(1, a.steps)
    n = reference_sample_n(steps + min(a.warmup, 1), a.drm)
    for _ in range(min(a.warmup, 1)):
        cpu_sample(1, n, a.drm)
    v, cores, sample, times = cpu_sample(steps, n, a.drm)
    line = {"impl": "reference", "metric": METRIC, "value": v, "unit": "entries/s", "n_gpus": a.gpus,
            "steps": steps, "warmup": a.warmup, "ms_per_step": 1e3 * statistics.median(times),
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic",
            "config": {"workload": f"Hilbert-type d=4 n=256 FP32 (bounded sample per step: n={n})",
                       "test_matrices": a.drm, "sample": sample},
            "cpu_baseline": {"value": v, "unit": "entries/s", "cores": cores, "kind": "oracle", "sample": sample},
            "e2e": {"value": v, "unit": "entries/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


# ---------------------------------------------------------------- GPU arm
def batched_inputs(count, dev, seed=5):
    """The batched workload on the device: `count` FP32 tensors, d in {3..6},
    n in {8..32} (n^d <= 2e6), random N(0,1) TT cores of ranks in {2..16}
    (data seed 1000 + b), plus 1e-7 relative Gaussian noise; eps = 1e-5,
    p = 5, rmax = 16, test-matrix seed 1000 + b."""
    import numpy as np
    import torch
    import ttinputs as ti
    xs, probs = [], []
    for b, (dims, r) in enumerate(ti.batch_specs(count=count, seed=seed, cap=2_000_000)):
        xs.append(device_tt(dims, r, 1000 + b, 1e-7, dev, noise_seed=seed + b))
        probs.append(dict(dims=dims, eps=1e-5, rmax=16, p=5, seed=1000 + b))
    return xs, probs


def run_batched(a, dev, P, stream):
    """Batched workload: one plan, one persistent sketch launch over all
    tensors + batched finalize, per precision; autotuned launch shape."""
    import numpy as np
    import torch
    import ttinputs as ti
    xs, probs = batched_inputs(a.batch, dev)
    torch.cuda.synchronize(dev)  # inputs come from torch's stream; the library runs on `stream`
    ntot = sum(x.numel() for x in xs)
    out = {"workload": f"{a.batch} FP32 tensors, d in 3..6, n in 8..32 (n^d <= 2e6), TT ranks 2..16 + 1e-7 noise; "
                       f"eps=1e-5 p=5 rmax=16; {ntot} entries ({ntot * 4 / 1e9:.2f} GB)", "entries": ntot}
    for prec in a.batch_prec.split(","):
        t = P.TTSketch(None, batch=probs, x_dtype=torch.float32, prec=prec)
        if a.batch_shape:
            best = tuple(int(v) for v in a.batch_shape.split(","))
            t.batch_config(*best)
        else:
            best = t.autotune(xs, stream)
        stream.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        k = max(3, min(a.steps, 10))
        t.batched(xs, stream)
        e0.record(stream)
        for _ in range(k):
            t.batched(xs, stream)
        e1.record(stream)
        stream.synchronize()
        eager_ms = e0.elapsed_time(e1) / k
        # the served form: the whole batched call captured once as a CUDA
        # graph and replayed (the workspace tables were uploaded above)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            t.batched(xs, stream)
        with torch.cuda.stream(stream):
            graph.replay()
            e0.record(stream)
            for _ in range(k):
                graph.replay()
            e1.record(stream)
        stream.synchronize()
        ms = e0.elapsed_time(e1) / k
        # accuracy on a sample of items (host contraction of the cores)
        errs = []
        for b in range(0, len(xs), max(1, len(xs) // 8)):
            xt = ti.contract_tt(t.core_list(b))
            xh = xs[b].double().cpu().numpy()
            errs.append(float(np.linalg.norm(xt - xh) / np.linalg.norm(xh)))
        out[prec] = {"value": ntot / (ms * 1e-3), "unit": "entries/s", "ms_per_step": ms,
                     "mode": "CUDA-graph replay of one tt_pstt2_batched call", "eager_ms_per_step": eager_ms,
                     "hbm_frac_of_measured": ntot * 4 / (ms * 1e-3) / 1e9 / measured_peaks()[0],
                     "launch_shape": {"ta": best[0], "chunk": best[1], "ctas_per_sm": best[2]},
                     "max_rel_err_sampled": max(errs), "items_sampled": len(errs)}
        del graph, t
    return out


def whole_job(ms_local, units_local, world, device=None):
    """Whole-job rate over `world` ranks: the step time is the MAX over ranks,
    the units are the SUM over ranks.  Returns (ms, units, units/s)."""
    if world > 1:
        import torch
        import torch.distributed as dist
        t = torch.tensor([ms_local], dtype=torch.float64, device=device)
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
        u = torch.tensor([float(units_local)], dtype=torch.float64, device=device)
        dist.all_reduce(u, op=dist.ReduceOp.SUM)
        ms_local, units_local = float(t.item()), float(u.item())
    return ms_local, units_local, units_local / (ms_local * 1e-3)


def device_tt(dims, ranks, seed, noise, dev, noise_seed=2):
    """Random-TT tensor (cores of ttinputs.random_tt_cores, contracted on the
    device in FP64) plus relative Gaussian noise from a seeded torch
    generator, as FP32 (column-major flat)."""
    import numpy as np
    import torch
    import ttinputs as ti
    L = torch.ones(1, 1, dtype=torch.float64, device=dev)
    for G in ti.random_tt_cores(dims, ranks, seed=seed):
        a_, n_, c_ = G.shape
        Gd = torch.from_numpy(np.asfortranarray(G).reshape(a_, n_ * c_, order="F")).to(dev)
        L = (L @ Gd).T.reshape(c_, n_, -1).permute(1, 2, 0).reshape(-1, c_)  # rows u + N i
    x = L[:, 0]
    if noise > 0:
        gen = torch.Generator(device=dev)
        gen.manual_seed(noise_seed)
        e = torch.randn(x.numel(), dtype=torch.float64, device=dev, generator=gen)
        x = x + e * (noise * x.norm() / e.norm())
    return x.to(torch.float32).contiguous()


def run_precision(a, dev, P, stream):
    """Precision form: d = 6, n = 24 random TT (internal ranks 10) + 1e-6
    relative noise, FP32; eps = 1e-5, p = 10, rmax = 16.  FP64 GPU path, TF32
    and BF16 sketches; errors against X and against the FP64 GPU result."""
    import torch
    dims = [24] * 6
    X = device_tt(dims, [1, 10, 10, 10, 10, 10, 1], 0, 1e-6, dev)
    torch.cuda.synchronize(dev)  # X comes from torch's stream; the library runs on `stream`
    out = {"workload": "random TT d=6 n=24 (1.91e8 FP32 entries), ranks 10, +1e-6 noise; eps=1e-5 p=10 rmax=16"}
    ref = None
    # "<prec>_kr": the same with Khatri-Rao test matrices (cheap per-plane rows
    # on the small planes of this tensor); its error is reported against X
    precs = a.precision_only.split(",") if a.precision_only else ["fp64", "tf32", "bf16", "fp16", "bf16_kr"]
    xs_log2 = P.x_scale_log2(X, stream)  # FP16 split scale of this tensor
    for form in precs:
        prec, _, drm = form.partition("_")
        t = P.TTSketch(dims, eps=1e-5, rmax=16, p=10, seed=1, x_dtype=torch.float32, prec=prec, drm=drm or "gauss",
                       x_scale_log2=xs_log2)
        t.pstt2(X, stream)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        t.pstt2(X, stream)
        e1.record(stream)
        err = t.error(X, stream)
        stream.synchronize()
        ms = e0.elapsed_time(e1)
        err = err.cpu().numpy()
        r = {"value": X.numel() / (ms * 1e-3), "unit": "entries/s", "ms_per_step": ms,
             "rel_err_vs_X": float((err[0] / err[1]) ** 0.5), "ranks": t.status(stream)[1],
             "kernel": t.kernel_name()}
        if form == "fp64":
            ref = t.reconstruct(torch.float32, stream=stream)
        elif ref is not None and not drm:
            d2 = t.error(ref, stream)
            stream.synchronize()
            d2 = d2.cpu().numpy()
            r["rel_err_vs_fp64_gpu"] = float((d2[0] / err[1]) ** 0.5)
        out[form] = r
        stream.synchronize()  # nothing of t may still run when its buffers go back to torch
        del t
    del X, ref
    return out


def run_diff(a, dev, P, stream):
    """Differentiation form: d = 5, n = 32 FP32 random TT (rank 8, seed 0),
    loss ||TT_pstt2(X) - T||^2 with a fixed N(0,1) target (seed 3), target
    ranks 8, p = 5; forward + hand-written backward through autograd."""
    import torch
    import ttinputs as ti
    dims = [32] * 5
    X = device_tt(dims, [1, 8, 8, 8, 8, 1], 0, 0.0, dev)
    T = torch.tensor(ti.target_tensor(X.numel(), seed=3), device=dev)
    torch.cuda.synchronize(dev)
    out = {"workload": "random TT d=5 n=32 (3.36e7 FP32 entries), rank 8; target ranks 8, p=5"}
    for prec in ("fp64", "bf16"):
        t = P.TTSketch(dims, ranks=[1, 8, 8, 8, 8, 1], p=5, seed=1, x_dtype=torch.float32, prec=prec, diff=True)

        def fwd_bwd():
            Xg = X.detach().requires_grad_(True)
            cores = P.PSTT2Fn.apply(Xg, t)
            Xt = P.TTReconstructFn.apply(cores, t, torch.float32)
            L = torch.sum((Xt.double() - T) ** 2)
            L.backward()
            return Xg.grad

        with torch.cuda.stream(stream):
            fwd_bwd()
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            g = fwd_bwd()
            e1.record(stream)
        stream.synchronize()
        # the sketch adjoint alone: dX written once (4 bytes per entry)
        dcores = torch.randn(t.cores.numel(), dtype=torch.float64, device=dev)
        dX = torch.empty_like(X)
        t.backward(dcores, dX, stream)
        b0, b1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        b0.record(stream)
        t.backward(dcores, dX, stream)
        b1.record(stream)
        stream.synchronize()
        bms = b0.elapsed_time(b1)
        out[prec] = {"fwd_bwd_ms": e0.elapsed_time(e1), "backward_ms": bms,
                     "backward_dX_write_GBs": X.numel() * 4 / (bms * 1e-3) / 1e9,
                     "grad_norm": float(g.double().norm())}
        stream.synchronize()
        del t
    return out


SECOND = {
    # the paper's Hilbert tensor at the three Table 1 shapes with its ranks, and
    # the Gaussian-bumps tensor of Sec. 4.4 (100 bumps, gamma = 10) at d = 3
    "hilbert3": dict(kind="hilbert", dims=[960] * 3, ranks=[1, 25, 25, 1]),
    "hilbert5": dict(kind="hilbert", dims=[96] * 5, ranks=[1, 17, 18, 18, 17, 1]),
    "hilbert9": dict(kind="hilbert", dims=[12] * 9, ranks=[1, 12, 18, 18, 19, 19, 18, 18, 12, 1]),
    "bumps3": dict(kind="bumps", dims=[960] * 3, eps=1e-5, rmax=54),
}


def median_ms(call, stream, reps=3):
    """Device time of `call` on `stream`: `reps` runs enqueued back to back
    (the host stays ahead of the GPU), each bracketed by CUDA events; the
    median and every run in ms."""
    import torch
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(reps)]
    for e0, e1 in ev:
        e0.record(stream)
        call()
        e1.record(stream)
    stream.synchronize()
    runs = [e0.elapsed_time(e1) for e0, e1 in ev]
    return sorted(runs)[reps // 2], runs


def run_second(a, dev, P, stream):
    """The paper's second workloads (Sec. 4.3-4.4) at full size, FP32 X
    generated on the device (not timed), BF16 sketches, p = 10: one untimed
    pstt2 and the median of three timed ones each, error against X."""
    import ctypes as C
    import torch
    import ttinputs as ti
    from paper_2111_10448_gb300 import _native as N
    L = P.lib()
    out = {}
    names = a.second_only.split(",") if a.second_only else list(SECOND)
    for name in names:
        w = SECOND[name]
        dims = w["dims"]
        d = len(dims)
        ntot = 1
        for v in dims:
            ntot *= v
        r = {"dims": dims, "entries": ntot}
        try:
            X = torch.empty(ntot, dtype=torch.float32, device=dev)
            nn = (C.c_int64 * d)(*dims)
            sp = C.c_void_p(stream.cuda_stream)
            if w["kind"] == "hilbert":
                N.check(L.tt_generate_hilbert(d, nn, 0, dims[-1], C.c_void_p(X.data_ptr()), N.TT_F32, sp), "gen")
                kw = dict(ranks=w["ranks"])
            else:
                import numpy as np
                c = np.ascontiguousarray(ti.bump_centres(d, 100, seed=4))
                N.check(L.tt_generate_gaussian_bumps(d, nn, 100, 10.0, c.ctypes.data_as(C.c_void_p), 0, dims[-1],
                                                     C.c_void_p(X.data_ptr()), N.TT_F32, sp), "gen")
                kw = dict(eps=w["eps"], rmax=w["rmax"])
            stream.synchronize()
            t = P.TTSketch(dims, p=10, seed=1, x_dtype=torch.float32, prec="bf16", device=dev, **kw)
            t.pstt2(X, stream)
            ms, runs = median_ms(lambda: t.pstt2(X, stream), stream)
            err = t.error(X, stream)
            stream.synchronize()
            err = err.cpu().numpy()
            st, ranks = t.status(stream)
            r.update({"value": ntot / (ms * 1e-3), "unit": "entries/s", "ms_per_step": ms, "ms_runs": runs,
                      "hbm_frac_of_measured": ntot * 4 / (ms * 1e-3) / 1e9 / measured_peaks()[0],
                      "rel_err_vs_X": float((err[0] / err[1]) ** 0.5), "ranks": ranks, "status": st,
                      "kernel": t.kernel_name(),
                      "mode": {k: v for k, v in kw.items()}})
            stream.synchronize()
            del t
        except Exception as ex:  # reported in the line, the rest of the bench goes on
            r["error"] = f"{type(ex).__name__}: {ex}"
        X = None
        torch.cuda.empty_cache()
        out[name] = r
    return out


def run_onesided(a, dev, P, stream):
    """One-sided PSTT-onepass (every unfolding sketched from the right, last
    core by least squares) and two-pass PSTT (last core Q^T X_{d-1} from a
    second pass) against the two-sided PSTT2-onepass on the same X:
    the precision-form tensor (random TT d=6 n=24, eps 1e-5, rmax 16, p 10)
    and the streaming Hilbert-type tensor (d=4 n=256, eps 1e-6, rmax 6, p 10);
    BF16 sketches, one untimed pstt2 and the median of three timed ones
    each, errors against X."""
    import ctypes as C
    import torch
    from paper_2111_10448_gb300 import _native as N
    out = {}
    cases = [("randomtt_d6_n24", [24] * 6, dict(eps=1e-5, rmax=16, p=10)),
             ("hilbert_type_d4_n256", [256] * 4, dict(eps=1e-6, rmax=6, p=10))]
    for name, dims, kw in cases:
        ntot = 1
        for v in dims:
            ntot *= v
        r = {"dims": dims, "entries": ntot, **{k: v for k, v in kw.items()}}
        try:
            if name.startswith("randomtt"):
                X = device_tt(dims, [1, 10, 10, 10, 10, 10, 1], 0, 1e-6, dev)
                torch.cuda.synchronize(dev)
            else:
                X = torch.empty(ntot, dtype=torch.float32, device=dev)
                nn = (C.c_int64 * 4)(*dims)
                N.check(P.lib().tt_generate_hilbert_type(4, nn, 0, dims[-1], C.c_void_p(X.data_ptr()), N.TT_F32,
                                                         C.c_void_p(stream.cuda_stream)), "gen")
                stream.synchronize()
            for label, one, passes in (("one_sided", True, 1), ("one_sided_twopass", True, 2), ("two_sided", False, 1)):
                t = P.TTSketch(dims, seed=1, x_dtype=torch.float32, prec="bf16", device=dev, one_sided=one,
                               passes=passes, **kw)
                t.pstt2(X, stream)
                ms, runs = median_ms(lambda: t.pstt2(X, stream), stream)
                err = t.error(X, stream)
                stream.synchronize()
                err = err.cpu().numpy()
                r[label] = {"value": ntot / (ms * 1e-3), "unit": "entries/s", "ms_per_step": ms, "ms_runs": runs,
                            "rel_err_vs_X": float((err[0] / err[1]) ** 0.5), "ranks": t.status(stream)[1],
                            "sketch_MB": sum(S.numel() for _, _, S in t.sketches(0)) * 8 / 1e6,
                            "kernel": t.kernel_name()}
                stream.synchronize()
                del t
        except Exception as ex:  # reported in the line, the rest of the bench goes on
            r["error"] = f"{type(ex).__name__}: {ex}"
        X = None
        torch.cuda.empty_cache()
        out[name] = r
    return out


def run_tucker(a, dev, P, stream):
    """Tucker2TT (Algorithm 3) of X = G x_1 A_1 ... x_4 A_4 with a 64^4 FP64
    Tucker core G (random TT, ranks 8, + 1e-6 noise) and orthonormal 256 x 64
    factors: X (256^4) is never formed.  FP64, eps 1e-6, rmax 12, p 10; one
    untimed and one timed call; the error ||G - G~|| / ||G|| equals ||X - X~|| /
    ||X|| since the factors are isometries.  Then TT2Tucker (Algorithm 4) of
    the resulting train with multilinear ranks 54, timed the same way."""
    import torch
    s, n = [64] * 4, 256
    G = device_tt(s, [1, 8, 8, 8, 1], 0, 1e-6, dev).double()
    gen = torch.Generator(device=dev)
    gen.manual_seed(7)
    A = [torch.linalg.qr(torch.randn(n, s[k], dtype=torch.float64, device=dev, generator=gen))[0] for k in range(4)]
    torch.cuda.synchronize(dev)
    kw = dict(eps=1e-6, rmax=12, p=10, seed=1)
    out = {"workload": "Tucker core 64^4 FP64 (random TT ranks 8 + 1e-6 noise), factors 256 x 64 orthonormal: "
                       "X = 256^4 never formed; eps=1e-6 rmax=12 p=10, FP64"}
    try:
        P.tucker2tt(G, A, prec="fp64", stream=stream, **kw)
        stream.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        cores, t = P.tucker2tt(G, A, prec="fp64", stream=stream, **kw)
        e1.record(stream)
        err = t.error(G, stream)
        stream.synchronize()
        err = err.cpu().numpy()
        # and back (Algorithm 4): the TT cores to a Tucker format with multilinear ranks 54 (width 54 + 10)
        P.tt2tucker(cores, [54] * 4, p=10, seed=3, stream=stream)
        stream.synchronize()
        f0, f1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        f0.record(stream)
        Hs, As = P.tt2tucker(cores, [54] * 4, p=10, seed=3, stream=stream)
        f1.record(stream)
        stream.synchronize()
        out.update({"tt2tucker_ms": f0.elapsed_time(f1), "tt2tucker_tucker_ranks": [int(A.shape[1]) for A in As]})
        out.update({"ms": e0.elapsed_time(e1), "rel_err_vs_X": float((err[0] / err[1]) ** 0.5),
                    "ranks": t.status(stream)[1], "x_entries_not_formed": n ** 4, "core_entries": G.numel(),
                    "kernel": t.kernel_name()})
        stream.synchronize()
        del t, cores
    except Exception as ex:  # reported in the line, the rest of the bench goes on
        out["error"] = f"{type(ex).__name__}: {ex}"
    return out


def run_tucker_only(a):
    import torch
    import paper_2111_10448_gb300 as P
    dev = torch.device("cuda", int(os.environ.get("LOCAL_RANK", "0")))
    torch.cuda.set_device(dev)
    stream = torch.cuda.Stream(device=dev)
    print(json.dumps({"tucker2tt": run_tucker(a, dev, P, stream)}), flush=True)


def run_onesided_only(a):
    import torch
    import paper_2111_10448_gb300 as P
    dev = torch.device("cuda", int(os.environ.get("LOCAL_RANK", "0")))
    torch.cuda.set_device(dev)
    stream = torch.cuda.Stream(device=dev)
    print(json.dumps({"one_sided": run_onesided(a, dev, P, stream)}), flush=True)


def run_second_only(a):
    import torch
    import paper_2111_10448_gb300 as P
    dev = torch.device("cuda", int(os.environ.get("LOCAL_RANK", "0")))
    torch.cuda.set_device(dev)
    stream = torch.cuda.Stream(device=dev)
    print(json.dumps({"second_workloads": run_second(a, dev, P, stream)}), flush=True)


def run_precision_only(a):
    import torch
    import paper_2111_10448_gb300 as P
    dev = torch.device("cuda", int(os.environ.get("LOCAL_RANK", "0")))
    torch.cuda.set_device(dev)
    stream = torch.cuda.Stream(device=dev)
    print(json.dumps({"precision_form": run_precision(a, dev, P, stream)}), flush=True)


def run_diff_only(a):
    import torch
    import paper_2111_10448_gb300 as P
    dev = torch.device("cuda", int(os.environ.get("LOCAL_RANK", "0")))
    torch.cuda.set_device(dev)
    stream = torch.cuda.Stream(device=dev)
    print(json.dumps({"diff_form": run_diff(a, dev, P, stream)}), flush=True)


def run_batched_only(a):
    import torch
    import paper_2111_10448_gb300 as P
    dev = torch.device("cuda", int(os.environ.get("LOCAL_RANK", "0")))
    torch.cuda.set_device(dev)
    stream = torch.cuda.Stream(device=dev)
    out = run_batched(a, dev, P, stream)
    print(json.dumps({"batched": out}), flush=True)


def run_gpu(a):
    import torch
    import paper_2111_10448_gb300 as P
    from paper_2111_10448_gb300 import _native as N
    import ctypes as C

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=dev)
    L = P.lib()
    n = a.n
    m = a.mid or n
    nl = a.nlast or n
    dims = [n, m, m, nl]
    ntot = n * m * m * nl
    Nd1 = n * m * m
    stream = torch.cuda.Stream(device=dev)
    sp = C.c_void_p(stream.cuda_stream)

    # X resident in HBM (generated on the device, not timed)
    X = torch.empty(ntot, dtype=torch.float32, device=dev)
    nn = (C.c_int64 * 4)(*dims)
    N.check(L.tt_generate_hilbert_type(4, nn, 0, nl, C.c_void_p(X.data_ptr()), N.TT_F32, sp), "gen")
    stream.synchronize()

    # FP16 split of X 2^s: s from the largest |X| (one reduction over the
    # resident tensor, before any timing); 16 for this tensor, |X| <= 1/4
    xs_log2 = P.x_scale_log2(X, stream) if a.prec == "fp16" else 0
    kw = dict(eps=WORKLOAD["eps"], rmax=WORKLOAD["rmax"], p=WORKLOAD["p"], seed=WORKLOAD["seed"] + rank,
              x_dtype=torch.float32, device=dev, x_scale_log2=xs_log2)
    slab = a.slab if nl % a.slab == 0 else nl

    def stream_step(t, sl, evs=None):
        """begin + one accumulate per slab of `sl` last-mode slices + finalize;
        evs: a (start, end) event pair per slab around its accumulate."""
        t.begin(stream)
        for k, s0 in enumerate(range(0, nl, sl)):
            if evs is not None:
                evs[k][0].record(stream)
            t.accumulate(X[s0 * Nd1:(s0 + sl) * Nd1], s0, sl, stream)
            if evs is not None:
                evs[k][1].record(stream)
        t.finalize(stream)

    STATUS = {0: "TT_OK", 5: "TT_ERR_RANK_DEFICIENT", 6: "TT_ERR_TIMEOUT", 7: "TT_WARN_RANK_CAP",
              9: "TT_ERR_NONFINITE"}

    def measure_form(t, sl, steps, warmup):
        """Whole-step and per-slab sketch times of one form (CUDA events on
        the launching stream), its status, ranks and error against X."""
        for _ in range(warmup):
            stream_step(t, sl)
        stream.synchronize()
        nsl = nl // sl
        evs = [[(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(nsl)]
               for _ in range(steps)]
        f0, f1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        f0.record(stream)
        for i in range(steps):
            stream_step(t, sl, evs[i])
        f1.record(stream)
        torch.cuda.synchronize(dev)
        per_slab = [s_.elapsed_time(e_) for ev in evs for s_, e_ in ev]
        st_, rk_ = t.status(stream)
        e2 = t.error(X, stream)
        stream.synchronize()
        e2 = e2.cpu().numpy()
        sk_ms = sum(per_slab) / steps
        return {"step_ms": f0.elapsed_time(f1) / steps, "sketch_ms": sk_ms,
                "sketch_ms_per_launch": statistics.mean(per_slab), "launches_per_step": nsl,
                "hbm_frac_of_measured": ntot * 4 / (sk_ms * 1e-3) / 1e9 / measured_peaks()[0],
                "status": STATUS.get(st_, st_), "ranks": rk_, "rel_err_vs_X": float((e2[0] / e2[1]) ** 0.5)}

    # the headline: the test matrices of --drm, 1 GiB slabs (16 slices) streamed
    t = P.TTSketch(dims, prec=a.prec, drm=a.drm, **kw)
    for _ in range(a.warmup):
        stream_step(t, slab)
    stream.synchronize()
    if world > 1:
        torch.distributed.barrier()
    nsl = nl // slab
    evs = [[(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(nsl)]
           for _ in range(a.steps)]
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    clk = ClockSampler(torch.cuda.get_device_properties(dev).index if hasattr(torch.cuda.get_device_properties(dev), "index") else local)
    clk.start()
    time.sleep(0.3)
    l0 = L.tt_kernel_launches()
    torch.cuda.synchronize(dev)
    if world > 1:
        torch.distributed.barrier()
    e0.record(stream)
    for i in range(a.steps):
        stream_step(t, slab, evs[i])
    e1.record(stream)
    torch.cuda.synchronize(dev)
    if world > 1:
        torch.distributed.barrier()
    l1 = L.tt_kernel_launches()
    clocks = clk.stop()
    ms, _, value = whole_job(e0.elapsed_time(e1) / a.steps, ntot, world, dev)
    per_slab = [s_.elapsed_time(e_) for ev in evs for s_, e_ in ev]
    sketch_ms = sum(per_slab) / a.steps
    launch_ms = statistics.mean(per_slab)
    st, ranks = t.status(stream)

    # accuracy of this run: ||X - X~|| / ||X|| on the device
    err2 = t.error(X, stream)
    stream.synchronize()
    err2 = err2.cpu().numpy()
    rel_err = float((err2[0] / err2[1]) ** 0.5)

    out = {}
    # ---- the other forms of the same workload: dense Gaussian / Khatri-Rao
    # test matrices, 1 GiB slabs / the whole last mode in one accumulate
    if not a.no_forms:
        forms = {}
        for drm_, sl_ in (("gauss", nl), ("gauss", slab), ("kr", slab), ("kr", nl)):
            if drm_ == a.drm and sl_ == slab:
                continue
            tf = P.TTSketch(dims, prec=a.prec, drm=drm_, **kw)
            forms[f"{drm_}_{sl_}_slices_per_accumulate"] = measure_form(tf, sl_, max(3, min(a.steps, 10)), 2)
            del tf
        # the headline with TT_FLAG_SHORT_CHAINS: FP32 tensor-memory chains of
        # 32 MMAs instead of 256 in the column sketches (accuracy for time)
        tf = P.TTSketch(dims, prec=a.prec, drm=a.drm, short_chains=True, **kw)
        forms[f"{a.drm}_{slab}_slices_short_chains"] = measure_form(tf, slab, max(3, min(a.steps, 10)), 2)
        del tf
        # the headline's other 16-bit split: BF16 (2^-17, below the rank threshold's resolution)
        other = "bf16" if a.prec == "fp16" else "fp16"
        tf = P.TTSketch(dims, prec=other, drm=a.drm, **kw)
        forms[f"{a.drm}_{slab}_slices_{other}"] = measure_form(tf, slab, max(3, min(a.steps, 10)), 2)
        del tf
        out["forms"] = forms

    # ---- FP64 GPU path, same eps, same slabs (one step after one warm-up)
    if not a.no_fp64:
        f = P.TTSketch(dims, prec="fp64", drm=a.drm, **kw)
        stream_step(f, slab)
        stream.synchronize()
        g0, g1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        g0.record(stream)
        stream_step(f, slab)
        g1.record(stream)
        torch.cuda.synchronize(dev)
        f_ms = g0.elapsed_time(g1)
        fe = f.error(X, stream)
        # mixed vs FP64: ||X~_mixed - X~_fp64|| / ||X||
        Xf = f.reconstruct(torch.float32, stream=stream)
        d2 = t.error(Xf, stream)
        stream.synchronize()
        fe, d2 = fe.cpu().numpy(), d2.cpu().numpy()
        del Xf
        shapes64 = [tuple(S.shape) for _, _, S in f.sketches(0)]
        fl64 = 2 * sum(w for _, w in shapes64)  # FP64 FMA flops per entry, every sketch
        out["fp64_gpu"] = {"value": ntot / (f_ms * 1e-3), "unit": "entries/s", "ms_per_step": f_ms,
                           "rel_err_vs_X": float((fe[0] / fe[1]) ** 0.5),
                           "mixed_vs_fp64_rel": float((d2[0] / err2[1]) ** 0.5),
                           "ranks": f.status(stream)[1],
                           "roofline": {"bound": "fp64 alu", "flops_per_entry": fl64,
                                        "achieved_tflops": ntot * fl64 / (f_ms * 1e-3) / 1e12,
                                        "peak_tflops": FP64_PEAK_TFLOPS, "peak_kind": "nominal GB300 FP64",
                                        "frac": ntot * fl64 / (f_ms * 1e-3) / 1e12 / FP64_PEAK_TFLOPS}}
        del f

    # ---- e2e: X from pinned host memory, one 1 GiB slab at a time, cores back
    if not a.no_e2e:
        Xh = torch.empty(ntot, dtype=torch.float32, pin_memory=True)
        Xh.copy_(X)
        Xd = torch.empty_like(X)
        cores_h = torch.empty(t.cores.numel(), dtype=torch.float64, pin_memory=True)
        ranks_h = torch.empty(t.ranks.numel(), dtype=torch.int32, pin_memory=True)
        copy = torch.cuda.Stream(device=dev)
        SL = SLAB if nl % SLAB == 0 else nl

        def e2e_step():
            # each slab is copied on a second stream and sketched as soon as
            # its copy has landed
            t.begin(stream)
            for s0 in range(0, nl, SL):
                with torch.cuda.stream(copy):
                    Xd[s0 * Nd1:(s0 + SL) * Nd1].copy_(Xh[s0 * Nd1:(s0 + SL) * Nd1], non_blocking=True)
                    ev = torch.cuda.Event()
                    ev.record(copy)
                stream.wait_event(ev)
                t.accumulate(Xd[s0 * Nd1:(s0 + SL) * Nd1], s0, SL, stream)
            t.finalize(stream)
            with torch.cuda.stream(stream):
                cores_h.copy_(t.cores, non_blocking=True)
                ranks_h.copy_(t.ranks, non_blocking=True)

        def e2e_direct_step():
            # the sketch kernel reads each pinned host slab itself (over the
            # host link), no staging copy
            t.begin(stream)
            for s0 in range(0, nl, SL):
                t.accumulate(Xh[s0 * Nd1:(s0 + SL) * Nd1], s0, SL, stream)
            t.finalize(stream)
            with torch.cuda.stream(stream):
                cores_h.copy_(t.cores, non_blocking=True)
                ranks_h.copy_(t.ranks, non_blocking=True)

        def timed(fn):
            fn()
            torch.cuda.synchronize(dev)
            h0 = time.perf_counter()
            k = max(1, min(a.steps, 3))
            for _ in range(k):
                fn()
            torch.cuda.synchronize(dev)
            return (time.perf_counter() - h0) * 1e3 / k

        e_copy = timed(e2e_step)
        e_direct = timed(e2e_direct_step)
        e_ms = min(e_copy, e_direct)
        out["e2e"] = {"value": world * ntot / (e_ms * 1e-3), "unit": "entries/s", "ms_per_step": e_ms,
                      "h2d_bytes_per_step": ntot * 4,
                      "d2h_bytes_per_step": t.cores.numel() * 8 + t.ranks.numel() * 4,
                      "mode": "kernel reads each pinned host slab directly" if e_direct <= e_copy
                      else "1 GiB pinned-host slabs copied on a second stream, each sketched when it lands",
                      "ms_copy_slabs": e_copy, "ms_direct_host_reads": e_direct}
        del Xh, Xd

    peak, peak_kind = measured_peaks()
    # the dominant kernel: one launch sketches one slab (4 bytes per entry read once)
    achieved = ntot // nsl * 4 / (launch_ms * 1e-3) / 1e9
    # the two other ceilings of the sketch, beside HBM: tensor pipe (every entry
    # feeds l MACs per sketch, twice for the hi + lo split of X) and test-matrix
    # generation (each test-matrix row once: sum over sketches of l * rows)
    shapes = [tuple(S.shape) for _, _, S in t.sketches(0)]
    flops_pe = 2 * 2 * sum(w for _, w in shapes)
    normals = sum((ntot // rows) * w for rows, w in shapes)
    tpeak, tkind = measured_tensor_peak(a.prec)
    tflops = ntot * flops_pe / (sketch_ms * 1e-3) / 1e12
    kname = {"slab": "sketch_slab_kernel", "plane": "sketch_tc_kernel", "strip": "sketch_strip_kernel",
             "small-plane": "sketch_sp_kernel", "tile": "sketch_mma_kernel", "fp64": "sketch_f64_kernel"}[
                 t.kernel_name(slab)]
    roofline = {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s", "frac": achieved / peak,
                "traffic": traffic_record(f"{kname}_{a.prec}_{a.drm}_{n}x{m}x{m}x{slab}"),
                "peak_kind": f"{peak_kind} hbm_gbs", "kernel": kname,
                "kernel_ms": launch_ms, "algorithmic_bytes": ntot // nsl * 4,
                "tensor": {"flops_per_entry": flops_pe, "achieved_tflops": tflops, "peak_tflops": tpeak,
                           "peak_kind": tkind, "frac": tflops / tpeak},
                "rng": {"normals_per_entry": normals / ntot, "normals_per_step": normals}}

    if not a.no_batched:
        out["batched"] = run_batched(a, dev, P, stream)
    if not a.no_forms:
        out["precision_form"] = run_precision(a, dev, P, stream)
        out["diff_form"] = run_diff(a, dev, P, stream)
    if not a.no_second:
        out["second_workloads"] = run_second(a, dev, P, stream)
    if not a.no_onesided:
        out["one_sided"] = run_onesided(a, dev, P, stream)
    if not a.no_tucker:
        out["tucker2tt"] = run_tucker(a, dev, P, stream)

    cpu = None
    if rank == 0 and not a.no_cpu:
        v, cores, sample, _ = cpu_sample(1, 128, a.drm)
        cpu = {"value": v, "unit": "entries/s", "cores": cores, "kind": "oracle", "sample": sample,
               "one_core": cpu_sample_one_core(64, a.drm)}

    if rank == 0:
        line = {"metric": METRIC, "value": value, "unit": "entries/s", "n_gpus": world, "steps": a.steps,
                "warmup": a.warmup, "ms_per_step": ms, "higher_is_better": True, "scaling": "weak",
                "vs_baseline": None, "dtype": a.prec, "data": "synthetic",
                "config": {"workload": f"Hilbert-type d=4 dims={dims} FP32 ({ntot * 4 / 1e9:.2f} GB) one-pass PSTT2, "
                                       f"streamed in {nl // slab} slabs of {slab} last-mode slices "
                                       f"({slab * Nd1 * 4 / 2 ** 30:.2f} GiB each), eps=1e-6 p=10 rmax=6, "
                                       f"{'Khatri-Rao' if a.drm == 'kr' else 'dense Gaussian'} test matrices, "
                                       f"{a.prec} tensor-core sketch with X split hi+lo"
                                       f"{f' (X 2^{xs_log2})' if a.prec == 'fp16' else ''}, FP64 solves",
                           "test_matrices": a.drm, "slab_slices": slab, "x_scale_log2": xs_log2,
                           "l2": "inputs larger than L2 (no flush needed)",
                           "ranks": ranks, "status": STATUS.get(st, st), "rel_err_vs_X": rel_err,
                           "meets_eps": rel_err <= WORKLOAD["eps"],
                           "status_note": None if st == 0 else (
                               "the rank rule stopped at rmax: the BF16 hi+lo sketch (about 2^-17 relative) "
                               "cannot resolve the threshold eps/sqrt(d-1); the result is within 10 eps"
                               if a.prec == "bf16" else "see status"),
                           "parallelism": "replicas" if world > 1 else "single GPU"},
                "roofline": roofline, "cpu_baseline": cpu, "e2e": out.get("e2e"),
                "gpu_launches": int(l1 - l0), "clocks": clocks, "fp64_gpu": out.get("fp64_gpu"),
                "batched": out.get("batched"), "forms": out.get("forms"),
                "precision_form": out.get("precision_form"), "diff_form": out.get("diff_form"),
                "second_workloads": out.get("second_workloads"), "one_sided": out.get("one_sided"),
                "tucker2tt": out.get("tucker2tt")}
        print(json.dumps(line), flush=True)
    if world > 1:
        torch.distributed.destroy_process_group()


def main():
    a = parse()
    if a.impl == "reference":
        run_reference(a)
    elif a.batched_only:
        run_batched_only(a)
    elif a.diff_only:
        run_diff_only(a)
    elif a.precision_only:
        run_precision_only(a)
    elif a.second_only:
        run_second_only(a)
    elif a.onesided_only:
        run_onesided_only(a)
    elif a.tucker_only:
        run_tucker_only(a)
    else:
        run_gpu(a)


if __name__ == "__main__":
    main()
