#!/usr/bin/env python
"""Benchmark of the SLSE-FRS hot path on one GB300: time to reach a relative error of
1e-8 in beta-hat (mixed-precision path) and the HBM throughput of its dominant kernel,
with the plain FP64 GPU path measured beside it.

Workload: N = 2^22 rows, d = 512 columns, X stored FP32 (8.6 GB, larger than L2),
rows i.i.d. N(0, Sigma) with Sigma_ij = 0.5^|i-j|, beta ~ N(0, I), noise sd 0.1;
the paper's schedule rule (r = 6d, m_1 = 8d doubling to N/2, a_i = 2, T = 100).
Each timed step is one slse_fit call with a fresh sketch seed.  The accuracy
reference is the CPU oracle's OLS estimate (FP64 normal equations; cond(X) ~ 3).

Usage: python bench.py [--gpus N] [--steps K] [--warmup W] [--impl reference]
Prints one JSON line (rank 0).  Multi-GPU runs are independent replicas.
"""
import argparse
import dataclasses
import hashlib
import json
import math
import os
import statistics
import subprocess
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "time-to-1e-8 rel-err β̂ (ms) & HBM GB/s, mixed vs FP64 GPU, N=2^22 d=512"
TARGET = 1e-8
def workload_name(log2n: int, d: int) -> str:
    return f"AR(1) rho=0.5 Gaussian rows, N=2^{log2n}, d={d}, X fp32, sigma=0.1, beta~N(0,I)"
FALLBACK_HBM = 6800.0
FALLBACK_BF16_TFLOPS = 1900.0


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=30)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--log2n", type=int, default=22)
    ap.add_argument("--d", type=int, default=512)
    ap.add_argument("--fp64-steps", type=int, default=2)
    ap.add_argument("--cs-steps", type=int, default=2, help="CountSketch-variant fits reported beside the SRHT line")
    ap.add_argument("--fp8-steps", type=int, default=2, help="fits with the FP8 form of the sketch")
    ap.add_argument("--full-steps", type=int, default=2, help="fits with the full form of the 2nd stage")
    ap.add_argument("--cfg2-steps", type=int, default=2, help="FP64 fits at N=2^20, d=256, cond 1e4")
    ap.add_argument("--cfg4-steps", type=int, default=1, help="fits per form at N=2^24, d=256, heavy tails")
    ap.add_argument("--one-fit", default=None, metavar="PREC:KIND",
                    help="run one untimed fit of the workload at --log2n (e.g. mixed_bf16:srht) and exit; "
                         "the command the committed kernel profiles were captured with")
    ap.add_argument("--tuning-steps", type=int, default=2, help="fits with the SLSE-FRS-tuning schedule")
    ap.add_argument("--gauss-steps", type=int, default=2, help="fits with the Gaussian Hessian sketch")
    ap.add_argument("--diff-steps", type=int, default=2, help="forward+backward passes of the differentiation block")
    ap.add_argument("--e2e-steps", type=int, default=3, help="end-to-end fits from pinned host inputs (median reported)")
    ap.add_argument("--sample-log2n", type=int, default=15, help="rows (log2) of each reference-arm step")
    ap.add_argument("--cpu-rungs", default="16,17,18,19", help="log2 row counts of the oracle ladder")
    ap.add_argument("--cpu-full", action="store_true", help="also time the oracle on the full workload (needs ~40 GB)")
    ap.add_argument("--no-cpu", action="store_true", help="skip the CPU baseline timing (accuracy reference still runs)")
    return ap.parse_args()


def dist_init(backend: str = "nccl"):
    """Replica setup from the torchrun environment (RANK, LOCAL_RANK, WORLD_SIZE, MASTER_*).
    The replicas exchange only timing scalars; the library itself runs on one GPU per rank."""
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    if ws <= 1:
        return 0, 1, 0
    import torch.distributed as dist
    dist.init_process_group(backend=backend)
    return dist.get_rank(), ws, int(os.environ.get("LOCAL_RANK", "0"))


def _scalar_device():
    import torch.distributed as dist
    return "cuda" if dist.get_backend() == "nccl" else "cpu"


def barrier(ws):
    if ws > 1:
        import torch.distributed as dist
        dist.barrier()


def reduce_max(v, ws):
    if ws <= 1:
        return v
    import torch
    import torch.distributed as dist
    t = torch.tensor([float(v)], dtype=torch.float64, device=_scalar_device())
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def reduce_sum(v, ws):
    if ws <= 1:
        return v
    import torch
    import torch.distributed as dist
    t = torch.tensor([float(v)], dtype=torch.float64, device=_scalar_device())
    dist.all_reduce(t, op=dist.ReduceOp.SUM)
    return float(t.item())


def replica_summary(ms_local: float, units_local: float, ws: int) -> dict:
    """Whole-job numbers from per-rank results: the slowest rank's time (after the barrier
    that brackets the timed region) and the units all ranks processed."""
    barrier(ws)
    return {"ms": reduce_max(ms_local, ws), "units": reduce_sum(units_local, ws), "ranks": ws}


# ----------------------------------------------------------------------------- clocks
class ClockSampler:
    FIELDS = "index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active," \
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown," \
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap"

    def __init__(self, gpu_index):
        self.gpu = gpu_index
        self.proc = None
        self.lines = []

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--id={self.gpu}", f"--query-gpu={self.FIELDS}",
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.thread = threading.Thread(target=self._read, daemon=True)
            self.thread.start()
        except OSError:
            self.proc = None

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        self.thread.join(timeout=5)
        sm, smax, reasons, power = [], [], set(), []
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            parts = [x.strip() for x in ln.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                smax.append(float(parts[2]))
                power.append(float(parts[3]))
            except ValueError:
                continue
            for name, val in zip(names, parts[5:9]):
                if val.lower() in ("active", "1"):
                    reasons.add(name)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(smax) if smax else None,
                "power_w_max": max(power) if power else None, "samples": len(sm), "reasons": sorted(reasons)}


# ----------------------------------------------------------------------------- helpers
def measured_hbm_peak():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(path) as f:
            v = json.load(f).get("hbm_gbs")
        if v:
            return float(v), "measured"
    except (OSError, ValueError):
        pass
    return FALLBACK_HBM, "fallback"


def measured_bf16_peak():
    """Dense BF16 tensor peak (TFLOP/s) for a kernel timed on its own: the burst figure."""
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            v = json.load(f).get("bf16_tflops")
        if v:
            return float(v), "measured"
    except (OSError, ValueError):
        pass
    return FALLBACK_BF16_TFLOPS, "fallback"


def profile_traffic(kernel_key, source_files):
    """DRAM bytes per launch from the committed ncu summary, if the kernel source is unchanged."""
    path = os.path.join(ROOT, "profiles", "traffic.json")
    try:
        with open(path) as f:
            prof = json.load(f)
    except (OSError, ValueError):
        return None
    ent = prof.get(kernel_key)
    if not ent:
        return None
    h = hashlib.sha256()
    for sf in source_files:
        with open(os.path.join(ROOT, sf), "rb") as f:
            h.update(f.read())
    if ent.get("source_sha256") != h.hexdigest():
        return None
    return ent.get("dram_bytes_per_launch")


def make_data(log2n, d):
    import workloads
    return workloads.cfg3(N=1 << log2n, d=d, seed=1003)


def e4m3_values():
    """The 256 values of the OCP E4M3 format (1 sign, 4 exponent bits with bias 7, 3 mantissa
    bits; exponent field 0 is subnormal; S.1111.111 is NaN), indexed by the code byte."""
    v = np.empty(256)
    for c in range(256):
        sgn = -1.0 if c & 0x80 else 1.0
        e, f = (c >> 3) & 0xF, c & 0x7
        if e == 0xF and f == 0x7:
            v[c] = np.nan
        elif e == 0:
            v[c] = sgn * f * 2.0 ** -9
        else:
            v[c] = sgn * (1.0 + f / 8.0) * 2.0 ** (e - 7)
    return v


def link_rates(nbytes, ms_pass1, ms_copy):
    """GB/s at which pass 1 read X from host memory, of a plain copy of the same X, and the share."""
    read, copy = (nbytes / statistics.median(ms) / 1e6 for ms in (ms_pass1, ms_copy))
    return {"pass1_host_read_gbs": read, "link_copy_gbs": copy, "pass1_frac_of_link": read / copy}


def first_crossing(hist, ms, bh, target):
    nb = np.linalg.norm(bh)
    errs = np.linalg.norm(hist - bh[None, :], axis=1) / nb
    idx = np.nonzero(errs <= target)[0]
    if idx.size == 0:
        return None, float(errs[-1]) if errs.size else float("nan")
    return float(ms[idx[0]]), float(errs[idx[0]])


# ----------------------------------------------------------------------------- oracle legs
def oracle_fit_seconds(X, Y, n, d, seed=0):
    """Wall time of the oracle's Algorithm 2 (FP64, numpy) on the first n rows, with the
    schedule rule of the workload at that size."""
    from oracle import slse as osl
    Xs, Ys = X[:n].astype(np.float64), Y[:n].astype(np.float64)
    sched = osl.default_schedule(n, d, T=100, tol=1e-9)
    t0 = time.time()
    osl.slse_fit(Xs, Ys, sched, seed=seed)
    return time.time() - t0


def cost_model_fit(ns, ts):
    """Least-squares fit of t(N) = c + a N log2 N + b N (Thm 4.4: the transform costs
    N d log2 N, the passes O(N d) at fixed d; c is the size-independent QR of the r x d
    Hessian sketch).  Returns a callable model."""
    A = np.array([[1.0, n * math.log2(n), float(n)] for n in ns])
    coef, *_ = np.linalg.lstsq(A, np.asarray(ts, np.float64), rcond=None)
    return lambda n: float(coef[0] + coef[1] * n * math.log2(n) + coef[2] * n)


def cpu_ladder(X, Y, log2n, d, rungs):
    """The oracle timed on the first 2^k rows for each k in rungs (all host cores); the cost
    model fitted on every rung but the largest predicts the largest (the check), and the fit
    on all rungs gives the estimate at the full size."""
    ts = [oracle_fit_seconds(X, Y, 1 << k, d) for k in rungs]
    ns = [1 << k for k in rungs]
    held = cost_model_fit(ns[:-1], ts[:-1])(ns[-1])
    model = cost_model_fit(ns, ts)
    return {"rungs": [{"rows": n, "seconds": t} for n, t in zip(ns, ts)],
            "check": {"rows": ns[-1], "predicted_seconds": held, "measured_seconds": ts[-1],
                      "rel_error": abs(held - ts[-1]) / ts[-1]},
            "estimate_seconds": model(1 << log2n), "model": model}


def cpu_leg(X, Y, log2n, d, rungs, full, time_it):
    """The only place the benchmark runs the oracle: the accuracy reference (OLS of the
    full workload) and, optionally, the oracle's own SLSE-FRS timed on the host cores: a
    ladder of row counts fitted to the cost model (and, with ``full``, the full workload)."""
    from oracle import linalg
    t0 = time.time()
    bh = linalg.ols_normal(X, Y)
    t_ref = time.time() - t0
    base = None
    if time_it:
        lad = cpu_ladder(X, Y, log2n, d, rungs)
        est = lad.pop("model")(1 << log2n)
        base = {"value": est * 1000.0, "unit": "ms", "cores": os.cpu_count(), "kind": "oracle",
                "sample": (f"oracle slse_fit (FP64, numpy, BLAS on all cores) on the first 2^k rows of the workload "
                           f"(d={d}, same schedule rule) for k in {list(rungs)}; value = the fit "
                           f"t(N) = c + a N log2 N + b N of those times at N = 2^{log2n}; check: the fit "
                           f"without the largest rung predicts it within rel_error"),
                "ladder": lad}
        if full:
            tf = oracle_fit_seconds(X, Y, 1 << log2n, d)
            base["value"] = tf * 1000.0
            base["sample"] = f"oracle slse_fit on the full workload (2^{log2n} rows, d={d}), measured"
            base["ladder_estimate_ms"] = est * 1000.0
        # one thread: the same oracle in a fresh interpreter at the two smallest rungs; the
        # estimate scales the all-core value by the measured one-thread / all-core ratio
        k1 = rungs[1] if len(rungs) > 1 else rungs[0]
        dt1 = oracle_one_thread(X[:1 << k1].astype(np.float64), Y[:1 << k1].astype(np.float64))
        if dt1 is not None:
            tm = lad["rungs"][1 if len(rungs) > 1 else 0]["seconds"]
            base["value_1_thread"] = base["value"] * dt1 / tm
            base["one_thread"] = {"rows": 1 << k1, "seconds": dt1, "all_cores_seconds": tm}
    return bh, t_ref, base


def oracle_one_thread(Xs, Ys):
    """Wall time of the same oracle fit in a fresh interpreter with every BLAS/OpenMP pool
    limited to one thread (the limit must be set before numpy loads); None if it fails."""
    import tempfile
    with tempfile.TemporaryDirectory() as td:
        fx, fy = os.path.join(td, "x.npy"), os.path.join(td, "y.npy")
        np.save(fx, Xs)
        np.save(fy, Ys)
        code = ("import sys, time, numpy as np; sys.path.insert(0, %r); from oracle import slse as osl; "
                "X = np.load(%r); Y = np.load(%r); "
                "s = osl.default_schedule(X.shape[0], X.shape[1], T=100, tol=1e-9); "
                "t0 = time.time(); osl.slse_fit(X, Y, s, seed=0); print(time.time() - t0)") % (ROOT, fx, fy)
        env = dict(os.environ, OMP_NUM_THREADS="1", OPENBLAS_NUM_THREADS="1", MKL_NUM_THREADS="1",
                   NUMEXPR_NUM_THREADS="1")
        try:
            r = subprocess.run([sys.executable, "-c", code], env=env, capture_output=True, text=True, timeout=600)
            return float(r.stdout.strip().splitlines()[-1]) if r.returncode == 0 else None
        except (subprocess.TimeoutExpired, ValueError, IndexError):
            return None


def cpu_leg_cfg2(p):
    """Oracle leg of the cfg2 block: the least-squares reference by Householder QR (cond(X) = 1e4)."""
    from oracle import linalg
    t0 = time.time()
    bh = linalg.ols(p["X"], p["Y"])
    return bh, time.time() - t0


def cpu_leg_cfg4(p, m, seed, rows, cols):
    """Oracle leg of the cfg4 block: the OLS reference (FP64 normal equations) and single sketch
    entries from the definition with the oracle's own draws."""
    from oracle import linalg, sketch as osk
    t0 = time.time()
    bh = linalg.ols_normal(p["X"], p["Y"])
    D, P, sigma = osk.draws(osk.padded_size(p["X"].shape[0]), seed)
    ref = osk.sketch_entries(p["X"], p["Y"], D, P, sigma, m, rows, cols)
    return bh, ref, time.time() - t0


def sketch_form_errors(slse, torch, seed=4):
    """Reference leg (oracle): error of one SRHT sketch in each stored form -- FP64, BF16 and
    FP8 (E4M3 with 32-column block scales) -- against the oracle's FP64 sketch, on a
    2^16 x 64 sample of the workload (m = 4096): max and mean of |error| / column rms."""
    import workloads
    from oracle import fp8 as ofp8, sketch as osk
    n, d, m = 1 << 16, 64, 4096
    p = workloads.cfg3(N=n, d=d, seed=1003)
    X, Y = p["X"], p["Y"]
    ref = osk.sketch(X.astype(np.float64), Y.astype(np.float64), m, seed)[0]
    rms = np.sqrt((ref ** 2).mean(0))
    Xd, Yd = torch.from_numpy(X).cuda(), torch.from_numpy(Y).cuda()
    out = {}
    for form in ("fp64", "mixed_bf16", "mixed_fp8"):
        if form == "fp64":
            g = slse.sketch(Xd.double(), Yd.double(), m, seed=seed, prec="fp64")[0].cpu().numpy()
        elif form == "mixed_bf16":
            g = slse.sketch(Xd, Yd, m, seed=seed, prec=form)[0].float().cpu().numpy().astype(np.float64)
        else:
            codes, k, _ = slse.sketch(Xd, Yd, m, seed=seed, prec=form)
            q = ofp8.decode_e4m3(codes.cpu().numpy().astype(np.int64))
            g = q * np.repeat(np.ldexp(1.0, k.cpu().numpy().astype(np.int64) - 127), 32, axis=1)[:, :d]
        e = np.abs(g - ref) / rms
        out[form] = {"max": float(e.max()), "mean": float(e.mean())}
    return {"sample": f"cfg3 rows, N=2^16, d={d}, m={m}, error / column rms vs the oracle's FP64 sketch",
            "by_form": out}


def run_reference(args, rank, ws):
    """The reference arm: the oracle as it stands on the host cores (rank 0 only).  Each
    step times the oracle fit on the first 2^sample rows of the workload; the step's
    full-size figure scales that time by the cost model's ratio t(2^log2n) / t(2^sample),
    the model fitted on a ladder of row counts timed once before the steps."""
    if rank != 0:
        return
    import workloads
    d = args.d
    ns = 1 << args.sample_log2n
    rungs = [args.sample_log2n + k for k in range(4)]
    p = workloads.cfg3(N=1 << rungs[-1], d=d, seed=1003)
    X, Y = p["X"], p["Y"]
    lad = cpu_ladder(X, Y, args.log2n, d, rungs)
    model = lad.pop("model")
    ratio = model(1 << args.log2n) / model(ns)
    for w in range(args.warmup):
        oracle_fit_seconds(X, Y, ns, d, seed=100 + w)
    times = [oracle_fit_seconds(X, Y, ns, d, seed=k) for k in range(args.steps)]
    val = statistics.mean(times) * 1000.0 * ratio
    sample = (f"oracle slse_fit (FP64, numpy) per step on the first 2^{args.sample_log2n} rows of the workload "
              f"(d={d}, same schedule rule), times the ratio {ratio:.1f} of the cost model t(N) = c + a N log2 N "
              f"+ b N fitted on rungs 2^{rungs[0]}..2^{rungs[-1]} at N = 2^{args.log2n} and 2^{args.sample_log2n}")
    out = {"metric": METRIC, "value": val, "unit": "ms", "n_gpus": args.gpus, "steps": args.steps,
           "warmup": args.warmup, "ms_per_step": statistics.mean(times) * 1000.0, "higher_is_better": False,
           "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic", "impl": "reference",
           "config": {"workload": workload_name(args.log2n, d), "N": 1 << args.log2n, "d": d, "sample_rows": ns},
           "cpu_baseline": {"value": val, "unit": "ms", "cores": os.cpu_count(), "kind": "oracle", "sample": sample,
                            "ladder": lad},
           "e2e": {"value": val, "unit": "ms", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(out), flush=True)


# ----------------------------------------------------------------------------- our arm
def run_ours(args, rank, ws, local_rank):
    import torch
    torch.cuda.set_device(local_rank)
    import paper_2509_06856_gb300 as slse

    N, d = 1 << args.log2n, args.d
    t0 = time.time()
    data = make_data(args.log2n, d)
    X, Y = data["X"], data["Y"]
    t_gen = time.time() - t0

    Xh = torch.empty((N, d), dtype=torch.float32, pin_memory=True)
    Yh = torch.empty(N, dtype=torch.float32, pin_memory=True)
    Xh.numpy()[:] = X
    Yh.numpy()[:] = Y
    Xd = Xh.cuda()
    Yd = Yh.cuda()

    # accuracy reference (and CPU baseline at N = 1) from the oracle, rank 0
    bh, t_ref, cpu_base = (None, None, None)
    if rank == 0:
        rungs = [int(k) for k in args.cpu_rungs.split(",")]
        bh, t_ref, cpu_base = cpu_leg(X, Y, args.log2n, d, rungs, args.cpu_full, time_it=(ws == 1 and not args.no_cpu))

    sched = slse.default_schedule(N, d, prec="mixed_bf16", T=100, tol=5e-9)
    wsz = slse.workspace_size(Xd, Yd, slse.OP_FIT, sched)
    wbuf = slse.alloc_workspace(wsz)
    cap = sched.T

    for w in range(max(3, args.warmup)):
        slse.fit(Xd, Yd, sched, seed=1000 + w, workspace=wbuf, trace_cap=cap)
    barrier(ws)
    torch.cuda.synchronize()
    clocks = ClockSampler(local_rank)
    clocks.start()
    time.sleep(0.3)
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    results = []
    e0.record()
    for k in range(args.steps):
        results.append(slse.fit(Xd, Yd, sched, seed=k, workspace=wbuf, trace_cap=cap))
    e1.record()
    torch.cuda.synchronize()
    barrier(ws)
    clk = clocks.stop()
    ms_total = e0.elapsed_time(e1)

    # time-to-accuracy from the per-iteration CUDA events of each fit
    tta, errs_final, crossed = [], [], True
    for r in results:
        hist = r.beta_hist.cpu().numpy() if rank == 0 else None
        if rank == 0:
            t, e = first_crossing(hist, np.array(r.ms_hist), bh, TARGET)
            if t is None:
                crossed = False
                t = r.report["ms_total"]
            tta.append(t)
            errs_final.append(float(np.linalg.norm(r.beta - bh) / np.linalg.norm(bh)))
    value_local = statistics.mean(tta) if rank == 0 else 0.0
    value = reduce_max(value_local, ws)
    ms_per_step = reduce_max(ms_total / args.steps, ws)
    launches = int(reduce_sum(sum(r.report["kernels"] for r in results), ws))

    # dominant kernel: the largest of the main path's kernels by summed CUDA-event time (the 2nd-stage
    # passes over X, the two sketch passes); the Gram build of the correction form runs on a second
    # stream beside the main path (its time overlaps other kernels) and is listed, not chosen
    rep = results[-1].report
    k_times = {
        "grad_stage2": (rep["ms_grad2"], rep["n_grad2"], rep["bytes_grad2"]),
        "gram": (rep["ms_gram"], 1 if rep["ms_gram"] > 0 else 0, rep["bytes_gram"]),
        "srht_pass1": (rep["ms_srht_pass1"], 1, N * (d + 1) * 4.0 + N * (d + 1) * 2.0),
        "srht_pass2": (rep["ms_srht_pass2"], 1, N * (d + 1) * 2.0 + (sched.m[-1] + sched.r) * (d + 1) * 2.0),
    }
    peak, peak_kind = measured_hbm_peak()
    kernels_gbs = {}
    for k, (ms, n, by) in k_times.items():
        if ms > 0 and n > 0:
            kernels_gbs[k] = {"ms_per_launch": ms / n, "launches": n, "alg_bytes_per_launch": by,
                              "gbs": by / (ms / n) / 1e6, "frac_of_" + peak_kind: by / (ms / n) / 1e6 / peak}
    dom = max((k for k in k_times if k != "gram"), key=lambda k: k_times[k][0])
    ms_d, n_d, by_d = k_times[dom]
    achieved = by_d / (ms_d / n_d) / 1e6
    src = {"grad_stage2": ["paper_2509_06856_gb300/csrc/grad.cu"],
           "srht_pass1": ["paper_2509_06856_gb300/csrc/srht_tc.cu"],
           "srht_pass2": ["paper_2509_06856_gb300/csrc/srht_tc.cu"]}[dom]
    roofline = {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s", "frac": achieved / peak,
                "traffic": profile_traffic(dom, src), "kernel": dom, "peak_source": peak_kind,
                "frac_of_nominal_8000": achieved / 8000.0}

    # FP64 GPU path on the same workload (X widened exactly to FP64 in the kernels)
    fp64 = None
    if args.fp64_steps > 0:
        s64 = slse.default_schedule(N, d, prec="fp64", T=100, tol=1e-11)
        w64 = slse.alloc_workspace(slse.workspace_size(Xd, Yd, slse.OP_FIT, s64))
        slse.fit(Xd, Yd, s64, seed=999, workspace=w64, trace_cap=cap)
        t8, t10, tot, fin = [], [], [], []
        for k in range(args.fp64_steps):
            r = slse.fit(Xd, Yd, s64, seed=k, workspace=w64, trace_cap=cap)
            if rank == 0:
                h = r.beta_hist.cpu().numpy()
                a8, _ = first_crossing(h, np.array(r.ms_hist), bh, 1e-8)
                a10, _ = first_crossing(h, np.array(r.ms_hist), bh, 1e-10)
                t8.append(a8)
                t10.append(a10)
                tot.append(r.report["ms_total"])
                fin.append(float(np.linalg.norm(r.beta - bh) / np.linalg.norm(bh)))
        del w64
        if rank == 0:
            r64 = r.report
            fp64 = {"time_to_1e-8_ms": statistics.mean(t8) if all(v is not None for v in t8) else None,
                    "time_to_1e-10_ms": statistics.mean(t10) if all(v is not None for v in t10) else None,
                    "ms_per_fit": statistics.mean(tot), "final_rel_err": max(fin),
                    "phases_ms": {k: r64[k] for k in ("ms_draws", "ms_sketch", "ms_qr", "ms_stage1", "ms_stage2")},
                    "grad_stage2_ms_per_pass": r64["ms_grad2"] / max(1, r64["n_grad2"]),
                    "iters": [r64["iters_stage1"], r64["iters_stage2"]]}
        torch.cuda.empty_cache()

    # the same fit with every 2nd-stage pass streaming X in FP32 (the full form), for comparison with
    # the default correction form (passes over a BF16 copy between exact FP32 passes)
    s2full = None
    if args.full_steps > 0:
        sf = slse.default_schedule(N, d, prec="mixed_bf16", T=100, tol=5e-9, stage2="full")
        tf, fin = [], []
        for k in range(args.full_steps + 1):
            r = slse.fit(Xd, Yd, sf, seed=k, workspace=wbuf, trace_cap=cap)
            if rank == 0 and k > 0:
                a8, _ = first_crossing(r.beta_hist.cpu().numpy(), np.array(r.ms_hist), bh, TARGET)
                tf.append(a8)
                fin.append(float(np.linalg.norm(r.beta - bh) / np.linalg.norm(bh)))
        if rank == 0:
            rf = r.report
            s2full = {"time_to_1e-8_ms": statistics.mean(tf) if all(v is not None for v in tf) else None,
                      "final_rel_err": max(fin), "ms_stage2": rf["ms_stage2"],
                      "passes_over_x": rf["n_grad2"], "iters": [rf["iters_stage1"], rf["iters_stage2"]],
                      "grad_ms_per_pass": rf["ms_grad2"] / max(1, rf["n_grad2"])}

    # FP8 form of the sketch on the same workload (1st-stage sketches in E4M3 + block scales)
    f8 = None
    if args.fp8_steps > 0:
        s8 = slse.default_schedule(N, d, prec="mixed_fp8", T=100, tol=5e-9)
        w8 = slse.alloc_workspace(slse.workspace_size(Xd, Yd, slse.OP_FIT, s8))
        slse.fit(Xd, Yd, s8, seed=997, workspace=w8, trace_cap=cap)
        t8s, fin = [], []
        for k in range(args.fp8_steps):
            r = slse.fit(Xd, Yd, s8, seed=k, workspace=w8, trace_cap=cap)
            if rank == 0:
                a8, _ = first_crossing(r.beta_hist.cpu().numpy(), np.array(r.ms_hist), bh, TARGET)
                t8s.append(a8)
                fin.append(float(np.linalg.norm(r.beta - bh) / np.linalg.norm(bh)))
        del w8
        if rank == 0:
            r8 = r.report
            f8 = {"time_to_1e-8_ms": statistics.mean(t8s) if all(v is not None for v in t8s) else None,
                  "final_rel_err": max(fin),
                  "phases_ms": {k: r8[k] for k in ("ms_sketch", "ms_qr", "ms_stage1", "ms_stage2", "ms_total")},
                  "iters": [r8["iters_stage1"], r8["iters_stage2"]],
                  "sketch_error_by_form": sketch_form_errors(slse, torch)}
        torch.cuda.empty_cache()

    # the SLSE-FRS-tuning schedule (Sec. 5) on the same workload
    tun = None
    if args.tuning_steps > 0:
        stn = slse.tuning_schedule(N, d, prec="mixed_bf16", T=100, tol=5e-9)
        wtn = slse.alloc_workspace(slse.workspace_size(Xd, Yd, slse.OP_FIT, stn))
        slse.fit(Xd, Yd, stn, seed=996, workspace=wtn, trace_cap=cap)
        ttn = []
        for k in range(args.tuning_steps):
            r = slse.fit(Xd, Yd, stn, seed=k, workspace=wtn, trace_cap=cap)
            if rank == 0:
                a8, _ = first_crossing(r.beta_hist.cpu().numpy(), np.array(r.ms_hist), bh, TARGET)
                ttn.append(a8)
        del wtn
        if rank == 0:
            rt = r.report
            tun = {"schedule": f"m={stn.m}, a_i=3", "time_to_1e-8_ms": statistics.mean(ttn) if all(v is not None for v in ttn) else None,
                   "phases_ms": {k: rt[k] for k in ("ms_sketch", "ms_qr", "ms_stage1", "ms_stage2", "ms_total")},
                   "iters": [rt["iters_stage1"], rt["iters_stage2"]]}
        torch.cuda.empty_cache()

    # CountSketch variant (SLSE-FRS-CS, Sec. 5) on the same workload and schedule sizes
    cs = None
    if args.cs_steps > 0:
        scs = slse.default_schedule(N, d, prec="mixed_bf16", T=100, tol=5e-9, kind="countsketch")
        wcs = slse.alloc_workspace(slse.workspace_size(Xd, Yd, slse.OP_FIT, scs))
        slse.fit(Xd, Yd, scs, seed=998, workspace=wcs, trace_cap=cap)
        tcs, fin = [], []
        for k in range(args.cs_steps):
            r = slse.fit(Xd, Yd, scs, seed=k, workspace=wcs, trace_cap=cap)
            if rank == 0:
                a8, _ = first_crossing(r.beta_hist.cpu().numpy(), np.array(r.ms_hist), bh, TARGET)
                tcs.append(a8)
                fin.append(float(np.linalg.norm(r.beta - bh) / np.linalg.norm(bh)))
        del wcs
        if rank == 0:
            rc = r.report
            # the sketch reads X twice (nested sizes and S-hat) and writes every sketch once
            by = 2.0 * N * (d + 1) * 4.0 + (sum(scs.m) + scs.r) * (d + 1) * 2.0
            cs = {"time_to_1e-8_ms": statistics.mean(tcs) if all(v is not None for v in tcs) else None,
                  "final_rel_err": max(fin),
                  "phases_ms": {k: rc[k] for k in ("ms_sketch", "ms_qr", "ms_stage1", "ms_stage2", "ms_total")},
                  "iters": [rc["iters_stage1"], rc["iters_stage2"]],
                  "sketch_alg_bytes": by, "sketch_gbs": by / rc["ms_sketch"] / 1e6,
                  "sketch_frac_of_" + peak_kind: by / rc["ms_sketch"] / 1e6 / peak}
        torch.cuda.empty_cache()

    # Gaussian Hessian sketch (Sec. 2) on the same workload: SRHT subproblems, S-hat X = G X / sqrt(r)
    # formed on the tensor cores; the sketch call alone is timed against the dense BF16 peak
    gau = None
    if args.gauss_steps > 0:
        sg = slse.default_schedule(N, d, prec="mixed_bf16", T=100, tol=5e-9, kind="gaussian")
        wg = slse.alloc_workspace(slse.workspace_size(Xd, Yd, slse.OP_FIT, sg))
        slse.fit(Xd, Yd, sg, seed=995, workspace=wg, trace_cap=cap)
        tg, fin = [], []
        for k in range(args.gauss_steps):
            r = slse.fit(Xd, Yd, sg, seed=k, workspace=wg, trace_cap=cap)
            if rank == 0:
                a8, _ = first_crossing(r.beta_hist.cpu().numpy(), np.array(r.ms_hist), bh, TARGET)
                tg.append(a8)
                fin.append(float(np.linalg.norm(r.beta - bh) / np.linalg.norm(bh)))
        del wg
        torch.cuda.empty_cache()
        wsk = slse.alloc_workspace(slse.workspace_size(Xd, Yd, slse.OP_SKETCH, sg, sg.r))
        for w in range(3):
            slse.sketch(Xd, Yd, sg.r, seed=w, prec="mixed_bf16", kind="gaussian", workspace=wsk, want_y=False)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        ng = 5
        torch.cuda.synchronize()
        e0.record()
        for k in range(ng):
            slse.sketch(Xd, Yd, sg.r, seed=k, prec="mixed_bf16", kind="gaussian", workspace=wsk, want_y=False)
        e1.record()
        torch.cuda.synchronize()
        ms_sk = e0.elapsed_time(e1) / ng
        del wsk
        torch.cuda.empty_cache()
        if rank == 0:
            rg = r.report
            tpk, tkind = measured_bf16_peak()
            flops = 2.0 * sg.r * N * d
            gau = {"time_to_1e-8_ms": statistics.mean(tg) if all(v is not None for v in tg) else None,
                   "final_rel_err": max(fin),
                   "phases_ms": {k: rg[k] for k in ("ms_sketch", "ms_srht_pass1", "ms_srht_pass2", "ms_qr",
                                                    "ms_stage1", "ms_stage2", "ms_total")},
                   "iters": [rg["iters_stage1"], rg["iters_stage2"]],
                   "sketch_call_ms": ms_sk,
                   "sketch_call": f"G X / sqrt(r), r={sg.r}: pack X to BF16, tensor-core product, split sum",
                   "tensor_tflops": flops / ms_sk / 1e9, "tensor_peak_tflops": tpk,
                   "frac_of_" + tkind: flops / ms_sk / 1e9 / tpk}
        torch.cuda.empty_cache()

    # differentiation through the estimate at the N = 2^21, d = 128 FP32 workload (forward
    # fit, backward normal-equation solve and the one-pass input gradients)
    diff = None
    if args.diff_steps > 0:
        import workloads
        n5, d5 = 1 << 21, 128
        p5 = workloads.cfg5(N=n5, d=d5, seed=1005)
        X5, Y5 = torch.from_numpy(p5["X"]).cuda(), torch.from_numpy(p5["Y"]).cuda()
        s5 = slse.default_schedule(n5, d5, prec="mixed_bf16", T=100, tol=1e-10)
        sa = dataclasses.replace(s5, tol=1e-9)
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(5)]
        fw, sv, svd, vj, its = [], [], [], [], []
        # the backward's buffers are allocated once, as a training loop would hold them
        ws5 = slse.alloc_workspace(slse.solve_normal_workspace(X5, sa))
        dX5 = torch.empty_like(X5)
        dY5 = torch.empty_like(Y5)
        for k in range(args.diff_steps + 1):
            ev[0].record()
            r5 = slse.fit(X5, Y5, s5, seed=k, hinv=True)
            ev[1].record()
            v5 = torch.from_numpy(r5.beta - p5["beta_true"]).cuda()
            b5 = torch.from_numpy(r5.beta).cuda()
            w5, rep5 = slse.solve_normal(X5, r5.hinv, v5, sa, workspace=ws5)
            ev[2].record()
            slse.ols_vjp(X5, Y5, b5, w5, out=(dX5, dY5))
            ev[3].record()
            torch.cuda.synchronize()
            if k > 0:
                fw.append(ev[0].elapsed_time(ev[1]))
                sv.append(ev[1].elapsed_time(ev[2]))
                svd.append(rep5["ms_total"])
                vj.append(ev[2].elapsed_time(ev[3]))
                its.append(rep5["iters_stage2"])
        vjp_bytes = 2.0 * n5 * d5 * 4 + 2.0 * n5 * 4
        diff = {"workload": f"N=2^21, d={d5}, X fp32, L = 1/2 ||beta-hat - beta*||^2",
                "forward_fit_ms": statistics.mean(fw), "backward_solve_ms": statistics.mean(sv),
                "backward_solve_device_ms": statistics.mean(svd),
                "backward_solve_iters": statistics.mean(its), "vjp_ms": statistics.mean(vj),
                "vjp_gbs": vjp_bytes / statistics.mean(vj) / 1e6,
                "vjp_frac_of_" + peak_kind: vjp_bytes / statistics.mean(vj) / 1e6 / peak}
        del X5, Y5, dX5, dY5
        torch.cuda.empty_cache()

    # plain FP64 on the GPU at N = 2^20, d = 256, cond(X) = 1e4, sketch sizes 2d .. 64d (a_i = 2,
    # r = 6d): time to 1e-10 and the final error against the oracle's QR least-squares solution
    c2 = None
    if args.cfg2_steps > 0:
        import workloads
        t0 = time.time()
        p2 = workloads.cfg2()
        gen2 = time.time() - t0
        bh2, tref2 = cpu_leg_cfg2(p2) if rank == 0 else (None, None)
        n2, d2 = p2["X"].shape
        X2, Y2 = torch.from_numpy(p2["X"]).cuda(), torch.from_numpy(p2["Y"]).cuda()
        m2 = [2 * d2 * 2 ** t for t in range(6)]
        r2 = 6 * d2
        s2 = slse.Schedule(m=m2, a=[2] * len(m2), r=r2, mu=(1 - d2 / r2) ** 2, eta=d2 / r2, T=100, tol=1e-13)
        w2 = slse.alloc_workspace(slse.workspace_size(X2, Y2, slse.OP_FIT, s2))
        t10, t8, fin, tot = [], [], [], []
        for k in range(args.cfg2_steps + 1):
            r = slse.fit(X2, Y2, s2, seed=k, workspace=w2, trace_cap=s2.T)
            if rank == 0 and k > 0:
                h, ms = r.beta_hist.cpu().numpy(), np.array(r.ms_hist)
                t10.append(first_crossing(h, ms, bh2, 1e-10)[0])
                t8.append(first_crossing(h, ms, bh2, 1e-8)[0])
                fin.append(float(np.linalg.norm(r.beta - bh2) / np.linalg.norm(bh2)))
                tot.append(r.report["ms_total"])
        if rank == 0:
            rr = r.report
            c2 = {"workload": f"N=2^20, d={d2}, X fp64 = G diag(s) V^T, cond 1e4, sigma=1e-2",
                  "schedule": f"m={m2[0]}..{m2[-1]} (x2), a_i=2, r={r2}, T=100, tol=1e-13",
                  "time_to_1e-10_ms": statistics.mean(t10) if all(v is not None for v in t10) else None,
                  "time_to_1e-8_ms": statistics.mean(t8) if all(v is not None for v in t8) else None,
                  "ms_per_fit": statistics.mean(tot), "final_rel_err": max(fin),
                  "reference": "oracle OLS by Householder QR", "reference_seconds": tref2,
                  "data_gen_seconds": gen2,
                  "phases_ms": {k: rr[k] for k in ("ms_draws", "ms_sketch", "ms_qr", "ms_stage1", "ms_stage2")},
                  "iters": [rr["iters_stage1"], rr["iters_stage2"]],
                  "grad_ms_per_pass": rr["ms_grad2"] / max(1, rr["n_grad2"]),
                  "grad_fp64_tflops": 4.0 * n2 * d2 / (rr["ms_grad2"] / max(1, rr["n_grad2"])) / 1e9}
        del X2, Y2, w2, p2
        torch.cuda.empty_cache()

    # heavy tails at N = 2^24, d = 256 (X FP32, Student-t(3), 0.1% of rows x100): per stored form of
    # the sketch (FP64, BF16, FP8) the fit's time to its target and final error against the FP64
    # oracle, and sampled entries of one m = 4096 sketch against the definition
    c4 = None
    if args.cfg4_steps > 0:
        import workloads
        t0 = time.time()
        p4 = workloads.cfg4()
        gen4 = time.time() - t0
        n4, d4 = p4["X"].shape
        m4, seed4 = 4096, 7
        rows4, cols4 = [0, 1, 2047, m4 - 1], [0, 1, 100, d4 - 1, d4]
        bh4, ref4, tref4 = cpu_leg_cfg4(p4, m4, seed4, rows4, cols4) if rank == 0 else (None, None, None)
        X4, Y4 = torch.from_numpy(p4["X"]).cuda(), torch.from_numpy(p4["Y"]).cuda()
        c4 = {"workload": "N=2^24, d=256, X fp32 Student-t(3), 0.1% of rows x100, beta~U(-1,1), sigma=1",
              "reference": "oracle OLS, FP64 normal equations; sketch entries from the definition",
              "reference_seconds": tref4, "data_gen_seconds": gen4, "by_form": {}}
        colrms = np.sqrt(np.mean(ref4 ** 2, axis=0)) if rank == 0 else None
        for prec, target in (("fp64", 1e-10), ("mixed_bf16", 1e-8), ("mixed_fp8", 1e-8)):
            s4 = slse.default_schedule(n4, d4, prec=prec, T=100, tol=1e-13 if prec == "fp64" else 5e-9)
            w4 = slse.alloc_workspace(slse.workspace_size(X4, Y4, slse.OP_FIT, s4))
            tt, fin = [], []
            for k in range(args.cfg4_steps + 1):
                r = slse.fit(X4, Y4, s4, seed=k, workspace=w4, trace_cap=s4.T)
                if rank == 0 and k > 0:
                    tt.append(first_crossing(r.beta_hist.cpu().numpy(), np.array(r.ms_hist), bh4, target)[0])
                    fin.append(float(np.linalg.norm(r.beta - bh4) / np.linalg.norm(bh4)))
            del w4
            torch.cuda.empty_cache()
            # the stored sketch of this form at sampled entries
            if prec == "mixed_fp8":
                codes, scales, sy = slse.sketch(X4, Y4, m4, seed=seed4, prec=prec)
                c8, s8, y8 = codes.cpu().numpy(), scales.cpu().numpy(), sy.float().cpu().numpy()
                e4m3 = e4m3_values()
                got = np.array([[e4m3[c8[i, c]] * 2.0 ** (int(s8[i, c // 32]) - 127) if c < d4 else y8[i]
                                 for c in cols4] for i in rows4])
            else:
                sx, sy = slse.sketch(X4, Y4, m4, seed=seed4, prec=prec)
                a_ = sx.double().cpu().numpy()
                b_ = sy.double().cpu().numpy()
                got = np.array([[a_[i, c] if c < d4 else b_[i] for c in cols4] for i in rows4])
            torch.cuda.empty_cache()
            if rank == 0:
                rr = r.report
                e = np.abs(got - ref4) / colrms
                c4["by_form"][prec] = {
                    "target": target,
                    "time_to_target_ms": statistics.mean(tt) if all(v is not None for v in tt) else None,
                    "final_rel_err_vs_fp64_oracle": max(fin),
                    "phases_ms": {k: rr[k] for k in ("ms_sketch", "ms_qr", "ms_stage1", "ms_stage2", "ms_total")},
                    "iters": [rr["iters_stage1"], rr["iters_stage2"]],
                    "sketch_entry_err_over_col_rms": {"max": float(e.max()), "mean": float(e.mean()),
                                                      "m": m4, "entries": len(rows4) * len(cols4)}}
        del X4, Y4, p4
        torch.cuda.empty_cache()

    # end to end through the public API with pinned host inputs (copy inside the call)
    e2e = None
    if args.e2e_steps > 0:
        wsz_h = slse.workspace_size(Xh, Yh, slse.OP_FIT, sched)
        wh = slse.alloc_workspace(wsz_h)
        slse.fit(Xh, Yh, sched, seed=2000, workspace=wh, trace_cap=cap)
        ev = []
        for k in range(args.e2e_steps):
            r = slse.fit(Xh, Yh, sched, seed=k, workspace=wh, trace_cap=cap)
            if rank == 0:
                t, _ = first_crossing(r.beta_hist.cpu().numpy(), np.array(r.ms_hist), bh, TARGET)
                ev.append((t if t is not None else r.report["ms_total"], r.report["ms_copy_in"],
                           r.report["ms_srht_pass1"]))
        del wh
        # the link of this box beside it: copies of the same pinned X by the copy engine
        buf, copies = torch.empty(Xh.shape, dtype=Xh.dtype, device="cuda"), []
        for k in range(4):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            buf.copy_(Xh, non_blocking=True)
            e1.record()
            torch.cuda.synchronize()
            copies.append(e0.elapsed_time(e1))
        del buf
        if rank == 0:
            e2e = {"value": reduce_max(statistics.median(v for v, _, _ in ev), 1), "unit": "ms",
                   "h2d_bytes_per_step": int(Xh.numel() * 4 + Yh.numel() * 4), "d2h_bytes_per_step": d * 8,
                   "steps_ms": [round(v, 3) for v, _, _ in ev],
                   "ms_copy_in": statistics.mean(c for _, c, _ in ev),
                   "ms_srht_pass1_from_host": statistics.median(p1 for _, _, p1 in ev),
                   **link_rates(Xh.numel() * 4, [p1 for _, _, p1 in ev], copies[1:]),
                   "how": "slse_fit with pinned host X, Y: Y copied on a side stream during the draws, X read from host "
                          "memory by the first SRHT pass, which also writes its device copy; "
                          "time from the call's first CUDA event to the first iterate within 1e-8; median of the "
                          "steps; pass1_host_read_gbs is the rate at which that pass reads X over the host link, "
                          "link_copy_gbs the rate of a copy of the same pinned X by the copy engine in this run"}

    if rank != 0:
        return
    out = {
        "metric": METRIC, "value": value, "unit": "ms", "n_gpus": ws, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": ms_per_step, "higher_is_better": False, "scaling": "weak", "vs_baseline": None,
        "dtype": "f32", "data": "synthetic",
        "config": {"workload": workload_name(args.log2n, d), "N": N, "d": d, "X_dtype": "fp32", "precision": "mixed_bf16",
                   "schedule": f"m={sched.m[0]}..{sched.m[-1]} (x2), a_i=2, r={sched.r}, T=100, tol=5e-9, 2nd stage {sched.stage2} form",
                   "parallelism": "replicas" if ws > 1 else "single GPU",
                   "l2": "inputs larger than L2 (X is 8.6 GB)", "seeds": f"sketch seeds 0..{args.steps - 1}"},
        "roofline": roofline,
        "cpu_baseline": cpu_base,
        "e2e": e2e,
        "gpu_launches": launches,
        "clocks": clk,
        "accuracy": {"target": TARGET, "crossed_every_step": crossed, "final_rel_err_max": max(errs_final),
                     "reference": "oracle OLS, FP64 normal equations", "reference_seconds": t_ref},
        "fp64": fp64,
        "countsketch": cs,
        "tuning": tun,
        "fp8": f8,
        "gaussian": gau,
        "differentiation": diff,
        "cfg2": c2,
        "cfg4": c4,
        "phases_ms": {k: rep[k] for k in ("ms_draws", "ms_sketch", "ms_srht_pass1", "ms_srht_pass2", "ms_qr",
                                          "ms_stage1", "ms_stage2", "ms_total")},
        "iters": [rep["iters_stage1"], rep["iters_stage2"]], "rebases": rep["rebases"],
        "stage2": {"form": sched.stage2, "exact_passes": rep["n_grad2"], "correction_steps": rep["n_corr"],
                   "ms_correction_steps": rep["ms_corr"], "ms_gram": rep["ms_gram"],
                   "gram_tflops": rep["flops_gram"] / rep["ms_gram"] / 1e9 if rep["ms_gram"] > 0 else None,
                   "gram_frac_of_bf16_peak": (rep["flops_gram"] / rep["ms_gram"] / 1e9 / measured_bf16_peak()[0]
                                              if rep["ms_gram"] > 0 else None),
                   "fell_back_to_full": rep["stage2_full"], "full_form": s2full},
        "kernels": kernels_gbs, "data_gen_seconds": t_gen,
    }
    print(json.dumps(out), flush=True)


def one_fit(args):
    """One fit of the benchmark workload (rows at --log2n, d = --d, data seed 1003, sketch seed 0)
    with the default schedule of the given precision and kind; prints its report.  Precision
    "fp64" stores X, Y in FP64; "fp64_x32" runs the FP64 path on the FP32 storage."""
    import torch
    import paper_2509_06856_gb300 as slse
    prec, kind = args.one_fit.split(":")
    N, d = 1 << args.log2n, args.d
    data = make_data(args.log2n, d)
    X, Y = torch.from_numpy(data["X"]).cuda(), torch.from_numpy(data["Y"]).cuda()
    if prec == "fp64":
        X, Y = X.double(), Y.double()
    elif prec == "fp64_x32":
        prec = "fp64"
    s = slse.default_schedule(N, d, prec=prec, T=100, tol=5e-9 if prec != "fp64" else 1e-13, kind=kind)
    r = slse.fit(X, Y, s, seed=0)
    print(json.dumps({"one_fit": args.one_fit, "N": N, "d": d, "status": r.status,
                      "report": {k: v for k, v in r.report.items() if k.startswith(("ms_", "iters", "n_"))}}))


def main():
    args = parse()
    if args.one_fit:
        one_fit(args)
        return
    rank, ws, local_rank = dist_init()
    if args.impl == "reference":
        run_reference(args, rank, ws)
    else:
        run_ours(args, rank, ws, local_rank)
    if ws > 1:
        import torch.distributed as dist
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
