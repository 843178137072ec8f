#!/usr/bin/env python
"""Benchmark of the directional scale-discretized wavelet transform on GB300.

One step = one analysis + one synthesis (a round trip) of a real signal at
L = 1024, N = 5, lambda = 2, J0 = 0 (11 wavelet scales) on the full-resolution
Driscoll-Healy SO(3) grid, f_lm Gaussian with C_l = 1/(l(l+1)) (seed 2),
mixed precision (FP32 arithmetic, FP64-generated Delta).  The metric is
transforms/s; the plain FP64 path is timed beside it, and the error of both
against the CPU oracle (spot rows) is reported.

Usage: python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]
For N > 1, launch under torch.distributed.run: every rank runs its own
independent transforms (replicas; no data-path collective), rank 0 prints.
"""
from __future__ import annotations

import argparse
import json
import math
import os
import statistics
import subprocess
import sys
import tempfile
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

from paper_1308_5706_gb300.inputs import flm_gaussian  # noqa: E402

L, N, LAM, J0, SEED = 1024, 5, 2.0, 0, 2
METRIC = "wavelet analysis+synthesis transforms/s at L=1024,N=5 (mixed vs FP64, 1 GB300) @max rel err; p99"
UNIT = "transforms/s"
WORKLOAD = "L=1024, N=5, lambda=2, J0=0 (11 scales), real Gaussian f_lm C_l=1/(l(l+1)), seed 2"
FP32_LANES_PER_SM, N_SM = 128, 152
SIDE = {"ana": 0, "syn": 1}  # direction index of s2dw_alpha_method


def peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        d = json.load(open(path))
        return d.get("hbm_gbs", 6800.0), d.get("sm_max_mhz", 2070.0), "measured"
    return 6800.0, 2070.0, "fallback"


# ---------------------------------------------------------------------------
# Oracle timing (CPU): bounded samples, spawn pool over host cores
# ---------------------------------------------------------------------------

_ORACLE = {}


def _init_worker():
    """Spawned oracle worker: one thread, the workload's f_lm and kernels."""
    os.environ["OMP_NUM_THREADS"] = "1"
    import oracle as O
    _ORACLE["O"] = O
    _ORACLE["f"] = flm_gaussian(L, SEED, "cl")
    _ORACLE["kern"] = O.kernels(L, N, LAM, J0)


def _oracle_task(b):
    """One sample unit: the analysis of beta-row b and the synthesis
    contribution of beta-row b (a round trip is 2L of each)."""
    O, f, kern = _ORACLE["O"], _ORACLE["f"], _ORACLE["kern"]
    t0 = time.perf_counter()
    O.analysis_rows(f, L, N, LAM, J0, [b], kern)
    t1 = time.perf_counter()
    J1 = kern[0].shape[0]
    rng = np.random.default_rng(b)
    # only row b is read by the partial sum: a broadcast view stands for the full array
    row = rng.standard_normal((J1, N, 1, 2 * L - 1))
    W = np.broadcast_to(row, (J1, N, 2 * L, 2 * L - 1))
    Wphi = np.broadcast_to(rng.standard_normal((1, 2 * L - 1)), (2 * L, 2 * L - 1))
    O.synthesis(W, Wphi, L, N, LAM, J0, kern, b_list=[b])
    t2 = time.perf_counter()
    return t1 - t0, t2 - t1


def _oracle_full(Ls):
    """A full oracle round trip (analysis of every beta row, then synthesis)
    of the workload's parameters at band-limit Ls; returns its seconds."""
    O = _ORACLE["O"]
    f = flm_gaussian(Ls, SEED, "cl")
    kern = O.kernels(Ls, N, LAM, J0)
    t0 = time.perf_counter()
    W, Wphi = O.analysis(f, Ls, N, LAM, J0, kern)
    fr = O.synthesis(W, Wphi, Ls, N, LAM, J0, kern)
    dt = time.perf_counter() - t0
    assert np.abs(fr - f).max() < 1e-10
    return dt


def oracle_full_round_trips(pool, workers: int, Ls=(16, 32, 64)):
    """Full oracle round trips at small band-limits, one per host core at a
    time: {L: {transforms/s over all cores, seconds per round trip}}."""
    out = {}
    for Ls_ in Ls:
        t0 = time.perf_counter()
        res = pool.map(_oracle_full, [Ls_] * workers, chunksize=1)
        wall = time.perf_counter() - t0
        out[str(Ls_)] = {"transforms_per_s": workers / wall, "s_per_round_trip": statistics.mean(res)}
    return out


def oracle_pool(workers: int):
    """Spawned pool (safe after CUDA initialisation), warmed outside timing."""
    import multiprocessing as mp
    # one thread per worker: the spawned workers import numpy (and its BLAS)
    # before their initializer runs, so the limits go in their environment
    for var in ("OMP_NUM_THREADS", "OPENBLAS_NUM_THREADS", "MKL_NUM_THREADS"):
        os.environ[var] = "1"
    pool = mp.get_context("spawn").Pool(workers, initializer=_init_worker)
    pool.map(_oracle_task, [1] * workers, chunksize=1)
    return pool


def oracle_run(pool, ntasks: int):
    """Run ntasks sample units (rows spread over the 2L beta rows) on the
    pool; returns (transforms/s, wall s, mean analysis-row s, mean synthesis-row s)."""
    rows = [int(x) for x in np.linspace(1, 2 * L - 2, max(1, ntasks))][:ntasks]
    t0 = time.perf_counter()
    res = pool.map(_oracle_task, rows, chunksize=1)
    wall = time.perf_counter() - t0
    ana = statistics.mean(r[0] for r in res)
    syn = statistics.mean(r[1] for r in res)
    return (ntasks / (2 * L)) / wall, wall, ana, syn


def run_reference(args):
    """The oracle as the reference arm: each step is one sample unit (one
    analysis beta-row and one synthesis beta-row of the L=1024 workload);
    the K timed steps run in parallel on the host cores."""
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return 0
    workers = max(1, os.cpu_count() or 1)
    pool = oracle_pool(workers)
    if args.warmup > 0:
        oracle_run(pool, args.warmup)
    value, wall, ana, syn = oracle_run(pool, args.steps)
    pool.close()
    pool.join()
    sample = (f"{args.steps} steps, each one analysis beta-row and one synthesis beta-row of the L=1024 "
              f"workload (a round trip is 2L = {2 * L} of each), run on {workers} spawn workers in "
              f"{wall:.1f} s (row: analysis {ana:.2f} s, synthesis {syn:.2f} s); extrapolated")
    out = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
           "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * wall / max(1, args.steps),
           "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
           "data": "synthetic", "config": {"workload": WORKLOAD},
           "cpu_baseline": {"value": value, "unit": UNIT, "cores": workers, "kind": "oracle", "sample": sample},
           "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(out))
    return 0


# ---------------------------------------------------------------------------
# GPU arm
# ---------------------------------------------------------------------------

class Clocks:
    """nvidia-smi sampling of SM clocks and throttle reasons during a region."""

    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,clocks_event_reasons.hw_slowdown,"
         "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
         "clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.proc = None
        # the raw samples go to $S2DW_CLOCKS_DIR when set (to keep them), else a temporary folder
        out_dir = os.environ.get("S2DW_CLOCKS_DIR") or tempfile.gettempdir()
        self.path = os.path.join(out_dir, f"clocks_bench_{index}_{os.getpid()}.csv")

    def __enter__(self):
        try:
            os.makedirs(os.path.dirname(self.path), exist_ok=True)
            self.fh = open(self.path, "w")
            self.proc = subprocess.Popen(["nvidia-smi", f"--id={self.index}", f"--query-gpu={self.Q}",
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=self.fh, stderr=subprocess.DEVNULL)
        except (OSError, FileNotFoundError):
            self.proc = None
        return self

    def __exit__(self, *exc):
        if self.proc is not None:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()
            self.fh.close()

    def summary(self):
        if self.proc is None or not os.path.exists(self.path):
            return None
        sm, mx, reasons = [], 0.0, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in open(self.path):
            parts = [x.strip() for x in line.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                mx = max(mx, float(parts[2]))
            except ValueError:
                continue
            for nm, v in zip(names, parts[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(nm)
        if not sm:
            return None
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": mx, "reasons": sorted(reasons), "samples": len(sm)}


def aggregate_replicas(total_ms: float, steps: int, dist=None, device=None):
    """Whole-job throughput of independent replicas: every rank ran `steps`
    transforms in `total_ms`; the job time is the maximum over ranks (one
    all-reduce, outside the data path) and the value counts all ranks' work."""
    world = 1
    if dist is not None and dist.is_initialized():
        import torch
        world = dist.get_world_size()
        t = torch.tensor([float(total_ms)], dtype=torch.float64, device=device)
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
        total_ms = float(t.item())
    return total_ms, steps * world / (total_ms / 1e3)


def contraction_flops(plan) -> float:
    """Algorithmic flops of one contraction launch (analysis or synthesis):
    per scale j and l in its support, (l+1)^2 (m', m >= 0) triples, each Delta * f (2 flops) plus one
    complex-by-real multiply-add (4 flops) per order n: 2 + 4N per triple
    (1.58e10 at L=1024, N=5).  The kernel shares one multiply-add between
    the orders +-n (the rows of -n equal those of n up to (-1)^{l+m'}), so it
    executes fewer flops than this count."""
    tot = 0.0
    for j in range(plan.nscale):
        lo, hi = plan.support(j)
        if hi < 0:
            continue
        ls = np.arange(lo, hi + 1, dtype=np.float64)
        tot += float(((ls + 1.0) ** 2).sum()) * (2 + 4 * plan.N)
    return tot


def delta_eighth_bytes(L_: int) -> float:
    """FP32 bytes of Delta^l_{m'm}, 0 <= m' <= m <= l < L (the eighth domain the
    symmetries reduce the table to): read once per contraction."""
    ls = np.arange(L_, dtype=np.float64)
    return float(((ls + 1) * (ls + 2) / 2).sum()) * 4


def scale_rows(plan, j):
    """(gamma samples, beta rows per gamma sample, band L_j) of scale j (j = nscale: scaling part)."""
    lo, hi = plan.support(j)
    return (1 if j == plan.nscale else N), 2 * L, hi + 1


def alpha_bytes(plan, elem: int, method: int, side: str) -> float:
    """Algorithmic bytes of one alpha launch over the scales it handles
    (method 0 direct sums, 1 full-band chirp-z, 2 segmented chirp-z, as the
    plan reports): W written (or read) once plus the [N][2L][L_j] complex
    rows of X (or V) read (or written) once."""
    n = 2 * L - 1
    tot = 0.0
    for j in range(plan.nscale + 1):
        g, rows, Lj = scale_rows(plan, j)
        if Lj <= 0 or plan.alpha_method(j, SIDE[side])[0] != method:
            continue
        tot += g * rows * n * elem + g * rows * Lj * 2 * elem
    return tot


def beta_bytes(plan, elem: int) -> float:
    """Algorithmic bytes of one beta launch: the cube Y [N][L_j][L_j] and the
    rows X [N][2L][L_j] (complex) of every scale, each moved once."""
    tot = 0.0
    for j in range(plan.nscale + 1):
        g, rows, Lj = scale_rows(plan, j)
        if Lj > 0:
            tot += g * (Lj * Lj + rows * Lj) * 2 * elem
    return tot


TRAFFIC_RECORD = os.path.join(ROOT, "profiles", "dram_traffic.json")


def source_fingerprint(files) -> str:
    import hashlib
    h = hashlib.sha256()
    for f in files:
        with open(os.path.join(ROOT, f), "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()[:16]


def recorded_traffic(stage: str):
    """DRAM bytes per launch of the kernel behind `stage`, from the ncu record,
    if the kernel's sources are unchanged since that capture (else None)."""
    try:
        rec = json.load(open(TRAFFIC_RECORD)).get(stage)
    except (OSError, ValueError):
        return None, None
    if not rec:
        return None, None
    try:
        same = source_fingerprint(rec["files"]) == rec["fingerprint"]
    except OSError:  # a source file is gone
        same = False
    if not same:
        return None, "sources changed since the capture of " + rec["date"]
    return rec["bytes_per_launch"], f"ncu capture of {rec['date']} ({rec['kernel']})"


def roofline(pm, mean_stage, ms_per_step):
    """Roofline of every timed stage and of the dominant one (largest mean
    duration), from the live CUDA-event durations (a stage is one launch or a few:
    f packing and contraction, conversion and products, products and chirp-z); and the round trip against
    the sum of the stage roofs: per direction the
    contraction at max(Delta bytes / HBM, 2+4N flops per triple / FP32 peak)
    and the FFT passes at (W + f bytes) / HBM."""
    hbm, sm_max, peak_src = peaks()
    fp32_peak = N_SM * FP32_LANES_PER_SM * 2 * sm_max * 1e6 / 1e12  # TFLOP/s at max SM clock
    alu_src = f"derived FP32: {N_SM} SMs x {FP32_LANES_PER_SM} lanes x 2 flop x {sm_max:.0f} MHz"
    work = {
        "ana_contract": ("alu", contraction_flops(pm)), "syn_contract": ("alu", contraction_flops(pm)),
        # one roof for the launches of all scales above 32: those that run as matrix products on
        # the tensor cores launch with the chirp-z group whatever the method the plan reports
        "ana_alpha_czt+seg": ("hbm", alpha_bytes(pm, 4, 1, "ana") + alpha_bytes(pm, 4, 2, "ana")),
        "syn_alpha_czt+seg": ("hbm", alpha_bytes(pm, 4, 1, "syn") + alpha_bytes(pm, 4, 2, "syn")),
        "ana_alpha_direct": ("hbm", alpha_bytes(pm, 4, 0, "ana")),
        "syn_alpha_direct": ("hbm", alpha_bytes(pm, 4, 0, "syn")),
        "ana_beta": ("hbm", beta_bytes(pm, 4)), "syn_beta": ("hbm", beta_bytes(pm, 4)),
    }
    per = {}
    for k, (bound, w) in work.items():
        ms = mean_stage.get(k, 0.0)
        if k.endswith("czt+seg"):
            ms = mean_stage.get(k[:-4], 0.0) + mean_stage.get(k[:4] + "alpha_seg", 0.0)
        if ms <= 0 or w <= 0:
            continue
        if bound == "alu":
            a = w / (ms * 1e-3) / 1e12
            per[k] = {"bound": "alu", "ms": round(ms, 4), "achieved": a, "peak": fp32_peak, "unit": "TFLOP/s",
                      "frac": a / fp32_peak}
        else:
            a = w / (ms * 1e-3) / 1e9
            per[k] = {"bound": "hbm", "ms": round(ms, 4), "achieved": a, "peak": hbm, "unit": "GB/s",
                      "frac": a / hbm}
    dom = max(per, key=lambda k: per[k]["ms"])
    r = dict(per[dom])
    r["kernel"] = dom
    r["timed"] = "stage"
    r["traffic"], r["traffic_source"] = recorded_traffic(dom)
    r["peak_source"] = alu_src if r["bound"] == "alu" else f"hbm_gbs of {peak_src} peaks"
    r["work_per_launch"] = work[dom][1]
    r["kernels"] = {k: {"ms": v["ms"], "frac": round(v["frac"], 4), "bound": v["bound"]} for k, v in per.items()}
    r["stage_ms"] = {k: round(v, 4) for k, v in mean_stage.items()}
    # round trip against the stage roofs (both directions)
    t_con = max(delta_eighth_bytes(pm.L) / (hbm * 1e9), contraction_flops(pm) / (fp32_peak * 1e12))
    w_bytes = 4.0 * (pm.nscale * N * 2 * L * (2 * L - 1) + 2 * L * (2 * L - 1)) + 8.0 * L * L
    t_fft = w_bytes / (hbm * 1e9)
    r["round_trip_roof_ms"] = 2e3 * (t_con + t_fft)
    r["round_trip_ms"] = ms_per_step
    r["round_trip_frac"] = r["round_trip_roof_ms"] / ms_per_step
    return r


def time_path(torch, plan, f_dev, steps, warmup, stream, profile=False):
    W, Wphi = plan.alloc_w()
    fr = plan.alloc_flm()
    for _ in range(warmup):
        plan.analysis(f_dev, W, Wphi, stream)
        plan.synthesis(W, Wphi, fr, stream)
    torch.cuda.synchronize()
    if profile:
        plan.profile(True)
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(steps)]
    with torch.cuda.stream(stream):
        for k in range(steps):
            ev[k][0].record(stream)
            plan.analysis(f_dev, W, Wphi, stream)
            plan.synthesis(W, Wphi, fr, stream)
            ev[k][1].record(stream)
    torch.cuda.synchronize()
    per = [a.elapsed_time(b) for a, b in ev]
    total = ev[0][0].elapsed_time(ev[-1][1])
    prof = None
    if profile:
        prof = plan.profile_read()
        plan.profile(False)
    return per, total, W, Wphi, fr, prof


def run_batch_workload(args):
    """64 real signals, L from {64,128,256,512}, N from {1,3,5}, lambda=2,
    C_l spectrum (seed 3): batched analysis + synthesis of all signals, both
    launch sets captured once in a CUDA graph and replayed."""
    import torch
    from paper_1308_5706_gb300 import binding as B
    rng = np.random.default_rng(3)
    Ls, Ns = rng.choice([64, 128, 256, 512], 64), rng.choice([1, 3, 5], 64)
    plans = [B.Plan(int(a), int(b), 2.0, 0, "mixed", autotune=True) for a, b in zip(Ls, Ns)]
    fs = [torch.from_numpy(flm_gaussian(p.L, 300 + i, "cl")).to(torch.complex64).cuda() for i, p in enumerate(plans)]
    Ws = [p.alloc_w() for p in plans]
    fr = [p.alloc_flm() for p in plans]
    hs = [p.handle for p in plans]
    stream = torch.cuda.Stream()

    def step():
        B.s2dw_analysis_batch(hs, fs, [w[0] for w in Ws], [w[1] for w in Ws], stream)
        B.s2dw_synthesis_batch(hs, [w[0] for w in Ws], [w[1] for w in Ws], fr, stream)

    with torch.cuda.stream(stream):
        for _ in range(args.warmup):
            step()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        step()
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    with torch.cuda.stream(stream):
        e0.record(stream)
        for _ in range(args.steps):
            graph.replay()
        e1.record(stream)
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1) / args.steps
    eps = max(float((f.to(torch.complex128).cpu() - torch.from_numpy(flm_gaussian(p.L, 300 + i, "cl"))).abs().max())
              for i, (p, f) in enumerate(zip(plans, fr)))
    out = {"metric": "batched signals/s (64 signals, analysis+synthesis per signal)", "value": 64 / (ms / 1e3),
           "unit": "signals/s", "ms_per_step": ms, "steps": args.steps, "warmup": args.warmup,
           "config": {"workload": "64 real signals, L in {64,128,256,512}, N in {1,3,5}, lambda=2, C_l, seed 3",
                      "launch_methods": "autotuned per configuration (s2dw_plan_tune, cached)",
                      "launches_per_step": "analysis: 1 contraction per distinct N + scaling + beta + alpha; "
                                           "synthesis: alpha + beta + contractions + scaling + reduction; "
                                           "one CUDA graph replay", "precision": "mixed"},
           "round_trip_eps_max": eps}
    print(json.dumps(out))
    for p in plans:
        p.close()
    return 0


def serve_report(torch, rate: float, seconds: float):
    """The serving workload (Poisson arrivals, analysis/synthesis 50/50, L =
    round(exp U[ln 32, ln 2048]), N 1..8, lambda {2, 3}, seed 4) for a few
    seconds: p50/p99 latency from arrival to completion, transforms/s,
    admission deferrals.  The server builds the process-wide Wigner tables up
    to L = 2048 when it starts; plans are made on demand while serving."""
    from paper_1308_5706_gb300.serve import Server, poisson_workload
    reqs = poisson_workload(rate=rate, duration=seconds, seed=4, L_range=(32, 2048))
    srv = Server("mixed", slots=4, max_batch=16, table_L=2048)
    bank = [torch.from_numpy(flm_gaussian(2048, 100 + k, "cl")).to(torch.complex64).pin_memory() for k in range(4)]
    torch.cuda.synchronize()
    rep = srv.run(reqs, payload=lambda r: bank[r.seed % 4][: r.L * r.L])
    srv.close()
    torch.cuda.synchronize()
    return {"transforms_per_s": rep["transforms_per_s"], "latency_ms": rep["latency_ms"],
            "requests": rep["requests"], "admission_deferrals": rep["admission_deferrals"],
            "mean_batch": rep["mean_batch"], "plans_created": rep["plans_created"],
            "plan_create_ms_mean": rep["plan_create_ms_mean"],
            "distinct_configurations": len({(r.L, r.N, r.lam) for r in reqs}),
            "workload": (f"Poisson {rate:g} req/s for {seconds:g} s, analysis/synthesis 50/50, L = round(exp "
                         f"U[ln 32, ln 2048]), N 1..8, lambda {{2,3}}, seed 4, mixed precision")}


def run_serve_workload(args):
    """Poisson arrivals of analysis/synthesis requests (50/50, a synthesis
    consumes an earlier analysis' W), L = round(exp U[ln 32, ln 2048]), N
    uniform in 1..8, lambda in {2, 3}, seed 4.  Plans are created on demand
    (no pre-warming: with ~1,000 distinct configurations per 10 s almost every
    analysis needs a new plan) on the server's worker threads, so plan
    creation is inside the measured latencies."""
    import torch
    from paper_1308_5706_gb300.serve import Server, poisson_workload
    reqs = poisson_workload(rate=args.serve_rate, duration=args.serve_seconds, seed=4, L_range=(32, 2048))
    srv = Server("mixed", slots=4, max_batch=16, table_L=2048)
    # client payloads: four pinned host signals at L = 2048; a request of
    # band-limit L sends the first L^2 coefficients (l < L) of one of them
    from paper_1308_5706_gb300.inputs import flm_gaussian
    bank = [torch.from_numpy(flm_gaussian(2048, 100 + k, "cl")).to(torch.complex64).pin_memory()
            for k in range(4)]
    torch.cuda.synchronize()
    rep = srv.run(reqs, payload=lambda r: bank[r.seed % 4][: r.L * r.L])
    srv.close()
    torch.cuda.synchronize()
    rep["distinct_configurations"] = len({(r.L, r.N, r.lam) for r in reqs})
    out = {"metric": "served transforms/s with p50/p99 latency", "value": rep["transforms_per_s"],
           "unit": "transforms/s", "latency_ms": rep["latency_ms"], "report": rep,
           "config": {"workload": f"Poisson {args.serve_rate:g} req/s for {args.serve_seconds:g} s, "
                                  "analysis/synthesis 50/50, L = round(exp U[ln 32, ln 2048]), N 1..8, "
                                  "lambda {2,3}, seed 4; plans made on demand; payloads pinned on the host",
                      "precision": "mixed"}}
    print(json.dumps(out))
    return 0


def run_multires_workload(args):
    """The L=1024, N=5, lambda=2 round trip with every scale on the grid of its
    own band-limit (S2DW_MULTIRES): mixed timed with CUDA events, checked
    against the FP64 multi-resolution plan and by the round trip."""
    import torch
    from paper_1308_5706_gb300 import binding as B
    pm = B.Plan(L, N, LAM, J0, "mixed", multires=True)
    f = torch.from_numpy(flm_gaussian(L, SEED, "cl")).to(torch.complex64).cuda()
    stream = torch.cuda.Stream()
    per, total, Wm, Wpm, frm, prof = time_path(torch, pm, f, args.steps, args.warmup, stream, profile=True)
    stage_ms, nana, nsyn = prof
    mean_stage = {k: round(v / (nana if k.startswith("ana") else nsyn), 4) for k, v in stage_ms.items()}
    p64 = B.Plan(L, N, LAM, J0, "fp64", multires=True)
    W64, Wp64 = p64.alloc_w()
    p64.analysis(f.to(torch.complex128), W64, Wp64)
    f64r = p64.alloc_flm()
    p64.synthesis(W64, Wp64, f64r)
    torch.cuda.synchronize()
    err = max(float((pm.w_scale(Wm, j).double() - p64.w_scale(W64, j)).abs().max()
                    / p64.w_scale(W64, j).abs().max().clamp_min(1e-300)) for j in range(pm.nscale))
    f0 = f.to(torch.complex128)
    eps_m = float((frm.to(torch.complex128) - f0).abs().max() / f0.abs().max())
    eps_64 = float((f64r - f0).abs().max() / f0.abs().max())
    full = pm.nscale * N * 2 * L * (2 * L - 1)
    out = {"metric": "multi-resolution wavelet analysis+synthesis transforms/s (L=1024, N=5, mixed)",
           "value": args.steps / (total / 1e3), "unit": "transforms/s", "ms_per_step": total / args.steps,
           "steps": args.steps, "warmup": args.warmup,
           "config": {"workload": WORKLOAD + "; every scale on the grid of its own band-limit",
                      "samples": int(pm.w_shape[0]), "samples_full_resolution": int(full)},
           "max_rel_err": {"mixed_vs_fp64_W_max_rel_per_scale": err, "round_trip_eps_mixed": eps_m,
                           "round_trip_eps_fp64": eps_64},
           "stage_ms": mean_stage}
    print(json.dumps(out))
    pm.close()
    p64.close()
    return 0


def run_precision_workload(args):
    """Error of the mixed path against the FP64 path as the band-limit grows
    (N=5, lambda=2, J0=0, C_l spectrum): the largest normwise error over the
    scales of W (max|W_mixed - W_fp64| / max|W_fp64| per scale), of W^Phi, and
    of the round trip f (max|f_rec - f| / max|f|), at L = 256, 512, 1024, 2048."""
    import torch
    from paper_1308_5706_gb300 import binding as B
    rows = []
    for Ls in (256, 512, 1024, 2048):
        f64 = flm_gaussian(Ls, SEED, "cl")
        res = {}
        for prec in ("mixed", "fp64"):
            p = B.Plan(Ls, N, LAM, J0, prec)
            cd, _ = p.torch_dtypes()
            f = torch.from_numpy(f64).to(cd).cuda()
            W, Wp = p.alloc_w()
            p.analysis(f, W, Wp)
            fr = p.alloc_flm()
            p.synthesis(W, Wp, fr)
            torch.cuda.synchronize()
            res[prec] = (W, fr.to(torch.complex128), p.nscale)
            p.close()
        Wm, frm, ns = res["mixed"]
        W64, fr64, _ = res["fp64"]
        per_scale = []
        for j in range(ns):
            ref = W64[j].abs().max()
            if float(ref) > 0:
                per_scale.append(float((Wm[j].double() - W64[j]).abs().max() / ref))
        f0 = torch.from_numpy(f64).cuda()
        rows.append({"L": Ls, "W_max_rel_over_scales": max(per_scale), "W_rel_per_scale": per_scale,
                     "round_trip_mixed": float((frm - f0).abs().max() / f0.abs().max()),
                     "round_trip_fp64": float((fr64 - f0).abs().max() / f0.abs().max())})
        del res, Wm, W64
        torch.cuda.empty_cache()
    print(json.dumps({"metric": "mixed-precision error against the FP64 path vs band-limit (N=5, lambda=2)",
                      "rows": rows}))
    return 0


def run_mw_workload(args):
    """The L=1024, N=5, lambda=2 round trip sampled on the McEwen-Wiaux grid
    (S2DW_MW: L beta samples instead of 2L): mixed timed with CUDA events,
    checked against the FP64 MW plan and by the round trip."""
    import torch
    from paper_1308_5706_gb300 import binding as B
    pm = B.Plan(L, N, LAM, J0, "mixed", mw=True)
    f = torch.from_numpy(flm_gaussian(L, SEED, "cl")).to(torch.complex64).cuda()
    stream = torch.cuda.Stream()
    per, total, Wm, Wpm, frm, prof = time_path(torch, pm, f, args.steps, args.warmup, stream, profile=True)
    stage_ms, nana, nsyn = prof
    mean_stage = {k: round(v / (nana if k.startswith("ana") else nsyn), 4) for k, v in stage_ms.items()}
    p64 = B.Plan(L, N, LAM, J0, "fp64", mw=True)
    W64, Wp64 = p64.alloc_w()
    p64.analysis(f.to(torch.complex128), W64, Wp64)
    f64r = p64.alloc_flm()
    p64.synthesis(W64, Wp64, f64r)
    torch.cuda.synchronize()
    err = max(float((Wm[j].double() - W64[j]).abs().max() / W64[j].abs().max().clamp_min(1e-300))
              for j in range(pm.nscale))
    f0 = f.to(torch.complex128)
    eps_m = float((frm.to(torch.complex128) - f0).abs().max() / f0.abs().max())
    eps_64 = float((f64r - f0).abs().max() / f0.abs().max())
    out = {"metric": "MW-grid wavelet analysis+synthesis transforms/s (L=1024, N=5, mixed)",
           "value": args.steps / (total / 1e3), "unit": "transforms/s", "ms_per_step": total / args.steps,
           "steps": args.steps, "warmup": args.warmup,
           "config": {"workload": WORKLOAD + "; beta sampled at pi(2b+1)/(2L-1), b < L",
                      "samples": int(Wm.numel()), "samples_dh": int(pm.nscale * N * 2 * L * (2 * L - 1))},
           "max_rel_err": {"mixed_vs_fp64_W_max_rel_per_scale": err, "round_trip_eps_mixed": eps_m,
                           "round_trip_eps_fp64": eps_64},
           "stage_ms": mean_stage}
    print(json.dumps(out))
    pm.close()
    p64.close()
    return 0


def run_sht_workload(args):
    """Inverse then forward spherical harmonic transform of the L=1024 signal
    on the DH sphere grid (mixed), timed with CUDA events; error of the round
    trip."""
    import torch
    from paper_1308_5706_gb300 import binding as B
    pm = B.Plan(L, N, LAM, J0, "mixed")
    f = torch.from_numpy(flm_gaussian(L, SEED, "cl")).to(torch.complex64).cuda()
    pix = pm.alloc_pix()
    g = pm.alloc_flm()
    stream = torch.cuda.current_stream()
    for _ in range(args.warmup):
        pm.sht_inverse(f, pix)
        pm.sht_forward(pix, g)
    torch.cuda.synchronize()
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(3)]
    ti = tf = 0.0
    for _ in range(args.steps):
        ev[0].record(stream)
        pm.sht_inverse(f, pix)
        ev[1].record(stream)
        pm.sht_forward(pix, g)
        ev[2].record(stream)
        torch.cuda.synchronize()
        ti += ev[0].elapsed_time(ev[1])
        tf += ev[1].elapsed_time(ev[2])
    f0 = f.to(torch.complex128)
    eps = float((g.to(torch.complex128) - f0).abs().max() / f0.abs().max())
    out = {"metric": "spherical harmonic transform pairs/s (L=1024, DH grid, mixed)",
           "value": args.steps / ((ti + tf) / 1e3), "unit": "pairs/s",
           "ms_per_step": (ti + tf) / args.steps, "ms_inverse": ti / args.steps, "ms_forward": tf / args.steps,
           "steps": args.steps, "warmup": args.warmup,
           "config": {"workload": "L=1024 real Gaussian f_lm C_l=1/(l(l+1)), seed 2; 2048 x 2047 samples"},
           "round_trip_eps": eps}
    print(json.dumps(out))
    pm.close()
    return 0


def run_steer_workload(args):
    """Steering (Eq. (10)) of the L=1024, N=5 mixed W to one arbitrary
    orientation per step: one pass over W (read) and out (write)."""
    import torch
    from paper_1308_5706_gb300 import binding as B
    pm = B.Plan(L, N, LAM, J0, "mixed")
    f = torch.from_numpy(flm_gaussian(L, SEED, "cl")).to(torch.complex64).cuda()
    W, Wp = pm.alloc_w()
    pm.analysis(f, W, Wp)
    gam = [0.3141]
    out = pm.steer(W, gam)
    stream = torch.cuda.current_stream()
    for _ in range(args.warmup):
        pm.steer(W, gam, out)
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    for _ in range(args.steps):
        pm.steer(W, gam, out)
    e1.record(stream)
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1) / args.steps
    nbytes = (W.numel() + out.numel()) * 4
    hbm, _, src = peaks()
    achieved = nbytes / (ms * 1e-3) / 1e9
    out_line = {"metric": "steering passes/s (W of 11 scales to one orientation)", "value": 1e3 / ms,
                "unit": "passes/s", "ms_per_step": ms, "steps": args.steps, "warmup": args.warmup,
                "config": {"workload": "L=1024, N=5, lambda=2, 11 scales, mixed; 1 orientation per pass",
                           "l2": "W (0.92 GB) larger than L2"},
                "roofline": {"kernel": "k_steer", "bound": "hbm", "achieved": achieved, "peak": hbm,
                             "unit": "GB/s", "frac": achieved / hbm, "traffic": None,
                             "peak_source": f"{src} hbm_gbs"}}
    print(json.dumps(out_line))
    pm.close()
    return 0


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=200)
    ap.add_argument("--warmup", type=int, default=10)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--fp64-steps", type=int, default=3)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--workload", default="roundtrip",
                    choices=["roundtrip", "batch", "serve", "steer", "multires", "sht", "mw", "precision"])
    ap.add_argument("--serve-seconds", type=float, default=60.0)
    ap.add_argument("--serve-rate", type=float, default=200.0)
    ap.add_argument("--serve-line-seconds", type=float, default=10.0,
                    help="seconds of the served mixed-L Poisson run reported in the roundtrip line (0: none)")
    ap.add_argument("--L", type=int, default=1024,
                    help="band-limit of the roundtrip workload; values other than 1024 are for profiling "
                         "captures at a smaller size and give no bench line of the metric")
    args = ap.parse_args()
    args.warmup = max(3, args.warmup)
    global L, WORKLOAD
    if args.L != L:
        L = args.L
        WORKLOAD = WORKLOAD.replace("L=1024", f"L={L}") + " (profiling size, not the metric's workload)"
    if args.impl == "reference":
        return run_reference(args)
    if args.workload == "batch":
        return run_batch_workload(args)
    if args.workload == "serve":
        return run_serve_workload(args)
    if args.workload == "steer":
        return run_steer_workload(args)
    if args.workload == "multires":
        return run_multires_workload(args)
    if args.workload == "sht":
        return run_sht_workload(args)
    if args.workload == "mw":
        return run_mw_workload(args)
    if args.workload == "precision":
        return run_precision_workload(args)

    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))

    # CPU baseline first (spawned pool, before the first GPU call)
    cpu = None
    if rank == 0 and not args.no_cpu_baseline:
        workers = max(1, os.cpu_count() or 1)
        pool = oracle_pool(workers)
        v, wall, ana, syn = oracle_run(pool, workers)
        full = oracle_full_round_trips(pool, workers)
        pool.close()
        pool.join()
        cpu = {"value": v, "unit": UNIT, "cores": workers, "kind": "oracle",
               "sample": (f"{workers} sample units (1 analysis beta-row + 1 synthesis beta-row each) of the "
                          f"L={L} workload on {workers} spawn workers in {wall:.1f} s (row: analysis "
                          f"{ana:.2f} s, synthesis {syn:.2f} s); a round trip is 2L = {2 * L} rows of each, "
                          f"extrapolated"),
               "full_round_trips": full,
               "full_round_trips_note": (f"complete oracle round trips (N={N}, lambda={LAM:g}, J0={J0}, same "
                                         f"spectrum and seed), {workers} at a time on the {workers} workers")}

    import torch
    from paper_1308_5706_gb300 import binding as B

    torch.cuda.set_device(local)
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl")

    f64 = flm_gaussian(L, SEED + rank, "cl")
    stream = torch.cuda.Stream()
    pm = B.Plan(L, N, LAM, J0, "mixed", autotune=True)  # launch methods tuned (or cached) before timing
    f_mixed = torch.from_numpy(f64).to(torch.complex64).cuda()

    if dist:
        dist.barrier()
    torch.cuda.synchronize()
    with Clocks(local) as clk:
        per, total, Wm, Wpm, frm, _ = time_path(torch, pm, f_mixed, args.steps, args.warmup, stream)
    torch.cuda.synchronize()
    if dist:
        dist.barrier()
    total, value = aggregate_replicas(total, args.steps, dist, device="cuda")
    # the per-stage breakdown from a separate run with the library's stage
    # events on (they add about 1% to a round trip, so not in the timed one)
    _, _, _, _, _, prof = time_path(torch, pm, f_mixed, min(args.steps, 50), 2, stream, profile=True)

    # end to end through the C ABI with pinned host buffers: every step copies
    # its f_lm in and its result out; the copies run on their own streams
    # (double-buffered), so that step k+1's upload and step k's download
    # overlap the transforms as a serving pipeline would
    fh = torch.from_numpy(f64).to(torch.complex64).pin_memory()
    fo = [torch.empty_like(fh).pin_memory() for _ in range(2)]
    fd = [torch.empty(L * L, dtype=torch.complex64, device="cuda") for _ in range(2)]
    Wd, Wpd = pm.alloc_w()
    frd = [pm.alloc_flm() for _ in range(2)]
    up, down = torch.cuda.Stream(), torch.cuda.Stream()
    ev_in = [torch.cuda.Event() for _ in range(2)]     # f uploaded
    ev_read = [torch.cuda.Event() for _ in range(2)]   # analysis has read f
    ev_done = [torch.cuda.Event() for _ in range(2)]   # result written
    ev_out = [torch.cuda.Event() for _ in range(2)]    # result downloaded
    started = [False, False]

    def e2e_step(k):
        i = k & 1
        if started[i]:
            up.wait_event(ev_read[i])
        with torch.cuda.stream(up):
            fd[i].copy_(fh, non_blocking=True)
            ev_in[i].record(up)
        stream.wait_event(ev_in[i])
        pm.analysis(fd[i], Wd, Wpd, stream)
        ev_read[i].record(stream)
        if started[i]:
            stream.wait_event(ev_out[i])
        pm.synthesis(Wd, Wpd, frd[i], stream)
        ev_done[i].record(stream)
        down.wait_event(ev_done[i])
        with torch.cuda.stream(down):
            fo[i].copy_(frd[i], non_blocking=True)
            ev_out[i].record(down)
        started[i] = True

    for k in range(args.warmup):
        e2e_step(k)
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    for k in range(args.steps):
        e2e_step(k)
    for i in range(2):
        stream.wait_event(ev_out[i])
    e1.record(stream)
    torch.cuda.synchronize()
    e2e_ms = e0.elapsed_time(e1)
    e2e = {"value": args.steps * world / (e2e_ms / 1e3), "unit": UNIT,
           "h2d_bytes_per_step": int(fh.numel() * fh.element_size()),
           "d2h_bytes_per_step": int(fo[0].numel() * fo[0].element_size()),
           "copies": "pinned host buffers, on their own streams, overlapping the previous step's transforms"}

    # FP64 path (the baseline the mixed path is compared with)
    p64 = None
    err = {}
    Wm_d = Wm.double()
    err["round_trip_eps_mixed"] = float((frm.to(torch.complex128).cpu() - torch.from_numpy(f64)).abs().max())
    # the last downloaded end-to-end result (host memory)
    err["round_trip_eps_e2e"] = float((fo[(args.steps - 1) & 1].to(torch.complex128) - torch.from_numpy(f64)).abs().max())
    if args.fp64_steps > 0:
        p64 = B.Plan(L, N, LAM, J0, "fp64", autotune=True)
        f_d64 = torch.from_numpy(f64).cuda()
        per64, total64, W64, Wp64, fr64, _ = time_path(torch, p64, f_d64, args.fp64_steps, 1, stream)
        # accuracy: mixed vs FP64 (whole arrays), both vs the oracle on spot rows, round trips
        err["mixed_vs_fp64_W_max_rel_per_scale"] = max(
            float((Wm_d[j] - W64[j]).abs().max() / W64[j].abs().max()) for j in range(pm.nscale))
        err["round_trip_eps_fp64"] = float((fr64.cpu() - torch.from_numpy(f64)).abs().max())
    if rank == 0 and p64 is not None:
        import oracle as O
        b_spot = [700]
        kern = O.kernels(L, N, LAM, J0)
        Wo, Wpo, _ = O.analysis_rows(f64, L, N, LAM, J0, b_spot, kern)
        w64s = W64[:, :, b_spot, :].cpu().numpy()
        wms = Wm_d[:, :, b_spot, :].cpu().numpy()
        nz = [j for j in range(pm.nscale) if np.abs(Wo[j]).max() > 0]   # W^j = 0 where f vanishes on supp j
        err["fp64_vs_oracle_spot_max_rel"] = max(
            float(np.abs(w64s[j] - Wo[j]).max() / np.abs(Wo[j]).max()) for j in nz)
        err["mixed_vs_oracle_spot_max_rel"] = max(
            float(np.abs(wms[j] - Wo[j]).max() / np.abs(Wo[j]).max()) for j in nz)
        err["zero_scales_max_abs"] = max([float(np.abs(w64s[j]).max()) for j in range(pm.nscale) if j not in nz]
                                         + [0.0])
        err["oracle_spot"] = "beta row b=700, all scales, gamma and alpha samples"

    # served latency: a short run of the mixed-L Poisson serving workload
    serve = None
    if rank == 0 and args.serve_line_seconds > 0 and L == 1024:
        serve = serve_report(torch, args.serve_rate, args.serve_line_seconds)

    # roofline of the dominant kernel, from the stage events of the timed region
    stage_ms, nana, nsyn = prof
    mean_stage = {k: (v / (nana if k.startswith("ana") else nsyn)) for k, v in stage_ms.items()}
    roof = roofline(pm, mean_stage, total / args.steps)

    per_sorted = sorted(per)
    out = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": total / args.steps, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f32",
        "data": "synthetic",
        "config": {"workload": WORKLOAD, "precision": "mixed (FP32 arithmetic, FP64-generated Delta)",
                   "grid": "full-resolution DH SO(3) grid per scale: 5 x 2048 x 2047",
                   "parallelism": f"replicas x{world}",
                   "launch_methods": {"choices": pm.tuned[0], "source": pm.tuned[1],
                                      "layout": "beta ana, beta syn, alpha ana / syn per scale, then a value kept for saved choices (s2dw.h)"},
                   "l2": "inputs larger than L2 (W 0.92 GB, Delta pair table 0.78 GB per direction)"},
        "latency_ms": {"p50": per_sorted[len(per) // 2],
                       "p99": per_sorted[min(len(per) - 1, int(round(0.99 * (len(per) - 1))))]},
        "fp64": ({"value": args.fp64_steps / (total64 / 1e3), "ms_per_step": total64 / args.fp64_steps,
                  "steps": args.fp64_steps} if p64 else None),
        "speedup_vs_fp64": ((value / world) / (args.fp64_steps / (total64 / 1e3)) if p64 else None),
        "max_rel_err": err,
        "roofline": roof,
        "cpu_baseline": cpu,
        "serve": serve,
        "e2e": e2e,
        "gpu_launches": args.steps * sum(pm.launch_counts()),
        "clocks": clk.summary(),
    }
    if rank == 0:
        print(json.dumps(out))
    pm.close()
    if p64:
        p64.close()
    if dist:
        dist.destroy_process_group()
    return 0


if __name__ == "__main__":
    sys.exit(main())
