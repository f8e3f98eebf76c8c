"""Benchmark of the GB300 FT-GCR(k) library.

Workload (one "step"): one mixed-precision FT-GCR(4) solve of the 1024 x 512
latitude-longitude hill problem (h0 = 0.1, half-width 20 deg, flow RHS,
mu = 0.3 / dtheta^2, tol 1e-10 relative): FP32 inner vectors, stencil,
preconditioner and axpys; FP64 inner products, norm test and outer refinement
residual.  Inputs are resident in HBM; L2 (129 MB) is flushed between timed
steps by writing a 256 MB buffer.  Reported beside it: the plain FP64 GPU path
on the same problem, per-solve p50/p99 latency, the roofline of the
persistent iteration kernel, the end-to-end number through the C ABI with
host buffers, and the CPU oracle timed on this host's cores.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]
"""
from __future__ import annotations

import argparse
import hashlib
import json
import math
import os
import subprocess
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

from paper_2103_07210_gb300 import inputs  # noqa: E402

METRIC = "GCR iters/s, solves/s at 1024x512 (mixed vs FP64), HBM % peak; p50/p99 latency"
NLON, NLAT, K, TOL = 1024, 512, 4, 1e-10
# Every solve of the benchmark starts from x = 0 and says so
# (FTGCR_FLAG_ZERO_GUESS): x is not read (host x not copied in), and the mixed
# path takes R for its first inner solve directly.
ZG = True
WORKLOAD = "ftgcr4_mixed_1024x512_hill_tol1e-10"

# Algorithmic bytes of one inner step, averaged over a Krylov cycle of length
# k: (14 + 1.5 (k + 1)) vectors of s bytes (s = 4 for the FP32 inner vectors);
# each refinement round adds 6 FP64 vectors (x, d, R, r_out, Tx, Ty): `outer`
# sweeps, plus the round forming the first r_out unless the solve declared a
# zero initial guess (which skips that round).
def algorithmic_bytes(steps: int, outer: int, k: int = K, s: int = 4, N: int = NLON * NLAT, mixed: bool = True) -> float:
    refine = (outer + (0 if ZG else 1)) * 6 * 8 * N if mixed else 0
    return steps * (14 + 1.5 * (k + 1)) * s * N + refine


# DRAM traffic of a solve (zero initial guess) from one ncu capture, valid
# only for the kernel sources it was taken on (sha256 of the CUDA sources).
NCU_TRAFFIC = {"sources_sha256": "1d5b5fb458376f0f2cb2db005b41915501fb39e97b3dcd7015435c26383e0c76",
               "bytes_per_launch": 42429440 + 93857536,  # mixed 1024x512 (read + write)
               "large": {"2048x1024": 2780000000 + 1860000000, "4096x2048": 12320000000 + 5110000000}}


def sources_hash() -> str:
    """sha256 of the solve kernels' sources: their device code and the
    translation units that instantiate them (host code and set-up kernels in
    ftgcr.cu do not change their DRAM traffic)."""
    h = hashlib.sha256()
    d = os.path.join(ROOT, "paper_2103_07210_gb300", "csrc")
    for f in sorted(os.listdir(d)):
        if f in ("ftgcr_device.cuh", "ftgcr_phases.cuh", "ftgcr_stream.cuh", "ftgcr_band.cuh", "ftgcr_instances.h") or \
                (f.startswith(("ftgcr_k", "ftgcr_b")) and f.endswith(".cu")):
            h.update(open(os.path.join(d, f), "rb").read())
    return h.hexdigest()


def read_peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            pk = json.load(f)
        return float(pk["hbm_gbs"]), "measured"
    except Exception:
        return 6800.0, "fallback"


def measure_peaks_in_run(torch, ftgcr, dev, reps=5):
    """The two ceilings measured in this process, beside MEASURED_PEAKS.json:
    a 2 GiB device-to-device copy (read + write bytes over the event time,
    best of `reps`) and the library's FP64 FMA-rate probe (best of 3)."""
    n = (1 << 31) // 4
    a = torch.empty(n, dtype=torch.float32, device=dev).fill_(1.0)
    b = torch.empty_like(a)
    b.copy_(a)
    stream = torch.cuda.current_stream()
    best = 1e30
    for _ in range(reps):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        b.copy_(a)
        e1.record(stream)
        torch.cuda.synchronize()
        best = min(best, e0.elapsed_time(e1))
    copy_gbs = 2 * 4 * n / (best * 1e-3) / 1e9
    del a, b
    fma = max(ftgcr.fp64_fma_rate(4096) for _ in range(3))
    return {"copy_gbs": copy_gbs, "copy_bytes": 2 * 4 * n, "fp64_fma_tflops": fma}


class ClockSampler:
    """nvidia-smi clock / throttle sampling during the timed region."""

    FIELDS = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.hw_slowdown,"
              "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
              "clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.proc = None
        self.lines = []

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.index), f"--query-gpu={self.FIELDS}",
                                          "--format=csv,noheader,nounits", "-lms", "100"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            threading.Thread(target=self._read, daemon=True).start()
        except Exception:
            self.proc = None
        time.sleep(0.3)
        return self

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def __exit__(self, *a):
        time.sleep(0.25)
        if self.proc:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=2)
            except Exception:
                self.proc.kill()

    def summary(self):
        sm, mx, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            parts = [p.strip() for p in ln.split(",")]
            if len(parts) < 7:
                continue
            try:
                sm.append(float(parts[0]))
                mx = float(parts[1])
            except ValueError:
                continue
            for nm, v in zip(names, parts[3:7]):
                if v.lower() == "active":
                    reasons.add(nm)
        return {"sm_mhz": float(np.median(sm)) if sm else None, "sm_max_mhz": mx, "reasons": sorted(reasons),
                "samples": len(sm)}


def max_over_ranks(x, device):
    """The largest of x over the ranks of the initialised process group (x
    itself without one): the slowest rank's time is the job's time."""
    import torch
    import torch.distributed as dist
    if not (dist.is_available() and dist.is_initialized()) or dist.get_world_size() == 1:
        return float(x)
    t = torch.tensor([float(x)], device=device, dtype=torch.float64)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def dist_env():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


# ------------------------------------------------------------------ oracle arm
def _oracle_solve(_):
    import oracle

    p = inputs.hill_problem(NLON, NLAT)
    t = time.perf_counter()
    o = oracle.ftgcr(p.D, p.R, p.mu, K, TOL)
    return time.perf_counter() - t, o["steps"]


def oracle_throughput(seconds_budget: float = 12.0, cores: int | None = None):
    """Independent oracle solves of the benchmark problem, one process per
    core, for about `seconds_budget` of wall time: solves/s and steps/s."""
    import multiprocessing as mp

    import oracle

    oracle.build()
    cores = cores or os.cpu_count() or 1
    one, steps = _oracle_solve(0)
    per_core = max(1, int(seconds_budget / max(one, 1e-3)))
    n = cores * per_core
    ctx = mp.get_context("spawn")
    with ctx.Pool(cores) as pool:
        pool.map(_oracle_solve, range(cores))  # warm the workers
        t = time.perf_counter()
        res = pool.map(_oracle_solve, range(n), chunksize=1)
        wall = time.perf_counter() - t
    return dict(value=n / wall, steps_per_s=sum(r[1] for r in res) / wall, cores=cores,
                latency_s=float(np.median([r[0] for r in res])), steps=steps, n=n, wall=wall)


def _oracle_x(args):
    """FP64 oracle solution of the default hill problem (flow RHS) at
    (nlon, nlat, k, tol), run in a spawned worker."""
    import oracle

    nlon, nlat, k, tol = args
    p = inputs.hill_problem(nlon, nlat)
    o = oracle.ftgcr(p.D, p.R, p.mu, k, tol)
    return o["x"], o["steps"], o["converged"]


def rel_err(a, b) -> float:
    """Relative 2-norm error of a against the reference b."""
    a = np.asarray(a, dtype=np.float64).ravel()
    b = np.asarray(b, dtype=np.float64).ravel()
    nb = float(np.linalg.norm(b))
    return float(np.linalg.norm(a - b) / nb) if nb > 0 else float(np.linalg.norm(a))


def errors_vs_oracle(results):
    """Each result's relative error against the FP64 oracle's solution of the
    same problem at the same tolerance.  `results` maps a name to
    ((nlon, nlat, k, tol), x); the oracle solves (after the timed region) run
    in a spawned pool, one process per distinct problem."""
    import multiprocessing as mp

    import oracle

    oracle.build()
    cfgs = sorted({c for c, _ in results.values()})
    with mp.get_context("spawn").Pool(max(1, min(len(cfgs), os.cpu_count() or 1))) as pool:
        refs = dict(zip(cfgs, pool.map(_oracle_x, cfgs)))
    out = {}
    for name, (c, x) in results.items():
        xr, steps, conv = refs[c]
        out[name] = {"err_vs_oracle": rel_err(x, xr), "tol": c[3], "oracle_steps": steps, "oracle_converged": conv}
    return out


def physical_cores():
    """Distinct (package, core) pairs of the host's online CPUs, or None."""
    seen = set()
    base = "/sys/devices/system/cpu"
    try:
        for d in os.listdir(base):
            if not (d.startswith("cpu") and d[3:].isdigit()):
                continue
            t = os.path.join(base, d, "topology")
            try:
                pkg = open(os.path.join(t, "physical_package_id")).read().strip()
                core = open(os.path.join(t, "core_id")).read().strip()
            except OSError:
                continue
            seen.add((pkg, core))
    except OSError:
        return None
    return len(seen) or None


def run_reference(args):
    ws, rank, _ = dist_env()
    if rank != 0:
        return 0
    import multiprocessing as mp

    import oracle

    oracle.build()
    cores = os.cpu_count() or 1
    ctx = mp.get_context("spawn")
    times = []
    with ctx.Pool(cores) as pool:
        for i in range(args.warmup + args.steps):
            t = time.perf_counter()
            pool.map(_oracle_solve, range(cores), chunksize=1)
            dt = time.perf_counter() - t
            if i >= args.warmup:
                times.append(dt)
    ms = 1e3 * float(np.mean(times))
    value = cores / (ms * 1e-3)
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": "solves/s", "n_gpus": ws,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": WORKLOAD, "nlon": NLON, "nlat": NLAT, "k": K, "tol": TOL},
            "cpu_baseline": {"value": value, "unit": "solves/s", "cores": cores, "kind": "oracle",
                             "sample": f"each step: {cores} independent FP64 oracle solves of the {NLON}x{NLAT} "
                                       f"problem, one per core"},
            "e2e": {"value": value, "unit": "solves/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line))
    return 0


# ------------------------------------------------------------------ larger grids
def bench_large(torch, ftgcr, dev, flush, sizes=((2048, 1024), (4096, 2048)), reps=3, keep=None):
    """Single mixed solves on grids whose working set exceeds the 129 MB L2
    (1024x512 stays L2-resident), so that the roofline fraction measures HBM:
    per size the event-timed solve, inner steps, algorithmic bytes and
    achieved bandwidth against the measured copy peak.  `keep` (a dict), if
    given, receives each size's solution for the comparison with the oracle."""
    peak, peak_kind = read_peaks()
    stream = torch.cuda.current_stream()
    out = {}
    for nlon, nlat in sizes:
        p = inputs.hill_problem(nlon, nlat)
        R = torch.from_numpy(p.R).to(dev)
        x = torch.zeros_like(R)
        with ftgcr.Solver(p.D, p.mu, k=K, tol=TOL, precision="mixed", zero_guess=ZG) as s:
            s.solve_async(R, x, stream=stream)  # warm
            ms = []
            for _ in range(reps):
                x.zero_()
                flush.fill_(3)
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record(stream)
                s.solve_async(R, x, stream=stream)
                b.record(stream)
                torch.cuda.synchronize()
                ms.append(a.elapsed_time(b))
            info = s.stats()
        t = float(np.median(ms))
        nb = algorithmic_bytes(info["steps"], info["outer"], N=nlon * nlat)
        gbs = nb / (t * 1e-3) / 1e9
        traffic = NCU_TRAFFIC["large"].get(f"{nlon}x{nlat}") if NCU_TRAFFIC["sources_sha256"] == sources_hash() else None
        if keep is not None:
            keep[(nlon, nlat)] = x.cpu().numpy()
        out[f"{nlon}x{nlat}"] = {"ms": t, "solves_per_s": 1e3 / t, "inner_steps": info["steps"], "traffic": traffic,
                                 "refinement_sweeps": info["outer"], "tiles": info["tiles"],
                                 "algorithmic_bytes": nb, "achieved_gbs": gbs, "frac": gbs / peak,
                                 "peak_kind": peak_kind, "converged": info["converged"],
                                 "residual_rel": info["res_final_true"] / info["norm_R"]}
    return out


# ------------------------------------------------------------------ steady state: a window of inner steps
def bench_steady(torch, ftgcr, dev, flush, sizes=((1024, 512), (2048, 1024)), window=(100, 600), reps=3):
    """Time per inner step away from the solve's start and end: the singular
    mu = 0 hill problem (Section 4's pure Poisson form) needs thousands of
    fault-free steps, so solves capped at window[0] and at window[1] executed
    steps differ by window[1] - window[0] steps of the iteration proper
    (whole Krylov cycles: both ends are multiples of k).  Per size and
    precision: the event-timed difference per step, its algorithmic bytes
    (14 + 1.5(k+1)) s N, and the bandwidth against the measured copy peak.
    `clean` says the window held no detection and no refinement sweep."""
    peak, peak_kind = read_peaks()
    stream = torch.cuda.current_stream()
    n0, n1 = window
    assert n0 % K == 0 and n1 % K == 0
    out = {}
    for nlon, nlat in sizes:
        p = inputs.hill_problem(nlon, nlat)
        R = torch.from_numpy(p.R).to(dev)
        N = nlon * nlat
        for precision, s_bytes in (("mixed", 4), ("fp64", 8)):
            t, infos = {}, {}
            for cap in window:
                x = torch.zeros_like(R)
                with ftgcr.Solver(p.D, 0.0, k=K, tol=TOL, precision=precision, max_steps=cap, zero_guess=ZG) as s:
                    s.solve_async(R, x, stream=stream)  # warm
                    ms = []
                    for _ in range(reps):
                        x.zero_()
                        flush.fill_(3)
                        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                        a.record(stream)
                        s.solve_async(R, x, stream=stream)
                        b.record(stream)
                        torch.cuda.synchronize()
                        ms.append(a.elapsed_time(b))
                    t[cap], infos[cap] = float(np.median(ms)), s.stats()
            i0, i1 = infos[n0], infos[n1]
            per_step_us = (t[n1] - t[n0]) * 1e3 / (n1 - n0)
            nb = (14 + 1.5 * (K + 1)) * s_bytes * N
            gbs = nb / (per_step_us * 1e-6) / 1e9
            clean = (i0["steps"] == n0 and i1["steps"] == n1 and not i1["detect_steps"]
                     and i1["outer"] == i0["outer"] and not i1["converged"])
            out[f"{precision}_{nlon}x{nlat}"] = {
                "us_per_step": per_step_us, "algorithmic_bytes_per_step": nb, "achieved_gbs": gbs,
                "frac": gbs / peak, "peak_kind": peak_kind, "clean": clean,
                "ms": {str(n0): t[n0], str(n1): t[n1]}}
    return out


# ------------------------------------------------------------------ k sweep, cost of the protection
def bench_ksweep(torch, ftgcr, dev, flush, ks=(1, 2, 4, 5, 8), reps=5):
    """Fault-free mixed solves of the 1024x512 problem for several Krylov
    cycle lengths, protected (FT-GCR(k)) and unprotected (plain GCR(k)): the
    cost of the fault test and backup (Section 4 expects it near zero)."""
    p = inputs.hill_problem(NLON, NLAT)
    R = torch.from_numpy(p.R).to(dev)
    stream = torch.cuda.current_stream()
    out = {}
    for k in ks:
        row = {}
        for mode, protect in (("ftgcr", True), ("gcr", False)):
            with ftgcr.Solver(p.D, p.mu, k=k, tol=TOL, precision="mixed", protect=protect, zero_guess=ZG) as s:
                x = torch.zeros_like(R)
                s.solve_async(R, x, stream=stream)
                ms = []
                for _ in range(reps):
                    x.zero_()
                    flush.fill_(5)
                    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                    a.record(stream)
                    s.solve_async(R, x, stream=stream)
                    b.record(stream)
                    torch.cuda.synchronize()
                    ms.append(a.elapsed_time(b))
                info = s.stats()
            row[mode + "_ms"] = float(np.median(ms))
            row[mode + "_steps"] = info["steps"]
        row["overhead"] = row["ftgcr_ms"] / row["gcr_ms"] - 1.0
        out[f"k{k}"] = row
    return out


# ------------------------------------------------------------------ batch and serving mixes
def bench_batch(torch, ftgcr, dev, n=128, seed=42, reps=3):
    """128 independent mixed-precision solves of sizes U{128x64, 256x128,
    512x256, 1024x512} (hills: centre, height and width drawn per solve) in
    ONE persistent launch, against the same solves launched one by one; the
    launch also captured into a CUDA graph and replayed.  Row bands and round
    layout per size from the autotuner (ftgcr_tune, timed for as many solves
    of that size as the batch holds), beside the layout ftgcr_create picks by
    itself."""
    import collections

    sizes = inputs.batch_sizes(seed, n)
    probs = [inputs.hill_problem(nlon, nlat, **inputs.random_hill(seed * 1000 + q))
             for q, (nlon, nlat) in enumerate(sizes)]
    Rs = [torch.from_numpy(p.R).to(dev) for p in probs]
    stream = torch.cuda.current_stream()
    tuned = {}
    for (nlon, nlat), cnt in sorted(collections.Counter(sizes).items()):
        p0 = probs[sizes.index((nlon, nlat))]
        t = ftgcr.tune(p0.D, p0.mu, k=K, tol=TOL, precision="mixed", concurrency=min(cnt, 256), zero_guess=ZG)
        tuned[(nlon, nlat)] = t

    def run(layout):
        solvers = []
        for (nlon, nlat), p in zip(sizes, probs):
            t = layout.get((nlon, nlat)) if layout else None
            solvers.append(ftgcr.Solver(p.D, p.mu, k=K, tol=TOL, precision="mixed", tiles=t["tiles"] if t else 0,
                                        rounds=t["rounds"] if t else "auto", zero_guess=ZG))
        xs = [torch.zeros_like(R) for R in Rs]
        alone_ms, alone_x = [], []
        for s, R, x in zip(solvers, Rs, xs):
            s.solve_async(R, x, stream=stream)  # warm
            x.zero_()
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record(stream)
            s.solve_async(R, x, stream=stream)
            b.record(stream)
            torch.cuda.synchronize()
            alone_ms.append(a.elapsed_time(b))
            alone_x.append(x.clone())
        times = []
        for rep in range(reps + 1):
            for x in xs:
                x.zero_()
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record(stream)
            ftgcr.solve_batch(solvers, Rs, xs, stream=stream)
            b.record(stream)
            torch.cuda.synchronize()
            if rep:
                times.append(a.elapsed_time(b))
        same = all(bool(torch.equal(x, y)) for x, y in zip(xs, alone_x))
        steps = sum(s.stats()["steps"] for s in solvers)
        # the same launch captured into a CUDA graph and replayed
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            ftgcr.solve_batch(solvers, Rs, xs, stream=torch.cuda.current_stream())
        gtimes = []
        for rep in range(reps + 1):
            for x in xs:
                x.zero_()
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record(stream)
            g.replay()
            b.record(stream)
            torch.cuda.synchronize()
            if rep:
                gtimes.append(a.elapsed_time(b))
        gsame = all(bool(torch.equal(x, y)) for x, y in zip(xs, alone_x))
        del g
        for s in solvers:
            s.close()
        ms = float(np.median(times))
        return {"launch_ms": ms, "solves_per_s": n * 1e3 / ms, "iters_per_s": steps * 1e3 / ms,
                "sequential_ms": float(np.sum(alone_ms)), "speedup_vs_sequential": float(np.sum(alone_ms)) / ms,
                "bitwise_equal_to_alone": same, "graph_replay_ms": float(np.median(gtimes)),
                "graph_bitwise_equal_to_alone": gsame}

    default = run(None)
    auto = run(tuned)
    out = {"solves": n, "sizes": "U{128x64,256x128,512x256,1024x512}", "seed": seed, "precision": "mixed",
           "tiles": "autotuned (ftgcr_tune per size, concurrency = solves of that size)"}
    out.update(auto)
    out["autotuner"] = {f"{a}x{b}": {"tiles": t["tiles"], "rounds": t["rounds"], "default_tiles": t["default_tiles"],
                                     "tuned_ms": t["ms"], "default_ms": t["default_ms"], "candidates": t["candidates"]}
                        for (a, b), t in tuned.items()}
    out["default_tiles"] = {k: default[k] for k in ("launch_ms", "solves_per_s", "graph_replay_ms",
                                                    "bitwise_equal_to_alone")}
    return out


def bench_serving(torch, ftgcr, dev, n_req=2000, load=0.8, seed=7, hills_per_size=4, n_cap=300,
                  sweep_loads=(0.5, 1.0, 1.2), n_sweep=400, tune_concurrency=16, n_tuned=600, n_limited=1000,
                  n_isolated=400):
    """Open-loop serving: n_req requests with Poisson arrivals at `load` x the
    measured capacity; sizes U{256x128, 512x256, 1024x512, 2048x1024}, mixed
    precision, hills drawn per problem, 1% carrying one bit flip.  Right-hand
    side and solution in pinned host memory, coefficients resident on the
    device and identified by a key (a model's operator is fixed across its time
    steps, so pooled handles keep their set-up); latency = arrival -> solution
    on the host.  Then shorter runs at other fractions of the capacity
    (load_sweep).  Beside it, a shorter run with row bands per size from the
    autotuner (ftgcr_tune at `tune_concurrency` solves per launch, passed with
    each request): taller bands raise throughput a little but lengthen a lone
    request's solve, so the default bands stay the headline.  And a run with
    the admission limit (ftgcr_server_set_max_points) at 1.1 x the largest
    request's points, at 0.8 x its own measured capacity.  And `isolated`: the
    first n_isolated requests served one at a time, whose p99 / p50 is what
    the size mix alone gives with no contention."""
    import threading

    sizes = [(256, 128), (512, 256), (1024, 512), (2048, 1024)]
    probs = []
    for si, (nlon, nlat) in enumerate(sizes):
        for hq in range(hills_per_size):
            p = inputs.hill_problem(nlon, nlat, **inputs.random_hill(seed * 100 + si * 10 + hq))
            probs.append((p, torch.from_numpy(p.D).to(dev), torch.from_numpy(p.R).pin_memory()))
    g = inputs.SplitMix64(seed)
    reqs = []
    for i in range(max(n_req, n_cap)):
        pi = g.below(len(sizes)) * hills_per_size + g.below(hills_per_size)
        faults = ()
        if g.below(100) == 0:
            N = probs[pi][0].R.size
            faults = [inputs.sweep_flip(seed, i, 10, N, nbits=32, vecs=("r", "ap"))]
        reqs.append((pi, faults))
    pool_lock = threading.Lock()
    xpool = {}  # pinned solution buffers per problem shape, reused

    def take_x(shape):
        with pool_lock:
            lst = xpool.setdefault(shape, [])
            x = lst.pop() if lst else None
        if x is None:
            x = torch.zeros(shape, dtype=torch.float64).pin_memory()
        else:
            x.zero_()
        return x

    def give_x(x):
        with pool_lock:
            xpool.setdefault(tuple(x.shape), []).append(x)

    tuned = {}
    for si, (nlon, nlat) in enumerate(sizes):
        p0 = probs[si * hills_per_size][0]
        tuned[(nlon, nlat)] = ftgcr.tune(p0.D, p0.mu, k=K, tol=TOL, precision="mixed", concurrency=tune_concurrency,
                                         zero_guess=ZG)
    tiling = {}  # the layout the current run submits with, per shape

    def layout(p):
        t = tiling.get((p.nlon, p.nlat))
        return (t["tiles"], t["rounds"]) if t else (0, "auto")

    def submit_p(srv, pi, faults=()):
        p, Dd, Rh = probs[pi]
        x = take_x(tuple(p.R.shape))
        tl, rd = layout(p)
        return srv.submit(Dd, p.mu, Rh, x, k=K, tol=TOL, precision="mixed", faults=faults, coeff_key=pi + 1, zero_guess=ZG,
                          tiles=tl, rounds=rd), x

    def submit(srv, i):
        pi, faults = reqs[i]
        return submit_p(srv, pi, faults)

    def isolated(srv, n):
        """The same request stream served one request at a time (each waits
        for the previous to finish): latency with no contention at all, the
        floor the size mix itself sets under p50 and p99."""
        lat, by = [], {}
        for i in range(n):
            t0 = time.perf_counter()
            t, x = submit(srv, i)
            r = srv.next(timeout=30)
            dt = 1e3 * (time.perf_counter() - t0)
            give_x(x)
            if r is None or r[0] != t:
                return None
            p = probs[reqs[i][0]][0]
            lat.append(dt)
            by.setdefault(f"{p.nlon}x{p.nlat}", []).append(dt)
        lat = np.array(lat)
        p50, p99 = float(np.percentile(lat, 50)), float(np.percentile(lat, 99))
        return {"requests": n, "p50_ms": p50, "p99_ms": p99, "p99_over_p50": p99 / p50,
                "median_ms_by_size": {k: float(np.median(v)) for k, v in sorted(by.items())}}

    def serve(n_req, sweep_loads, max_points=0, n_isolated=0):
        with ftgcr.Server(max_slots=64, epoch_rounds=24) as srv:
            srv.set_max_points(max_points)
            warm = [submit_p(srv, pi) for pi in range(len(probs))]  # a handle set up for every problem
            for _ in warm:
                srv.next()
            for _, x in warm:
                give_x(x)
            # capacity: closed loop, everything queued at once
            t0 = time.perf_counter()
            xs0 = [submit(srv, i) for i in range(n_cap)]
            for _ in range(n_cap):
                srv.next()
            cap = n_cap / (time.perf_counter() - t0)
            for _, x in xs0:
                give_x(x)
            def open_loop(ld, n, seed_arr, keep_sample):
                arr = inputs.poisson_arrivals(seed_arr, n, ld * cap)
                sample = set(range(0, n, max(1, n // 8))) if keep_sample else set()  # kept for the equality check
                t_arr, xs, kept, lat = {}, {}, {}, []
                lock = threading.Lock()
                start = time.perf_counter()

                def producer():
                    for i in range(n):
                        d = start + arr[i] - time.perf_counter()
                        if d > 0:
                            time.sleep(d)
                        ta = time.perf_counter()
                        t, x = submit(srv, i)
                        with lock:
                            t_arr[t] = ta
                            xs[t] = (i, x)

                th = threading.Thread(target=producer)
                th.start()
                done, results = 0, {}
                while done < n:
                    r = srv.next(timeout=30)
                    if r is None:
                        break
                    now = time.perf_counter()
                    t, st, ss = r
                    with lock:
                        ta = t_arr.get(t)
                    while ta is None:  # the producer has not recorded it yet
                        time.sleep(1e-5)
                        with lock:
                            ta = t_arr.get(t)
                    lat.append(now - ta)
                    results[t] = (st, ss)
                    with lock:
                        i, x = xs.pop(t)
                    if i in sample:
                        kept[t] = (i, x.numpy().copy(), ss["tiles"])
                    give_x(x)
                    done += 1
                th.join()
                wall = time.perf_counter() - start
                return results, kept, 1e3 * np.array(lat), wall

            iso = isolated(srv, n_isolated) if n_isolated else None
            results, kept, lat_ms, wall = open_loop(load, n_req, seed, True)
            info = srv.info()
            # latency against offered load: shorter runs at other fractions of capacity
            sweep = []
            for q, ld in enumerate(sweep_loads):
                r2, _, l2, w2 = open_loop(ld, n_sweep, seed + 1 + q, False)
                sweep.append({"load": ld, "requests": n_sweep, "offered_per_s": ld * cap, "achieved_solves_per_s": n_sweep / w2,
                              "completed_ok": sum(1 for st, _ in r2.values() if st == 0),
                              "p50_ms": float(np.percentile(l2, 50)), "p99_ms": float(np.percentile(l2, 99))})
        # a sample of served results against the same request solved alone
        same = True
        for t in sorted(kept):
            i, x, tl = kept[t]  # the bands the server reported for the request
            pi, faults = reqs[i]
            p = probs[pi][0]
            _, rd = layout(p)
            with ftgcr.Solver(p.D, p.mu, k=K, tol=TOL, precision="mixed", tiles=tl, rounds=rd, zero_guess=ZG) as s:
                xa = np.zeros_like(p.R)
                s.solve(p.R, xa, faults=faults)
            same = same and np.array_equal(x, xa)
        ok = sum(1 for st, _ in results.values() if st == 0)
        return {"requests": n_req, "completed_ok": ok, "load": load, "capacity_solves_per_s": cap,
                "offered_per_s": load * cap, "achieved_solves_per_s": n_req / wall,
                "latency_ms": {"p50": float(np.percentile(lat_ms, 50)), "p99": float(np.percentile(lat_ms, 99)),
                               "max": float(lat_ms.max())},
                "faulty_requests": sum(1 for _, f in reqs[:n_req] if f), "epochs": info["epochs"],
                "handles": info["handles"], "sizes": "U{256x128,512x256,1024x512,2048x1024}", "precision": "mixed",
                "io": "rhs and x in pinned host memory, D resident with a coefficient key",
                "bitwise_equal_to_alone_sample": same, "load_sweep": sweep,
                **({"isolated": iso} if n_isolated else {})}

    out = serve(n_req, sweep_loads, n_isolated=n_isolated)
    out["tiles"] = "default (ftgcr_create's own choice)"
    tiling.update(tuned)
    d = serve(n_tuned, ())
    out["autotuned_tiles"] = {k: d[k] for k in ("requests", "completed_ok", "capacity_solves_per_s",
                                                "achieved_solves_per_s", "latency_ms",
                                                "bitwise_equal_to_alone_sample")}
    out["autotuned_tiles"]["tiles"] = {f"{a}x{b}": {"tiles": t["tiles"], "rounds": t["rounds"],
                                                    "default_tiles": t["default_tiles"]} for (a, b), t in tuned.items()}
    out["autotuned_tiles"]["tuned_for"] = f"ftgcr_tune at {tune_concurrency} solves per launch"
    tiling.clear()
    lim = int(1.1 * max(a * b for a, b in sizes))
    d = serve(n_limited, (), max_points=lim)
    out["max_points_limit"] = {k: d[k] for k in ("requests", "completed_ok", "capacity_solves_per_s",
                                                 "achieved_solves_per_s", "latency_ms",
                                                 "bitwise_equal_to_alone_sample")}
    out["max_points_limit"]["max_points"] = lim
    return out


# ------------------------------------------------------------------ GPU arm
def run_ours(args):
    import torch

    from paper_2103_07210_gb300 import ftgcr

    ws, rank, local = dist_env()
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    if ws > 1:
        import torch.distributed as dist

        dist.init_process_group("nccl", device_id=dev)

    def barrier():
        if ws > 1:
            import torch.distributed as dist

            dist.barrier()
        torch.cuda.synchronize()

    p = inputs.hill_problem(NLON, NLAT)
    R = torch.from_numpy(p.R).to(dev)
    stream = torch.cuda.current_stream()
    flush = torch.empty(256 << 20, dtype=torch.uint8, device=dev)

    def measure(precision, nsteps, nwarm):
        s = ftgcr.Solver(p.D, p.mu, k=K, tol=TOL, precision=precision, zero_guess=ZG)
        xs = [torch.zeros_like(R) for _ in range(2)]
        for i in range(nwarm):
            xs[0].zero_()
            s.solve_async(R, xs[0], stream=stream)
        torch.cuda.synchronize()
        ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(nsteps)]
        barrier()
        for i in range(nsteps):
            x = xs[i % 2]
            x.zero_()
            flush.fill_(i & 0xFF)  # evict L2 between timed steps
            ev[i][0].record(stream)
            s.solve_async(R, x, stream=stream)
            ev[i][1].record(stream)
        barrier()
        ms = np.array([a.elapsed_time(b) for a, b in ev])
        info = s.stats()
        return s, ms, info, xs[(nsteps - 1) % 2]

    with ClockSampler(local) as clk:
        s_mx, ms_mx, info_mx, x_mx = measure("mixed", args.steps, args.warmup)
    clocks = clk.summary()
    s64, ms_64, info_64, x_64 = measure("fp64", max(3, args.steps // 4), max(1, args.warmup // 2))
    x_mx, x_64 = x_mx.cpu().numpy(), x_64.cpu().numpy()

    # the parity configuration: the same mixed solve to tol 1e-13, where its
    # solution must match the FP64 oracle's to 1e-10 relative (at the
    # headline's tol 1e-10 both sides only bound the residual, and their
    # solutions may differ by up to cond x tol)
    PAR_TOL = 1e-13
    with ftgcr.Solver(p.D, p.mu, k=K, tol=PAR_TOL, precision="mixed", zero_guess=ZG) as s_par:
        x_par = torch.zeros_like(R)
        for _ in range(args.warmup):
            x_par.zero_()
            s_par.solve_async(R, x_par, stream=stream)
        ms_par = []
        for i in range(max(5, args.steps // 2)):
            x_par.zero_()
            flush.fill_(i & 0xFF)
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record(stream)
            s_par.solve_async(R, x_par, stream=stream)
            b.record(stream)
            torch.cuda.synchronize()
            ms_par.append(a.elapsed_time(b))
        info_par = s_par.stats()
        x_par = x_par.cpu().numpy()

    # max over ranks
    tot = float(ms_mx.sum())
    tot = max_over_ranks(tot, dev)
    ms_step = tot / args.steps
    value = ws * 1e3 / ms_step

    # e2e: host buffers through the C ABI (blocking ftgcr_solve), copies inside
    Rh = torch.from_numpy(p.R).pin_memory()
    xh = torch.zeros(NLAT, NLON, dtype=torch.float64).pin_memory()
    for _ in range(2):
        xh.zero_()
        s_mx.solve(Rh, xh)
    e2e = []
    for _ in range(args.steps):
        xh.zero_()
        flush.fill_(1)
        torch.cuda.synchronize()
        t = time.perf_counter()
        s_mx.solve(Rh, xh)
        e2e.append(time.perf_counter() - t)
    e2e_blocking = ws / float(np.mean(e2e))

    # e2e, pipelined: the same host-array solves enqueued with
    # ftgcr_solve_host_async on NH handles taken in turn on two streams, so one
    # step's copies (R and x0 in from pinned memory, x out) overlap the
    # previous step's solve.  Every step still copies its inputs in and its
    # solution out.  The NH handles' Krylov state (about 50 MB each) exceeds
    # the 129 MB L2, so no step finds the previous use of its data in L2.
    NH = 4
    hs = [s_mx] + [ftgcr.Solver(p.D, p.mu, k=K, tol=TOL, precision="mixed", zero_guess=ZG) for _ in range(NH - 1)]
    xhs = [torch.zeros(NLAT, NLON, dtype=torch.float64).pin_memory() for _ in range(NH)]
    e2e_streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    e2e_ev = [torch.cuda.Event() for _ in range(NH)]

    def pipeline(nsteps):
        for i in range(nsteps):
            b = i % NH
            e2e_ev[b].synchronize()  # this handle's previous solve (and copy out) has ended
            xhs[b].zero_()
            st = e2e_streams[i % 2]
            hs[b].solve_host_async(Rh, xhs[b], stream=st)
            e2e_ev[b].record(st)

    pipeline(NH)
    torch.cuda.synchronize()
    t = time.perf_counter()
    pipeline(args.steps)
    torch.cuda.synchronize()
    e2e_val = ws * args.steps / (time.perf_counter() - t)
    e2e_ok = all(h.stats()["status"] == ftgcr.OK for h in hs) and \
        all(bool(torch.equal(xh_, xhs[0])) for xh_ in xhs[1:])
    for h in hs[1:]:
        h.close()

    peak, peak_kind = read_peaks()
    bytes_launch = algorithmic_bytes(info_mx["steps"], info_mx["outer"])
    kern_ms = float(np.mean(ms_mx))
    achieved = bytes_launch / (kern_ms * 1e-3) / 1e9
    traffic = NCU_TRAFFIC["bytes_per_launch"] if NCU_TRAFFIC["sources_sha256"] == sources_hash() else None

    # the FP64 path against the two ceilings measured in this run: its
    # algorithmic flops, about (32 + 6m) per point and step with m = (k+1)/2
    # directions on average (stencil 10, line solve 8, axpy and norm 6, the
    # dots and recurrences 6m), over the FP64 FMA rate; its algorithmic bytes,
    # 21.5 FP64 vectors per step, over the copy rate
    peaks_run = measure_peaks_in_run(torch, ftgcr, dev) if ws == 1 else None
    t64 = float(np.mean(ms_64)) * 1e-3
    fl64 = info_64["steps"] * (32 + 6 * (K + 1) / 2) * NLON * NLAT
    by64 = algorithmic_bytes(info_64["steps"], 0, s=8, mixed=False)
    fp64_roof = None
    if peaks_run:
        fp64_roof = {"bound": "alu", "achieved": fl64 / t64 / 1e12, "peak": peaks_run["fp64_fma_tflops"],
                     "unit": "TFLOP/s", "frac": fl64 / t64 / 1e12 / peaks_run["fp64_fma_tflops"],
                     "peak_kind": "measured in this run (FP64 FMA probe)", "flops_per_launch": fl64,
                     "hbm_achieved_gbs": by64 / t64 / 1e9, "hbm_frac_of_copy": by64 / t64 / 1e9 / peaks_run["copy_gbs"]}

    # correctness of the timed result, by a property that holds at any size
    res_rel = info_mx["res_final_true"] / info_mx["norm_R"]

    if rank == 0:
        line = {
            "metric": METRIC, "value": value, "unit": "solves/s", "n_gpus": ws, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": ms_step, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f32+f64", "data": "synthetic",
            "config": {"workload": WORKLOAD, "nlon": NLON, "nlat": NLAT, "k": K, "tol": TOL,
                       "precision": "mixed (FP32 inner, FP64 dots/norm/refinement)",
                       "l2": "flushed between timed steps (256 MB write)", "tiles": info_mx["tiles"],
                       "x0": "zero, declared (FTGCR_FLAG_ZERO_GUESS)" if ZG else "zero"},
            "iters_per_s": info_mx["steps"] * value, "inner_steps_per_solve": info_mx["steps"],
            "refinement_sweeps": info_mx["outer"],
            "latency_ms": {"p50": float(np.percentile(ms_mx, 50)), "p99": float(np.percentile(ms_mx, 99))},
            "fp64_path": {"solves_per_s": 1e3 / float(np.mean(ms_64)),
                          "iters_per_s": info_64["steps"] * 1e3 / float(np.mean(ms_64)),
                          "steps_per_solve": info_64["steps"],
                          "roofline": fp64_roof},
            "mixed_over_fp64": float(np.mean(ms_64)) / float(np.mean(ms_mx)),
            "residual_rel": res_rel,
            "parity_config": {"tol": PAR_TOL, "ms": float(np.median(ms_par)),
                              "solves_per_s": 1e3 / float(np.median(ms_par)), "inner_steps": info_par["steps"],
                              "refinement_sweeps": info_par["outer"], "converged": info_par["converged"],
                              "residual_rel": info_par["res_final_true"] / info_par["norm_R"]},
            # the 1024x512 launch's working set stays in the 129 MB L2 (ncu:
            # DRAM traffic a few % of the algorithmic bytes), so its bound is
            # L2 and round latency; the fraction is still taken against the
            # measured HBM copy rate.  roofline_hbm below is the HBM figure.
            "roofline": {"bound": "l2", "achieved": achieved, "peak": peak, "unit": "GB/s",
                         "frac": achieved / peak, "traffic": traffic, "peak_kind": peak_kind + " HBM copy",
                         "dram_over_algorithmic": (traffic / bytes_launch) if traffic else None,
                         "kernel": "k_ftgcr_band<float>",
                         "algorithmic_bytes_per_launch": bytes_launch},
            "e2e": {"value": e2e_val, "unit": "solves/s", "h2d_bytes_per_step": (1 if ZG else 2) * 8 * NLON * NLAT,
                    "pipelined": f"ftgcr_solve_host_async, {NH} handles in turn on 2 streams (state > L2)",
                    "results_ok": e2e_ok, "blocking_value": e2e_blocking,
                    "d2h_bytes_per_step": 8 * NLON * NLAT + 2 * 4096},
            "gpu_launches": 2 * args.steps,
            "peaks_in_run": peaks_run,
            "clocks": clocks,
        }
        large_x = {}
        if not args.no_large and ws == 1:
            line["large_grids"] = bench_large(torch, ftgcr, dev, flush, keep=large_x)
            big = line["large_grids"].get("4096x2048")
            if big:
                nb = big["algorithmic_bytes"]
                line["roofline_hbm"] = {
                    "bound": "hbm", "achieved": big["achieved_gbs"], "peak": peak, "unit": "GB/s",
                    "frac": big["frac"], "traffic": big["traffic"], "peak_kind": peak_kind + " HBM copy",
                    "dram_over_algorithmic": (big["traffic"] / nb) if big["traffic"] else None,
                    "kernel": "k_ftgcr_persistent<float> (4096x2048 mixed solve, HBM-resident)",
                    "algorithmic_bytes_per_launch": nb, "ms": big["ms"]}
        if not args.no_ksweep and ws == 1:
            line["k_sweep"] = bench_ksweep(torch, ftgcr, dev, flush)
        if not args.no_steady and ws == 1:
            line["steady_state"] = bench_steady(torch, ftgcr, dev, flush)
        if not args.no_batch and ws == 1:
            line["batch"] = bench_batch(torch, ftgcr, dev)
        if not args.no_serving and ws == 1:
            line["serving"] = bench_serving(torch, ftgcr, dev, n_req=args.serving_requests, load=args.serving_load)
        if not args.no_oracle_check and ws == 1:
            res = {"headline": ((NLON, NLAT, K, TOL), x_mx), "fp64_path": ((NLON, NLAT, K, TOL), x_64),
                   "parity_config": ((NLON, NLAT, K, PAR_TOL), x_par)}
            for (a, b), xl in large_x.items():
                res[f"large_{a}x{b}"] = ((a, b, K, TOL), xl)
            ev = errors_vs_oracle(res)
            line["err_vs_oracle"] = ev["headline"]["err_vs_oracle"]
            line["fp64_path"]["err_vs_oracle"] = ev["fp64_path"]["err_vs_oracle"]
            line["parity_config"]["err_vs_oracle"] = ev["parity_config"]["err_vs_oracle"]
            for (a, b) in large_x:
                line["large_grids"][f"{a}x{b}"]["err_vs_oracle"] = ev[f"large_{a}x{b}"]["err_vs_oracle"]
            line["oracle_check"] = ev
        if not args.no_cpu_baseline and ws == 1:
            cb = oracle_throughput()
            line["cpu_baseline"] = {"value": cb["value"], "unit": "solves/s", "cores": cb["cores"], "kind": "oracle",
                                    "sample": f"{cb['n']} FP64 oracle solves of the {NLON}x{NLAT} problem, "
                                              f"one process per core, {cb['wall']:.1f} s",
                                    "latency_s_per_solve_one_core": cb["latency_s"],
                                    "latency_s_per_step_one_core": cb["latency_s"] / max(1, cb["steps"]),
                                    "steps_per_s": cb["steps_per_s"], "physical_cores": physical_cores()}
        print(json.dumps(line))
    if ws > 1:
        import torch.distributed as dist

        dist.destroy_process_group()
    return 0


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-batch", action="store_true", help="skip the 128-solve batched launch")
    ap.add_argument("--no-large", action="store_true", help="skip the 2048x1024 and 4096x2048 solves")
    ap.add_argument("--no-ksweep", action="store_true", help="skip the k sweep (protected vs unprotected)")
    ap.add_argument("--no-serving", action="store_true", help="skip the open-loop serving run")
    ap.add_argument("--no-steady", action="store_true", help="skip the steady-state step window (mu = 0)")
    ap.add_argument("--no-oracle-check", action="store_true",
                    help="skip the per-result comparison with the FP64 oracle (after the timed region)")
    ap.add_argument("--serving-requests", type=int, default=2000)
    ap.add_argument("--serving-load", type=float, default=0.8, help="arrival rate / measured capacity")
    args = ap.parse_args()
    if args.warmup < 3:
        args.warmup = 3
    if args.impl == "reference":
        return run_reference(args)
    return run_ours(args)


if __name__ == "__main__":
    sys.exit(main())
