"""Benchmark of the PDMCF hot path on GB300: PDHG iterations per second.

Default workload (one GPU): the large single solve, n = 10^4 nodes, m = 10^5 edges (directed
ring plus 9 random out-edges per node), capacities lognormal(0, 0.5), power utility
w s^0.5 with w ~ U[0.5, 1.5]; F is 10^4 x 10^5 (10^9 variables) in FP32. A step is one PDHG
iteration (edge phase, node phase, scalar tail; every k_check-th iteration also the
residual check), launched through the C ABI on torch's current stream.

Printed JSON line (rank 0):
  value     iterations/s of the whole job (sum over ranks / max time), inputs resident in HBM,
            by the launches that mcf_solve_timed puts events around (one per phase)
  solve     the same number of iterations by one plain mcf_solve on this rank, whose automatic
            kernels are others on shorter rows (the resident iteration, the flat node phase);
            on the default workload they are the same launches
  e2e       the same metric through the public API with host buffers: problem creation
            (host -> device copies), the solve, and the read-back of T inside the timed region
  roofline  the dominant kernel: algorithmic bytes per launch / its mean CUDA-event duration,
            against the measured HBM copy bandwidth
  cpu_baseline  the FP64 CPU oracle timed on a bounded sample (the same recipe at n = 1000),
            scaled to this workload by the ratio of n m
  --impl reference  times that oracle alone as the reference arm.
"""
from __future__ import annotations

import os

os.environ.setdefault("OMP_NUM_THREADS", "1")
os.environ.setdefault("OPENBLAS_NUM_THREADS", "1")
os.environ.setdefault("MKL_NUM_THREADS", "1")

import argparse  # noqa: E402
import hashlib  # noqa: E402
import json  # noqa: E402
import math  # noqa: E402
import statistics  # noqa: E402
import subprocess  # noqa: E402
import sys  # noqa: E402
import tempfile  # noqa: E402
import time  # noqa: E402

import numpy as np  # noqa: E402

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

from paper_2501_17996_gb300 import instances as I  # noqa: E402

METRIC = "PDHG iters/s, HBM GB/s vs peak; served p50/p99 solve latency @1e-4 KKT"

WORKLOADS = {
    "large": dict(factory=lambda seed: I.large(seed), sample=lambda seed: I.large_slice(seed),
                  desc="n=10000, m=100000 (ring + 9 random out-edges per node), "
                       "c~lognormal(0,0.5), u = w s^0.5, w~U[0.5,1.5]"),
    # profiling case: the large per-edge vector length (n = 10^4, same kernel shape) with
    # out-degree 2, so one capture holds ~4 GB on the device
    "prof": dict(factory=lambda seed: I.ring_random_instance(10000, 2, seed, "lognormal", "pow",
                                                             gamma=0.5, name="prof"),
                 sample=lambda seed: I.large_slice(seed),
                 desc="n=10000, m=20000 (ring + 1 random out-edge per node), large recipe"),
    "batched": dict(factory=None, sample=None, desc="64 uneven instances (see run_batched)"),
    "served": dict(factory=None, sample=None, desc="Poisson request stream (see run_served)"),
    "mid": dict(factory=lambda seed: I.mid(seed), sample=lambda seed: I.mid(seed),
                desc="n=100, m=1000 (ring + 9 random out-edges per node), c~U[1,10], "
                     "u = w log s, w~U[0.5,1.5]"),
    # the paper's own family (Sec. 3.1); sizes come from --knn-n / --knn-q (set in main)
    "knn": dict(factory=None, sample=None, desc=None),
}


def knn_connected(n: int, q: int, seed: int):
    """The kNN instance of the first seed >= `seed` whose graph is strongly connected."""
    import scipy.sparse as sp
    from scipy.sparse.csgraph import connected_components

    for s in range(seed, seed + 100):
        inst = I.knn(n, q, s)
        g = sp.coo_matrix((np.ones(inst.m), (inst.tail, inst.head)), shape=(n, n))
        if connected_components(g, directed=True, connection="strong")[0] == 1:
            return inst
    raise RuntimeError(f"no strongly connected kNN graph for n={n}, q={q}")


def peaks():
    try:
        d = json.load(open(os.path.join(ROOT, "MEASURED_PEAKS.json")))
        return float(d["hbm_gbs"]), "measured"
    except Exception:
        return 6800.0, "fallback"


def kernel_source_hash() -> str:
    """Hash of the per-iteration kernels' sources (their definitions and instantiation
    units) with comments and whitespace removed: it changes when the kernels' code changes,
    not when their comments or the host code do."""
    import re

    h = hashlib.sha256()
    csrc = os.path.join(ROOT, "paper_2501_17996_gb300", "csrc")
    kernel_files = ("pdmcf_device.cuh", "pdmcf_types.h", "pdmcf_kernels.h")
    for f in sorted(os.listdir(csrc)):
        if f in kernel_files or (f.startswith("pdmcf_kernels_") and f.endswith(".cu")):
            text = open(os.path.join(csrc, f), encoding="utf-8").read()
            text = re.sub(r"/\*.*?\*/", " ", text, flags=re.S)
            text = re.sub(r"//[^\n]*", " ", text)
            h.update(f.encode() + b"\0" + " ".join(text.split()).encode())
    return h.hexdigest()[:16]


def algorithmic_bytes(n: int, m: int, s_f: int, s_p: int = 4, kind: int = 0) -> dict:
    """Bytes the method must move per launch (each array touched once):
    edge:   read F^{k-1/2}, write F^{k+1/2} (2 s_F n m), read Y once (s_P n^2), 16 m of
            incidence, capacity and mu;
    node:   read F^{k+1/2} once (s_F n m), read Y, W, P and write Y, P (5 s_P n^2), 4(m+2n);
    check:  read F^{k-1/2} once (s_F n m), read Y, U', Y^ once (3 s_P n^2), 12 m;
    iteration floor: 2 s_F n m + 3 s_P n^2 (read and write F once; read Y, W, write Y).
    `design_extra` is what this design adds on top: kinds 1 and 2 write the per-head in-sums
    in the edge phase and read them in the node phase (s_P n^2 each). The roofline uses the
    method's bytes only."""
    nm, n2 = float(n) * m, float(n) * n
    pin = s_p * n2 if kind in (1, 2) else 0.0
    return {
        "edge": 2 * s_f * nm + s_p * n2 + 16 * m,
        "node": s_f * nm + 5 * s_p * n2 + 4 * (m + 2 * n),
        "check": s_f * nm + 3 * s_p * n2 + 12 * m,
        "scalar": 0.0,
        "iteration_floor": 2 * s_f * nm + 3 * s_p * n2,
        "design_extra": {"edge": pin, "node": pin},
    }


# ------------------------------------------------------------------ clocks sampler

class ClockSampler:
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, device: int):
        self.device = device
        self.proc = None
        self.path = None

    def __enter__(self):
        try:
            fd, self.path = tempfile.mkstemp(suffix=".csv")
            os.close(fd)
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
                 "-i", str(self.device), "-lms", "200"],
                stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
            time.sleep(0.3)
        except Exception:
            self.proc = None
        return self

    def __exit__(self, *exc):
        if self.proc is not None:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except Exception:
                self.proc.kill()

    def summary(self) -> dict:
        if not self.path or not os.path.exists(self.path):
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["unavailable"]}
        sm, smax, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in open(self.path):
            parts = [p.strip() for p in line.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                smax.append(float(parts[2]))
            except ValueError:
                continue
            for nm_, v in zip(names, parts[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(nm_)
        os.unlink(self.path)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["no samples"]}
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(smax),
                "reasons": sorted(reasons), "samples": len(sm)}


# ------------------------------------------------------------------ CPU oracle timing

def oracle_iters_per_s(sample, k_check: int, steps: int, warmup: int):
    """Time `steps` oracle iterations on the sample instance (cold start each call):
    t(warmup + steps) - t(warmup) so start-up work cancels."""
    from oracle import pdmcf as O

    def run(k):
        t0 = time.perf_counter()
        O.pdmcf(sample.n, sample.tail, sample.head, sample.cap, sample.kind, sample.w,
                sample.gamma, stop_mode="none", max_iters=k, k_check=k_check)
        return time.perf_counter() - t0

    t_w = run(warmup) if warmup > 0 else 0.0
    t_all = run(warmup + steps)
    dt = max(t_all - t_w, 1e-9)
    return steps / dt, dt


def host_description() -> str:
    """nproc and the CPU model of this host (the oracle's timing context)."""
    model = ""
    try:
        out = subprocess.run(["lscpu"], capture_output=True, text=True, timeout=10).stdout
        for line in out.splitlines():
            if line.lower().startswith("model name:"):
                model = line.split(":", 1)[1].strip()
                break
    except (OSError, subprocess.SubprocessError):
        pass
    try:
        for line in ([] if model else open("/proc/cpuinfo")):
            key = line.split(":")[0].strip().lower()
            if key in ("model name", "cpu model", "hardware") and ":" in line:
                model = line.split(":", 1)[1].strip()
                break
    except OSError:
        pass
    if not model:
        import platform

        model = platform.machine()
    return f"{os.cpu_count()} host cores, {model}"


def oracle_parallel_iters_per_s(sample, steps: int, warmup: int, workers: int):
    """Time `steps` iterations of the oracle spread over `workers` processes
    (oracle.parallel, spawn start: safe after CUDA has been initialised)."""
    from oracle.parallel import ParallelPDMCF

    with ParallelPDMCF(sample, workers=workers) as pp:
        pp.run(max(warmup, 1))
        t0 = time.perf_counter()
        pp.run(steps)
        dt = max(time.perf_counter() - t0, 1e-9)
    return steps / dt, dt


def cpu_baseline(wl, inst, seed, k_check, steps=20, warmup=1):
    """The FP64 oracle on the host cores, on a bounded sample: the same recipe at the
    sample size (the n = 1000 slice for the large workload). The oracle's work per iteration
    is proportional to n m (dense F, one sort per column), so the sample's rate is scaled by
    the ratio of n m to the full workload. value/cores: all host cores (oracle.parallel, the
    paper's "PDMCF (CPU)" configuration); single_core: the single-threaded oracle as it is."""
    sample = wl["sample"](seed)
    scale = (sample.n * sample.m) / float(inst.n * inst.m)
    ips1, dt1 = oracle_iters_per_s(sample, k_check, steps, warmup)
    cores = os.cpu_count() or 1
    ipsn, dtn = oracle_parallel_iters_per_s(sample, steps, warmup, cores)
    return {
        "value": ipsn * scale,
        "unit": "iters/s",
        "cores": cores,
        "kind": "oracle",
        "host": host_description(),
        "sample": (f"{steps} FP64 oracle iterations on the same recipe at n={sample.n}, "
                   f"m={sample.m}, measured at that size and scaled by the n m ratio "
                   f"{scale:.3g} to the full workload (the oracle's per-iteration work is "
                   f"proportional to n m): {cores} worker processes (oracle.parallel) "
                   f"{ipsn:.3g} iters/s at the sample size ({dtn:.1f} s)"),
        "measured_at_sample_size": {"all_cores_iters_per_s": ipsn, "single_core_iters_per_s": ips1,
                                    "n": sample.n, "m": sample.m},
        "single_core": {"value": ips1 * scale, "unit": "iters/s", "cores": 1,
                        "sample": f"single-threaded oracle.pdmcf, {steps} iterations "
                                  f"({dt1:.1f} s) at n={sample.n}, m={sample.m}, scaled the same way"},
    }


# ------------------------------------------------------------------ arms

def run_reference(args, rank, world):
    if rank != 0:
        return
    wl = WORKLOADS[args.workload]
    if args.workload == "knn":
        full = wl["factory"](args.seed)
        inst_n, inst_m = full.n, full.m
    else:
        inst_n, inst_m = {"large": (10000, 100000), "prof": (10000, 20000), "mid": (100, 1000)}[args.workload]
    sample = wl["sample"](args.seed)
    if args.workload == "large" and args.steps + args.warmup > 60:
        sample = I.large(args.seed, n=500)
    ips, dt = oracle_iters_per_s(sample, args.k_check, args.steps, args.warmup)
    scale = (sample.n * sample.m) / float(inst_n * inst_m)
    value = ips * scale
    line = {
        "impl": "reference",
        "metric": METRIC, "value": value, "unit": "iters/s", "n_gpus": args.gpus,
        # a step is one oracle iteration on the sample; value is that rate scaled to the
        # full workload by the n m ratio (stated in config)
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * dt / args.steps,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
        "data": "synthetic",
        "config": {"workload": f"{args.workload}: {wl['desc']}", "n": inst_n, "m": inst_m,
                   "sample": {"n": sample.n, "m": sample.m, "iters_per_s_at_sample": ips,
                              "scale_to_full_by_nm_ratio": scale}},
        "cpu_baseline": {"value": value, "unit": "iters/s", "cores": 1, "kind": "oracle",
                         "host": host_description(),
                         "sample": (f"each step one FP64 oracle iteration on the same recipe at "
                                    f"n={sample.n}, m={sample.m}; {args.steps} steps took "
                                    f"{dt:.1f} s; scaled by n m ratio {scale:.3g}")},
        "e2e": {"value": value, "unit": "iters/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)


def run_ours(args, rank, world, local_rank):
    import torch
    import torch.distributed as dist

    from paper_2501_17996_gb300 import binding as B

    torch.cuda.set_device(local_rank)
    stream = torch.cuda.current_stream()
    wl = WORKLOADS[args.workload]
    seed = args.seed + rank
    inst = wl["factory"](seed)
    n, m = inst.n, inst.m
    prec = args.precision
    s_f = {"fp32": 4, "bf16": 2, "fp64": 8}[prec]
    s_p = 8 if prec == "fp64" else 4
    common = dict(precision=prec, device=local_rank, k_check=args.k_check,
                  cuda_stream=stream.cuda_stream, stop_mode="none", shape=args.shape,
                  compensated_duals=args.compensated_duals)

    def barrier():
        if world > 1:
            dist.barrier()

    # ---- device-resident timed region
    prob = B.Problem(inst)
    prob.solve(want_T=False, max_iters=max(args.warmup, 1), **common)     # allocate, upload, warm
    # The cold-start window (iterations W .. W+20 of a cold solve), reported beside the main
    # number: the projection needs 4.3 Newton passes per edge in the first iterations and 1.1
    # once the multipliers settle, so the first iterations are the slowest of a solve.
    torch.cuda.synchronize()
    kc = min(args.steps, 20)
    cold_res, cold_times = prob.solve_timed(max_iters=kc, warm_start=1, **common)
    cold = {"iterations": [args.warmup, args.warmup + kc],
            "value": kc / (cold_times["ms_total"] / 1e3),
            "ms_per_launch": {k: v[0] / v[1] for k, v in cold_times.items()
                              if k != "ms_total" and v[1]}}
    # The main window starts at iteration --prepare of the same solve (untimed iterations in
    # between, then W warm-up iterations): the regime of almost all of a solve's iterations.
    start = max(args.prepare, 2 * args.warmup + kc)
    if start > 2 * args.warmup + kc:
        prob.solve(want_T=False, max_iters=start - 2 * args.warmup - kc, warm_start=1, **common)
    prob.solve(want_T=False, max_iters=args.warmup, warm_start=1, **common)
    torch.cuda.synchronize()
    barrier()
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    with ClockSampler(local_rank) as clk:
        ev0.record(stream)
        res, times = prob.solve_timed(max_iters=args.steps, warm_start=1, **common)
        ev1.record(stream)
        torch.cuda.synchronize()
    barrier()
    ms = ev0.elapsed_time(ev1)
    # the iterations after them as a caller's solve runs them (a first run captures its graphs)
    plain_ms = []
    for _ in range(2):
        ev0.record(stream)
        prob.solve(want_T=False, max_iters=args.steps, warm_start=1, **common)
        ev1.record(stream)
        torch.cuda.synchronize()
        plain_ms.append(ev0.elapsed_time(ev1))
    from paper_2501_17996_gb300.sharding import aggregate_rate

    value, t_max = aggregate_rate(args.steps, ms / 1e3, world, device="cuda")
    ms_max = t_max * 1e3
    launches = sum(v[1] for k, v in times.items() if k != "ms_total")

    # ---- roofline of the dominant kernel
    used_shape = res.get("shape", -1)
    kind = B.mcf_shape_info()[used_shape][3] if used_shape >= 0 else 0
    alg = algorithmic_bytes(n, m, s_f, s_p, kind)
    dom = max(("edge", "node", "check"), key=lambda k: times[k][0])
    dom_ms = times[dom][0] / max(times[dom][1], 1)
    peak, peak_kind = peaks()
    achieved = alg[dom] / (dom_ms / 1e3) / 1e9
    traffic = None
    prof = os.path.join(ROOT, "profiles", f"{dom}_kernel_{args.workload}_{prec}.json")
    if os.path.exists(prof):
        try:
            pj = json.load(open(prof))
            if pj.get("kernel_source_hash") == kernel_source_hash():
                traffic = pj.get("dram_bytes_per_launch")
        except Exception:
            traffic = None
    iter_ms = ms / args.steps
    per_kernel = {k: {"ms_per_launch": (v[0] / v[1]) if v[1] else None, "launches": v[1],
                      "share": v[0] / max(times["ms_total"], 1e-9),
                      "alg_gbs": (alg[k] / (v[0] / v[1] / 1e3) / 1e9) if v[1] and alg[k] else None,
                      "alg_frac": (alg[k] / (v[0] / v[1] / 1e3) / 1e9 / peak) if v[1] and alg[k] else None,
                      "design_extra_bytes": alg["design_extra"].get(k, 0.0)}
                  for k, v in times.items() if k != "ms_total"}
    prob.close()

    # ---- end to end through the public API with host buffers
    e2e_value = None
    if not args.no_e2e:
        torch.cuda.synchronize()
        barrier()
        t0 = time.perf_counter()
        with B.Problem(inst) as p2:
            p2.solve(want_T=True, max_iters=args.steps, **common)
        t_e2e = time.perf_counter() - t0
        from paper_2501_17996_gb300.sharding import aggregate_rate

        e2e_value, _ = aggregate_rate(args.steps, t_e2e, world, device="cuda")
    ld = (n + 7) // 8 * 8
    h2d = (n * ld * s_p) + m * s_p + (3 * m + 2 * (n + 1)) * 4     # W, cap, incidence
    d2h = n * ld * s_p                                             # T

    # ---- time to tolerance (optional)
    ttt = None
    if args.ttt:
        with B.Problem(inst) as p3:
            t0 = time.perf_counter()
            if args.ttt_stop == "paper":
                eps = args.ttt_eps if args.ttt_eps is not None else \
                    (0.01 if n <= 1000 else 0.03) / (n * (n - 1.0))
            else:
                eps = args.ttt_eps if args.ttt_eps is not None else 1e-4
            r3 = p3.solve(want_T=False, max_iters=args.ttt_max_iters,
                          **{**common, "stop_mode": args.ttt_stop}, eps=eps, raise_on_error=False)
            ttt = {"seconds": time.perf_counter() - t0, "iters": r3["iters"],
                   "rel_kkt": r3["rel_kkt"], "r_over_nm": r3["r_over_nm"], "stop": args.ttt_stop,
                   "eps": eps, "status": r3["rc"]}

    if rank != 0:
        return
    line = {
        "metric": METRIC, "value": value, "unit": "iters/s", "n_gpus": world,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms_max / args.steps,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "f32" if prec != "fp64" else "f64",
        "data": "synthetic",
        "config": {"workload": f"{args.workload}: {wl['desc']}", "n": n, "m": m,
                   "precision": prec, "storage_F": {"fp32": "f32", "bf16": "bf16", "fp64": "f64"}[prec],
                   "k_check": args.k_check, "seed": args.seed, "shape": used_shape,
                   "timed_iterations": [start, start + args.steps],
                   "compensated_duals": args.compensated_duals,
                   "kernel_kind": ["register", "bulk-copy pipelined", "register with in-sums"][kind],
                   "l2": "inputs larger than L2 (F alone is %.1f GB)" % (2 * s_f * n * m / 1e9),
                   "parallelism": "replicas" if world > 1 else "single"},
        "roofline": {"bound": "hbm", "kernel": dom, "achieved": achieved, "peak": peak,
                     "peak_kind": peak_kind, "unit": "GB/s", "frac": achieved / peak,
                     "traffic": traffic, "alg_bytes_per_launch": alg[dom],
                     "ms_per_launch": dom_ms,
                     # the kernel's own DRAM bytes (ncu) over the same event time
                     "traffic_frac": (traffic / (dom_ms / 1e3) / 1e9 / peak) if traffic else None},
        "hbm": {"iteration_floor_gbs": alg["iteration_floor"] / (iter_ms / 1e3) / 1e9,
                "iteration_alg_gbs": (alg["edge"] + alg["node"]) / (iter_ms / 1e3) / 1e9,
                "peak_gbs": peak, "kernels": per_kernel},
        "e2e": {"value": e2e_value, "unit": "iters/s", "h2d_bytes_per_step": h2d / args.steps,
                "d2h_bytes_per_step": d2h / args.steps,
                "note": ("problem creation + upload, %d iterations, T read-back (after the device-resident "
                         "leg in the same process, so the device memory pool is warm)" % args.steps)},
        "gpu_launches": launches,
        "solve": {"value": args.steps / (plain_ms[1] / 1e3), "ms_per_step": plain_ms[1] / args.steps},
        "clocks": clk.summary(),
        "cold_start": cold,
    }
    if ttt:
        line["time_to_tolerance"] = ttt
    if world == 1 and not args.no_cpu_baseline:
        line["cpu_baseline"] = cpu_baseline(wl, inst, args.seed, args.k_check)
    print(json.dumps(line), flush=True)


def run_batched(args, rank, world, local_rank):
    """cfg4: 64 instances, n ~ U[50,400], out-degree ~ U[4,16], half log / half power,
    solved to relative KKT 1e-4 by one batched engine, against one-at-a-time solves."""
    import torch

    from paper_2501_17996_gb300 import binding as B

    torch.cuda.set_device(local_rank)
    insts = I.batched(seed=args.seed + rank, count=64)
    probs = [B.Problem(i) for i in insts]
    kw = dict(stop_mode="kkt", eps=1e-4, max_iters=200000, k_check=args.k_check, device=local_rank)
    # warm-up: allocate device state for every problem, build graphs
    B.mcf_solve_batch(probs, B.mcf_options_default(**{**kw, "stop_mode": "none", "max_iters": 50}))
    torch.cuda.synchronize()
    if args.batched_iters > 0:
        # fixed-length form (for profiling): K more iterations of all 64 instances, timed
        K = args.batched_iters
        t0 = time.perf_counter()
        B.mcf_solve_batch(probs, B.mcf_options_default(**{**kw, "stop_mode": "none", "max_iters": K}))
        torch.cuda.synchronize()
        dt = time.perf_counter() - t0
        for p in probs:
            p.close()
        if rank == 0:
            print(json.dumps({
                "metric": METRIC, "value": K / dt, "unit": "batched iterations/s (64 instances)",
                "n_gpus": world, "steps": K, "warmup": 50, "ms_per_step": dt / K * 1e3,
                "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
                "data": "synthetic",
                "config": {"workload": "batched, fixed length: 64 instances, n~U[50,400], "
                                       "out-degree~U[4,16], %d iterations after 50" % K}}), flush=True)
        return
    t0 = time.perf_counter()
    rc, res = B.mcf_solve_batch(probs, B.mcf_options_default(**kw))
    t_batch = time.perf_counter() - t0
    iters = [r["iters"] for r in res]
    # the same 64 solves submitted together (continuous batching): each one's completion
    # time from the common start
    t0 = time.perf_counter()
    pending = {p.submit(**kw): i for i, p in enumerate(probs)}
    done_at = [None] * len(probs)
    status = [None] * len(probs)
    while pending:
        for tk in list(pending):
            r = B.mcf_poll(tk)
            if r is not None:
                i = pending.pop(tk)
                done_at[i] = time.perf_counter() - t0
                status[i] = r["status"]
        time.sleep(0.0005)
    t_served = max(done_at)
    # one at a time from the same common start: solve i completes after solves 0..i
    t0 = time.perf_counter()
    seq_done = []
    for p in probs:
        p.solve(want_T=False, **kw)
        seq_done.append(time.perf_counter() - t0)
    t_seq = seq_done[-1]
    for p in probs:
        p.close()
    if rank != 0:
        return

    def pct(x):
        return {"p50_s": float(np.percentile(x, 50)), "p99_s": float(np.percentile(x, 99)),
                "max_s": float(np.max(x))}

    line = {
        "metric": METRIC, "value": len(insts) / t_batch, "unit": "solves/s", "n_gpus": world,
        "steps": 1, "warmup": 1, "ms_per_step": t_batch * 1e3, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": {"workload": "batched: 64 instances, n~U[50,400], out-degree~U[4,16], "
                               "c~U[1,10], half log / half power gamma~U[0.3,0.7]",
                   "stop": "rel_kkt < 1e-4", "k_check": args.k_check,
                   "latency": "completion time of each solve from the common start of its arm"},
        "batched": {"seconds": t_batch, "solves_per_s": len(insts) / t_batch, "rc": rc,
                    "iters_total": int(sum(iters)), "iters_max": int(max(iters)),
                    "all_converged": all(r["status"] == 0 for r in res),
                    "note": "mcf_solve_batch returns when every solve is done"},
        "submitted_together": {"seconds": t_served, "solves_per_s": len(insts) / t_served,
                               "all_converged": all(s_ == 0 for s_ in status), **pct(done_at)},
        "one_at_a_time": {"seconds": t_seq, "solves_per_s": len(insts) / t_seq, **pct(seq_done)},
        "speedup": t_seq / t_batch,
    }
    print(json.dumps(line), flush=True)


def run_served(args, rank, world, local_rank):
    """cfg5: Poisson stream of solves (mean --rate req/s for --window s) over resident
    networks with n in {100, 300, 1000, 3000} (out-degree 8, log utility): 70% warm
    re-solves after a +-10% perturbation of capacities or weights, 30% cold solves (a cold
    start of a resident network stands for a new network of that size; the host-side
    creation of new networks is left out of the trace). Served by continuous batching
    (mcf_submit/mcf_poll), then the same trace one request at a time with mcf_solve.
    Latency = completion time - arrival time; stop rule rel_kkt < 1e-4."""
    import threading

    from paper_2501_17996_gb300 import binding as B

    rng = np.random.default_rng(args.seed + 1000 * rank)
    sizes = [100, 300, 1000, 3000]
    per = args.pool
    nets = []
    for n in sizes:
        for k in range(per):
            inst = I.served_network(n, seed=args.seed * 100003 + n * 97 + k)
            nets.append((inst, B.Problem(inst)))
    kw = dict(stop_mode="kkt", eps=1e-4, max_iters=100000, k_check=args.k_check, device=local_rank)
    # warm-up: every network solved once (device state resident, graphs built)
    for t in [p.submit(**kw) for _, p in nets]:
        B.mcf_wait(t, -1)
    # trace
    arrivals = []
    tcur = 0.0
    while True:
        tcur += rng.exponential(1.0 / args.rate)
        if tcur > args.window:
            break
        warm = rng.random() < 0.7
        what = "cap" if rng.random() < 0.5 else "w"
        arrivals.append((tcur, int(rng.integers(len(nets))), warm, what, int(rng.integers(1 << 30))))
    originals = [(inst.cap.copy(), inst.w.copy()) for inst, _ in nets]

    def apply(idx, what, seed):
        inst, p = nets[idx]
        prng = np.random.default_rng(seed)
        base = I.Instance(inst.n, inst.tail, inst.head, originals[idx][0], inst.kind, originals[idx][1])
        pert = I.perturb(base, 0.1, what, prng)
        if what == "cap":
            p.update_capacities(pert.cap)
        else:
            p.update_weights(pert.w)

    def run_trace(mode):
        lat = [None] * len(arrivals)
        busy = set()
        pending = {}
        lock = threading.Lock()
        t0 = time.perf_counter()
        deferred = []
        idx = 0
        done = 0
        iters = []
        while done < len(arrivals):
            now = time.perf_counter() - t0
            # submit everything that has arrived and whose network is idle
            while idx < len(arrivals) and arrivals[idx][0] <= now:
                deferred.append(idx)
                idx += 1
            still = []
            for r in deferred:
                ta, net, warm, what, seed = arrivals[r]
                if net in busy or time.perf_counter() - t0 > args.window + args.drain_limit:
                    still.append(r)
                    continue
                apply(net, what, seed)
                opts = dict(kw, warm_start=1 if warm else 0)
                if mode == "served":
                    pending[nets[net][1].submit(**opts)] = (r, net)
                    busy.add(net)
                else:
                    res = nets[net][1].solve(want_T=False, raise_on_error=False, **opts)
                    lat[r] = time.perf_counter() - t0 - ta
                    iters.append(res["iters"])
                    done += 1
            deferred = still
            if mode == "served":
                for tk in list(pending):
                    res = B.mcf_poll(tk)
                    if res is None:
                        continue
                    r, net = pending.pop(tk)
                    lat[r] = time.perf_counter() - t0 - arrivals[r][0]
                    iters.append(res["iters"])
                    busy.discard(net)
                    done += 1
                time.sleep(0.0005)
            if time.perf_counter() - t0 > args.window + args.drain_limit:
                break
        wall = time.perf_counter() - t0
        for tk in list(pending):   # past the drain limit: cancel and collect what still runs
            B.mcf_cancel(tk)
            B.mcf_wait(tk, -1)
            pending.pop(tk)
        got = [x for x in lat if x is not None]
        # a request that did not finish counts as slower than any that did: its latency is
        # at least the time it waited (window + drain limit - arrival)
        lim = [x if x is not None else wall - arrivals[i][0] for i, x in enumerate(lat)]
        unfinished = len(lat) - len(got)
        return {"completed": len(got), "offered": len(arrivals), "unfinished": unfinished,
                "wall_s": wall, "solves_per_s": len(got) / wall if wall > 0 else None,
                "p50_s": float(np.percentile(lim, 50)) if lim else None,
                "p99_s": float(np.percentile(lim, 99)) if lim else None,
                "p99_is_lower_bound": unfinished > 0,
                "mean_iters": float(np.mean(iters)) if iters else None}

    served = run_trace("served")
    serial = run_trace("serial")
    for _, p in nets:
        p.close()
    if rank != 0:
        return
    line = {
        "metric": METRIC, "value": served["p99_s"], "unit": "s (p99 latency)", "n_gpus": world,
        "steps": served["completed"], "warmup": 1, "ms_per_step": None,
        "higher_is_better": False, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
        "data": "synthetic",
        "config": {"workload": "served: Poisson %g req/s for %g s, n in {100,300,1000,3000}, "
                               "out-degree 8, 70%% warm (+-10%% c or w), 30%% cold, "
                               "rel_kkt < 1e-4, 120 GB budget" % (args.rate, args.window),
                   "networks": len(nets)},
        "served": served, "one_at_a_time": serial,
    }
    print(json.dumps(line), flush=True)


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=500)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--prepare", type=int, default=1000,
                    help="iteration of the solve at which the timed window starts (untimed "
                         "iterations before it; a cold-start window is reported as well)")
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default="large", choices=list(WORKLOADS))
    ap.add_argument("--precision", default="fp32", choices=["fp32", "bf16", "fp64"])
    ap.add_argument("--k-check", dest="k_check", type=int, default=50)
    ap.add_argument("--seed", type=int, default=0)
    ap.add_argument("--shape", type=int, default=-1, help="kernel shape index (-1 = automatic)")
    ap.add_argument("--compensated-duals", dest="compensated_duals", type=int, default=1,
                    help="FP32 head + BF16 tail duals (1, the library default) or plain FP32 (0)")
    ap.add_argument("--no-ttt", dest="ttt", action="store_false",
                    help="skip the time-to-tolerance solve (a cold solve to --ttt-eps, "
                         "timed through the public API; on by default)")
    ap.add_argument("--ttt-eps", dest="ttt_eps", type=float, default=None,
                    help="kkt: relative KKT target (default 1e-4); paper: epsilon of r < n m eps "
                         "(default 0.01/(n(n-1)) for n <= 1000, 0.03/(n(n-1)) above, Sec. 3.1)")
    ap.add_argument("--ttt-stop", dest="ttt_stop", default="kkt", choices=["kkt", "paper"])
    ap.add_argument("--ttt-max-iters", dest="ttt_max_iters", type=int, default=40000)
    ap.add_argument("--no-cpu-baseline", dest="no_cpu_baseline", action="store_true")
    ap.add_argument("--no-e2e", dest="no_e2e", action="store_true")
    ap.add_argument("--rate", type=float, default=200.0, help="served: mean arrivals per s")
    ap.add_argument("--window", type=float, default=5.0, help="served: arrival window (s)")
    ap.add_argument("--pool", type=int, default=6, help="served: networks per size")
    ap.add_argument("--drain-limit", dest="drain_limit", type=float, default=60.0)
    ap.add_argument("--batched-iters", dest="batched_iters", type=int, default=0,
                    help="batched: run this many iterations of the 64 instances instead of "
                         "solving them (a short fixed-length form for profiling)")
    ap.add_argument("--knn-n", dest="knn_n", type=int, default=1000, help="knn: nodes")
    ap.add_argument("--knn-q", dest="knn_q", type=int, default=10, help="knn: neighbours")
    args = ap.parse_args()
    WORKLOADS["knn"] = dict(
        factory=lambda seed: knn_connected(args.knn_n, args.knn_q, seed),
        sample=lambda seed: knn_connected(min(args.knn_n, 300), args.knn_q, seed),
        desc=(f"kNN (Sec. 3.1): n={args.knn_n} uniform points in the unit square, edges both "
              f"ways to the {args.knn_q} nearest neighbours, log c~U[log 0.5, log 5], "
              f"log w~U[log 0.3, log 3], u = w log s"))
    if args.warmup < 3:
        raise SystemExit("--warmup must be >= 3")
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local_rank = int(os.environ.get("LOCAL_RANK", "0"))
    if args.impl == "reference":
        run_reference(args, rank, world)
        return
    if world > 1:
        import torch
        import torch.distributed as dist

        torch.cuda.set_device(local_rank)
        dist.init_process_group("nccl")
    if args.workload == "batched":
        run_batched(args, rank, world, local_rank)
    elif args.workload == "served":
        run_served(args, rank, world, local_rank)
    else:
        run_ours(args, rank, world, local_rank)
    if world > 1:
        import torch.distributed as dist

        dist.destroy_process_group()


if __name__ == "__main__":
    main()
