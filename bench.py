"""Benchmark: converged JFNK NLTE column solves on the GPU (one JSON line).

Default workload (config 4): 4,096 independent Ca II-like columns of 64 to
256 depths (about 1,000 frequencies, 5 mu per hemisphere), solved together in
one persistent batch plan in the mixed precision mode, from LTE through a
capped RH92 warm-up and Algorithm 2 to the paper's stopping rule (Sect. 3.1).
One step = one batched solve of every column: every F-class evaluation
(opacity, formal solution, rates, assembly, preconditioner) and every
Krylov/Newton update, on the device.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]
                  [--workload batch|ca|two-level|h|serve] [--precision fp64|mixed]

Metric: formal-solution ray-points/s (= F-class evaluations x N_nu x 2 N_mu x
N_z per second, summed over columns); the line also carries converged
columns/s, the FP64 one-column-per-launch path's columns/s on a sample of
the same columns, and the error against the oracle on a sample. ``--workload
ca`` is the FP64 single-column line (config 2), ``serve`` the continuous-
batching stream (config 5, p50/p99 latency).
N > 1 (torchrun): every rank solves its own columns (weak scaling, no
collective on the data path); value = ray-points of all ranks / max time.
``--impl reference`` times the CPU oracle on the host cores instead.
"""
from __future__ import annotations

import argparse
import hashlib
import json
import re
import math
import os
import subprocess
import sys
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

import workloads as W  # noqa: E402

METRIC = "formal-solution ray-points/s"


def parse():
    p = argparse.ArgumentParser()
    p.add_argument("--gpus", type=int, default=1)
    p.add_argument("--steps", type=int, default=None,
                   help="timed steps (default: 40 single-column solves, 10 batched solves or oracle steps)")
    p.add_argument("--warmup", type=int, default=3)
    p.add_argument("--impl", default="ours", choices=["ours", "reference"])
    p.add_argument("--workload", default="batch",
                   choices=["batch", "ca", "two-level", "h", "ca-velocity", "serve", "rtol"])
    p.add_argument("--columns", type=int, default=4096, help="batch workload: number of columns")
    p.add_argument("--requests", type=int, default=10000, help="serve workload: number of requests")
    p.add_argument("--rate", type=float, default=2000.0, help="serve workload: Poisson arrival rate [1/s]")
    p.add_argument("--slots", type=int, default=512, help="serve workload: columns in flight")
    p.add_argument("--producers", type=int, default=4, help="serve workload: threads building requests")
    p.add_argument("--precision", default=None, choices=[None, "fp64", "mixed"])
    p.add_argument("--no-cpu-baseline", action="store_true")
    args = p.parse_args()
    if args.steps is None:
        # a single-column solve takes tens of ms: 40 of them give the clock
        # sampler a timed region of about a second
        single = args.workload in ("ca", "two-level", "h", "ca-velocity")
        args.steps = 40 if (single and args.impl == "ours") else 10
    return args


def workload(name):
    if name == "two-level":
        return W.config1(), "fp64"
    if name == "ca-velocity":
        return W.config2_velocity(), "fp64"
    if name == "h":
        return W.config3(), "mixed"
    return W.config2(), "fp64"


def workload_config(wl, m_info, precision):
    nq, nz, nmu = m_info
    return {"workload": f"{wl.name}: {wl.atom.name} atom, {nz} depths, {nq} frequencies, "
                        f"{nmu} mu per hemisphere, JFNK from {wl.init.upper()} to the paper's "
                        f"stopping rule ({precision})",
            "atom": wl.atom.name, "n_levels": int(wl.atom.n_levels), "n_depth": nz, "n_nu": nq,
            "n_mu": nmu, "init": wl.init, "rtol": 1e-2, "ftol": 1e-4, "fdrop": 1e-2,
            "l2": "flushed by a 256 MiB device write before every timed step"}


def dist_setup():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    if ws <= 1:
        return 0, 1, 0, None
    import torch
    import torch.distributed as dist
    rank = int(os.environ["RANK"])
    local = int(os.environ.get("LOCAL_RANK", rank))
    torch.cuda.set_device(local)
    dist.init_process_group("nccl")
    return rank, ws, local, dist


def reduce_ranks(dist, values, device="cuda"):
    """Whole-job aggregates over the ranks of a weak-scaling run: the maximum
    (times: the slowest rank sets the job's time) and the sum (work done) of
    each value. Returns (max list, sum list); a single process returns its own."""
    if dist is None:
        return list(values), list(values)
    import torch
    t = torch.tensor([float(v) for v in values], dtype=torch.float64, device=device)
    tmax = t.clone()
    dist.all_reduce(tmax, op=dist.ReduceOp.MAX)
    tsum = t.clone()
    dist.all_reduce(tsum, op=dist.ReduceOp.SUM)
    return tmax.tolist(), tsum.tolist()


def rank_seed(base, rank):
    """Seed of a rank's share of a sharded workload (distinct columns per rank)."""
    return base + rank


def clocks_start():
    try:
        return subprocess.Popen(
            ["nvidia-smi", "--query-gpu=index,clocks.sm,clocks.max.sm,power.draw,"
             "clocks_event_reasons.active,clocks_event_reasons.hw_slowdown,"
             "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
             "clocks_event_reasons.sw_power_cap", "--format=csv,noheader,nounits", "-lms", "50"],
            stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
    except Exception:
        return None


def clocks_stop(proc, device):
    if proc is None:
        return None
    proc.terminate()
    try:
        out, _ = proc.communicate(timeout=5)
    except Exception:
        proc.kill()
        out, _ = proc.communicate()
    sm, mx, reasons = [], [], set()
    names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
    for line in out.strip().splitlines():
        f = [x.strip() for x in line.split(",")]
        if len(f) < 9 or f[0] != str(device):
            continue
        try:
            sm.append(float(f[1]))
            mx.append(float(f[2]))
        except ValueError:
            continue
        for nm, v in zip(names, f[5:9]):
            if v.lower() == "active":
                reasons.add(nm)
    if not sm:
        return None
    return {"sm_mhz": float(np.median(sm)), "sm_max_mhz": float(max(mx)), "reasons": sorted(reasons),
            "samples": len(sm)}


# the arithmetic of the mixed mode: FP32 formal solution and tangents, float
# pairs (about 48 bits, FP32 pipe) for S, J and the base rate sums, FP64 for
# the rate-equation assembly, the block inverses, GMRES and the Newton update
MIXED_DTYPE = "f32 formal solution / f32-pair S, J, rate sums / f64 assembly, Krylov, Newton"

# the sources each formal kernel is compiled from (its translation unit and the
# ray-step coefficient header): a change to any of them voids its ncu traffic
KERNEL_SOURCES = {
    "formal_fp64": ("formal_fused.cu", "formal_coef.cuh"),
    "formal_fp32_tan": ("formal_sweep.cu", "formal_coef.cuh", "dfloat.cuh"),
    "formal_fp32_base": ("formal_sweep.cu", "formal_coef.cuh", "dfloat.cuh"),
}


def _code_only(text):
    """Source text without comments and blank space (a comment edit leaves the kernel as it was)."""
    text = re.sub(r"/\*.*?\*/", " ", text, flags=re.S)
    text = re.sub(r"//[^\n]*", " ", text)
    return " ".join(text.split())


def source_hash(kernel_key):
    h = hashlib.sha256()
    csrc = os.path.join(ROOT, "paper_2406_17234_gb300", "csrc")
    for f in KERNEL_SOURCES[kernel_key]:
        with open(os.path.join(csrc, f), encoding="utf-8") as fh:
            h.update(_code_only(fh.read()).encode())
    return h.hexdigest()[:16]


def measured_traffic(kernel_key):
    """DRAM bytes per launch of the formal kernel from a committed ncu summary, if current."""
    path = os.path.join(ROOT, "profiles", "formal_traffic.json")
    try:
        d = json.load(open(path))
    except Exception:
        return None
    e = d.get(kernel_key)
    if not e or e.get("source_hash") != source_hash(kernel_key):
        return None
    return e.get("bytes_per_ray_point")


def host_cpu():
    """CPU model and logical core count of this host (for the baseline's record)."""
    fields = {}
    try:
        out = subprocess.run(["lscpu"], capture_output=True, text=True, timeout=10).stdout
        for line in out.splitlines():
            if ":" in line:
                k, v = line.split(":", 1)
                fields.setdefault(k.strip(), v.strip())
    except Exception:
        pass
    model = fields.get("Model name") or fields.get("Vendor ID") or "unknown"
    return model, os.cpu_count() or 1


def cpu_baseline(wl, budget_s=20.0):
    """The oracle as it stands, on the host cores: a bounded sample of the same workload."""
    from oracle import model as OM
    from oracle.residual import jvp_complex, residual
    m = OM.build_model(wl.atom, wl.columns[0], wl.n_mu)
    J0 = OM.initial_J(m)
    rng = np.random.default_rng(0)
    t0 = time.perf_counter()
    evals = 0
    residual(m, m.nstar, J0)
    evals += 1
    while time.perf_counter() - t0 < budget_s:
        v = rng.normal(size=m.nstar.shape) * m.nstar
        jvp_complex(m, m.nstar, J0, v)
        evals += 1
    dt = time.perf_counter() - t0
    model, ncpu = host_cpu()
    return {"value": evals * m.ray_points / dt, "unit": "ray-points/s", "cores": 1, "kind": "oracle",
            "host_cores": ncpu, "cpu_model": model,
            "sample": f"{evals} oracle F-class evaluations (1 residual + {evals - 1} complex-step JVPs) "
                      f"of the same column at LTE, {dt:.1f} s, numpy FP64/complex128 single thread "
                      f"(one column is one thread's work)"}


def _oracle_column_solve(atom, col, n_mu, start):
    """One column solved by the oracle with the batch's options (hybrid start,
    paper stopping rule): populations, F-class evaluations, ray-points, seconds."""
    from oracle import model as OM
    from oracle.hybrid import hybrid
    m = OM.build_model(atom, col, n_mu)
    t0 = time.perf_counter()
    r = hybrid(m, m.nstar, switch_tol=start["rh92_switch"], rh92_max=start["rh92_warmup"])
    dt = time.perf_counter() - t0
    return dict(n=r.n, converged=bool(r.converged), F_calls=int(r.F_calls),
                ray_points=float(r.F_calls) * m.ray_points, seconds=dt)


def _oracle_evals(atom, col, n_mu, k):
    """k oracle F-class evaluations (1 residual + k - 1 complex-step JVPs) of one column at LTE."""
    from oracle import model as OM
    from oracle.residual import jvp_complex, residual
    m = OM.build_model(atom, col, n_mu)
    J0 = OM.initial_J(m)
    rng = np.random.default_rng(0)
    residual(m, m.nstar, J0)
    for _ in range(k - 1):
        jvp_complex(m, m.nstar, J0, rng.normal(size=m.nstar.shape) * m.nstar)
    return k * m.ray_points


def oracle_pool(workers):
    """Process pool for the oracle: spawn-started (a child forked from a process
    that holds a CUDA context can hang), one BLAS thread per worker."""
    import multiprocessing as mp
    from concurrent.futures import ProcessPoolExecutor
    for v in ("OMP_NUM_THREADS", "OPENBLAS_NUM_THREADS", "MKL_NUM_THREADS"):
        os.environ.setdefault(v, "1")
    return ProcessPoolExecutor(max_workers=workers, mp_context=mp.get_context("spawn"))


def cpu_baseline_batch(wl, start, pool, futures, workers, t0):
    """The oracle solving the first ``workers`` columns of the batch to
    convergence, one column per host core (started before the GPU run; the
    wall time counts from the pool's start)."""
    res = [f.result() for f in futures]
    wall = max(time.perf_counter() - t0, max(r["seconds"] for r in res))
    model, ncpu = host_cpu()
    pts = sum(r["ray_points"] for r in res)
    conv = sum(r["converged"] for r in res)
    return {"value": pts / wall, "unit": "ray-points/s", "cores": workers, "kind": "oracle",
            "host_cores": ncpu, "cpu_model": model, "columns_per_s": conv / wall,
            "sample": f"the first {len(res)} columns of the batch solved to the paper's stopping rule by the "
                      f"oracle (hybrid start, complex-step JVPs, numpy FP64), one column per process, "
                      f"{workers} processes in parallel, {wall:.1f} s wall; {conv} converged"}, res


# Algorithmic work per ray-point (value / JVP evaluation): FP32-pipe
# instructions and MUFU operations (exp and reciprocal), after the unit count
# of the path (Delta tau, exp, 1/Delta tau, w a b, I update, J accumulation;
# the tangent adds the differentiated recurrence).
ALG_OPS = {"value": (10, 2), "jvp": (26, 2)}
# ... of the cached FP64 evaluations, which form an exponential and a reciprocal
# per layer and angle for both hemispheres (moving columns: per ray and layer) in
# base evaluations only: a product is three FMAs per ray-point (moving: five)
CACHED_OPS = {"value": (10, 1), "jvp": (3, 0)}
CACHED_MOVING_OPS = {"value": (10, 2), "jvp": (5, 0)}
FORMAL_KERNELS = {0: "k_formal<double> + k_ray_sum (per-ray buffers)", 1: "k_formal_fused<double>",
                  2: "k_formal_sweep (thread per frequency)", 3: "k_formal_sweep_warp (warp per frequency pair)",
                  4: "k_mv_formal / k_eval64_moving (moving column)",
                  6: "k_eval64 (opacity, formal solution and rate integrals per tile of frequencies)"}


FP32_LANES_PER_SM = 128   # FP32 FMA lanes per SM per clock (Blackwell SM: 4 x 32)


def nominal_fp32_fma(device=0):
    """FP32 FMA lane instructions per second from the unit count and the maximum
    SM clock: multiprocessors x 128 lanes x the clock (MEASURED_PEAKS.json's
    sm_max_mhz, else nvidia-smi's clocks.max.sm)."""
    import torch
    n_sm = torch.cuda.get_device_properties(device).multi_processor_count
    mhz = None
    try:
        mhz = float(json.load(open(os.path.join(ROOT, "MEASURED_PEAKS.json")))["sm_max_mhz"])
    except Exception:
        try:
            out = subprocess.run(["nvidia-smi", "--query-gpu=clocks.max.sm", "--format=csv,noheader,nounits",
                                  "-i", str(device)], capture_output=True, text=True, timeout=20).stdout
            mhz = float(out.split()[0])
        except Exception:
            mhz = None
    return None if mhz is None else n_sm * FP32_LANES_PER_SM * mhz * 1e6


def measured_peaks(B, ctx, device=0):
    """Pipe rates measured on this GPU by the library's probe kernels
    (jfnk_probe_alu): FP32 and FP64 fused multiply-adds per second (lane
    instructions) and MUFU exponentials per second. The FP32 rate taken as the
    roofline denominator is the larger of the probe's and the nominal one, so a
    probe that ran below the maximum clock cannot inflate a fraction."""
    p = {"fp32_fma_per_s": B.probe_alu(ctx, 1) / 2.0, "fp64_fma_per_s": B.probe_alu(ctx, 0) / 2.0,
         "fp64_exp_per_s": B.probe_alu(ctx, 2), "mufu_per_s": B.probe_alu(ctx, 3)}
    nom = nominal_fp32_fma(device)
    p["fp32_fma_probe_per_s"] = p["fp32_fma_per_s"]
    p["fp32_fma_nominal_per_s"] = nom
    if nom is not None:
        p["fp32_fma_per_s"] = max(p["fp32_fma_per_s"], nom)
    return p


def peak_rate(kind, fp64, peaks, counts=ALG_OPS):
    """Roofline ray-points/s of one evaluation kind ('value' or 'jvp') from the
    algorithmic unit counts and the measured pipe rates: the mixed path is bound
    by the slower of the FP32 lanes and the MUFU; in FP64 mode every operation
    goes to the FP64 pipe, with exp and the reciprocal costed by the probe."""
    ops, mufu = counts[kind]
    if fp64:
        c_exp = peaks["fp64_fma_per_s"] / peaks["fp64_exp_per_s"]   # one exp in FMA-instruction time
        return peaks["fp64_fma_per_s"] / (ops + mufu * c_exp)
    return 1.0 / max(ops / peaks["fp32_fma_per_s"], mufu / peaks["mufu_per_s"])


STAGES = ("opacity", "tangent_sweep", "base_formal", "rate_integrals", "assembly", "krylov_step")


def stage_breakdown(st):
    """Mean duration per active tick of each stage of a profiled solve (all
    kernels on one stream, in-graph CUDA events), with each stage's share."""
    n = max(1, int(st["formal_launches"]))
    ms = [float(x) / n for x in st["stage_ms"]]
    tot = sum(ms) or 1.0
    return {"per_tick": {k: v for k, v in zip(STAGES, ms)}, "tick_total": sum(ms),
            "share": {k: v / tot for k, v in zip(STAGES, ms)}}


def kernel_roofline(name, kind, fp64, points, kern_ms, launches, peaks, traffic_key=None):
    """One formal kernel: achieved = algorithmic ray-points of its launches /
    their summed CUDA-event duration, against the roofline of its evaluation kind."""
    peak = peak_rate(kind, fp64, peaks)
    avg_s = kern_ms * 1e-3 / max(1, launches)
    achieved = points / (kern_ms * 1e-3) if kern_ms > 0 else 0.0
    tpp = measured_traffic(traffic_key) if traffic_key else None
    return {"kernel": name, "kind": kind, "achieved": achieved / 1e9, "peak": peak / 1e9,
            "frac": achieved / peak, "avg_launch_us": avg_s * 1e6, "launches": launches,
            "ray_points_per_launch": points / max(1, launches),
            "traffic": None if tpp is None else tpp * points / max(1, launches)}


def peak_source(fp64, peaks):
    if fp64:
        return (f"measured FP64 FMA {peaks['fp64_fma_per_s'] * 2 / 1e12:.3f} TFLOP/s and FP64 exp "
                f"{peaks['fp64_exp_per_s'] / 1e9:.1f} G/s (jfnk_probe_alu kinds 0, 2)")
    nom = peaks.get("fp32_fma_nominal_per_s")
    return (f"FP32 FMA {peaks['fp32_fma_per_s'] * 2 / 1e12:.1f} TFLOP/s (the larger of the probe's "
            f"{peaks.get('fp32_fma_probe_per_s', peaks['fp32_fma_per_s']) * 2 / 1e12:.1f} and the nominal "
            f"{'n/a' if nom is None else f'{nom * 2 / 1e12:.1f}'}: SMs x 128 lanes x max clock) and measured "
            f"MUFU exp {peaks['mufu_per_s'] / 1e12:.3f} T/s (jfnk_probe_alu kinds 1, 3) with unit counts "
            f"value {ALG_OPS['value']}, jvp {ALG_OPS['jvp']} (FP32 ops, MUFU ops) per ray-point")


def kernel_ops(kernel, qb):
    """Unit counts of a single column's formal kernel (qb > 0: a tiled one, of the
    moving kernels the cached one)."""
    if kernel == 6:
        return CACHED_OPS
    return CACHED_MOVING_OPS if kernel == 4 and qb > 0 else ALG_OPS


def alu_roofline(B, ctx, fp64, n_value, n_jvp, pts_per_launch, kern_ms, launches, clocks, kernel, qb, device):
    """Roofline of the single-column formal-solution kernel (one launch per
    tick, value and JVP evaluations mixed): achieved = ray-points per launch /
    mean launch time (in-graph CUDA events around the formal kernel of every
    tick), peak = the mix of the two kinds' rooflines at the measured rates."""
    peaks = measured_peaks(B, ctx, device)
    w_v, w_j = n_value / max(1, n_value + n_jvp), n_jvp / max(1, n_value + n_jvp)
    counts = kernel_ops(kernel, qb)
    peak = 1.0 / (w_v / peak_rate("value", fp64, peaks, counts) + w_j / peak_rate("jvp", fp64, peaks, counts))
    avg_s = kern_ms * 1e-3 / max(1, launches)
    achieved = pts_per_launch / avg_s if avg_s > 0 else 0.0
    traffic_pp = measured_traffic("formal_fp64" if fp64 else "formal_fp32_tan")
    return {"bound": "alu", "kernel": FORMAL_KERNELS.get(kernel, str(kernel)),
            "achieved": achieved / 1e9, "peak": peak / 1e9, "unit": "G ray-points/s",
            "frac": achieved / peak,
            "traffic": None if traffic_pp is None or not fp64 or kernel != 1 else traffic_pp * pts_per_launch,
            "ops_per_ray_point": {"value": counts["value"], "jvp": counts["jvp"],
                                  "mix": {"value": w_v, "jvp": w_j}},
            "avg_launch_us": avg_s * 1e6, "launches": launches, "peak_source": peak_source(fp64, peaks),
            "measured_peaks": peaks}


def run_reference(args, rank, ws, dist):
    """The oracle as it stands on the host cores (rank 0 only): each step is a
    bounded sample of the workload's F-class evaluations. Batch workload: one
    residual + one complex-step JVP of each of the batch's first P columns, one
    column per process on P host cores; single-column workloads: one residual
    + 3 JVPs of the column on one core."""
    if rank != 0:
        return
    model, ncpu = host_cpu()
    if args.workload == "batch":
        wl = W.config4(n_columns=args.columns, seed=rank_seed(20240624, 0))
        workers = max(1, min(16, ncpu))
        cols = wl.columns[:workers]
        pool = oracle_pool(workers)

        def step():
            return sum(f.result() for f in [pool.submit(_oracle_evals, wl.atom, c, wl.n_mu, 2) for c in cols])

        cores, sample = workers, (f"per step: 1 residual + 1 complex-step JVP of each of the batch's first "
                                  f"{workers} columns at LTE, one column per process on {workers} cores")
        from oracle import model as OM
        cfg = batch_config(wl.columns, OM.build_model(wl.atom, cols[0], wl.n_mu).nq, "FP64 oracle")
    else:
        wl, prec = workload(args.workload)
        from oracle import model as OM
        m = OM.build_model(wl.atom, wl.columns[0], wl.n_mu)
        pool = None

        def step():
            return _oracle_evals(wl.atom, wl.columns[0], wl.n_mu, 4)

        cores, sample = 1, "per step: 1 residual + 3 complex-step JVPs of the column at LTE"
        cfg = workload_config(wl, (m.nq, m.nz, m.nmu), "fp64 oracle")
    for _ in range(args.warmup):
        step()
    t0 = time.perf_counter()
    pts = 0.0
    for _ in range(args.steps):
        pts += step()
    dt = time.perf_counter() - t0
    if pool is not None:
        pool.shutdown()
    value = pts / dt
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": "ray-points/s",
            "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": 1e3 * dt / args.steps, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64", "data": "synthetic", "config": cfg,
            "cpu_baseline": {"value": value, "unit": "ray-points/s", "cores": cores, "kind": "oracle",
                             "host_cores": ncpu, "cpu_model": model, "sample": sample},
            "e2e": {"value": value, "unit": "ray-points/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


def run_ours(args, rank, ws, local, dist):
    import torch
    from paper_2406_17234_gb300 import binding as B

    wl, default_prec = workload(args.workload)
    prec = args.precision or default_prec
    precision = B.JFNK_MIXED if prec == "mixed" else B.JFNK_FP64
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    ctx = B.Context(local)
    atom = B.Atom(ctx, wl.atom)
    atm = B.Atmosphere(ctx, atom, wl.columns[0], n_mu=wl.n_mu)
    N = atm.n_depth * atm.n_levels
    rh92 = 200 if wl.init == "hybrid" else 0
    lib = ctx.lib
    import ctypes as C

    def opts(profile=1):
        return B.default_options(precision=precision, profile=profile, rh92_warmup=rh92)

    n_dev = torch.zeros(N, dtype=torch.float64, device=dev)
    flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device=dev)
    stream = torch.cuda.current_stream(dev)
    st = B.jfnk_stats()

    def solve_device(o):
        rc = lib.jfnk_solve(ctx.h, atm.h, C.byref(o), n_dev.data_ptr(), None, C.byref(st),
                            B.JFNK_MEM_DEVICE, stream.cuda_stream)
        B.check(rc, "jfnk_solve")
        return st.as_dict()

    o = opts(profile=0)
    for _ in range(args.warmup):
        flush.zero_()
        solve_device(o)
    torch.cuda.synchronize()
    if dist is not None:
        dist.barrier()
    torch.cuda.synchronize()
    clk = clocks_start() if rank == 0 else None
    times, stats = [], []
    torch.cuda.nvtx.range_push("timed")   # lets ncu capture the timed steps only
    for _ in range(args.steps):
        flush.zero_()
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        s = solve_device(o)
        e1.record(stream)
        e1.synchronize()
        times.append(e0.elapsed_time(e1))
        stats.append(s)
    torch.cuda.nvtx.range_pop()
    torch.cuda.synchronize()
    clocks = clocks_stop(clk, local) if rank == 0 else None
    if dist is not None:
        dist.barrier()
    total_ms = float(sum(times))
    pts = float(sum(s["ray_points"] for s in stats))
    # roofline: a separate profiled solve (in-graph CUDA events around the
    # formal kernel of every tick), outside the timed region
    flush.zero_()
    prof = solve_device(opts(profile=1))
    # e2e: host buffers through the public API (pinned in / out), wall clock
    n_host = torch.from_numpy(atm.lte().ravel().copy()).pin_memory()
    n_out = torch.empty_like(n_host).pin_memory()
    e2e_times, e2e_pts = [], 0.0
    oe = opts(profile=0)
    oe.init = B.JFNK_INIT_USER
    st2 = B.jfnk_stats()
    for _ in range(max(1, min(10, args.steps // 2))):
        flush.zero_()
        torch.cuda.synchronize()
        n_out.copy_(n_host)
        t0 = time.perf_counter()
        rc = lib.jfnk_solve(ctx.h, atm.h, C.byref(oe), n_out.data_ptr(), None, C.byref(st2),
                            B.JFNK_MEM_HOST, stream.cuda_stream)
        e2e_times.append(time.perf_counter() - t0)
        B.check(rc, "jfnk_solve (host)")
        e2e_pts += st2.ray_points
    mx, sm = reduce_ranks(dist, [total_ms, pts, sum(e2e_times), e2e_pts], dev)
    total_ms, pts, e2e_s, e2e_pts_all = mx[0], sm[1], mx[2], sm[3]
    if rank != 0:
        return
    value = pts / (total_ms * 1e-3)
    lat = np.array(times)
    cols_per_s = ws * args.steps / (total_ms * 1e-3)
    s0 = stats[-1]
    # roofline of the formal-solution kernel (dominant), from the profiled solve
    launches = prof["formal_launches"]
    kern_ms = prof["formal_ms"] + prof["formal_tan_ms"]
    fp64 = precision == B.JFNK_FP64
    roofline = alu_roofline(B, ctx, fp64, prof["F_calls"] - prof["jvp_calls"], prof["jvp_calls"],
                            atm.ray_points, kern_ms, launches, clocks, prof["formal_kernel"],
                            prof["formal_qb"], local)
    roofline["share_of_step"] = kern_ms / (total_ms / args.steps)
    roofline["tick_stages_ms"] = stage_breakdown(prof)
    roofline["timed_in"] = "a separate profiled solve (in-graph events around the formal kernel of every tick)"
    gpu_launches = int(sum(s["kernel_launches"] for s in stats))
    line = {"metric": METRIC, "value": value, "unit": "ray-points/s", "n_gpus": ws,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": total_ms / args.steps,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "f64" if fp64 else MIXED_DTYPE,
            "data": "synthetic",
            "config": workload_config(wl, (atm.n_nu, atm.n_depth, atm.n_mu), prec),
            "columns_per_s": cols_per_s,
            "latency_ms": {"p50": float(np.percentile(lat, 50)), "p99": float(np.percentile(lat, 99))},
            "solve": {"newton_iters": s0["newton_iters"], "rh92_iters": s0["rh92_iters"],
                      "F_calls": s0["F_calls"], "jvp_calls": s0["jvp_calls"],
                      "F_norm_drop": s0["F_norm"] / s0["F_norm0"], "dn_norm": s0["dn_norm"],
                      "status": s0["status"]},
            "roofline": roofline,
            "e2e": {"value": e2e_pts_all / e2e_s, "unit": "ray-points/s",
                    "h2d_bytes_per_step": N * 8, "d2h_bytes_per_step": N * 8 + 0},
            "gpu_launches": gpu_launches,
            "clocks": clocks}
    if not args.no_cpu_baseline and ws == 1:
        line["cpu_baseline"] = cpu_baseline(wl)
    print(json.dumps(line), flush=True)


def batch_config(columns, nq, precision):
    nz = [c.n_depth for c in columns]
    return {"workload": f"batched 1.5D: {len(columns)} Ca II-like columns, depths {min(nz)}-{max(nz)}, "
                        f"{nq} frequencies, 5 mu, T noise 5 %, {precision}, one batched solve per step",
            "columns": len(columns), "init": "LTE, then <= 5 limited RH92 iterations (switch below 0.1 "
                                             "change), then JFNK to the paper's stopping rule",
            "rtol": 1e-2, "ftol": 1e-4, "fdrop": 1e-2,
            "l2": "flushed by a 256 MiB device write before every timed step (the batch's tables and "
                  "work buffers are also far larger than L2)"}


BATCH_START = dict(rh92_warmup=5, rh92_switch=0.1)


def run_batch(args, rank, ws, local, dist):
    """Batched 1.5D workload (config 4): every column of the batch solved
    together in one persistent batch plan (mixed precision), against the plain
    FP64 path that solves one column per launch sequence, with the oracle on
    the host cores beside it."""
    import ctypes as C
    import torch
    from paper_2406_17234_gb300 import binding as B
    wl = W.config4(n_columns=args.columns, seed=rank_seed(20240624, rank))
    # the oracle's sample solves start first and run on the host cores while the GPU works
    cpu = None
    if rank == 0 and ws == 1 and not args.no_cpu_baseline:
        workers = max(1, min(16, os.cpu_count() or 1))
        pool = oracle_pool(workers)
        t_cpu0 = time.perf_counter()
        futs = [pool.submit(_oracle_column_solve, wl.atom, c, wl.n_mu, BATCH_START)
                for c in wl.columns[:workers]]
        cpu = (pool, futs, workers, t_cpu0)
    torch.cuda.set_device(local)
    ctx = B.Context(local)
    atom = B.Atom(ctx, wl.atom)
    free0, total_mem = torch.cuda.mem_get_info()
    t0 = time.perf_counter()
    atms = [B.Atmosphere(ctx, atom, c, n_mu=wl.n_mu) for c in wl.columns]
    setup_s = time.perf_counter() - t0
    plan = B.BatchPlan(ctx, atms, precision=B.JFNK_MIXED)
    free1, _ = torch.cuda.mem_get_info()
    opts = B.default_options(precision=B.JFNK_MIXED, profile=0, **BATCH_START)
    stream = torch.cuda.current_stream()
    flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device="cuda")
    for _ in range(args.warmup):
        flush.zero_()
        plan.run(opts, raise_on_fail=False)
    torch.cuda.synchronize()
    if dist is not None:
        dist.barrier()
    torch.cuda.synchronize()
    clk = clocks_start() if rank == 0 else None
    times, allstats = [], []
    torch.cuda.nvtx.range_push("timed")
    for _ in range(args.steps):
        flush.zero_()
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        _, st = plan.run(opts, raise_on_fail=False)
        e1.record(stream)
        e1.synchronize()
        times.append(e0.elapsed_time(e1))
        allstats.append(st)
    torch.cuda.nvtx.range_pop()
    torch.cuda.synchronize()
    clocks = clocks_stop(clk, local) if rank == 0 else None
    if dist is not None:
        dist.barrier()
    n_gpu = [n.copy() for n in plan.ns]
    total_ms = float(sum(times))
    pts = float(sum(s["ray_points"] for st in allstats for s in st))
    conv = sum(1 for st in allstats for s in st if s["status"] == 0)
    # profiled pass (untimed): in-graph CUDA events around the two sweep
    # launches of every tick, on the streams they run on
    _, pst = plan.run(B.default_options(precision=B.JFNK_MIXED, profile=1, **BATCH_START), raise_on_fail=False)
    rp = [a.ray_points for a in atms]
    jvp_pts = float(sum(s["jvp_calls"] * r for s, r in zip(pst, rp)))
    val_pts = float(sum((s["F_calls"] - s["jvp_calls"]) * r for s, r in zip(pst, rp)))
    # e2e: jfnk_batch_run with pinned host buffers (populations in, populations out)
    Ns = [a.n_depth * a.n_levels for a in atms]
    offs = np.concatenate([[0], np.cumsum(Ns)])
    h_in = torch.from_numpy(np.concatenate([a.lte().ravel() for a in atms])).pin_memory()
    h_out = torch.empty_like(h_in).pin_memory()
    nps = (C.c_void_p * len(atms))(*[h_out.data_ptr() + 8 * int(o) for o in offs[:-1]])
    oe = B.default_options(precision=B.JFNK_MIXED, profile=0, **BATCH_START)
    oe.init = B.JFNK_INIT_USER
    st_e2e = (B.jfnk_stats * len(atms))()
    e2e_times, e2e_pts = [], 0.0
    for _ in range(min(3, args.steps)):
        flush.zero_()
        torch.cuda.synchronize()
        h_out.copy_(h_in)
        ta = time.perf_counter()
        rc = ctx.lib.jfnk_batch_run(plan.h, C.byref(oe), nps, None, st_e2e, B.JFNK_MEM_HOST, None)
        e2e_times.append(time.perf_counter() - ta)
        if rc in (B.JFNK_E_INVALID, B.JFNK_E_CUDA, B.JFNK_E_NOMEM):
            B.check(rc, "jfnk_batch_run (host buffers)")
        e2e_pts += sum(s.ray_points for s in st_e2e)
    # plain FP64 path: one column per launch sequence, a sample of the same columns
    nsample = min(8, len(atms))
    fp64_t = []
    for a in atms[:nsample]:
        B.solve(a, B.default_options(**BATCH_START), raise_on_fail=False)        # warm (allocation, tuning)
        flush.zero_()
        torch.cuda.synchronize()
        ta = time.perf_counter()
        _, _, s1 = B.solve(a, B.default_options(**BATCH_START), raise_on_fail=False)
        fp64_t.append(time.perf_counter() - ta)
    fp64_cols_s = nsample / sum(fp64_t)
    mx, sm = reduce_ranks(dist, [total_ms, pts, conv, sum(e2e_times), e2e_pts])
    total_ms, pts, conv, e2e_s, e2e_pts = mx[0], sm[1], sm[2], mx[3], sm[4]
    if rank != 0:
        return
    peaks = measured_peaks(B, ctx, local)
    tan_ms = float(sum(s["formal_tan_ms"] for s in pst[:1]))
    base_ms = float(sum(s["formal_ms"] for s in pst[:1]))
    launches = int(pst[0]["formal_launches"])
    kern = {"tangent": kernel_roofline("k_formal_sweep (tangent, JVP evaluations)", "jvp", False, jvp_pts,
                                       tan_ms, launches, peaks, "formal_fp32_tan"),
            "base": kernel_roofline("k_formal_sweep (base and RH92 evaluations)", "value", False, val_pts,
                                    base_ms, launches, peaks, "formal_fp32_base")}
    dom = max(kern.values(), key=lambda k: k["avg_launch_us"])
    prof_total = sum(s for s in [tan_ms, base_ms])
    roofline = {"bound": "alu", "kernel": dom["kernel"], "achieved": dom["achieved"], "peak": dom["peak"],
                "unit": "G ray-points/s", "frac": dom["frac"], "traffic": dom["traffic"],
                "avg_launch_us": dom["avg_launch_us"], "launches": dom["launches"],
                "peak_source": peak_source(False, peaks), "kernels": kern,
                "both_sweeps": {"achieved": (jvp_pts + val_pts) / (prof_total * 1e-3) / 1e9,
                                "frac": (jvp_pts + val_pts) / (prof_total * 1e-3) /
                                        (1.0 / ((val_pts / peak_rate("value", False, peaks) +
                                                 jvp_pts / peak_rate("jvp", False, peaks)) /
                                                (jvp_pts + val_pts)))},
                "measured_peaks": peaks, "timed_in": "a separate profiled batched solve (in-graph events)",
                "launch": {"threads": int(pst[0]["formal_threads"]), "variant": int(pst[0]["formal_kernel"]),
                           "blocks_per_sm_cap_tangent": int(pst[0]["formal_occ"]),
                           "blocks_per_sm_cap_base": int(pst[0]["formal_occ_base"]),
                           "tangent_opacity_in_sweep": int(pst[0]["formal_fuse"]),
                           "opacity_tangent_depths_per_thread": int(pst[0]["opacity_depths"])},
                "tick_stages_ms": stage_breakdown(pst[0])}
    st0 = allstats[-1]
    line = {"metric": METRIC, "value": pts / (total_ms * 1e-3), "unit": "ray-points/s", "n_gpus": ws,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": total_ms / args.steps,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": MIXED_DTYPE, "data": "synthetic",
            "config": batch_config(wl.columns, atms[0].n_nu, "mixed precision"),
            "columns_per_s": conv / (total_ms * 1e-3),
            "converged_fraction": conv / (len(atms) * args.steps * ws),
            "fp64_one_column_per_launch_columns_per_s": fp64_cols_s,
            "speedup_vs_fp64_per_column": (conv / (total_ms * 1e-3)) / (fp64_cols_s * ws),
            "latency_ms": {"p50": float(np.percentile(times, 50)), "p99": float(np.percentile(times, 99))},
            "solve": {"F_calls_max": max(s["F_calls"] for s in st0),
                      "F_calls_median": float(np.median([s["F_calls"] for s in st0])),
                      "F_norm_drop_max": max(s["F_norm"] / s["F_norm0"] for s in st0 if s["F_norm0"] > 0)},
            "setup_s": setup_s,
            "device_memory_gb": {"tables_and_batch": (free0 - free1) / 1e9, "device_total": total_mem / 1e9},
            "roofline": roofline,
            "e2e": {"value": e2e_pts / e2e_s, "unit": "ray-points/s",
                    "h2d_bytes_per_step": int(offs[-1]) * 8, "d2h_bytes_per_step": int(offs[-1]) * 8,
                    "steps": len(e2e_times), "call": "jfnk_batch_run with pinned host populations in and out"},
            "gpu_launches": int(st0[0]["kernel_launches"]) * args.steps,
            "clocks": clocks}
    if cpu is not None:
        pool, futs, workers, t_cpu0 = cpu
        cb, res = cpu_baseline_batch(wl, BATCH_START, pool, futs, workers, t_cpu0)
        pool.shutdown()
        line["cpu_baseline"] = cb
        errs = [float(np.max(np.abs(n_gpu[c] / r["n"] - 1.0))) for c, r in enumerate(res) if r["converged"]]
        line["oracle_error"] = {"max_rel": max(errs), "columns": len(errs),
                                "what": "GPU mixed batch vs FP64 oracle, both solved to the paper's stopping "
                                        "rule, populations of the sampled columns (max over elements)"}
    print(json.dumps(line), flush=True)


RTOLS = (1e-4, 3e-4, 1e-3, 3e-3, 1e-2, 3e-2, 1e-1)


def run_rtol(args, rank, ws, local, dist):
    """The experiment of Sect. 2.3 / Fig. 5 and Sect. 3.3 on the synthetic
    columns: formal solutions (F-class evaluations) to the paper's stopping
    rule for JFNK with GMRES and with BiCGSTAB over a range of Krylov
    tolerances r_tol, and for the reference method alone (RH92 iterations
    until the population change is below the same 1e-4), one column per solve
    on the GPU. Config 2 (Ca II-like, FP64, from LTE) and config 3 (H I-like,
    mixed, JFNK after the hybrid RH92 start). Accuracy reached = max relative
    difference from the same column solved far past the stopping rule
    (FP64, r_tol 1e-6, ftol 1e-10)."""
    import torch
    from paper_2406_17234_gb300 import binding as B
    if rank != 0:
        return
    torch.cuda.set_device(local)
    ctx = B.Context(local)
    cases = [("config 2 (Ca II-like, 82 depths, FP64, from LTE)", W.config2(), B.JFNK_FP64, {}),
             ("config 3 (H I-like, 82 depths, mixed, hybrid start)", W.config3(), B.JFNK_MIXED,
              dict(rh92_warmup=60, rh92_switch=0.03))]
    out, headline, total_ms = {}, None, 0.0

    def timed_solve(atm, o):
        B.solve(atm, o, raise_on_fail=False)              # warm: buffers, tuning, graphs
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record()
        n, _, st = B.solve(atm, o, raise_on_fail=False)
        e1.record()
        e1.synchronize()
        return n, st, e0.elapsed_time(e1)

    for name, wl, prec, start in cases:
        atom = B.Atom(ctx, wl.atom)
        atm = B.Atmosphere(ctx, atom, wl.columns[0], n_mu=wl.n_mu)
        ref, _, sref = B.solve(atm, B.default_options(rtol=1e-6, ftol=1e-10, **start))
        rows = {}
        for kname, kr in (("gmres", B.JFNK_KRYLOV_GMRES), ("bicgstab", B.JFNK_KRYLOV_BICGSTAB)):
            for rt in RTOLS:
                n, st, ms = timed_solve(atm, B.default_options(precision=prec, rtol=rt, krylov=kr, **start))
                total_ms += ms
                rows.setdefault(kname, {})[f"{rt:g}"] = {
                    "F_calls": st["F_calls"], "jvp_calls": st["jvp_calls"], "newton_iters": st["newton_iters"],
                    "rh92_iters": st["rh92_iters"], "status": st["status"], "ms": ms,
                    "F_norm_drop": st["F_norm"] / st["F_norm0"] if st["F_norm0"] > 0 else None,
                    "max_rel_err": float(np.max(np.abs(n / ref - 1.0)))}
        for key, pr in (("rh92", prec), ("rh92_fp64", B.JFNK_FP64)):
            if key == "rh92_fp64" and prec == B.JFNK_FP64:
                continue
            n, st, ms = timed_solve(atm, B.default_options(precision=pr, solver=B.JFNK_SOLVER_RH92, maxiter=5000))
            total_ms += ms
            rows[key] = {"F_calls": st["F_calls"], "status": st["status"], "ms": ms,
                         "F_norm_drop": st["F_norm"] / st["F_norm0"] if st["F_norm0"] > 0 else None,
                         "max_rel_err": float(np.max(np.abs(n / ref - 1.0)))}
        best = min((v["F_calls"], k, rt) for k in ("gmres", "bicgstab") for rt, v in rows[k].items()
                   if v["status"] == 0)
        rows["summary"] = {"best_jfnk": {"krylov": best[1], "rtol": float(best[2]), "F_calls": best[0]},
                           "rh92_over_best_jfnk_F_calls": rows["rh92"]["F_calls"] / best[0],
                           "reference_F_calls": sref["F_calls"]}
        out[name] = rows
        if headline is None:
            headline = rows["gmres"]["0.01"]["F_calls"]
    line = {"metric": "formal solutions to the paper's stopping rule (JFNK-GMRES, r_tol 1e-2, config 2)",
            "value": headline, "unit": "F-class evaluations", "n_gpus": 1, "steps": 1, "warmup": 1,
            "ms_per_step": total_ms, "higher_is_better": False, "scaling": "weak", "vs_baseline": None,
            "dtype": "f64 (config 2) / " + MIXED_DTYPE + " (config 3)", "data": "synthetic",
            "config": {"workload": "r_tol sweep: JFNK-GMRES, JFNK-BiCGSTAB and RH92 alone, configs 2 and 3",
                       "rtol": list(RTOLS), "stopping": "1/2 ||dn/n||_inf < 1e-4 (and ||F|| drop 1e-2 for JFNK)"},
            "sweep": out}
    print(json.dumps(line), flush=True)


def serve_options(atom):
    """Start options per atom kind of the serving stream: the H I-like columns
    need a longer RH92 warm-up (Sect. 3.5 hybrid) than the others."""
    from paper_2406_17234_gb300 import binding as B
    if atom.name.startswith("H"):
        return B.default_options(precision=B.JFNK_MIXED, rh92_warmup=60, rh92_switch=0.03)
    return B.default_options(precision=B.JFNK_MIXED, rh92_warmup=10, rh92_switch=0.1)


def run_serve(args, rank, ws, local, dist):
    """Serving stream (continuous batching): requests arrive on a seeded Poisson
    schedule; a producer thread builds each request's atom and atmosphere
    tables at its arrival time and submits it; the main thread steps the
    server and retires results. Latency = completion - scheduled arrival, so a
    request that waits (for the producer, a slot or memory) pays for it."""
    import threading
    import torch
    from paper_2406_17234_gb300 import binding as B
    wl = W.config5(n_requests=args.requests, rate=args.rate, seed=rank_seed(20240624, rank))
    torch.cuda.set_device(local)
    ctx = B.Context(local)
    # slot shape: the stream's largest column (frequency counts from the atoms)
    max_nq = max(sum(l.n_nu for l in a.lines) + sum(c.n_nu for c in a.conts) for a in wl.atoms)
    sv = B.Server(ctx, max_slots=args.slots, max_depth=max(c.n_depth for c in wl.columns), max_freq=max_nq,
                  max_levels=max(a.n_levels for a in wl.atoms),
                  max_trans=max(len(a.lines) + len(a.conts) for a in wl.atoms), max_mu=wl.n_mu,
                  opts=serve_options(wl.atoms[1]))
    n = len(wl.columns)
    live = {}                     # id -> (atom, atmosphere) until retired
    lock = threading.Lock()
    # requests built but not retired (their tables live on the device): a few
    # slots' worth of queue, capped so that large slot counts keep memory
    window = threading.Semaphore(min(4 * args.slots, 2048))
    err = []
    t_start = sv.clock()
    arrivals = t_start + np.asarray(wl.arrivals)

    def producer(first):
        try:
            for r in range(first, n, args.producers):
                window.acquire()
                wait = arrivals[r] - sv.clock()
                if wait > 0:
                    time.sleep(wait)
                atom = B.Atom(ctx, wl.atoms[r])
                atm = B.Atmosphere(ctx, atom, wl.columns[r], n_mu=wl.n_mu)
                with lock:
                    live[r] = (atom, atm)
                sv.submit(atm, r, serve_options(wl.atoms[r]))
        except Exception as e:   # surfaced by the main thread
            err.append(e)

    ths = [threading.Thread(target=producer, args=(i,), daemon=True) for i in range(args.producers)]
    clk = clocks_start() if rank == 0 else None
    for th in ths:
        th.start()
    done = []
    while len(done) < n and not err:
        active, queued = sv.step()
        res = sv.poll()
        for r in res:
            with lock:
                live.pop(r["id"], None)
            window.release()
        done += res
        if active == 0 and not res:
            time.sleep(2e-4)
    for th in ths:
        th.join()
    clocks = clocks_stop(clk, local) if rank == 0 else None
    if err:
        raise err[0]
    t_end = max(r["t_done"] for r in done)
    conv = [r for r in done if r["status"] == 0]
    lat = np.array([r["t_done"] - arrivals[r["id"]] for r in done])
    pts = float(sum(r["stats"]["ray_points"] for r in done))
    wall = t_end - t_start
    sv.close()
    mx, sm = reduce_ranks(dist, [wall, len(conv), pts])
    wall, nconv, pts = mx[0], sm[1], sm[2]
    if rank != 0:
        return
    line = {"metric": "converged NLTE columns/s", "value": nconv / wall, "unit": "columns/s", "n_gpus": ws,
            "steps": 1, "warmup": 0, "ms_per_step": wall * 1e3, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": MIXED_DTYPE, "data": "synthetic",
            "config": {"workload": f"serving: {n} column solves, Poisson arrivals at {args.rate:g}/s, atoms "
                                   "20 % two-level / 40 % Ca II-like / 40 % H I-like, depths 48-300, "
                                   "500-2000 frequencies, mixed precision, continuous batching",
                       "slots": args.slots, "requests": n,
                       "l2": "inputs of the in-flight columns exceed L2 (work buffers of hundreds of columns)"},
            "latency_ms": {"p50": float(np.percentile(lat, 50) * 1e3), "p99": float(np.percentile(lat, 99) * 1e3)},
            "queueing_ms": {  # where the latency goes: building the request, waiting for a slot, solving
                "submit_after_arrival_p50": float(np.median([r["t_submit"] - arrivals[r["id"]] for r in done]) * 1e3),
                "admit_after_submit_p50": float(np.median([r["t_admit"] - r["t_submit"] for r in done]) * 1e3),
                "solve_p50": float(np.median([r["t_done"] - r["t_admit"] for r in done]) * 1e3)},
            "producer_threads": args.producers,
            "converged_fraction": len(conv) / n, "ray_points_per_s": pts / wall,
            "not_converged": [{"id": int(r["id"]), "atom": wl.atoms[r["id"]].name,
                               "n_depth": int(wl.columns[r["id"]].n_depth),
                               "n_nu_lines_conts": int(sum(l.n_nu for l in wl.atoms[r["id"]].lines)
                                                       + sum(c.n_nu for c in wl.atoms[r["id"]].conts)),
                               "status": int(r["status"]), "F_calls": int(r["stats"]["F_calls"]),
                               "newton_iters": int(r["stats"]["newton_iters"]),
                               "rh92_iters": int(r["stats"]["rh92_iters"]),
                               "F_norm_drop": (r["stats"]["F_norm"] / r["stats"]["F_norm0"]
                                               if r["stats"]["F_norm0"] > 0 else None)}
                              for r in done if r["status"] != 0][:50],
            "offered_rate": args.rate, "clocks": clocks}
    print(json.dumps(line), flush=True)


def main():
    args = parse()
    rank, ws, local, dist = dist_setup()
    if args.impl == "reference":
        run_reference(args, rank, ws, dist)
    elif args.workload == "batch":
        run_batch(args, rank, ws, local, dist)
    elif args.workload == "serve":
        run_serve(args, rank, ws, local, dist)
    elif args.workload == "rtol":
        run_rtol(args, rank, ws, local, dist)
    else:
        run_ours(args, rank, ws, local, dist)
    if dist is not None:
        dist.barrier()
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
