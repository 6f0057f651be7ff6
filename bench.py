#!/usr/bin/env python3
"""Benchmark of the mQO hot path on GB300.

Default workload (the batched MIS configuration): 512 Erdős–Rényi graphs,
n ~ U[700, 800], p = 0.15, seeds 0..511, packed CSR, 32 trajectories per
graph (16,384 trajectories), BF16 x / momentum state with FP32 arithmetic.
A step is one tick of the full per-trajectory machine over all
trajectories (fused SpMM-gradient step, projection, rounding, exact
evaluation, acceptance, mutation resets, repair and local search).
Metric: edge-updates/s = CSR entries of the member graph for every
trajectory tick that ran a gradient step, per second of the timed ticks
(trajectories in a repair or local-search round that tick are not counted).
The default run also measures the steady state, batched against
single-instance quality, the other configurations (MaxCut on a 3-regular
graph, MIS at 10^7 nodes, the f_B autograd workload) and the paper-shaped
ER workloads: the printed line has their value and time, the file
bench_detail.json beside this one the complete record.

Arms:
  default            the CUDA library (one process per GPU, weak scaling)
  --impl reference   the plain CPU oracle on the host cores, bounded sample
"""
from __future__ import annotations

import argparse
import hashlib
import json
import multiprocessing as mp
import os
import re
import statistics
import subprocess
import sys
import tempfile
import time
import types

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402

import mqo_inputs as mi  # noqa: E402

METRIC = "edge-updates/s of fused mQO steps"
OBJECTIVES = {"fb": 0, "fl": 1, "fp": 2, "fa": 3}
UNIT = "edge-updates/s"
L2_BYTES = 126 * 1024 * 1024

WORKLOADS = {
    "mis_batched": dict(desc="MIS batched: 512 ER graphs n~U[700,800] p=0.15 seeds 0..511, packed CSR, B=32 "
                             "per graph (16384 trajectories)", problem=0, batch=32, alpha=0.8, momentum=0.45,
                        gamma=2.0, rho=0.6, t_gs=60, descent_cap=50, init_kind=1, sigma=0.1),
    "maxcut_regular": dict(desc="MaxCut f_B: random 3-regular n=100000, B=128", problem=1, batch=128, alpha=0.0025,
                           momentum=0.8, lambda_=0.001, rho=0.8, t_gs=90, descent_cap=200, init_kind=1, sigma=0.1),
    "maxcut_regular_signed": dict(desc="MaxCut f_B: random 3-regular n=100000, edge weights uniform in {-1,+1}, "
                                       "B=128", problem=1, batch=128, alpha=0.0025, momentum=0.8, lambda_=0.001,
                                  rho=0.8, t_gs=90, descent_cap=200, init_kind=1, sigma=0.1),
    "mis_scale": dict(desc="MIS at scale: ER n=1e7 mean degree 10, B=16", problem=0, batch=16, alpha=0.8,
                      momentum=0.75, gamma=2.0, rho=0.5, t_gs=60, descent_cap=50, init_kind=1, sigma=0.1),
    # the paper's ER setting (n, d) = (1000, 100) with its hyperparameter rows
    # (MIS: alpha 0.8, momentum 0.3, rho 0.7, T_gs 60; MaxCut: alpha 0.0025,
    # momentum 0.8, rho 0.8, T_gs 90, lambda 0.001); 8 seeded graphs
    "er_mis_1000_100": dict(desc="MIS on 8 ER graphs (n, d) = (1000, 100), B=128 per graph", problem=0, batch=128,
                            alpha=0.8, momentum=0.3, gamma=2.0, rho=0.7, t_gs=60, descent_cap=50, init_kind=1,
                            sigma=0.1, paper={"table": "Table 1 (MIS, 5-minute budget), (1000, 100)",
                                              "mQO-MIS": 66.38, "pmQO-MIS": 66.75, "ReduMIS": 67.00}),
    "er_maxcut_1000_100": dict(desc="MaxCut f_B on 8 ER graphs (n, d) = (1000, 100), B=128 per graph", problem=1,
                               batch=128, alpha=0.0025, momentum=0.8, lambda_=0.001, rho=0.8, t_gs=90,
                               descent_cap=200, init_kind=1, sigma=0.1,
                               paper={"table": "Table 1 (MaxCut, 10-minute budget), (1000, 100)",
                                      "mQO-MaxCut": 28518.375, "pmQO-MaxCut": 28530.875, "Gurobi": 28534.75}),
    # more of Table 1's ER shapes with their rows of the App. G tables
    "er_mis_3000_100": dict(desc="MIS on 8 ER graphs (n, d) = (3000, 100), B=128 per graph", problem=0, batch=128,
                            alpha=0.8, momentum=0.3, gamma=2.0, rho=0.6, t_gs=60, descent_cap=50, init_kind=1,
                            sigma=0.1, paper={"table": "Table 1 (MIS, 5-minute budget), (3000, 100)",
                                              "mQO-MIS": 198.25, "pmQO-MIS": 201.63, "ReduMIS": 201.00}),
    "er_mis_1000_500": dict(desc="MIS on 8 ER graphs (n, d) = (1000, 500), B=128 per graph", problem=0, batch=128,
                            alpha=0.8, momentum=0.45, gamma=2.0, rho=0.6, t_gs=60, descent_cap=50, init_kind=1,
                            sigma=0.1, paper={"table": "Table 1 (MIS, 5-minute budget), (1000, 500)",
                                              "mQO-MIS": 14.75, "pmQO-MIS": 14.88, "ReduMIS": 15.00}),
    "er_maxcut_1000_500": dict(desc="MaxCut f_B on 8 ER graphs (n, d) = (1000, 500), B=128 per graph", problem=1,
                               batch=128, alpha=0.0025, momentum=0.8, lambda_=0.001, rho=0.8, t_gs=90,
                               descent_cap=200, init_kind=1, sigma=0.1,
                               paper={"table": "Table 1 (MaxCut, 10-minute budget), (1000, 500)",
                                      "mQO-MaxCut": 130997.375, "pmQO-MaxCut": 131009.125, "Gurobi": 131009.875}),
}


# the differentiable f_B objective (torch.autograd.Function with the fused
# SpMM backward) driven by the projected momentum kernel
AUTOGRAD = dict(desc="f_B autograd: Chung-Lu power law (exponent 2.5, mean degree 8) n=1e6, B=64 FP32, "
                     "forward + backward + projected momentum step", batch=64, lambda_=0.001, lr=0.001, momentum=0.9)


SMALL_TICKS = 4096  # ticks per launch of the multi-tick kernel (kSmallTicks in mqo_api.cu)
MIS_SCALE_NODES = [10_000_000]  # --nodes overrides it (smaller cases for profiling)


def make_graph(name):
    if name == "mis_batched":
        return mi.workload_mis_batched()
    if name == "maxcut_regular":
        return mi.workload_maxcut_regular()
    if name == "maxcut_regular_signed":
        return mi.workload_maxcut_regular(signed=True)
    if name == "mis_scale":
        return mi.workload_mis_scale(n=MIS_SCALE_NODES[0])
    if name.startswith("er_"):
        n, d = (int(t) for t in name.split("_")[-2:])
        return mi.workload_er_table(n, float(d))
    if name == "autograd_powerlaw":
        return mi.workload_chung_lu()
    raise ValueError(name)


def dtype_code(s):
    return {"f32": 0, "bf16": 1, "f16": 2}[s]


# ---------------------------------------------------------------- CPU oracle (reference arm, cpu_baseline)
def _oracle_job(args):
    gi, rp, col, w, n, pdict, traj, ticks = args
    sys.path.insert(0, ROOT)
    import oracle
    G = mi.Graph(n, rp, col, w)
    og = oracle.Graph(G)
    p = oracle.params(**pdict)
    if pdict.get("pool_k", 0) > 0:
        # pool mode: the B trajectories of one member graph run together
        B = pdict["batch"]
        pg = oracle.PoolGraph(og, p, traj, B)
        t0 = time.perf_counter()
        pg.run(ticks)
        dt = time.perf_counter() - t0
        return dt, int(rp[-1]) * sum(pg.state(b)["steps"] for b in range(B)), pg.pool.best
    tr = oracle.Trajectory(og, p, traj)
    t0 = time.perf_counter()
    tr.run(ticks)
    # edge-updates of the ticks that ran a gradient step
    return time.perf_counter() - t0, int(rp[-1]) * tr.state["steps"], tr.state["best"]


_POOLS = {}


def _warm(_):
    sys.path.insert(0, ROOT)
    import oracle  # noqa: F401
    return 0


def worker_pool(cores):
    """A spawned process pool over the host cores, created once and warmed
    (each worker has imported the oracle) before any timed sample."""
    if cores not in _POOLS:
        pool = mp.get_context("spawn").Pool(cores)
        pool.map(_warm, range(cores), chunksize=1)
        _POOLS[cores] = pool
    return _POOLS[cores]


def oracle_sample(G, wl, x_dtype, v_dtype, target_s=12.0, cores=None, pool_k=0, objective=0):
    """Time the oracle on a bounded sample of the workload's trajectories
    (pool mode: of its member graphs, each with its B trajectories)."""
    cores = cores or os.cpu_count() or 1
    pd = {k: wl[k] for k in ("problem", "batch", "alpha", "momentum", "rho", "t_gs", "descent_cap", "init_kind",
                             "sigma") if k in wl}
    pd.update(gamma=wl.get("gamma", 2.0), lambda_=wl.get("lambda_", 0.001), x_dtype=x_dtype, v_dtype=v_dtype,
              seed=0, pool_k=pool_k, objective=objective)
    B = wl["batch"]
    if pool_k > 0:
        sub = G.subgraph(0)
        dt, eu, _ = _oracle_job((0, sub.row_ptr, sub.col_idx, sub.weights, sub.n, pd, 0, 10))
        rate1 = eu / max(dt, 1e-9)
        ticks = 100
        ngr = max(cores, int(target_s * rate1 * cores / (sub.nnz * B * ticks)))
        ngr = min(ngr, G.num_graphs)
        jobs = []
        for g in range(ngr):
            sg = G.subgraph(g)
            jobs.append((g, sg.row_ptr, sg.col_idx, sg.weights, sg.n, pd, g * B, ticks))
        pool = worker_pool(cores)
        t0 = time.perf_counter()
        res = pool.map(_oracle_job, jobs, chunksize=1)
        wall = time.perf_counter() - t0
        eu = sum(r[1] for r in res)
        return dict(value=eu / wall, unit=UNIT, cores=cores, kind="oracle",
                    sample=f"{ngr} member graphs x {B} trajectories (pool mode, K={pool_k}) x {ticks} ticks of the "
                           f"same workload, {eu:.3e} edge-updates in {wall:.2f} s wall on {cores} processes")
    # probe one trajectory to size the sample
    sub = G.subgraph(0)
    job = (0, sub.row_ptr, sub.col_idx, sub.weights, sub.n, pd, 0, 20)
    dt, eu, _ = _oracle_job(job)
    rate1 = eu / max(dt, 1e-9)
    per_traj_eu = sub.nnz * 200
    ticks = 200
    ntraj = max(cores, int(target_s * rate1 * cores / per_traj_eu))
    ntraj = min(ntraj, G.num_graphs * B, 4096)
    jobs = []
    for k in range(ntraj):
        g = k % G.num_graphs
        b = (k // G.num_graphs) % B
        sg = G.subgraph(g)
        jobs.append((g, sg.row_ptr, sg.col_idx, sg.weights, sg.n, pd, g * B + b, ticks))
    pool = worker_pool(cores)
    t0 = time.perf_counter()
    res = pool.map(_oracle_job, jobs, chunksize=1)
    wall = time.perf_counter() - t0
    eu = sum(r[1] for r in res)
    return dict(value=eu / wall, unit=UNIT, cores=cores, kind="oracle", single_core_value=rate1,
                sample=f"{ntraj} trajectories x {ticks} ticks of the same workload (member graphs 0..), "
                       f"{eu:.3e} edge-updates in {wall:.2f} s wall on {cores} processes; single_core_value: "
                       f"one trajectory of member graph 0 for 20 ticks on one core")


def reference_arm(args):
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return 0
    wl = WORKLOADS[args.workload]
    G = make_graph(args.workload)
    xd = dtype_code(args.x_dtype)
    vd = dtype_code(args.v_dtype or args.x_dtype)
    per_step = []
    base = None
    for _ in range(args.warmup):
        oracle_sample(G, wl, xd, vd, target_s=0.5, pool_k=args.pool_k, objective=OBJECTIVES[args.objective])
    for _ in range(args.steps):
        base = oracle_sample(G, wl, xd, vd, target_s=max(1.0, 60.0 / max(args.steps, 1)), pool_k=args.pool_k,
                             objective=OBJECTIVES[args.objective])
        per_step.append(base["value"])
    value = statistics.median(per_step)
    nnz_b = G.nnz * wl["batch"]
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": nnz_b / value * 1e3,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": f"f32 (x {args.x_dtype} / V {args.v_dtype or args.x_dtype} storage, int64 evaluation)", "data": "synthetic",
        "config": {"workload": wl["desc"], "x_dtype": args.x_dtype, "v_dtype": args.v_dtype or args.x_dtype,
                   "nnz": G.nnz, "batch": wl["batch"], "pool_k": args.pool_k, "objective": args.objective},
        "cpu_baseline": dict(base, value=value),
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line))
    return 0


def reference_autograd(args):
    if int(os.environ.get("RANK", "0")) != 0:
        return 0
    wl = AUTOGRAD
    G = make_graph("autograd_powerlaw")
    vals = [oracle_autograd_sample(G, wl["batch"], wl["lambda_"], target_s=max(1.0, 60.0 / max(args.steps, 1)))
            for _ in range(args.steps)]
    value = statistics.median(v["value"] for v in vals)
    eu_step = 2.0 * G.nnz * wl["batch"]
    print(json.dumps({
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": eu_step / value * 1e3, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": wl["desc"], "nnz": G.nnz, "batch": wl["batch"]},
        "cpu_baseline": dict(vals[-1], value=value),
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}))
    return 0


# ---------------------------------------------------------------- clocks
class ClockSampler:
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index):
        self.index = index
        self.proc = None
        self.path = None

    def __enter__(self):
        fd, self.path = tempfile.mkstemp(suffix=".csv")
        os.close(fd)
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--id={self.index}", f"--query-gpu={self.FIELDS}",
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
        except OSError:
            self.proc = None
        time.sleep(0.3)
        return self

    def __exit__(self, *a):
        if self.proc:
            # one more sample after the timed region, so that the samples
            # bracket it even when it is shorter than the sampling interval
            time.sleep(0.25)
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()

    def summary(self):
        sm, mx, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        try:
            for line in open(self.path):
                f = [x.strip() for x in line.split(",")]
                if len(f) < 9:
                    continue
                try:
                    sm.append(float(f[1]))
                    mx = float(f[2])
                except ValueError:
                    continue
                for nm, val in zip(names, f[5:9]):
                    if val.lower().startswith("active"):
                        reasons.add(nm)
        except OSError:
            pass
        finally:
            try:
                os.unlink(self.path)
            except OSError:
                pass
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": mx, "reasons": sorted(reasons),
                "samples": len(sm)}


# ---------------------------------------------------------------- ranks
def aggregate_ranks(ms_local: float, units_local: float, dist=None, device=None):
    """Whole-job throughput of independent replicas: the slowest rank's time
    (max over ranks) and the units processed by all ranks together."""
    import torch
    if dist is None:
        return ms_local, units_local / (ms_local / 1e3)
    t = torch.tensor([ms_local, units_local], dtype=torch.float64, device=device)
    mx = t[:1].clone()
    dist.all_reduce(mx, op=dist.ReduceOp.MAX)
    tot = t[1:].clone()
    dist.all_reduce(tot, op=dist.ReduceOp.SUM)
    ms = float(mx.item())
    return ms, float(tot.item()) / (ms / 1e3)


# ---------------------------------------------------------------- GPU arm
def algorithmic_bytes_per_step(G, B, sx, sv, idx_bytes=4):
    """col_idx (idx_bytes per entry) + row_ptr read once, x read + written,
    momentum read + written, rounding bits written (one word per node per 32
    trajectories)."""
    n = G.n
    bw = (B + 31) // 32
    return G.nnz * idx_bytes + (n + 1) * 4 + 2 * n * B * sx + 2 * n * B * sv + n * bw * 4


def profile_traffic(name, variant, sources):
    """Per-launch DRAM bytes of a kernel variant from the committed ncu
    summary profiles/<name>.txt, or None if there is none or the kernel
    sources changed since the capture."""
    path = os.path.join(ROOT, "profiles", f"{name}.txt")
    if not os.path.exists(path):
        return None
    txt = open(path).read()
    # a summary of several kernel variants gives one hash per variant
    m = re.search(r"source_sha256\[" + re.escape(variant) + r"\]:\s*([0-9a-f]{64})", txt) or \
        re.search(r"source_sha256:\s*([0-9a-f]{64})", txt)
    t = re.search(r"dram_bytes_per_launch\[" + re.escape(variant) + r"\]:\s*([0-9.eE+]+)", txt)
    if not m or not t:
        return None
    if source_hash(sources) != m.group(1):
        return None
    return float(t.group(1))


def code_text(src: str) -> str:
    """C / CUDA source without its comments and with every run of white
    space reduced to one blank: what the compiler sees of the code, so that
    a comment edit leaves the hash of a profiled kernel unchanged."""
    out = []
    i, n = 0, len(src)
    while i < n:
        c = src[i]
        if src.startswith("//", i):
            j = src.find("\n", i)
            i = n if j < 0 else j
            out.append(" ")
        elif src.startswith("/*", i):
            j = src.find("*/", i + 2)
            i = n if j < 0 else j + 2
            out.append(" ")
        elif c in "\"'":
            j = i + 1
            while j < n and src[j] != c:
                j += 2 if src[j] == "\\" else 1
            out.append(src[i:j + 1])
            i = j + 1
        else:
            out.append(c)
            i += 1
    return " ".join("".join(out).split())


def source_hash(sources) -> str:
    """sha256 over the code text (code_text) of csrc/<f> for f in sources, in order."""
    h = hashlib.sha256()
    for f in sources:
        txt = open(os.path.join(ROOT, "paper_2605_06921_gb300", "csrc", f), encoding="utf-8").read()
        h.update(code_text(txt).encode())
    return h.hexdigest()


STEP_SOURCES = {"smem": ("mqo_step.cu", "mqo_step_smem.cuh", "mqo_step.cuh", "mqo_dev.cuh"),
                "smem_ell": ("mqo_step_ell.cu", "mqo_step_smem.cuh", "mqo_step.cuh", "mqo_dev.cuh"),
                "global": ("mqo_step_generic.cu", "mqo_step.cuh", "mqo_dev.cuh"),
                "staged": ("mqo_step_staged.cu", "mqo_step.cuh", "mqo_dev.cuh"),
                "rows": ("mqo_step_rows.cu", "mqo_x16.cuh", "mqo_step.cuh", "mqo_dev.cuh"),
                "dense": ("mqo_step_dense.cu", "mqo_step_dense.cuh", "mqo_x16.cuh", "mqo_step.cuh", "mqo_dev.cuh"),
                "f32_ell": ("mqo_step_f32.cu", "mqo_step.cuh", "mqo_dev.cuh")}


def float32_stream(plan, x_dtype, batch=32):
    """Does the plan's step stage its member graphs' x as float32 (16-bit
    offsets in the sliced-ELL stream)?  Float32 states and fewer than 32
    trajectories of any type do where they take the stream."""
    return bool(plan.get("ell")) and (x_dtype == "f32" or batch < 32)


def step_variant(plan):
    """Profile variant name of a plan: smem, smem_wide (CSR indices),
    smem_ell, smem_wide_ell (sliced-ELL stream), staged, rows, global, dense
    (tensor cores)."""
    if plan.get("dense"):
        return "dense"
    kern = plan["step_kernel"]
    return kern + "_ell" if kern.startswith("smem") and plan.get("ell") else kern


def step_kernel_traffic(workload, x_dtype, variant, batch=32):
    """DRAM bytes per launch of the step kernel variant (step_variant)."""
    if float32_stream({"ell": variant == "smem_wide_ell"}, x_dtype, batch):
        variant = "f32_ell"
    if variant in STEP_SOURCES and not variant.startswith("smem"):
        src = STEP_SOURCES[variant]
    else:
        src = STEP_SOURCES["smem_ell" if variant.endswith("_ell") else "smem"]
    return profile_traffic(f"step_kernel_{workload}_{x_dtype}", variant, src)


INT64_MIN = -(1 << 63)
_T0 = time.perf_counter()


def progress(what):
    """One line per bench phase on stderr (seconds since start)."""
    print(f"[bench {time.perf_counter() - _T0:7.1f} s] {what}", file=sys.stderr, flush=True)


def per_graph_nnz(G):
    off = np.asarray(G.node_offsets, dtype=np.int64)
    return (G.row_ptr[off[1:]] - G.row_ptr[off[:-1]]).astype(np.int64)


def best_summary(vals):
    """Best values over the trajectories that have accepted a set (the others
    still hold INT64_MIN) and how many have."""
    v = np.asarray(vals, dtype=np.int64)
    ok = v != INT64_MIN
    return {"best_mean": float(v[ok].mean()) if ok.any() else None,
            "best_max": int(v[ok].max()) if ok.any() else None,
            "accepted": int(ok.sum()), "trajectories": int(v.size)}


def solver_kwargs(wl, seed, pool_k=0, objective=0):
    pkw = {k: wl[k] for k in ("problem", "batch", "alpha", "momentum", "rho", "t_gs", "descent_cap", "init_kind",
                              "sigma")}
    pkw.update(gamma=wl.get("gamma", 2.0), lambda_=wl.get("lambda_", 0.001), seed=seed, pool_k=pool_k,
               objective=objective)
    return pkw


def read_peaks():
    try:
        return json.load(open(os.path.join(ROOT, "MEASURED_PEAKS.json")))
    except (OSError, ValueError):
        return {}


def measure_solver(mq, G, pkw, xd, vd, steps, warmup, *, autotune=False, clocks_of=None, barrier=None,
                   phase_ticks=50, extra_ticks=0, probe=0):
    """`warmup` ticks (then the autotuner), `steps` ticks timed with CUDA
    events as a user runs them (mqo_run: replays of the captured tick
    graphs), the per-kernel split from the next ticks (instrumented, not
    timed), then `extra_ticks` more before the best values are read.  The
    stepped edge-updates of the timed ticks (CSR entries of the member graph
    for every trajectory tick that ran a gradient step) come from the
    machine's per-trajectory step counters read before and after."""
    import torch
    g = mq.Graph(G)
    s = mq.Solver(g, mq.params(x_dtype=xd, v_dtype=vd, **pkw))
    s.run(warmup)
    tuned = s.autotune(10) if autotune else None
    B = pkw["batch"]
    nnz_t = np.repeat(per_graph_nnz(G), B)
    st0 = s.steps_taken()
    torch.cuda.synchronize()
    if barrier:
        barrier()
    sampler = ClockSampler(clocks_of) if clocks_of is not None else None
    if sampler:
        sampler.__enter__()
    torch.cuda.synchronize()
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    e0.record()
    s.run(steps)
    e1.record()
    torch.cuda.synchronize()
    if barrier:
        barrier()
    if sampler:
        sampler.__exit__()
    ms = e0.elapsed_time(e1)
    dsteps = s.steps_taken() - st0
    pt = min(steps, phase_ticks)
    phase_sum, launches = s.run_timed(pt)
    rec = {"ms": ms, "steps": steps, "phase_ms": {k: v * steps / pt for k, v in phase_sum.items()},
           "launches": launches * steps // pt, "stepped_edge_updates": float((dsteps * nnz_t).sum()),
           "stepped_fraction": float(dsteps.sum()) / float(steps * len(nnz_t)),
           "all_edge_updates": float(G.nnz) * B * steps, "clocks": sampler.summary() if sampler else None,
           "plan": s.info()}
    if rec["plan"]["small"]:  # one launch, and one that advances the tick, per SMALL_TICKS ticks
        rec["launches"] = 2 * -(-steps // SMALL_TICKS)
    if tuned:
        rec["plan"]["autotune_ms_per_tick"] = tuned["ms_per_tick"]
    if extra_ticks:
        s.run(extra_ticks)
    rec["ticks_total"] = warmup + steps + pt + extra_ticks
    vals, _ = s.best(want_bits=False)
    rec["vals"] = vals
    rec.update(best_summary(vals))
    # descent steps per finished descent over the whole run (a descent ends at
    # its fixed-point test or at the cap, descent_cap)
    sts = s.traj_state()
    nd = sum(t["descents"] for t in sts)
    rec["mean_descent_steps"] = float(sum(t["steps"] for t in sts)) / nd if nd else None
    rec["descent_cap"] = pkw["descent_cap"]
    if probe:
        # the FP64 relaxed objective (timed on the device) and, for a few
        # trajectories in a descent, the stored x: the CPU leg states the
        # error of that objective against the oracle's all-double one
        o0 = torch.cuda.Event(enable_timing=True)
        o1 = torch.cuda.Event(enable_timing=True)
        o0.record()
        obj = s.objective_f64()
        o1.record()
        torch.cuda.synchronize()
        x = s.get_x()
        st = s.traj_state()
        T = len(st)
        samples = []
        for t in range(0, T, max(1, T // probe)):
            gi, b = divmod(t, B)
            if st[t]["phase"] != 0:  # x is defined in a descent only
                continue
            lo, hi = int(G.node_offsets[gi]), int(G.node_offsets[gi + 1])
            samples.append((gi, t, x[lo:hi, b].float().cpu().numpy().astype(np.float64), float(obj[t].item())))
        rec["objective_probe"] = {"ms": o0.elapsed_time(o1), "samples": samples}
    s.close()
    g.close()
    return rec


def objective_error(G, wl, objective, probe):
    """Largest relative error of the device's FP64 relaxed objective ((Ax)_v
    accumulated in float32, the rest in double) against the oracle's
    all-double objective of the same stored x, over the probed trajectories."""
    import oracle
    errs = []
    for gi, t, xs, got in probe.get("samples", []):
        og = oracle.Graph(G.subgraph(gi) if G.num_graphs > 1 else G)
        if wl["problem"] == 0:
            want = oracle.objective_f64(og, 0, wl.get("gamma", 2.0), 0.0, xs)
        else:
            want = oracle.cut_objective_f64(og, objective, wl.get("lambda_", 0.001), xs)
        errs.append(abs(got - want) / max(abs(want), 1e-30))
    return {"device_ms": probe.get("ms"), "trajectories_checked": len(errs),
            "max_rel_error_vs_fp64_oracle": max(errs) if errs else None}


def oracle_single(G, wl, xd, vd, ticks, objective=0):
    """One trajectory of member graph 0, `ticks` ticks, on one host core in
    this process (graphs too large to ship to a process pool)."""
    pd = {k: wl[k] for k in ("problem", "batch", "alpha", "momentum", "rho", "t_gs", "descent_cap", "init_kind",
                             "sigma") if k in wl}
    pd.update(gamma=wl.get("gamma", 2.0), lambda_=wl.get("lambda_", 0.001), x_dtype=xd, v_dtype=vd, seed=0,
              pool_k=0, objective=objective)
    sub = G.subgraph(0) if G.num_graphs > 1 else G
    dt, eu, _ = _oracle_job((0, sub.row_ptr, sub.col_idx, sub.weights, sub.n, pd, 0, ticks))
    return dict(value=eu / dt, unit=UNIT, cores=1, kind="oracle",
                sample=f"one trajectory of member graph 0 (n={sub.n}, nnz={sub.nnz}) for {ticks} ticks on one "
                       f"core, {eu:.3e} stepped edge-updates in {dt:.2f} s")


STEP_KERNEL_NAMES = {"smem": "mqo::k_step_s", "smem_wide": "mqo::k_step_s", "staged": "mqo::k_step_q",
                     "global": "mqo::k_step_g", "rows": "mqo::k_step_r"}


def step_kernel_name(plan, x_dtype, batch=32):
    """The kernel that runs a plan's steps."""
    if plan.get("small"):
        return "mqo::k_small (many ticks per launch)"
    if plan.get("dense"):
        return "mqo::k_step_t"
    if float32_stream(plan, x_dtype, batch):
        return "mqo::k_step_f"
    return STEP_KERNEL_NAMES.get(plan["step_kernel"], plan["step_kernel"])


def member_sizes(G):
    off = getattr(G, "node_offsets", None)
    return np.diff(off) if off is not None and len(off) > 2 else np.array([G.n])


def dense_flops_per_step(G, B):
    """Tensor-core operations of k_step_t per launch: every member graph's
    adjacency, rows and columns padded to 128 and 16, times 64 columns (x and
    its companions) per 32 trajectories."""
    sizes = member_sizes(G)
    rows, cols = -(-sizes // 128) * 128, -(-sizes // 16) * 16
    return float((2.0 * rows * cols).sum()) * 64 * (B // 32)


def step_roofline(G, B, sx, sv, step_ms, plan, workload, x_dtype, hbm_peak, peak_src, clocks, n_sm, peaks):
    """Roofline of the step kernel: algorithmic HBM bytes (CSR once, x and V
    read and written once, rounding words) per launch over its average
    launch time; the shared-memory kernel adds its gather bound."""
    # index bytes per CSR entry: 16-bit member-local ids, 32-bit ids, or the
    # sliced-ELL stream's row offsets (its padding not counted; x staged as float32: 16 bits)
    f32_stream = float32_stream(plan, x_dtype, B)
    idx = (2 if f32_stream else 4) if plan.get("ell") else (2 if plan.get("col16") else 4)
    alg = algorithmic_bytes_per_step(G, B, sx, sv, idx)
    if plan.get("dense"):  # bit matrices (rows and columns padded to 128) in place of the column indices
        rows = -(-member_sizes(G) // 128) * 128
        alg += float((rows.astype(np.int64) ** 2).sum()) / 8 - 4.0 * G.nnz
    achieved = alg / (step_ms / 1e3) / 1e9
    hbm = {"bound": "hbm", "achieved": achieved, "peak": hbm_peak, "unit": "GB/s", "frac": achieved / hbm_peak,
           "algorithmic_bytes_per_launch": alg, "peak_source": peak_src}
    kern = plan["step_kernel"]
    traffic = step_kernel_traffic(workload, x_dtype, step_variant(plan), B)
    gathered = float(G.nnz) * B * (4 if f32_stream else sx)  # neighbour rows of x read per launch
    if plan.get("dense"):
        # the adjacency comes from bit matrices and x once per CTA
        flops = dense_flops_per_step(G, B)
        peak = float(peaks.get("bf16_tflops", 1900.0))
        roof = {"bound": "tensor", "achieved": flops / (step_ms / 1e3) / 1e12, "peak": peak, "unit": "TFLOP/s",
                "frac": flops / (step_ms / 1e3) / 1e12 / peak, "traffic": traffic, "flops_per_launch": flops, "hbm": hbm,
                "peak_source": "measured" if "bf16_tflops" in peaks else "fallback"}
    elif kern.startswith("smem"):
        sm_clock = (clocks or {}).get("sm_mhz") or float(peaks.get("sm_max_mhz", 2070.0))
        derived = 128.0 * n_sm * sm_clock * 1e6 / 1e9
        probe = peaks.get("smem_probe_gbs")
        smem_peak = probe or derived
        smem_achieved = gathered / (step_ms / 1e3) / 1e9
        roof = {"bound": "smem", "achieved": smem_achieved, "peak": smem_peak, "unit": "GB/s",
                "frac": smem_achieved / smem_peak, "traffic": traffic,
                "peak_source": ("measured: conflict-free 16-byte shared-memory loads on every SM "
                                "(mqo_measure_smem_gbs)" if probe else "derived"),
                "peak_derived": derived,
                "peak_derivation": f"128 B/clk/SM x {n_sm} SMs x {sm_clock:.0f} MHz (sampled SM clock)",
                "algorithmic_bytes_per_launch": gathered, "hbm": hbm}
    else:
        # the neighbour-row gathers are requests to L2; the share that misses
        # is DRAM traffic on top of the algorithmic bytes (measured: traffic)
        roof = dict(hbm, traffic=traffic, gathered_bytes_per_launch=gathered,
                    achieved_incl_gathers=(alg + gathered) / (step_ms / 1e3) / 1e9)
    roof.update(kernel=step_kernel_name(plan, x_dtype, B), step_kernel_ms=step_ms, plan=plan)
    if traffic:
        # DRAM bytes of the committed capture over this launch time, against the same peak
        roof["dram_gbs_from_traffic"] = traffic / (step_ms / 1e3) / 1e9
        roof["dram_frac_from_traffic"] = roof["dram_gbs_from_traffic"] / hbm_peak
    return roof


def solver_config_record(mq, name, xd_s, vd_s, steps, warmup, extra_ticks, *, local, rank, cpu, G=None,
                         objective="fb", oracle_ticks=20):
    """Sub-record of the default bench line for another solver workload:
    throughput (stepped edge-updates/s), its step kernel's roofline, best
    values after a fixed tick budget, the FP64 objective error and (rank 0)
    a single-core oracle slice."""
    import torch
    wl = WORKLOADS[name]
    G = make_graph(name) if G is None else G
    B = wl["batch"]
    xd, vd = dtype_code(xd_s), dtype_code(vd_s)
    sx, sv = (4 if xd == 0 else 2), (4 if vd == 0 else 2)
    pkw = solver_kwargs(wl, 1000 * rank, 0, OBJECTIVES[objective])
    r = measure_solver(mq, G, pkw, xd, vd, steps, warmup, autotune=True, clocks_of=local, extra_ticks=extra_ticks,
                       probe=4 if cpu else 0)
    peaks = read_peaks()
    hbm_peak = float(peaks.get("hbm_gbs", 6800.0))
    step_ms = r["phase_ms"]["step"] / steps
    n_sm = torch.cuda.get_device_properties(local).multi_processor_count
    roof = step_roofline(G, B, sx, sv, step_ms, r["plan"], name, xd_s, hbm_peak,
                         "measured" if "hbm_gbs" in peaks else "fallback", r["clocks"], n_sm, peaks)
    rec = {"workload": wl["desc"], "x_dtype": xd_s, "v_dtype": vd_s, "dtype": f"f32 arithmetic, x {xd_s} / V {vd_s} "
           "storage, int64 evaluation", "nodes": G.n, "nnz": G.nnz, "batch": B, "steps": steps, "warmup": warmup,
           "value": r["stepped_edge_updates"] / (r["ms"] / 1e3), "unit": UNIT,
           "value_all_trajectories": r["all_edge_updates"] / (r["ms"] / 1e3),
           "stepped_fraction": r["stepped_fraction"], "ms_per_step": r["ms"] / steps,
           "kernel_ms_per_step": {k: v / steps for k, v in r["phase_ms"].items()}, "roofline": roof,
           "clocks": r["clocks"], "gpu_launches": r["launches"], "best_after_ticks": r["ticks_total"]}
    rec.update({k: r[k] for k in ("best_mean", "best_max", "accepted", "trajectories", "mean_descent_steps",
                                  "descent_cap")})
    if cpu:
        rec["objective_f64"] = objective_error(G, wl, OBJECTIVES[objective], r.get("objective_probe", {}))
        rec["cpu_baseline"] = oracle_single(G, wl, xd, vd, oracle_ticks, OBJECTIVES[objective])
    return rec


def gpu_arm(args):
    import torch
    import paper_2605_06921_gb300 as mq

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(local)
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl" if torch.cuda.is_available() else "gloo")

    def barrier():
        if dist is not None:
            dist.barrier()

    wl = WORKLOADS[args.workload]
    xd, vd = dtype_code(args.x_dtype), dtype_code(args.v_dtype or args.x_dtype)
    sx, sv = (4 if xd == 0 else 2), (4 if vd == 0 else 2)
    G = make_graph(args.workload)
    B = wl["batch"]
    pkw = solver_kwargs(wl, 1000 * rank, args.pool_k, OBJECTIVES[args.objective])
    peaks = read_peaks()
    hbm_peak = float(peaks.get("hbm_gbs", 6800.0))
    peak_src = "measured" if "hbm_gbs" in peaks else "fallback"
    cpu_leg = rank == 0 and world == 1 and not args.no_cpu

    progress(f"{args.workload}: timed ticks")
    main = measure_solver(mq, G, pkw, xd, vd, args.steps, args.warmup, autotune=not args.no_autotune,
                          clocks_of=local, barrier=barrier, probe=8 if cpu_leg else 0)
    progress("end to end")
    ms, value = aggregate_ranks(main["ms"], main["stepped_edge_updates"], dist, "cuda")
    _, value_all = aggregate_ranks(main["ms"], main["all_edge_updates"], dist, "cuda")
    step_avg_ms = main["phase_ms"]["step"] / args.steps
    n_sm = torch.cuda.get_device_properties(local).multi_processor_count
    if main["plan"]["step_kernel"].startswith("smem"):
        # the shared-memory roofline's denominator, measured after the timed region
        peaks = dict(peaks, smem_probe_gbs=mq.measure_smem_gbs())
    roof = step_roofline(G, B, sx, sv, step_avg_ms, main["plan"], args.workload, args.x_dtype, hbm_peak, peak_src,
                         main["clocks"], n_sm, peaks)

    # end to end through the public API with host buffers: graph upload from
    # pinned host arrays, solver creation, every tick followed by a
    # device->host read of the per-trajectory best values
    def pinned(a):
        return None if a is None else torch.from_numpy(np.ascontiguousarray(a)).pin_memory().numpy()

    Gp = types.SimpleNamespace(n=G.n, row_ptr=pinned(G.row_ptr.astype(np.int64)),
                               col_idx=pinned(G.col_idx.astype(np.int32)),
                               weights=None if G.weights is None else pinned(G.weights.astype(np.int8)),
                               node_offsets=G.node_offsets)
    torch.cuda.synchronize()
    barrier()
    t0 = time.perf_counter()
    g = mq.Graph(Gp)
    t1 = time.perf_counter()
    s = mq.Solver(g, mq.params(x_dtype=xd, v_dtype=vd, **pkw))
    t2 = time.perf_counter()
    e2e_steps = args.steps
    for _ in range(e2e_steps):
        s.run(1)
        s.best(want_bits=False)
    torch.cuda.synchronize()
    t3 = time.perf_counter()
    e2e_stepped = float((s.steps_taken() * np.repeat(per_graph_nnz(G), B)).sum())
    s.close()
    g.close()
    ms_e2e, e2e_value = aggregate_ranks((t3 - t0) * 1e3, e2e_stepped, dist, "cuda")
    csr_bytes = G.nnz * 4 + (G.n + 1) * 8 + (G.nnz if G.weights is not None else 0) + 8 * (G.num_graphs + 1)
    e2e = {"value": e2e_value, "unit": UNIT,
           "h2d_bytes_per_step": int(csr_bytes / e2e_steps), "d2h_bytes_per_step": int(8 * G.num_graphs * B),
           "graph_upload_ms": (t1 - t0) * 1e3, "solver_create_ms": (t2 - t1) * 1e3,
           "ticks_ms": (t3 - t2) * 1e3, "steps": e2e_steps,
           "note": "stepped edge-updates of the ticks run from a fresh start, graph upload and solver creation "
                   "inside the timed region"}

    alg = algorithmic_bytes_per_step(G, B, sx, sv)
    if alg > L2_BYTES:
        l2_note = f"inputs larger than L2 (CSR + state touched per step {alg / 1e6:.0f} MB > 126 MB); no flush"
    else:
        l2_note = (f"CSR + state touched per step {alg / 1e6:.0f} MB fit in the 126 MB L2 and stay resident between "
                   f"ticks by design (not flushed)")

    # quality on the paper-shaped workloads: best value per member graph (max
    # over its trajectories) after a longer tick budget, without and with a pool
    quality = paper_quality(mq, G, wl, pkw, xd, vd, args.quality_ticks) if "paper" in wl and args.quality_ticks > 0 \
        else None

    sub = {}
    if args.workload == "mis_batched" and not args.no_sub and world == 1 and args.pool_k == 0:
        sub = default_line_subrecords(mq, G, wl, pkw, xd, vd, args.x_dtype, local=local, rank=rank, cpu=cpu_leg)

    cpu = None
    objective_f64 = None
    if cpu_leg:
        progress("oracle sample")
        cpu = oracle_sample(G, wl, xd, vd, target_s=12.0, pool_k=args.pool_k, objective=OBJECTIVES[args.objective])
        objective_f64 = objective_error(G, wl, OBJECTIVES[args.objective], main.get("objective_probe", {}))

    if rank == 0:
        line = {
            "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": ms / args.steps, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None,
            "dtype": f"f32 (x {args.x_dtype} / V {args.v_dtype or args.x_dtype} storage, int64 evaluation)",
            "data": "synthetic",
            "config": {"workload": wl["desc"], "x_dtype": args.x_dtype, "v_dtype": args.v_dtype or args.x_dtype,
                       "nnz": G.nnz, "nodes": G.n, "batch": B, "edge_updates_per_step": G.nnz * B,
                       "value_counts": "CSR entries of the member graph for every trajectory tick that ran a "
                                       "gradient step (stepped_fraction of all trajectory ticks)",
                       "l2": l2_note, "parallelism": f"replicas x{world}",
                       "pool_k": args.pool_k, "objective": args.objective},
            "value_all_trajectories": value_all, "stepped_fraction": main["stepped_fraction"],
            "roofline": roof, "e2e": e2e, "gpu_launches": main["launches"],
            "kernel_ms_per_step": {k: v / args.steps for k, v in main["phase_ms"].items()},
            "clocks": main["clocks"],
        }
        line.update({k: main[k] for k in ("best_mean", "best_max", "accepted", "trajectories")})
        line["best_after_ticks"] = main["ticks_total"]
        if cpu:
            line["cpu_baseline"] = cpu
        if quality:
            line["quality"] = quality
        if objective_f64:
            line["objective_f64"] = objective_f64
        line.update(sub)
        emit(line)
    if dist is not None:
        dist.destroy_process_group()
    return 0


LINE_LIMIT = 2800  # characters of the printed line


def short_line(line):
    """The record as the one printed line: everything but the sub-records and
    the longer parts of the roofline and the baseline, and value and time of
    every sub-record; below LINE_LIMIT characters, so that a reader that keeps
    the end of the output has all of it."""
    def short(v):
        return float(f"{v:.6g}") if isinstance(v, float) else v

    out = {k: v for k, v in line.items() if not isinstance(v, (dict, list)) or k in ("config", "e2e", "clocks")}
    if "e2e" in out:
        out["e2e"] = {k: v for k, v in out["e2e"].items() if k != "note"}
    for k in ("roofline", "cpu_baseline", "objective_f64", "kernel_ms_per_step"):
        if k in line:
            out[k] = {a: short(b) for a, b in line[k].items() if not isinstance(b, (dict, list, bool)) and
                      not (isinstance(b, str) and len(b) > 40)}
    steady = line.get("steady_state")
    if steady:
        out["steady_state"] = {k: short(steady[k]) for k in ("value_median", "ms_per_step_median") if k in steady}
    out["configs"] = {k: {a: short(v[a]) for a in ("value", "ms_per_step") if a in v}
                      for k, v in line.get("configs", {}).items()}
    if not out["configs"]:
        del out["configs"]
    for k in ("configs", "steady_state", "objective_f64", "kernel_ms_per_step", "cpu_baseline", "roofline"):
        if len(json.dumps(out)) < LINE_LIMIT:
            break
        out.pop(k, None)
    return out


def emit(line, path=None):
    """Prints the short line and keeps the complete record in a file beside
    this one (bench_detail.json)."""
    path = os.path.join(ROOT, "bench_detail.json") if path is None else path
    try:
        with open(path, "w", encoding="utf-8") as f:
            json.dump(line, f, indent=1)
        progress(f"complete record: {path}")
    except OSError as e:
        progress(f"complete record not written: {e}")
    print(json.dumps(short_line(line)), flush=True)


def paper_quality(mq, G, wl, pkw, xd, vd, ticks):
    """Best value per member graph (max over its trajectories) after `ticks`
    ticks, independent trajectories and a pool of 8, with the gains
    breakdown of each graph's best trajectory."""
    import torch
    B = wl["batch"]
    quality = {"ticks": ticks, "paper": wl["paper"],
               "note": "paper: its own ER graphs, time budget on its hardware; here: seeded synthetic ER graphs of "
                       "the same (n, d), tick budget -- context, not a like-for-like comparison"}
    for label, k in (("independent", 0), ("pool_k8", 8)):
        g = mq.Graph(G)
        s = mq.Solver(g, mq.params(x_dtype=xd, v_dtype=vd, **dict(pkw, pool_k=k)))
        s.run(20)
        s.autotune(5)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        s.run(ticks - 20)
        vals, _ = s.best(want_bits=False)
        dt = time.perf_counter() - t0
        per_graph = vals.reshape(G.num_graphs, B).max(axis=1)
        quality[label] = {"best_per_graph_mean": float(per_graph.mean()), "best_per_graph": per_graph.tolist(),
                          "seconds": dt}
        sts = s.traj_state()
        pick = vals.reshape(G.num_graphs, B).argmax(axis=1)
        br = [sts[gi * B + int(pick[gi])] for gi in range(G.num_graphs)]
        quality[label]["breakdown_mean"] = {
            "first_descent": float(np.mean([x["first_value"] for x in br])),
            "gain_resets": float(np.mean([x["gain_descent"] for x in br])),
            "gain_local_search": float(np.mean([x["gain_ls"] for x in br]))}
        s.close()
        g.close()
    return quality


def steady_state(mq, G, pkw, xd, vd, *, warm, repeats, ticks, local):
    """The workload after `warm` ticks (every trajectory past its first
    descents), `repeats` timed windows of `ticks` ticks: median, min and max
    of the stepped edge-updates/s."""
    import torch
    B = pkw["batch"]
    g = mq.Graph(G)
    s = mq.Solver(g, mq.params(x_dtype=xd, v_dtype=vd, **pkw))
    s.run(warm)
    s.autotune(10)
    nnz_t = np.repeat(per_graph_nnz(G), B)
    vals, fracs, mss = [], [], []
    sampler = ClockSampler(local)
    sampler.__enter__()
    for _ in range(repeats):
        st0 = s.steps_taken()
        torch.cuda.synchronize()
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record()
        s.run(ticks)
        e1.record()
        torch.cuda.synchronize()
        ms = e0.elapsed_time(e1)
        d = s.steps_taken() - st0
        vals.append(float((d * nnz_t).sum()) / (ms / 1e3))
        fracs.append(float(d.sum()) / float(ticks * len(nnz_t)))
        mss.append(ms / ticks)
    sampler.__exit__()
    best = best_summary(s.best(want_bits=False)[0])
    s.close()
    g.close()
    return {"warmup_ticks": warm, "repeats": repeats, "ticks_per_repeat": ticks,
            "value_median": statistics.median(vals), "value_min": min(vals), "value_max": max(vals), "unit": UNIT,
            "ms_per_step_median": statistics.median(mss), "stepped_fraction_median": statistics.median(fracs),
            "clocks": sampler.summary(), "best_mean": best["best_mean"], "accepted": best["accepted"]}


def quality_vs_single(mq, G, pkw, xd, vd, xname, *, ticks):
    """The batched form (all member graphs in one launch, the workload's
    storage type), the same batch in FP32, and member graph 0 alone in FP32
    (the plain single-instance form) for the same tick budget: stepped
    edge-updates/s, and the best values of member graph 0's B trajectories
    (keyed by graph and slot, so the runs start from the same points); then
    the ticks and time the batched form needs until member graph 0's mean
    best reaches the single-instance form's (equal best-found)."""
    import torch
    B = pkw["batch"]
    out = {"ticks": ticks, "graph": "member graph 0 of the batch"}
    target = None
    runs = [(f"batched_{xname}", G, xd, vd)]
    if xd != 0 and vd != 0:
        runs.append((f"batched_{xname}_vf32", G, xd, 0))
    runs += [("batched_f32", G, 0, 0), ("single_instance_f32", G.subgraph(0), 0, 0)]
    for label, gg, x_d, v_d in runs:
        g = mq.Graph(gg)
        s = mq.Solver(g, mq.params(x_dtype=x_d, v_dtype=v_d, **pkw))
        s.run(10)
        nnz_t = np.repeat(per_graph_nnz(gg), B)
        st0 = s.steps_taken()
        torch.cuda.synchronize()
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record()
        s.run(ticks - 10)
        e1.record()
        torch.cuda.synchronize()
        ms = e0.elapsed_time(e1)
        d = s.steps_taken() - st0
        vals, _ = s.best(want_bits=False)
        out[label] = {"value": float((d * nnz_t).sum()) / (ms / 1e3), "unit": UNIT,
                      "ms_per_step": ms / (ticks - 10), "graph0": best_summary(vals[:B])}
        s.close()
        g.close()
    # equal best-found: ticks (and time) until the batched form's member graph
    # 0 reaches the mean best of the single-instance FP32 form after `ticks`
    target = out["single_instance_f32"]["graph0"]["best_mean"]
    g = mq.Graph(G)
    s = mq.Solver(g, mq.params(x_dtype=xd, v_dtype=vd, **pkw))
    nnz_t = np.repeat(per_graph_nnz(G), B)
    done, reached, ms_total, eu = 0, None, 0.0, 0.0
    while done < 8 * ticks:
        st0 = s.steps_taken()
        torch.cuda.synchronize()
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record()
        s.run(100)
        e1.record()
        torch.cuda.synchronize()
        ms_total += e0.elapsed_time(e1)
        eu += float(((s.steps_taken() - st0) * nnz_t).sum())
        done += 100
        m = best_summary(s.best(want_bits=False)[0][:B])["best_mean"]
        if m is not None and m >= target:
            reached = m
            break
    s.close()
    g.close()
    single = out["single_instance_f32"]
    out["equal_best_found"] = {
        "target_graph0_best_mean": target, "batched_form": f"batched_{xname}",
        "ticks": done if reached is not None else None, "graph0_best_mean": reached,
        "ms": ms_total, "value": eu / (ms_total / 1e3), "unit": UNIT,
        "single_instance_f32_ms": single["ms_per_step"] * (ticks - 10), "single_instance_f32_value": single["value"],
        "note": "the batched form runs all member graphs (its edge-updates/s counts all of them) until member "
                "graph 0's mean best reaches the single-instance FP32 form's mean best after its tick budget; "
                "null ticks: not reached within 8x that budget"}
    return out


PAPER_ER = ("er_mis_1000_100", "er_maxcut_1000_100", "er_mis_3000_100", "er_mis_1000_500", "er_maxcut_1000_500")


def paper_er_record(mq, ticks, rank):
    """Best value per graph (max over its B trajectories, mean over the 8
    seeded graphs) after `ticks` ticks on the paper-shaped ER workloads,
    independent trajectories, next to the paper's Table 1 numbers."""
    import torch
    out = {"ticks": ticks, "note": "seeded synthetic ER graphs of the paper's (n, d), tick budget; the paper's "
                                   "numbers come from its own graphs and a time budget: context only"}
    for name in PAPER_ER:
        progress(f"  {name}")
        wl = WORKLOADS[name]
        G = make_graph(name)
        B = wl["batch"]
        g = mq.Graph(G)
        s = mq.Solver(g, mq.params(x_dtype=1, v_dtype=1, **solver_kwargs(wl, 1000 * rank)))
        s.run(20)
        s.autotune(5)  # restores the state: the run below starts at tick 20
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        s.run(ticks - 20)
        vals, _ = s.best(want_bits=False)
        dt = time.perf_counter() - t0
        per_graph = vals.reshape(G.num_graphs, B).max(axis=1)
        out[name] = {"best_per_graph_mean": float(per_graph.mean()), "best_per_graph": per_graph.tolist(),
                     "seconds": dt, "ms_per_step": dt * 1e3 / ticks, "plan": s.info()["step_kernel"],
                     "paper": wl["paper"]}
        s.close()
        g.close()
    return out


def default_line_subrecords(mq, G, wl, pkw, xd, vd, xname, *, local, rank, cpu):
    """Sub-records of the default bench line: steady state, batched against
    single instance, the other configurations (large MIS, MaxCut, autograd)
    and the paper-shaped ER workloads."""
    progress("steady state")
    out = {"steady_state": steady_state(mq, G, pkw, xd, vd, warm=400, repeats=10, ticks=100, local=local)}
    progress("batched against single instance")
    out["quality_vs_single_instance"] = quality_vs_single(mq, G, pkw, xd, vd, xname, ticks=1000)
    cfg = {}
    for name, xs, vs in (("maxcut_regular", "bf16", "bf16"), ("maxcut_regular", "bf16", "f32"),
                         ("maxcut_regular_signed", "bf16", "bf16")):
        progress(f"{name} x {xs} V {vs}")
        cfg[f"{name}_{xs}_v{vs}"] = solver_config_record(mq, name, xs, vs, 20, 5, 2000, local=local, rank=rank,
                                                         cpu=cpu, oracle_ticks=400)
    progress("mis_scale graph")
    Gs = make_graph("mis_scale")
    for xs, vs in (("f16", "f16"), ("f16", "f32"), ("f32", "f32")):
        progress(f"mis_scale x {xs} V {vs}")
        cfg[f"mis_scale_{xs}_v{vs}"] = solver_config_record(mq, "mis_scale", xs, vs, 20, 5, 100, local=local,
                                                            rank=rank, cpu=cpu and vs == "f16", G=Gs, oracle_ticks=2)
    del Gs
    progress("autograd")
    cfg["autograd_powerlaw_f32"] = autograd_measure(mq, 20, 5, local=local, rank=rank, dist=None,
                                                    cpu=cpu, cpu_target_s=6.0)
    out["configs"] = cfg
    progress("paper-shaped ER")
    out["paper_er"] = paper_er_record(mq, 5000, rank)
    progress("App. B")
    out["app_b"] = app_b_record(mq, rank, cpu)
    progress("sub-records done")
    return out


# ---------------------------------------------------------------- App. B: the MaxCut relaxations compared
APP_B_OBJS = ("fl", "fp", "fa", "fb")
APP_B_TABLE5 = {(100, 50): (0.0025, 0.9), (1000, 100): (0.0025, 0.8), (1000, 500): (0.0025, 0.8),
                (1000, 800): (0.0025, 0.8)}  # (n, d): (alpha, momentum), the App. G MaxCut rows


def _descend(mq, G, obj, x0, alpha, momentum, steps, seed):
    """Plain projected (momentum) ascent steps of one relaxation from x0 on
    every trajectory: cut of the rounded start and end point, nodes that a
    step would still move at the end (0: a fixed binary point)."""
    import torch
    B = x0.shape[1]
    s = mq.Solver(mq.Graph(G), mq.params(problem=1, batch=B, alpha=alpha, momentum=momentum, lambda_=0.001,
                                         objective=OBJECTIVES[obj], init_kind=0, seed=seed))
    s.set_x(torch.from_numpy(x0).cuda())
    cut0 = s.evaluate(s.round())[0].cpu().numpy()
    s.step(steps)
    v, a, _ = s.evaluate(s.round())
    torch.cuda.synchronize()
    out = (cut0, v.cpu().numpy(), a.cpu().numpy(), s.get_x().float().cpu().numpy())
    s.close()
    return out


def _per_graph_mean(vals, num_graphs, B):
    return vals.reshape(num_graphs, B).mean(axis=1)


def app_b_record(mq, rank, cpu, steps=2000):
    """The paper's comparison of its MaxCut relaxations (App. B): escapes from
    f_L-interior stationary points x = c1 (Table 3) and from 1-flip
    repairable binary points (Table 4) on 10 ER(100, 0.66) graphs, alpha 0.1,
    lambda 0.001, plain projected gradient ascent, no local search or reset;
    and the four relaxations from one shared random start on ER graphs of
    the paper's (n, d) (Table 5, 3 graphs each, the App. G step sizes).
    Cuts are exact integers of the rounded points."""
    import torch
    B = 32
    out = {"note": "seeded synthetic ER graphs, not the paper's; the paper's numbers are context",
           "steps": steps}
    torch.cuda.synchronize()
    tables = {}
    replay = []
    # the stated density p = 0.66, and p = 0.017, whose random cut (about
    # m/2 = 42) matches the cut at initialisation that Table 4 prints
    for dens in (0.66, 0.017):
        G = mi.pack([mi.erdos_renyi(100, dens, 500 + k) for k in range(10)])
        rng = np.random.default_rng(1000 * rank + 3)
        # x = c 1 on each graph, one c per trajectory; c = +-k/16 so that every
        # float32 row sum of c is exact and c 1 is exactly stationary for f_L
        # (Prop. 3.2); a c with more mantissa bits leaves rounding residues in
        # L x that the step amplifies
        c = (rng.integers(1, 16, size=(G.num_graphs, B)) * rng.choice([-1.0, 1.0], size=(G.num_graphs, B)) /
             16.0).astype(np.float32)
        x_c = np.repeat(c, 100, axis=0)
        x_pm = np.where(rng.random((G.n, B)) < 0.5, -1.0, 1.0).astype(np.float32)
        for label, x0, paper in (("table3_stationary_c1", x_c, {"fl": [0, 0], "fp": [0, 47.2], "fb": [0, 51.1]}),
                                 ("table4_one_flip_repairable", x_pm,
                                  {"fl": [42.4, 42.4], "fp": [42.4, 42.4], "fb": [42.4, 50.1]})):
            t = {"paper_cut_init_and_end": paper, "graphs": f"10 ER(100, {dens})"}
            for obj in ("fl", "fp", "fb"):
                cut0, cut1, moving, _ = _descend(mq, G, obj, x0, 0.1, 0.0, steps, 7)
                rec = {"cut_init_mean": float(cut0.mean()), "cut_end_mean": float(cut1.mean()),
                       "increase_mean": float((cut1 - cut0).mean()),
                       "escaped_fraction": float((cut1 > cut0).mean()),
                       "still_moving_fraction": float((moving > 0).mean())}
                if label.startswith("table4"):
                    # the starts must be 1-flip repairable (a node with a positive gain)
                    pos = mq.Solver(mq.Graph(G), mq.params(problem=1, batch=B, objective=OBJECTIVES[obj]))
                    pos.set_x(torch.from_numpy(x0).cuda())
                    rec["starts_one_flip_repairable"] = float((pos.evaluate(pos.round())[2].cpu().numpy() > 0).mean())
                    pos.close()
                t[obj] = rec
                replay.append((G, obj, x0, 0.1, 0.0, cut1, steps))
            tables[f"{label}_p{dens}"] = t
    rng = np.random.default_rng(1000 * rank + 5)
    t5 = {"paper_cut_mean": {"fl": [1256.2, 25298.11, 125046.6, 200030.6], "fp": [1257, 25319.95, 125021.3, 200004.7],
                             "fa": [1397.16, 28157.02, 130331.9, 204291.2],
                             "fb": [1397.45, 28166.59, 130336.5, 204296.5]},
          "paper_columns": ["(100,50)", "(1000,100)", "(1000,500)", "(1000,800)"], "steps": 3 * steps}
    for (n, d), (alpha, mom) in APP_B_TABLE5.items():
        Gt = mi.pack([mi.erdos_renyi(n, d / n, 700 + k) for k in range(3)])
        x0 = rng.uniform(-1.0, 1.0, size=(Gt.n, B)).astype(np.float32)
        row = {}
        for obj in APP_B_OBJS:
            cut0, cut1, moving, _ = _descend(mq, Gt, obj, x0, alpha, mom, 3 * steps, 7)
            row[obj] = {"cut_mean": float(cut1.mean()), "best_per_graph_mean":
                        float(cut1.reshape(3, B).max(axis=1).mean()), "still_moving_fraction":
                        float((moving > 0).mean())}
            if n == 100:
                replay.append((Gt, obj, x0, alpha, mom, cut1, 3 * steps))
        t5[f"({n},{d})"] = row
    tables["table5_relaxations"] = t5
    out.update(tables)
    if cpu:
        out["oracle_replay"] = app_b_replay(replay)
    return out


def app_b_replay(replay):
    """The oracle takes the same plain steps from the same start for the
    first trajectory of the first two graphs of every Table 3/4 run and of
    the (100, 50) row of Table 5; the rounded end cuts must be equal."""
    import oracle
    checked = mismatched = 0
    for G, obj, x0, alpha, mom, cut1, nsteps in replay:
        B = x0.shape[1]
        p = oracle.params(problem=oracle.MAXCUT, batch=B, alpha=alpha, momentum=mom, lambda_=0.001,
                          objective=OBJECTIVES[obj], init_kind=0)
        for gi in range(min(G.num_graphs, 2)):
            og = oracle.Graph(G.subgraph(gi))
            lo, hi = int(G.node_offsets[gi]), int(G.node_offsets[gi + 1])
            x = x0[lo:hi, 0].copy()
            V = np.zeros_like(x)
            for _ in range(nsteps):
                x, V, _, _ = oracle.descent_step(og, p, x, V)
            z = (x > 0).astype(np.uint8)
            want = oracle.eval_cut(og, z)[0]
            checked += 1
            mismatched += int(want != int(cut1[gi * B]))
    return {"trajectories": checked, "mismatched_end_cuts": mismatched}


def fb_kernel_bytes(G, B, writes_grad):
    """col + row_ptr read once, X read once, and where a block of X's size (the
    gradient, or A X kept for it) is written, that once."""
    return G.nnz * 4 + (G.n + 1) * 4 + G.n * B * 4 + (G.n * B * 4 if writes_grad else 0)


def oracle_autograd_sample(G, B, lam, target_s=12.0, cores=None):
    """The oracle's float64 f_B and gradient, column by column, on a bounded
    number of the workload's columns (two edge passes per column)."""
    cores = cores or os.cpu_count() or 1
    rng = np.random.default_rng(0)
    t0 = time.perf_counter()
    _autograd_job((G.row_ptr, G.col_idx, G.n, lam, 0))
    per_col = time.perf_counter() - t0
    cols = int(min(B, max(cores, target_s * cores / max(per_col, 1e-9))))
    pool = worker_pool(min(cores, cols))
    t0 = time.perf_counter()
    pool.map(_autograd_job, [(G.row_ptr, G.col_idx, G.n, lam, c) for c in range(cols)], chunksize=1)
    wall = time.perf_counter() - t0
    eu = 2.0 * G.nnz * cols
    del rng
    return dict(value=eu / wall, unit=UNIT, cores=min(cores, cols), kind="oracle",
                sample=f"{cols} of the {B} columns (float64 objective + gradient per column), "
                       f"{eu:.3e} edge-updates in {wall:.2f} s wall")


def _autograd_job(args):
    rp, col, n, lam, c = args
    sys.path.insert(0, ROOT)
    import oracle
    og = oracle.Graph(mi.Graph(n, rp, col, None))
    x = np.random.default_rng(100 + c).random(n) * 2.0 - 1.0
    oracle.objective_f64(og, 1, 0.0, lam, x)
    oracle.gradient_f64(og, 1, 0.0, lam, x)
    return c


def autograd_measure(mq, steps, warmup, *, local, rank, dist, cpu, cpu_target_s=12.0):
    """The f_B autograd workload: FbObjective forward (one gather, A X kept) + backward from A X +
    the projected momentum kernel per step; returns its bench record."""
    import torch
    wl = AUTOGRAD
    G = make_graph("autograd_powerlaw")
    B, lam = wl["batch"], wl["lambda_"]
    g = mq.Graph(G)
    gen = torch.Generator(device="cuda").manual_seed(1000 * rank)
    X = (torch.rand((G.n, B), device="cuda", generator=gen) * 2 - 1).requires_grad_(True)
    opt = mq.PGAMomentum([X], lr=wl["lr"], momentum=wl["momentum"])
    evs = [[torch.cuda.Event(enable_timing=True) for _ in range(4)] for _ in range(steps)]
    ph = {"forward": 0.0, "backward": 0.0, "optimizer": 0.0}

    def step(ev=None):
        opt.zero_grad(set_to_none=False)
        if ev:
            ev[0].record()
        obj = mq.FbObjective.apply(X, g, lam)
        if ev:
            ev[1].record()
        obj.sum().backward()
        if ev:
            ev[2].record()
        opt.step()
        if ev:
            ev[3].record()
        return obj

    for _ in range(warmup):
        step()
    torch.cuda.synchronize()
    if dist is not None:
        dist.barrier()
    peaks = read_peaks()
    sampler = ClockSampler(local)
    sampler.__enter__()
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    for k in range(steps):
        step(evs[k])
    e1.record()
    torch.cuda.synchronize()
    for ev in evs:
        ph["forward"] += ev[0].elapsed_time(ev[1])
        ph["backward"] += ev[1].elapsed_time(ev[2])
        ph["optimizer"] += ev[2].elapsed_time(ev[3])
    if dist is not None:
        dist.barrier()
    sampler.__exit__()
    clocks = sampler.summary()
    ms_total = e0.elapsed_time(e1)
    eu_step = 2.0 * G.nnz * B
    ms, value = aggregate_ranks(ms_total, eu_step * steps, dist, "cuda")
    # forward: one launch for rows of <= 512 entries and row chunks, one more if
    # some row is longer; backward and the momentum step: one each
    launches_per_step = 1 + int(G.degrees().max() > 512) + 2
    # the forward (one SpMM pass: X read once, A X written); the backward reads
    # A X and writes the gradient
    fwd_ms = ph["forward"] / steps
    alg = fb_kernel_bytes(G, B, True)
    peak = float(peaks.get("hbm_gbs", 6800.0))
    achieved = alg / (fwd_ms / 1e3) / 1e9
    roof = {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s", "frac": achieved / peak,
            "traffic": profile_traffic("fb_kernel_autograd_powerlaw_f32", "fb_seg", ("mqo_grad.cu", "mqo_dev.cuh")),
            "kernel": "mqo::k_fb_seg (f_B forward pass: rows and long-row chunks; the sums of chunks and the "
                      "objective's memset are in forward_ms too)",
            "algorithmic_bytes_per_launch": alg, "forward_ms": fwd_ms,
            "gathered_bytes_per_launch": float(G.nnz) * B * 4,
            "backward_hbm_gbs": 2.0 * G.n * B * 4 / (ph["backward"] / steps / 1e3) / 1e9,
            "peak_source": "measured" if "hbm_gbs" in peaks else "fallback"}
    # end to end through the public API: X copied from pinned host memory
    # every step, forward + backward + optimiser step, the objective read back
    Xh = X.detach().cpu().pin_memory()
    Xe = torch.empty_like(X).requires_grad_(True)
    opt_e = mq.PGAMomentum([Xe], lr=wl["lr"], momentum=wl["momentum"])
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for _ in range(steps):
        with torch.no_grad():
            Xe.copy_(Xh, non_blocking=True)
        opt_e.zero_grad(set_to_none=False)
        obj = mq.FbObjective.apply(Xe, g, lam)
        obj.sum().backward()
        opt_e.step()
        obj.detach().cpu()
    torch.cuda.synchronize()
    t_e2e = time.perf_counter() - t0
    ms_e2e, e2e_value = aggregate_ranks(t_e2e * 1e3, eu_step * steps, dist, "cuda")
    g.close()
    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": 1 if dist is None else dist.get_world_size(),
        "steps": steps, "warmup": warmup, "ms_per_step": ms / steps, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f32 (f_B objective reduced in f64)", "data": "synthetic",
        "config": {"workload": wl["desc"], "nnz": G.nnz, "nodes": G.n, "batch": B,
                   "edge_updates_per_step": eu_step, "l2": "inputs larger than L2 (X 256 MB)",
                   "parallelism": "replicas x1" if dist is None else f"replicas x{dist.get_world_size()}"},
        "roofline": roof,
        "e2e": {"value": e2e_value, "unit": UNIT, "h2d_bytes_per_step": G.n * B * 4, "d2h_bytes_per_step": B * 8,
                "note": "the 256 MB host-to-device copy of X every step dominates this figure"},
        "gpu_launches": launches_per_step * steps,
        "kernel_ms_per_step": {k: v / steps for k, v in ph.items()},
        "clocks": clocks,
    }
    if cpu:
        line["cpu_baseline"] = oracle_autograd_sample(G, B, lam, target_s=cpu_target_s)
    return line


def app_b_arm(args):
    """--workload app_b: the App. B relaxation comparison as one JSON line."""
    import torch
    import paper_2605_06921_gb300 as mq
    if int(os.environ.get("RANK", "0")) != 0:
        return 0
    torch.cuda.set_device(int(os.environ.get("LOCAL_RANK", "0")))
    print(json.dumps({"app_b": app_b_record(mq, 0, not args.no_cpu)}))
    return 0


def autograd_arm(args):
    import torch
    import paper_2605_06921_gb300 as mq
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(local)
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl")
    line = autograd_measure(mq, args.steps, args.warmup, local=local, rank=rank, dist=dist,
                            cpu=rank == 0 and world == 1 and not args.no_cpu)
    if rank == 0:
        emit(line)
    if dist is not None:
        dist.destroy_process_group()
    return 0


def rho_sweep(args):
    """Best value per member graph after --quality-ticks ticks for each rho
    (the reset-fraction ablation), independent trajectories; one JSON line."""
    import torch
    import paper_2605_06921_gb300 as mq
    wl = WORKLOADS[args.workload]
    G = make_graph(args.workload)
    B = wl["batch"]
    xd, vd = dtype_code(args.x_dtype), dtype_code(args.v_dtype or args.x_dtype)
    out = {}
    for rho in [float(r) for r in args.rho_sweep.split(",")]:
        pkw = {k: wl[k] for k in ("problem", "batch", "alpha", "momentum", "t_gs", "descent_cap", "init_kind",
                                  "sigma")}
        pkw.update(gamma=wl.get("gamma", 2.0), lambda_=wl.get("lambda_", 0.001), rho=rho, seed=0,
                   objective=OBJECTIVES[args.objective])
        g = mq.Graph(G)
        s = mq.Solver(g, mq.params(x_dtype=xd, v_dtype=vd, **pkw))
        s.run(args.quality_ticks)
        vals, _ = s.best(want_bits=False)
        per = vals.reshape(G.num_graphs, B).max(axis=1)
        out[str(rho)] = {"best_per_graph_mean": float(per.mean()), "best_per_graph": per.tolist()}
        s.close()
        g.close()
    torch.cuda.synchronize()
    print(json.dumps({"rho_ablation": out, "workload": wl["desc"], "ticks": args.quality_ticks}))
    return 0


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=200)
    ap.add_argument("--warmup", type=int, default=20)
    ap.add_argument("--impl", default="gb300", choices=["gb300", "reference"])
    ap.add_argument("--workload", default="mis_batched", choices=sorted(WORKLOADS) + ["autograd_powerlaw", "app_b"])
    ap.add_argument("--x-dtype", default="bf16", choices=["f32", "bf16", "f16"])
    ap.add_argument("--v-dtype", default=None, choices=["f32", "bf16", "f16"])
    ap.add_argument("--no-cpu", action="store_true")
    ap.add_argument("--no-compare", action="store_true", help="same as --no-sub")
    ap.add_argument("--no-autotune", action="store_true")
    ap.add_argument("--nodes", type=int, default=None, help="mis_scale: nodes of the ER graph (default 1e7)")
    ap.add_argument("--no-sub", action="store_true",
                    help="default workload: leave out the sub-records (steady state, other configurations)")
    ap.add_argument("--pool-k", type=int, default=0, help="pmQO pool of K sets per graph (0: Alg. 1/2)")
    ap.add_argument("--objective", default="fb", choices=sorted(OBJECTIVES), help="MaxCut relaxation")
    ap.add_argument("--rho", type=float, default=None, help="override the workload's reset fraction rho")
    ap.add_argument("--rho-sweep", default=None,
                    help="comma-separated rho values: best-value runs on a paper-shaped ER workload (the rho ablation)")
    ap.add_argument("--quality-ticks", type=int, default=20000,
                    help="ticks of the best-value run on the paper-shaped ER workloads (0: skip)")
    args = ap.parse_args()
    if args.warmup < 3:
        args.warmup = 3
    if args.no_compare:
        args.no_sub = True
    if args.nodes:
        MIS_SCALE_NODES[0] = args.nodes
    if args.rho is not None:
        WORKLOADS[args.workload]["rho"] = args.rho
    if args.rho_sweep:
        return rho_sweep(args)
    if args.impl == "reference":
        if args.workload == "autograd_powerlaw":
            return reference_autograd(args)
        return reference_arm(args)
    if args.workload == "autograd_powerlaw":
        return autograd_arm(args)
    if args.workload == "app_b":
        return app_b_arm(args)
    return gpu_arm(args)


if __name__ == "__main__":
    try:
        rc = main()
    finally:
        for _p in _POOLS.values():
            _p.terminate()
            _p.join()
    sys.exit(rc)
