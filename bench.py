#!/usr/bin/env python
"""Benchmark of the Sphynx hot path on one GB300 (or N independent replicas).

A step is one whole partition (Algorithm 2: Laplacian setup, polynomial
preconditioner setup, LOBPCG, embedding, multi-jagged, cut and imbalance) of
the default workload: the 128^3 27-point mesh (2,097,152 vertices,
53,645,816 off-diagonal entries, synthetic stand-in for the paper's Brick3D
meshes), generalized Laplacian, polynomial preconditioner of degree 25,
K = 64 (d = 7), tol 1e-3.  The headline path stores blocks in FP32 and runs
the polynomial chain in BF16 (FP64 Gram / Rayleigh-Ritz / norms); the plain
FP64 path is timed beside it at the same tolerance.

Multi-GPU: the path does not shard in this build (one graph per GPU), so
N > 1 runs N independent replicas ("scaling": "weak").
"""

from __future__ import annotations

import argparse
import csv
import hashlib
import json
import math
import os
import subprocess
import sys
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402

METRIC = "partitions/sec + Laplacian SpMM HBM GB/s, mixed vs FP64 at equal residual"
UNIT = "partitions/s"

WORKLOADS = {
    "c2": dict(desc="3D 27-point mesh 128^3 (2,097,152 vertices, 53,645,816 off-diagonal nnz, unit weights), "
                    "generalized Laplacian, polynomial preconditioner degree 25, K=64 (d=7), LOBPCG tol 1e-3",
               K=64, laplacian="generalized", precond="poly", poly_degree=25, tol=1e-3, seed=2,
               precision="mixed_bf16", golden="c2_oracle.json"),
    "c1": dict(desc="2D 5-point mesh 64x64 (4096 vertices), combinatorial Laplacian, Jacobi, K=4 (d=3), tol 1e-2",
               K=4, laplacian="combinatorial", precond="jacobi", poly_degree=25, tol=1e-2, seed=1,
               precision="fp64", golden="c1_oracle.json"),
    "c3": dict(desc="R-MAT scale 22 (edge factor 16, a=.57 b=.19 c=.19), symmetrised, deduplicated, self-loops "
                    "dropped, largest component; normalized Laplacian, Jacobi, K=256 (d=9), tol 1e-2",
               K=256, laplacian="normalized", precond="jacobi", poly_degree=25, tol=1e-2, seed=3,
               precision="fp32", golden="c3_oracle.json"),
    "c4": dict(desc="2000 random geometric graphs in one batched call (n log-uniform in [1e3, 2e5], mean degree "
                    "about 8, largest component each), combinatorial Laplacian, polynomial preconditioner degree 25 "
                    "per graph, K=8 (d=4) each, FP32 blocks (graphs whose tol theta lies below the float floor "
                    "finish in FP64 blocks) with FP64 Rayleigh-Ritz, tol 1e-3; each phase's LOBPCG iterations in "
                    "one captured graph launch",
               K=8, laplacian="combinatorial", precond="poly", poly_degree=25, tol=1e-3, seed=4,
               precision="fp32", golden="c4_oracle.json", batch=2000, stall_window=0, max_iter=3000),
    "amg": dict(desc="3D 27-point mesh 128^3 (2,097,152 vertices), combinatorial Laplacian, aggregation multigrid "
                     "preconditioner (plain aggregation, degree-3 Chebyshev, ratio 7, <= 5 levels), K=64 (d=7), "
                     "LOBPCG tol 1e-2 (Sphynx's default for regular graphs with multigrid), FP32 blocks",
                K=64, laplacian="combinatorial", precond="amg", poly_degree=25, tol=1e-2, seed=2,
                precision="fp32", golden="amg_oracle.json"),
    "c5": dict(desc="R-MAT scale 24 (edge factor 16, a=.57 b=.19 c=.19), largest component, FP32 edge weights "
                    "uniform in [0.5, 1.5); normalized Laplacian, polynomial preconditioner degree 10, K=1024 "
                    "(d=11), BF16 polynomial chain, tol 1e-2",
               K=1024, laplacian="normalized", precond="poly", poly_degree=10, tol=1e-2, seed=5,
               precision="mixed_bf16", golden=None),
}


def make_graph(name: str):
    import workloads
    if name in ("c2", "amg"):
        return workloads.grid3d(128, 128, 128, 27)
    if name == "c1":
        return workloads.grid2d(64, 64)
    if name == "c3":
        return workloads.rmat(22, 16, 0.57, 0.19, 0.19, seed=3)
    if name == "c5":
        return workloads.random_edge_weights(workloads.rmat(24, 16, 0.57, 0.19, 0.19, seed=5), 0.5, 1.5, seed=5)
    raise ValueError(name)


def peaks() -> dict:
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        with open(p) as f:
            d = json.load(f)
        return {"hbm_gbs": d.get("hbm_gbs"), "src": "measured"}
    return {"hbm_gbs": 6800.0, "src": "fallback"}


# sources whose change invalidates a stored DRAM-traffic figure of the SpMM kernels
TRAFFIC_SOURCES = ("paper_2105_00578_gb300/csrc/spmm_kernels.cuh", "paper_2105_00578_gb300/csrc/spmm.cu",
                   "paper_2105_00578_gb300/csrc/spmm_bf16.cu", "paper_2105_00578_gb300/csrc/spmm_f32.cu",
                   "paper_2105_00578_gb300/csrc/spmm_f64.cu", "paper_2105_00578_gb300/csrc/graph.cu")


def kernel_source_hash() -> str:
    h = hashlib.sha256()
    for rel in TRAFFIC_SOURCES:
        with open(os.path.join(ROOT, rel), "rb") as f:
            h.update(f.read())
    return h.hexdigest()[:16]


def traffic_path(workload: str) -> str:
    return os.path.join(ROOT, "profiles", f"traffic_{workload}.json")


def profiled_traffic(workload: str):
    """DRAM bytes per launch of the workload's dominant kernel, from the JSON
    that `--ingest-ncu` wrote from an ncu capture; None when there is none or
    when the kernel sources changed after the capture."""
    p = traffic_path(workload)
    if not os.path.exists(p):
        return None, None
    with open(p) as f:
        d = json.load(f)
    if d.get("source_hash") != kernel_source_hash():
        return None, d
    return float(d["traffic_bytes_per_launch"]), d


_UNITS = {"byte": 1.0, "Kbyte": 1e3, "Mbyte": 1e6, "Gbyte": 1e9, "Tbyte": 1e12,
          "KB": 1e3, "MB": 1e6, "GB": 1e9, "B": 1.0}


def ingest_ncu(csv_path: str, kernel_regex: str, workload: str, command: str) -> dict:
    """Mean dram__bytes_read.sum + dram__bytes_write.sum per launch of the
    kernels matching kernel_regex in an ncu --csv log (metrics page), written
    to profiles/traffic_<workload>.json with the hash of the SpMM sources."""
    import re
    pat = re.compile(kernel_regex)
    per = {}
    with open(csv_path, newline="") as f:
        rows = [r for r in csv.reader(f) if r]
    names = ("dram__bytes_read.sum", "dram__bytes_write.sum")
    head = next((i for i, r in enumerate(rows) if "Metric Name" in r and "Kernel Name" in r), None)
    if head is not None:
        # the details page: one row per (launch, metric)
        cols = rows[head]
        ci = {c: cols.index(c) for c in ("ID", "Kernel Name", "Metric Name", "Metric Unit", "Metric Value")}
        for r in rows[head + 1:]:
            if len(r) < len(cols) or not pat.search(r[ci["Kernel Name"]]):
                continue
            name = r[ci["Metric Name"]]
            if name not in names:
                continue
            val = float(r[ci["Metric Value"]].replace(",", "")) * _UNITS.get(r[ci["Metric Unit"]], 1.0)
            per.setdefault(r[ci["ID"]], {})[name] = val
    else:
        # the raw page: one row per launch, metrics as columns, their units in the next row
        head = next(i for i, r in enumerate(rows) if "Kernel Name" in r and names[0] in r)
        cols, units = rows[head], rows[head + 1]
        ki, ii = cols.index("Kernel Name"), cols.index("ID")
        for r in rows[head + 2:]:
            if len(r) < len(cols) or not pat.search(r[ki]):
                continue
            for name in names:
                j = cols.index(name)
                per.setdefault(r[ii], {})[name] = float(r[j].replace(",", "")) * _UNITS.get(units[j], 1.0)
    launches = [v["dram__bytes_read.sum"] + v["dram__bytes_write.sum"] for v in per.values() if len(v) == 2]
    if not launches:
        raise SystemExit(f"no launch of {kernel_regex!r} with both DRAM metrics in {csv_path}")
    out = {"workload": workload, "kernel_regex": kernel_regex, "launches": len(launches),
           "traffic_bytes_per_launch": float(np.mean(launches)),
           "traffic_bytes_min": float(np.min(launches)), "traffic_bytes_max": float(np.max(launches)),
           "source_hash": kernel_source_hash(), "command": command, "csv": os.path.basename(csv_path)}
    with open(traffic_path(workload), "w") as f:
        json.dump(out, f, indent=1)
        f.write("\n")
    return out


def survey_bytes(n: int, nnz: int, b: int, s_in: int, s_out: int, s_diag: int, weighted: bool) -> float:
    """Algorithmic bytes of one Laplacian product as the scope table states
    them: 8 (n + 1) row offsets, nnz (4 + s_w) column indices and weights, the
    input and output blocks n b s and the diagonal n s_diag (X counted once)."""
    return 8.0 * (n + 1) + nnz * (4.0 + (4.0 if weighted else 0.0)) + n * b * (s_in + s_out) + n * s_diag


def config_of(w: dict, precision: str, col_bytes: float, world: int) -> dict:
    """The bench line's config (both arms print the same one)."""
    return {"workload": w["desc"], "K": w["K"], "precision": precision,
            "l2": (f"inputs larger than L2 (CSR column array {col_bytes / 1e6:.0f} MB > 129 MB)"
                   if col_bytes > 129e6 else "inputs within L2, no flush"),
            "parallelism": f"replicas x{world}" if world > 1 else "single GPU"}


class Clocks:
    """nvidia-smi sampling of SM clock and throttle reasons during the timed region."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, dev: int):
        self.dev = dev
        self.proc = None

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
                                          "-lms", "200", "-i", str(self.dev)], stdout=subprocess.PIPE,
                                         stderr=subprocess.DEVNULL, text=True)
        except OSError:
            self.proc = None
        return self

    def __exit__(self, *exc):
        self.out = ""
        if self.proc:
            self.proc.terminate()
            try:
                self.out, _ = self.proc.communicate(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()
                self.out, _ = self.proc.communicate()

    def summary(self):
        rows = [r.split(",") for r in (self.out or "").strip().splitlines() if r.count(",") >= 8]
        if not rows:
            return None
        sm = [float(r[1]) for r in rows if r[1].strip().replace(".", "").isdigit()]
        mx = [float(r[2]) for r in rows if r[2].strip().replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i - 5] for r in rows for i in range(5, 9) if "Active" in r[i] and "Not" not in r[i]})
        return {"sm_mhz": float(np.median(sm)) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": reasons, "samples": len(rows)}


def max_over_ranks(value: float, world: int, device: str = "cuda") -> float:
    """The largest of every rank's value (the slowest rank sets the job's
    time); the value itself on one rank."""
    if world <= 1:
        return value
    import torch
    import torch.distributed as dist
    t = torch.tensor([value], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def job_throughput(units_per_rank: float, ms_max: float, world: int) -> float:
    """Whole-job units per second: every rank's units over the slowest rank's time."""
    return world * units_per_rank / (ms_max / 1000.0)


def dist_env():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return world, rank, local


def oracle_timed_run(name: str, iterations: int):
    """One run of the FP64 oracle on the workload with the LOBPCG cap at
    `iterations`, timed piece by piece through the oracle's iteration
    callback: the fixed part (operator, preconditioner setup, initial
    Rayleigh-Ritz, embedding, multi-jagged and cut) and each iteration."""
    import oracle
    w = WORKLOADS[name]
    g = make_graph(name)
    marks = []
    t0 = time.perf_counter()
    oracle.partition(g, w["K"], problem=w["laplacian"], precond=w["precond"], tol=w["tol"], seed=w["seed"],
                     poly_degree=w["poly_degree"], maxit=iterations,
                     on_iteration=lambda it: marks.append(time.perf_counter()))
    t_end = time.perf_counter()
    iters = [b - a for a, b in zip(marks[:-1], marks[1:])]
    fixed = (marks[0] - t0) + (t_end - marks[-1])
    return fixed, iters, g


def oracle_iterations(name: str):
    """The oracle's own iteration count for the workload, from its full run
    stored in tests/golden (written by oracle code only), or None."""
    w = WORKLOADS[name]
    if not w.get("golden"):
        return None
    p = os.path.join(ROOT, "tests", "golden", w["golden"])
    if not os.path.exists(p):
        return None
    with open(p) as f:
        return json.load(f)["iterations"]


ORACLE_THREADS = ("scipy sparse products single-threaded; numpy BLAS (the small dense algebra) on up to "
                  f"{os.cpu_count()} threads")


def oracle_sample(name: str):
    """The FP64 oracle on the same workload, bounded to about 10-30 s: one
    run with the iteration cap at 2 gives the fixed part and the time of an
    iteration; partitions/s is extrapolated to the oracle's own iteration
    count (labelled as such)."""
    fixed, iters, _ = oracle_timed_run(name, 2)
    n_it = oracle_iterations(name) or len(iters)
    per_iter = float(np.mean(iters)) if iters else 0.0
    est = fixed + n_it * per_iter
    sample = (f"EXTRAPOLATED from one oracle.partition run with the LOBPCG cap at 2: fixed part {fixed:.1f} s "
              f"(operator, preconditioner setup, initial Rayleigh-Ritz, embedding, multi-jagged, cut) plus the "
              f"oracle's own {n_it} iterations at the measured {per_iter:.2f} s each; {ORACLE_THREADS}")
    return 1.0 / est, sample, fixed + sum(iters)


def vs_oracle(w, st, cut, precision):
    """Eigenvalue, residual and cut of one GPU partition against the FP64
    oracle's full run of the same workload and seed (tests/golden, written by
    oracle code only).  The eigenvalue-zero vector is compared absolutely, the
    others relatively; the tolerances are those the parity tests use."""
    if not w.get("golden"):
        return None
    p = os.path.join(ROOT, "tests", "golden", w["golden"])
    if not os.path.exists(p):
        return None
    with open(p) as f:
        d = json.load(f)
    ev, ev_o = st["eigenvalues"], d["eigenvalues"]
    rel = [abs(a - b) / abs(b) for a, b in zip(ev[1:], ev_o[1:])]
    return {"source": f"tests/golden/{w['golden']}", "oracle_iterations": d["iterations"],
            "eigenvalue_max_rel_err": max(rel) if rel else None, "eigenvalue_rel_tol": 1e-6 if precision == "fp64" else 1e-3,
            "null_eigenvalue_abs": abs(ev[0]),
            "max_resnorm_over_tol_theta": _res_ratio(st, w["tol"]),
            "oracle_cut": d["cut"], "cut_rel_err": abs(cut - d["cut"]) / d["cut"], "cut_rel_tol": 0.02}


def run_reference(args, world, rank):
    """The oracle arm, on the same workload, metric and config as ours.  A
    whole oracle partition of the large workloads takes minutes, so a step is
    one real piece of one oracle run: a single run with the LOBPCG cap at
    warmup + steps iterations, whose first `warmup` iterations are untimed
    warm-up and whose next `steps` iterations are the timed steps.  The fixed
    part of the same run (operator, preconditioner setup, initial
    Rayleigh-Ritz, embedding, multi-jagged, cut) is timed too, and the value
    is partitions/s for the fixed part plus the oracle's own iteration count
    at the measured per-iteration time.  Workloads whose whole oracle
    partition is short (the 64x64 mesh) time whole partitions per step."""
    if rank != 0:
        return 0
    w = WORKLOADS[args.workload]
    precision = args.precision or w["precision"]
    if w.get("batch"):
        import workloads
        graphs = workloads.rgg_batch(w["batch"])
        vals = []
        sample = ""
        for _ in range(args.steps):
            v, sample = oracle_batch_sample(graphs, w, budget_s=max(1.0, 150.0 / max(1, args.steps)))
            vals.append(v)
        value = float(np.median(vals))
        ms_step = 1000.0 * len(graphs) / value
        step_kind = "EXTRAPOLATED: the oracle on the batch's first graphs per step, scaled to the whole batch"
        col_bytes = sum(gq.col.nbytes for gq in graphs)
    elif args.workload == "c1":
        import oracle
        g = make_graph("c1")
        kw = dict(problem=w["laplacian"], precond=w["precond"], tol=w["tol"], seed=w["seed"])
        for _ in range(args.warmup):
            oracle.partition(g, w["K"], **kw)
        times = []
        for _ in range(args.steps):
            t = time.perf_counter()
            oracle.partition(g, w["K"], **kw)
            times.append(time.perf_counter() - t)
        ms_step = 1000.0 * float(np.mean(times))
        value = 1000.0 / ms_step
        sample = f"whole oracle partitions, one per step (timed, not extrapolated); {ORACLE_THREADS}"
        step_kind = "one whole oracle partition"
        col_bytes = g.col.nbytes
    else:
        fixed, iters, g = oracle_timed_run(args.workload, args.warmup + args.steps)
        timed = iters[args.warmup:args.warmup + args.steps]
        if len(timed) < args.steps:
            raise SystemExit("the oracle converged before the requested steps; use fewer steps")
        per_iter = float(np.mean(timed))
        n_it = oracle_iterations(args.workload) or len(iters)
        value = 1.0 / (fixed + n_it * per_iter)
        ms_step = 1000.0 * per_iter
        sample = (f"one oracle.partition run with the LOBPCG cap at {args.warmup}+{args.steps} iterations: the "
                  f"first {args.warmup} untimed, the next {args.steps} the timed steps ({per_iter:.2f} s each); "
                  f"value EXTRAPOLATED to a whole partition = fixed part {fixed:.1f} s (timed in the same run) + "
                  f"the oracle's own {n_it} iterations (tests/golden/{w['golden']}); {ORACLE_THREADS}")
        step_kind = "one LOBPCG iteration of the oracle's partition of this workload"
        col_bytes = g.col.nbytes
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms_step, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": config_of(w, precision, col_bytes, world), "step": step_kind,
            "cpu_baseline": {"kind": "oracle", "value": value, "unit": UNIT, "cores": os.cpu_count(),
                             "sample": sample},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)
    return 0


def oracle_batch_sample(graphs, w, budget_s: float = 20.0):
    """The oracle on the batch's first graphs (in order, until about budget_s
    of CPU work), extrapolated to the whole batch by vertex count."""
    import oracle
    done_n, t_used, used = 0, 0.0, 0
    for gq in graphs:
        t = time.perf_counter()
        oracle.partition(gq, w["K"], problem=w["laplacian"], precond=w["precond"], tol=w["tol"], seed=w["seed"])
        t_used += time.perf_counter() - t
        done_n += gq.n
        used += 1
        if t_used >= budget_s:
            break
    total_n = sum(gq.n for gq in graphs)
    est = t_used * total_n / done_n
    sample = (f"oracle.partition on the first {used} graphs ({done_n} vertices, {t_used:.1f} s), extrapolated "
              f"to the batch's {total_n} vertices by vertex count")
    return len(graphs) / est, sample


def batch_vs_oracle(w, eigs, cuts, status):
    """Per graph of the oracle's stored runs (tests/golden, written by oracle
    code only): eigenvalue and cut errors of the batch's result."""
    if not w.get("golden"):
        return None
    p = os.path.join(ROOT, "tests", "golden", w["golden"])
    if not os.path.exists(p):
        return None
    with open(p) as f:
        d = json.load(f)
    out = []
    for gq in d["graphs"]:
        q = gq["index"]
        ev, ev_o = eigs[q], gq["eigenvalues"]
        rel = max(abs(a - b) / abs(b) for a, b in zip(ev[1:], ev_o[1:]))
        out.append({"graph": q, "n": gq["n"], "status": int(status[q]), "eigenvalue_max_rel_err": rel,
                    "cut": float(cuts[q]), "oracle_cut": gq["cut"],
                    "cut_rel_err": abs(float(cuts[q]) - gq["cut"]) / gq["cut"]})
    return {"source": f"tests/golden/{w['golden']}", "eigenvalue_rel_tol": 1e-3, "cut_rel_tol": 0.02,
            "graphs": out}


def batch_chain_roofline(spx, h, w, big, stream, precision):
    """The batch's dominant kernel, the polynomial chain step over every
    graph's rows (the captured loop cannot hold per-launch events): 20 steps
    of sphynx_poly_step on the batch handle with the partition's block width
    and chain type, alternating the steps that add to y with those that do
    not, timed with CUDA events on the handle's stream."""
    import torch
    d = int(np.floor(np.log2(w["K"]))) + 1
    bp = (d + 3) // 4 * 4
    f64 = precision == "fp64"
    dt, tdt, s = (spx.DT_F64, torch.float64, 8) if f64 else (spx.DT_F32, torch.float32, 4)
    gen = torch.Generator(device="cuda").manual_seed(w["seed"])
    t = torch.randn(big.n, bp, dtype=tdt, device="cuda", generator=gen)
    tout = torch.empty_like(t)
    y = torch.zeros_like(t)
    lap = w["laplacian"]

    def chain_step(i):
        src, dst = (t, tout) if i % 2 == 0 else (tout, t)
        spx.sphynx_poly_step(h, lap, dt, src, dt, dst, y, bp, d, 2.0 + i, 3.0 + i, 2 if i % 2 == 0 else 0, 0)

    for i in range(4):
        chain_step(i)
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    e0.record(stream)
    for i in range(20):
        chain_step(i)
    e1.record(stream)
    torch.cuda.synchronize()
    us = e0.elapsed_time(e1) * 1000.0 / 20
    sb = survey_bytes(big.n, big.nnz, d, s, s, s, False)
    pk = peaks()
    return {"bound": "hbm", "achieved": sb / us / 1e3, "peak": pk["hbm_gbs"], "unit": "GB/s",
            "frac": sb / us / 1e3 / pk["hbm_gbs"], "frac_survey": sb / us / 1e3 / pk["hbm_gbs"],
            "peak_source": f"{pk['src']} (MEASURED_PEAKS.json copy bandwidth)" if pk["src"] == "measured" else pk["src"],
            "kernel": "polynomial chain step over the whole batch (sphynx_poly_step, %s)" % ("f64" if f64 else "f32"),
            "us_per_launch": us, "algorithmic_bytes_per_launch": sb,
            "algorithmic_bytes_formula": "8(n+1) + nnz(4+s_w) + n b (s_in+s_out) + n s_diag with n=%d, nnz=%d, b=%d, "
                                         "s_in=s_out=%d, s_w=0, s_diag=%d" % (big.n, big.nnz, d, s, s),
            "traffic": None, "traffic_source": None,
            "note": "rows in the generator's order: a geometric graph's neighbours have unrelated ids, so every "
                    "gather of a 16-byte row is its own 32-byte DRAM sector"}


def run_batch(args, world, rank, local):
    """The batch workload: all graphs partitioned by one sphynx_partition_batch
    call per step (replicas on N > 1 GPUs)."""
    import torch
    import workloads
    import paper_2105_00578_gb300 as spx

    torch.cuda.set_device(local)
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    w = WORKLOADS[args.workload]
    precision = args.precision or w["precision"]
    graphs = workloads.rgg_batch(w["batch"])
    big, gptr = workloads.concat_graphs(graphs)
    count = len(graphs)
    stream = torch.cuda.current_stream()
    h = spx.sphynx_create_batch(big.row_ptr, big.col, gptr, stream=stream)
    part = torch.empty(big.n, dtype=torch.int32, device="cuda")
    opt = spx.options(laplacian=w["laplacian"], precond=w["precond"], poly_degree=w["poly_degree"],
                      precision=precision, tol=w["tol"], seed=w["seed"], out_device=True,
                      stall_window=w.get("stall_window", 0), max_iter=w.get("max_iter", 1000))

    def step():
        return spx.sphynx_partition_batch(h, w["K"], opt, part, count)

    for _ in range(args.warmup):
        step()
    torch.cuda.synchronize()

    def barrier():
        if world > 1:
            torch.distributed.barrier()

    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    res = []
    with Clocks(local) as clk:
        barrier()
        torch.cuda.synchronize()
        e0.record(stream)
        for _ in range(args.steps):
            res.append(step())
        e1.record(stream)
        torch.cuda.synchronize()
        barrier()
    ms = max_over_ranks(e0.elapsed_time(e1) / args.steps, world)
    value = job_throughput(count, ms, world)
    code, cuts, imbs, eigs, iters, status, st = res[-1]
    roof = batch_chain_roofline(spx, h, w, big, stream, precision)

    # end to end: create from pinned host CSR, partition, read the part ids back
    rp = torch.from_numpy(big.row_ptr).pin_memory()
    cl = torch.from_numpy(big.col).pin_memory()
    hp = torch.empty(big.n, dtype=torch.int32).pin_memory()
    o_host = spx.options(laplacian=w["laplacian"], precond=w["precond"], poly_degree=w["poly_degree"],
                         precision=precision, tol=w["tol"], seed=w["seed"], stall_window=w.get("stall_window", 0),
                         max_iter=w.get("max_iter", 1000))
    torch.cuda.synchronize()
    barrier()
    t = time.perf_counter()
    e2e_steps = max(1, args.steps)
    for _ in range(e2e_steps):
        h2 = spx.sphynx_create_batch(rp.data_ptr(), cl.data_ptr(), gptr, stream=stream, nnz=big.nnz)
        spx.sphynx_partition_batch(h2, w["K"], o_host, hp.data_ptr(), count)
        spx.sphynx_destroy(h2)
    torch.cuda.synchronize()
    e2e_s = max_over_ranks((time.perf_counter() - t) / e2e_steps, world)
    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        v, sample = oracle_batch_sample(graphs, w)
        cpu = {"value": v, "unit": UNIT, "cores": os.cpu_count(), "kind": "oracle", "sample": sample}
    if rank == 0:
        line = {
            "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": ms, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f32" if precision != "fp64" else "f64", "data": "synthetic",
            "config": {"workload": w["desc"], "K": w["K"], "graphs": count, "vertices": big.n, "nnz": big.nnz,
                       "precision": precision,
                       "l2": f"inputs larger than L2 (CSR column array {big.col.nbytes / 1e6:.0f} MB > 129 MB)",
                       "parallelism": f"replicas x{world}" if world > 1 else "single GPU"},
            "graphs_converged": int(np.sum(status == 0)),
            "graphs_finished_in_fp64": int(st.get("fp64_finished", 0)),
            "graphs_noconv": int(np.sum(status != 0)),
            "noconv_graph_sizes": sorted((int(graphs[q].n) for q in np.flatnonzero(status != 0)), reverse=True)[:20],
            "ms_float_phase": float(st["ms_phase"][0]), "ms_fp64_phase": float(st["ms_phase"][1]),
            "loop_iterations": [int(v) for v in st["loop_iters"]],
            "vs_oracle": batch_vs_oracle(w, eigs, cuts, status),
            "stall_window": w.get("stall_window", 0), "max_iter": w.get("max_iter", 1000),
            "max_iterations": int(iters.max()),
            "median_iterations": float(np.median(iters)), "mean_cut": float(np.mean(cuts)),
            "max_imbalance": float(np.max(imbs)),
            "roofline": roof,
            "cpu_baseline": cpu,
            "e2e": {"value": world * count / e2e_s, "unit": UNIT,
                    "h2d_bytes_per_step": int(big.row_ptr.nbytes + big.col.nbytes),
                    "d2h_bytes_per_step": int(big.n * 4)},
            "gpu_launches": int(st["kernel_launches"]),
            "clocks": clk.summary(),
        }
        print(json.dumps(line), flush=True)
    spx.sphynx_destroy(h)
    if world > 1:
        torch.distributed.destroy_process_group()
    return 0


def run_ours(args, world, rank, local):
    import torch
    import paper_2105_00578_gb300 as spx

    torch.cuda.set_device(local)
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    w = WORKLOADS[args.workload]
    precision = args.precision or w["precision"]
    g = make_graph(args.workload)
    stream = torch.cuda.current_stream()
    graph = spx.Graph(g, stream=stream)

    def pin(h):
        # profiler captures pin the schedule: under a profiler the tuner's timings are distorted
        if args.spmm_variant is not None:
            spx.sphynx_set_spmm_variant(h, {"csr": 0, "sell": 1, "pattern": 2}[args.spmm_variant])
        if args.sell_stride is not None:
            spx.sphynx_set_spmm_sell_stride(h, args.sell_stride)

    pin(graph.h)
    n = g.n
    part = torch.empty(n, dtype=torch.int32, device="cuda")

    def opts(prec):
        return spx.options(laplacian=w["laplacian"], precond=w["precond"], poly_degree=w["poly_degree"],
                           precision=prec, tol=w["tol"], seed=w["seed"], out_device=True)

    o_main = opts(precision)

    def step(o):
        return spx.sphynx_partition(graph.h, w["K"], o, part)

    for _ in range(args.warmup):
        step(o_main)
    torch.cuda.synchronize()

    def barrier():
        if world > 1:
            torch.distributed.barrier()

    stats = []
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    with Clocks(local) as clk:
        barrier()
        torch.cuda.synchronize()
        e0.record(stream)
        for _ in range(args.steps):
            code, cut, imb, st = step(o_main)
            stats.append((code, cut, imb, st))
        e1.record(stream)
        torch.cuda.synchronize()
        barrier()
    ms = max_over_ranks(e0.elapsed_time(e1) / args.steps, world)
    value = job_throughput(1, ms, world)

    spmm_ms = sum(s[3]["ms_spmm"] for s in stats)
    spmm_bytes = sum(s[3]["spmm_bytes"] for s in stats)
    spmm_launches = sum(s[3]["spmm_launches"] for s in stats)
    launches = sum(s[3]["kernel_launches"] for s in stats)
    last = stats[-1]
    pk = peaks()
    achieved_all = spmm_bytes / (spmm_ms / 1000.0) / 1e9 if spmm_ms > 0 else None
    # the SpMM launches split by input precision (F64, F32, BF16)
    by_dt = {}
    for i, name in enumerate(("f64", "f32", "bf16")):
        ms_i = sum(s[3]["ms_spmm_by_dt"][i] for s in stats)
        by_i = sum(s[3]["spmm_bytes_by_dt"][i] for s in stats)
        la_i = sum(s[3]["spmm_launches_by_dt"][i] for s in stats)
        if la_i:
            by_dt[name] = {"launches_per_step": la_i / args.steps, "us_per_launch": 1000.0 * ms_i / la_i,
                           "bytes_per_launch": by_i / la_i, "gbs": by_i / (ms_i / 1000.0) / 1e9 if ms_i > 0 else None}
    # the dominant kernel: the SpMM flavour with the most device time
    dom = max(by_dt, key=lambda k: by_dt[k]["us_per_launch"] * by_dt[k]["launches_per_step"]) if by_dt else None
    info = spx.sphynx_get_info(graph.h)
    variant = {"csr": 0, "sell": 1, "pattern": 2}.get(args.spmm_variant, info["spmm_variant"])
    schedule = {0: "k_spmm_short", 1: "k_spmm_sell", 2: "k_spmm_block / k_spmm_sell (shared-pattern slices)"}[variant]
    kernel_name = f"{schedule}<{dom} in>"
    traffic, traffic_meta = profiled_traffic(args.workload)
    # achieved: the scope table's algorithmic bytes of one launch of the
    # dominant kernel (X read once and written once at the true block width b,
    # 8-byte row offsets, 4-byte column indices, 4-byte weights if any, the
    # diagonal) over its mean launch time from CUDA events on its stream
    roof = None
    if dom:
        s = {"f64": 8, "f32": 4, "bf16": 2}[dom]
        d_true = int(w["K"]).bit_length()
        sb = survey_bytes(g.n, g.nnz, d_true, s, s, 8 if dom == "f64" else 4, g.w is not None)
        us = by_dt[dom]["us_per_launch"]
        achieved = sb / (us * 1e-6) / 1e9
        layout_gbs = by_dt[dom]["gbs"]
        roof = {"bound": "hbm", "achieved": achieved, "peak": pk["hbm_gbs"], "unit": "GB/s",
                "frac": achieved / pk["hbm_gbs"], "frac_survey": achieved / pk["hbm_gbs"],
                "frac_of_nominal_8tbs": achieved / 8000.0,
                "peak_source": pk["src"] + " (MEASURED_PEAKS.json copy bandwidth)" if pk["src"] == "measured"
                else pk["src"],
                "kernel": kernel_name, "us_per_launch": us,
                "algorithmic_bytes_per_launch": sb,
                "algorithmic_bytes_formula": (f"8(n+1) + nnz(4+s_w) + n b (s_in+s_out) + n s_diag with n={g.n}, "
                                              f"nnz={g.nnz}, b={d_true}, s_in=s_out={s}, "
                                              f"s_w={4 if g.w is not None else 0}, "
                                              f"s_diag={8 if dom == 'f64' else 4}"),
                "layout_bytes_per_launch": by_dt[dom]["bytes_per_launch"],
                "achieved_layout": layout_gbs,
                "frac_layout": layout_gbs / pk["hbm_gbs"] if layout_gbs else None,
                "traffic": traffic,
                "traffic_source": (f"profiles/traffic_{args.workload}.json" if traffic is not None else
                                   ("stale: the SpMM sources changed after the capture" if traffic_meta else None))}

    # plain FP64 path at the same tolerance
    fp64 = None
    if args.fp64_steps > 0 and precision != "fp64":
        o64 = opts("fp64")
        step(o64)
        torch.cuda.synchronize()
        f0 = torch.cuda.Event(enable_timing=True)
        f1 = torch.cuda.Event(enable_timing=True)
        f0.record(stream)
        fst = []
        for _ in range(args.fp64_steps):
            fst.append(step(o64))
        f1.record(stream)
        torch.cuda.synchronize()
        fms = f0.elapsed_time(f1) / args.fp64_steps
        s64 = fst[-1][3]
        fp64 = {"ms_per_partition": fms, "partitions_per_s": 1000.0 / fms, "iterations": s64["iterations"],
                "max_resnorm_over_tol_theta": _res_ratio(s64, w["tol"]), "cut": fst[-1][1],
                "vs_oracle": vs_oracle(w, s64, fst[-1][1], "fp64"),
                "status": fst[-1][0], "speedup_of_mixed": fms / ms}

    # end to end through the C ABI with host buffers: create (H2D of the CSR
    # from pinned memory) + partition + read of the part ids (D2H) per step
    rp = torch.from_numpy(g.row_ptr).pin_memory()
    cl = torch.from_numpy(g.col).pin_memory()
    wp = torch.from_numpy(g.w).pin_memory() if g.w is not None else None
    hp = torch.empty(n, dtype=torch.int32).pin_memory()
    o_host = spx.options(laplacian=w["laplacian"], precond=w["precond"], poly_degree=w["poly_degree"],
                         precision=precision, tol=w["tol"], seed=w["seed"])
    e2e_steps = max(1, args.steps)
    torch.cuda.synchronize()
    barrier()
    t = time.perf_counter()
    for _ in range(e2e_steps):
        h = spx.sphynx_create(rp.data_ptr(), cl.data_ptr(), None if wp is None else wp.data_ptr(), None, n, g.nnz,
                              spx.HOST_PTRS, stream)
        pin(h)
        spx.sphynx_partition(h, w["K"], o_host, hp.data_ptr())
        spx.sphynx_destroy(h)
    torch.cuda.synchronize()
    e2e_s = max_over_ranks((time.perf_counter() - t) / e2e_steps, world)

    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        v, sample, _ = oracle_sample(args.workload)
        cpu = {"value": v, "unit": UNIT, "cores": os.cpu_count(), "kind": "oracle", "sample": sample,
               "threads": {"sparse_products": 1, "dense_blas": os.cpu_count()}}

    if rank == 0:
        line = {
            "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": ms, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f32" if precision != "fp64" else "f64",
            "data": "synthetic",
            "config": config_of(w, precision, g.col.nbytes, world),
            "iterations": last[3]["iterations"], "status": last[0], "cut": last[1], "imbalance": last[2],
            "eigenvalues": last[3]["eigenvalues"],
            "max_resnorm_over_tol_theta": _res_ratio(last[3], w["tol"]),
            "vs_oracle": vs_oracle(w, last[3], last[1], precision),
            "spmm": {"gbs": achieved_all, "launches_per_step": spmm_launches / args.steps,
                     "ms_per_step": spmm_ms / args.steps, "by_input_precision": by_dt,
                     "schedule": schedule, "sell_stride": info["sell_stride"] if variant > 0 else None,
                     "sell_pattern_slices": info["sell_pattern_slices"]},
            "fp64": fp64,
            "roofline": roof,
            "cpu_baseline": cpu,
            "e2e": {"value": world / e2e_s, "unit": UNIT,
                    "h2d_bytes_per_step": int(g.row_ptr.nbytes + g.col.nbytes + (0 if g.w is None else g.w.nbytes)),
                    "d2h_bytes_per_step": int(n * 4)},
            "gpu_launches": int(launches),
            "clocks": clk.summary(),
        }
        print(json.dumps(line), flush=True)
    graph.close()
    if world > 1:
        torch.distributed.destroy_process_group()
    return 0


def run_products(args) -> int:
    """No partition: time args.products Laplacian products Y = L X of the
    workload's graph (its Laplacian, blocks of width round4(d) in FP32, or FP64
    with --precision fp64), with an L2 flush before each, then run two more
    between cudaProfilerStart and cudaProfilerStop, the launches an
    `ncu --profile-from-start off` capture sees.  Prints one JSON line."""
    import torch
    import paper_2105_00578_gb300 as spx
    w = WORKLOADS[args.workload]
    g = make_graph(args.workload)
    d = int(np.floor(np.log2(w["K"]))) + 1
    bp = (d + 3) // 4 * 4
    f64 = args.precision == "fp64"
    dt, tdt, s = (spx.DT_F64, torch.float64, 8) if f64 else (spx.DT_F32, torch.float32, 4)
    h = spx.sphynx_create(g.row_ptr, g.col, g.w, None)
    if args.spmm_variant is not None:
        spx.sphynx_set_spmm_variant(h, {"csr": 0, "sell": 1, "pattern": 2}[args.spmm_variant])
    gen = torch.Generator(device="cuda").manual_seed(w["seed"])
    x = torch.randn(g.n, bp, dtype=tdt, device="cuda", generator=gen)
    y = torch.empty_like(x)
    lap = w["laplacian"]

    def apply():
        spx.sphynx_laplacian_apply(h, lap, dt, x, bp, y, bp, bp)

    for _ in range(3):
        apply()
    flush = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")   # twice L2
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    us = []
    for _ in range(args.products):
        flush.fill_(1)
        e0.record()
        apply()
        e1.record()
        torch.cuda.synchronize()
        us.append(e0.elapsed_time(e1) * 1000.0)
    torch.cuda.profiler.start()
    for _ in range(2):
        flush.fill_(1)
        apply()
    torch.cuda.synchronize()
    torch.cuda.profiler.stop()
    info = spx.sphynx_get_info(h)
    spx.sphynx_destroy(h)
    med = float(np.median(us))
    sb = survey_bytes(g.n, g.nnz, d, s, s, s, g.w is not None)
    pk = peaks()
    print(json.dumps({
        "workload": args.workload, "laplacian": lap, "n": g.n, "nnz": g.nnz, "block": d, "width": bp,
        "dtype": "f64" if f64 else "f32", "products": args.products, "us_median": med, "us_min": float(min(us)),
        "survey_bytes": sb, "gbs": sb / med / 1e3, "peak_gbs": pk["hbm_gbs"], "frac": sb / med / 1e3 / pk["hbm_gbs"],
        "l2": "256 MiB written between products",
        "schedule": {k: info[k] for k in ("spmm_variant", "spmm_med_max", "sell_stride", "long_rows")}}))
    return 0


def _res_ratio(st, tol):
    """max over the non-null columns of ||r|| / (tol |theta|)"""
    vals = [r / (tol * abs(t)) for r, t in zip(st["resnorm"][1:], st["eigenvalues"][1:]) if t != 0]
    return max(vals) if vals else None


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default="c2", choices=sorted(WORKLOADS))
    ap.add_argument("--precision", default=None, choices=[None, "fp64", "fp32", "mixed_bf16"])
    ap.add_argument("--fp64-steps", type=int, default=1)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--spmm-variant", default=None, choices=[None, "csr", "sell", "pattern"],
                    help="pin the short-row SpMM schedule instead of the one tuned at create "
                         "(used for profiler captures, where tuning times are distorted)")
    ap.add_argument("--sell-stride", type=int, default=None, choices=[1, 2, 4, 8, 16],
                    help="pin the SELL-32 slice stride instead of the one tuned at create (profiler captures)")
    ap.add_argument("--ingest-ncu", default=None, metavar="CSV",
                    help="no benchmark: read the per-launch dram__bytes_read.sum / dram__bytes_write.sum of an ncu "
                         "--csv log and write profiles/traffic_<workload>.json, which later runs report as "
                         "roofline.traffic")
    ap.add_argument("--kernel-regex", default=r"k_spmm_(block|sell)<((\(int\))?0, )?__nv_bfloat16, __nv_bfloat16",
                    help="kernels of the ncu log that --ingest-ncu averages")
    ap.add_argument("--ncu-command", default="", help="the ncu command that wrote the log (recorded by --ingest-ncu)")
    ap.add_argument("--products", type=int, default=0, metavar="N",
                    help="no partition: time N Laplacian products of the workload's graph (and profile two more "
                         "between cudaProfilerStart/Stop)")
    args = ap.parse_args()
    if args.ingest_ncu:
        print(json.dumps(ingest_ncu(args.ingest_ncu, args.kernel_regex, args.workload, args.ncu_command)))
        return 0
    if args.products > 0:
        return run_products(args)
    world, rank, local = dist_env()
    if args.impl == "reference":
        return run_reference(args, world, rank)
    if WORKLOADS[args.workload].get("batch"):
        return run_batch(args, world, rank, local)
    return run_ours(args, world, rank, local)


if __name__ == "__main__":
    sys.exit(main())
