#!/usr/bin/env python
"""Benchmark: conjugate-gradient throughput on the SEM Poisson operator.

Workload (one "step" = one complete solve): a 32x32x32 box of hexahedra
(E = 32768) of order N = 7, interior vertices jittered by +-5 % of the element
size (seed 2), Dirichlet boundary, right-hand side b = mask(QQ^T f) with
f ~ N(0, 1) per local node (seed 3, +rank for extra ranks), CG from x = 0 to
sqrt(<r,r>/<b,b>) <= 1e-8.  Throughput is the paper's GDOFS
(E N^3 iterations / time / 1e9, Section VIII-B).  Inputs already sit in HBM
when the timed region starts; the geometric factors alone (805 MB) exceed the
129 MB L2, so no flush is needed between steps.

Also reported on the same JSON line:
  e2e           the same metric through the public API with host buffers
                (pinned b copied in and x copied out every step)
  roofline      the dominant kernel (the fused CG operator kernel) timed with
                CUDA events on libsem's stream: against HBM bandwidth when the
                tuner picked the fixed-point operator (FP64 values evaluated
                as 64-bit integers), against the FP64 pipe for the DFMA kernels
  mixed         the same solve by mixed-precision iterative refinement (FP32
                inner CG, BF16 geometric factors, FP64 outer residual), with
                its own HBM roofline, solves/s against FP64, and a 1e-10 leg
  cpu_baseline  the FP64 CPU oracle on a bounded sample of the same workload:
                one core, and (all_cores) one oracle process per host core
  clocks        nvidia-smi samples taken during the timed region
  autotune      the per-order operator tuner's candidates and choices
  pcg           the same solve with the Jacobi preconditioner
  batched       256 uneven problems, one launch per order and CG phase
  serve         Poisson arrivals at 100..5000 req/s: p50/p99 latency, solves/s
  paper_sweep   the paper's protocol: GDOF/s against E = 2^1..2^14, N = 4, 6, 8
  vs_oracle     the small workload (E = 64, N = 7, sine source) solved on the
                GPU in FP64 and mixed precision to 1e-8 and 1e-10, each error
                stated against the oracle's stored solution (tol 1e-12)
  summary       the headline figures of every leg, last on the line

``--impl reference`` times the CPU oracle instead (the reference arm).
Multi-GPU (torchrun): every rank solves an independent problem (replicas,
no data-path collective); the value is the sum over ranks over the slowest
rank's time.
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import statistics
import subprocess
import sys
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "CG GDOF/s to 1e-8 rel. residual, mixed vs FP64 on GB300; serve p50/p99 ms"
# FP64 pipe: 152 SMs x 2 DFMA/clk x 2 flop x 2.07 GHz (max SM clock) = 1.259 TFLOP/s
FP64_PEAK_GFLOPS = 152 * 2 * 2 * 2.070
PEAKS_FILE = os.path.join(ROOT, "MEASURED_PEAKS.json")
TRAFFIC_FILE = os.path.join(ROOT, "profiles", "traffic.json")
AX_SOURCES = [os.path.join(ROOT, "paper_2606_12650_gb300", "csrc", f)
              for f in ("sem_ax_kernel.cuh", "sem_ax_lines.cuh", "sem_ax.cu", "sem_ax_lines64.cu", "sem_device.cuh",
                        "sem_internal.h", "sem_ax_fx.cuh", "sem_ax_fx.cu")]
GOLDEN_SMALL = os.path.join(ROOT, "tests", "golden", "oracle_cg_E64_N7.npz")
AX32_SOURCES = [os.path.join(ROOT, "paper_2606_12650_gb300", "csrc", f)
                for f in ("sem_ax_kernel.cuh", "sem_ax_lines.cuh", "sem_ax32.cu", "sem_ax_lines32.cu", "sem_ax32p.cuh", "sem_ax_f32.cuh",
                          "sem_device.cuh", "sem_internal.h")]
VARIANTS = {0: "columns", 1: "lines", 2: "persistent", 3: "lines_prefetch", 4: "lines_staged", 5: "lines_fx"}


def kernel_label(variant, epb, N, t, gt):
    """Name of the CG-operator kernel the tuner chose."""
    q = N + 1
    if variant == 5:
        return f"ax_fx_kernel<{q},CG> ({epb} elements/block, FP64 in 64-bit fixed point)"
    if variant in (1, 3, 4):
        pf = {1: "", 3: ", G prefetched", 4: ", G staged"}[variant]
        return f"ax_lines_kernel<{q},{t},{gt},CG> ({epb} elements/block{pf})"
    if variant == 2:
        return f"ax32p_kernel<{q},{gt},CG> (persistent)"
    return f"ax_kernel<{q},{t},{gt},CG> (columns)"


def parse():
    ap = argparse.ArgumentParser(description=__doc__.split("\n")[0])
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=3)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=("ours", "reference"), default="ours")
    ap.add_argument("--nx", type=int, default=32, help="elements per direction")
    ap.add_argument("--N", type=int, default=7, help="polynomial order")
    ap.add_argument("--tol", type=float, default=1e-8)
    ap.add_argument("--maxit", type=int, default=100000)
    ap.add_argument("--ax-reps", type=int, default=20, help="launches timed for the roofline")
    ap.add_argument("--cpu-iters", type=int, default=10, help="oracle CG iterations per CPU sample")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-cpu-allcores", action="store_true", help="single-core oracle timing only")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-mixed", action="store_true")
    ap.add_argument("--inner-tol", type=float, default=1e-3, help="inner FP32 CG residual reduction")
    ap.add_argument("--no-batched", action="store_true")
    ap.add_argument("--no-pcg", action="store_true")
    ap.add_argument("--no-serve", action="store_true")
    ap.add_argument("--serve-requests", type=int, default=2000, help="requests per arrival rate")
    ap.add_argument("--serve-rates", default="100,200,500,1000,2000,5000")
    ap.add_argument("--batch-count", type=int, default=256)
    ap.add_argument("--no-tune", action="store_true", help="keep the built-in operator table")
    ap.add_argument("--no-paper-sweep", action="store_true", help="skip the N in {4,6,8}, E = 2^1..2^14 sweep")
    ap.add_argument("--tune-reps", type=int, default=10, help="timed launches per tuner candidate")
    return ap.parse_args()


def workload_name(a):
    return (f"fp64 CG to {a.tol:g} rel. residual, box {a.nx}x{a.nx}x{a.nx} (E={a.nx ** 3}), N={a.N}, "
            f"jitter 5% seed 2, random-normal RHS seed 3")


def config_of(a, world, iters=None):
    c = {"workload": workload_name(a), "E": a.nx ** 3, "N": a.N, "tol": a.tol,
         "local_dofs": a.nx ** 3 * (a.N + 1) ** 3, "gdofs_per_iter": a.nx ** 3 * a.N ** 3,
         "l2": "inputs larger than L2 (805 MB of geometric factors per problem)",
         "parallelism": f"replicas x{world} (independent problems, no collective)"}
    if iters is not None:
        c["cg_iters"] = iters
    return c


def ax_flops_per_elem(N):
    q = N + 1
    return 12 * q ** 4 + 15 * q ** 3


def source_sha(paths):
    h = hashlib.sha256()
    for p in paths:
        with open(p, "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()[:16]


class ClockSampler:
    """nvidia-smi samples (200 ms) while the timed region runs."""

    FIELDS = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, device):
        self.device = device
        self.proc = None

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.device), f"--query-gpu={self.FIELDS}",
                 "--format=csv,noheader,nounits", "-lms", "200"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except (OSError, ValueError):
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
        rows = []
        for line in (self.out or "").splitlines():
            parts = [p.strip() for p in line.split(",")]
            if len(parts) < 8:
                continue
            try:
                rows.append((float(parts[0]), float(parts[1]), parts[4:8]))
            except ValueError:
                continue
        if not rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["no nvidia-smi samples"], "samples": 0}
        names = ("hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap")
        reasons = sorted({names[k] for _, _, flags in rows for k, f in enumerate(flags) if f.lower() == "active"})
        return {"sm_mhz": statistics.median(r[0] for r in rows), "sm_max_mhz": max(r[1] for r in rows),
                "reasons": reasons, "samples": len(rows)}


def dist_env():
    from paper_2606_12650_gb300.ranks import rank_env
    return rank_env()


# ------------------------------------------------------------------ oracle (CPU) timing
def time_oracle(a, iters, steps=1):
    """FP64 oracle CG on the full workload, `iters` iterations per step (set-up
    excluded).  Returns (GDOF/s, seconds per step)."""
    import oracle
    from paper_2606_12650_gb300.inputs import box_vertices, normal_field
    P = oracle.Problem(a.nx, a.nx, a.nx, a.N, box_vertices(a.nx, a.nx, a.nx, 0.05, seed=2))
    b = P.mask(P.gs(normal_field(P.nL, 3)))
    times = []
    for _ in range(steps):
        t0 = time.perf_counter()
        P.cg(b, maxit=iters, tol=0.0)
        times.append(time.perf_counter() - t0)
    return P.E * a.N ** 3 * iters / (sum(times) / len(times)) / 1e9, times


def _oracle_replica(nx, N, iters, steps, barrier, out):
    """One process of the all-core timing: the unchanged oracle on its own
    copy of the full problem, `steps` timed samples of `iters` CG iterations,
    each started together with the other processes."""
    import oracle
    from paper_2606_12650_gb300.inputs import box_vertices, normal_field
    P = oracle.Problem(nx, nx, nx, N, box_vertices(nx, nx, nx, 0.05, seed=2))
    b = P.mask(P.gs(normal_field(P.nL, 3)))
    times = []
    for _ in range(steps):
        barrier.wait()
        t0 = time.perf_counter()
        P.cg(b, maxit=iters, tol=0.0)
        times.append(time.perf_counter() - t0)
    out.put(times)


def _host_memory_bytes():
    """Memory this process may still use: MemAvailable, capped by a cgroup limit."""
    avail = None
    try:
        with open("/proc/meminfo") as fh:
            for ln in fh:
                if ln.startswith("MemAvailable:"):
                    avail = int(ln.split()[1]) * 1024
    except OSError:
        pass
    for lim, cur in (("/sys/fs/cgroup/memory.max", "/sys/fs/cgroup/memory.current"),
                     ("/sys/fs/cgroup/memory/memory.limit_in_bytes", "/sys/fs/cgroup/memory/memory.usage_in_bytes")):
        try:
            with open(lim) as fh:
                v = fh.read().strip()
            with open(cur) as fh:
                used = int(fh.read().strip())
            if v != "max" and int(v) < (1 << 60):
                room = int(v) - used
                avail = room if avail is None else min(avail, room)
            break
        except (OSError, ValueError):
            continue
    return avail


def time_oracle_replicas(a, iters, steps):
    """All host cores: one oracle process per core (spawned, not forked), each
    on its own copy of the full problem, capped so that the copies take at
    most half of the free host memory.  Returns (processes, per-step times of
    the slowest process, host cores) or None if fewer than two fit."""
    import multiprocessing as mp

    import oracle
    oracle.build()   # once here, not in every spawned process
    try:
        cores = len(os.sched_getaffinity(0))
    except AttributeError:
        cores = os.cpu_count() or 1
    per_proc = 160 * a.nx ** 3 * (a.N + 1) ** 3 + (512 << 20)   # arrays of the oracle's problem + interpreter
    mem = _host_memory_bytes()
    n = cores if mem is None else min(cores, int(0.5 * mem) // per_proc)
    if n < 2:
        return None
    ctx = mp.get_context("spawn")
    barrier = ctx.Barrier(n, timeout=1800)
    out = ctx.Queue()
    procs = [ctx.Process(target=_oracle_replica, args=(a.nx, a.N, iters, steps, barrier, out), daemon=True)
             for _ in range(n)]
    for p in procs:
        p.start()
    try:
        res = [out.get(timeout=3600) for _ in procs]
    finally:
        for p in procs:
            p.join(timeout=60)
            if p.is_alive():
                p.terminate()
    return n, [max(r[s] for r in res) for s in range(steps)], cores


def run_reference(a):
    rank, _, world = dist_env()
    if rank != 0:
        return
    iters = a.cpu_iters
    rep = time_oracle_replicas(a, iters, a.warmup + a.steps)
    if rep is not None:
        n, times, cores = rep
        sample = (f"{iters} FP64 CG iterations per step on the full E={a.nx ** 3}, N={a.N} problem, "
                  f"the single-threaded C oracle run as {n} independent processes on {cores} host cores "
                  f"(one problem each, started together; set-up excluded; time of the slowest)")
    else:
        n = 1
        _, times = time_oracle(a, iters, steps=a.warmup + a.steps)
        sample = (f"{iters} FP64 CG iterations per step on the full E={a.nx ** 3}, N={a.N} problem, "
                  f"single-threaded C oracle, set-up excluded")
    timed = times[a.warmup:]
    value = n * a.nx ** 3 * a.N ** 3 * iters * len(timed) / sum(timed) / 1e9
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": "GDOF/s", "n_gpus": a.gpus,
            "steps": a.steps, "warmup": a.warmup, "ms_per_step": 1e3 * sum(timed) / len(timed),
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic", "config": config_of(a, 1),
            "cpu_baseline": {"value": value, "unit": "GDOF/s", "cores": n, "kind": "oracle", "sample": sample},
            "e2e": {"value": value, "unit": "GDOF/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


# ------------------------------------------------------------------ our arm
def run_ours(a):
    import numpy as np
    import torch
    import torch.distributed as dist

    import __graft_entry__
    __graft_entry__.build()
    from paper_2606_12650_gb300 import Mesh, sem
    from paper_2606_12650_gb300.inputs import box_vertices, normal_field
    from paper_2606_12650_gb300.ranks import Job, rank_seed

    rank, local, world = dist_env()
    torch.cuda.set_device(local)
    if world > 1:
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    sem.init([f"--device={local}"])
    stream = sem.stream()
    torch.cuda.set_stream(stream)
    job = Job(world, dist, device=torch.device("cuda", local), local=local)
    barrier = job.barrier

    nx, N = a.nx, a.N
    E = nx ** 3
    M = Mesh(nx, nx, nx, N, box_vertices(nx, nx, nx, 0.05, seed=2))
    f = torch.from_numpy(normal_field(M.nL, rank_seed(3, rank))).cuda()
    b = f.clone()
    M.gs(b)
    M.mask(b)
    x = torch.empty_like(b)

    # ---- per-order operator tuner: every variant of the FP64 operator and of
    # the mixed path's FP32 (BF16 G) operator timed on this problem, fastest kept
    tune = None
    if not a.no_tune:
        tune = {"N": N, "reps": a.tune_reps}
        for kind, name in ((sem.TUNE_F64, "fp64"), (sem.TUNE_F32_G16, "fp32_bf16")):
            cands = M.autotune(kind, reps=a.tune_reps)
            v, e, us = sem.autotune_get(kind, N)
            tune[name] = {"chosen": {"variant": VARIANTS[v], "epb": e, "us": us},
                          "candidates": [{"variant": VARIANTS[c[0]], "epb": c[1], "us": c[2]} for c in cands]}

    for _ in range(a.warmup):
        iters, rel = M.cg_solve(b, x, a.tol, a.maxit)

    # ---- timed region: K complete solves, inputs resident in HBM
    n_launch0 = sem.launch_count()
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    iters_total = 0
    barrier()
    torch.cuda.synchronize()
    with ClockSampler(local) as clk:
        ev0.record(stream)
        for _ in range(a.steps):
            it, rel = M.cg_solve(b, x, a.tol, a.maxit)
            iters_total += it
        ev1.record(stream)
        torch.cuda.synchronize()
    barrier()
    launches = sem.launch_count() - n_launch0
    t_max, dofs = job.aggregate(ev0.elapsed_time(ev1), float(E * N ** 3 * iters_total))
    value = dofs / (t_max * 1e-3) / 1e9
    true_res = M.true_res(b, x)

    # ---- dominant kernel: the fused CG operator kernel, timed alone on libsem's stream
    for _ in range(3):
        sem.run("cg_ax", M.handle)
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    for _ in range(a.ax_reps):
        sem.run("cg_ax", M.handle)
    e1.record(stream)
    torch.cuda.synchronize()
    ax_ms = e0.elapsed_time(e1) / a.ax_reps
    flops = E * ax_flops_per_elem(N)
    achieved = flops / (ax_ms * 1e-3) / 1e9
    bytes_alg = E * (N + 1) ** 3 * 96  # r, p, x in; p, w, x out (x: the deferred update); 6 FP64 factors
    fp64 = sem.OutDouble()
    sem.run("peak_fma", 0, 4096, fp64)
    traffic = None
    try:
        with open(TRAFFIC_FILE) as fh:
            t = json.load(fh).get("ax_f64_cg", {})
        if t.get("source_sha") == source_sha(AX_SOURCES) and t.get("E") == E and t.get("N") == N:
            traffic = t.get("bytes_per_launch")
    except (OSError, ValueError):
        pass
    v64, e64, _ = sem.autotune_get(sem.TUNE_F64, N)
    hbm, hbm_how = hbm_peak()
    gbs = bytes_alg / (ax_ms * 1e-3) / 1e9
    if v64 == 5:
        # 64-bit fixed-point arithmetic on the integer multiplier: the FP64 pipe no longer
        # bounds the kernel; HBM bandwidth is its roofline
        roofline = {"bound": "hbm", "achieved": gbs, "peak": hbm, "unit": "GB/s", "frac": gbs / hbm,
                    "traffic": traffic, "kernel": kernel_label(v64, e64, N, "double", "double"),
                    "launch_ms": ax_ms, "alg_bytes_per_launch": bytes_alg,
                    "alg_bytes_note": "96 B per local node: r, p, x read; p, w, x written (x: the deferred "
                                      "update); 6 geometric factors of 8 B (as 64-bit integers with one "
                                      "scale per element)",
                    "peak_source": hbm_how,
                    "fp64_equiv_gflops": achieved, "fp64_pipe_peak_gflops": FP64_PEAK_GFLOPS,
                    "fp64_equiv_note": "the operator's direct-evaluation flops, 12(N+1)^4 + 15(N+1)^3 per "
                                       "element, per second: above the FP64 pipe's peak because the kernel "
                                       "computes in 64-bit fixed point on the integer multiply-add pipe"}
    else:
        roofline = {"bound": "alu", "achieved": achieved, "peak": FP64_PEAK_GFLOPS, "unit": "GFLOP/s",
                    "frac": achieved / FP64_PEAK_GFLOPS, "traffic": traffic,
                    "kernel": kernel_label(v64, e64, N, "double", "double"), "launch_ms": ax_ms,
                    "flops_note": "achieved counts the operator's direct-evaluation flops, 12(N+1)^4 + "
                                  "15(N+1)^3 per element; the line kernel's even-odd split executes fewer (48 "
                                  "instead of 64 operations per 1d line at N = 7)",
                    "flops_per_launch": flops, "alg_bytes_per_launch": bytes_alg,
                    "hbm_gbs_at_alg_bytes": gbs, "hbm_frac_at_alg_bytes": gbs / hbm,
                    "peak_note": "FP64 pipe from unit counts and the maximum SM clock (152 SMs x 2 DFMA/clk x "
                                 "2 flop x 2.07 GHz); fp64_probe_gflops is the same pipe measured live"}
    roofline["fp64_probe_gflops"] = fp64.value / 1e9

    # ---- Jacobi-preconditioned CG (FP64), the original Nekbone method
    pcg = None
    if not a.no_pcg:
        xp = torch.empty_like(b)
        M.pcg_solve(b, xp, a.tol, a.maxit)   # warm-up: preconditioner and graph
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        itp = 0
        for _ in range(a.steps):
            it_p, rel_p = M.pcg_solve(b, xp, a.tol, a.maxit)
            itp += it_p
        e1.record(stream)
        torch.cuda.synchronize()
        ms_p = e0.elapsed_time(e1) / a.steps
        pcg = {"workload": "same problem, Jacobi-preconditioned FP64 CG to the same tolerance",
               "ms_per_solve": ms_p, "iters_per_solve": itp // a.steps,
               "gdofs": E * N ** 3 * (itp // a.steps) / (ms_p * 1e-3) / 1e9,
               "speedup_solves_vs_cg": (t_max / a.steps) / ms_p, "rel_res": rel_p,
               "rel_res_true": M.true_res(b, xp),
               "err_vs_fp64_cg_inf": float((xp - x).abs().max().item() / x.abs().max().item())}

    # ---- mixed precision: FP32 inner CG (BF16 geometric factors), FP64 refinement
    mixed = None
    if not a.no_mixed:
        mixed = run_mixed(a, M, b, x, t_max, job, stream, sem, torch)

    # ---- batched: many uneven problems, one launch per order and CG phase
    batched = None
    if not a.no_batched:
        batched = run_batched(a, job, rank, stream, sem, torch)

    # ---- served: Poisson arrivals, continuous batching, HBM-budget admission
    served = None
    if not a.no_serve and rank == 0:
        from paper_2606_12650_gb300.serve import sweep
        rates = [float(r) for r in a.serve_rates.split(",")]
        rows = sweep(rates, a.serve_requests, seed=5, mode=1, budget_gb=40.0, K=16, tol=a.tol)
        served = {"workload": f"Poisson arrivals, {a.serve_requests} requests per rate, E log-uniform [8, 8192] "
                              f"(near-cubic boxes), N in {{5,7}}, jitter 5%, random source, tol {a.tol:g}, "
                              "mixed precision (BF16 G), 40 GB admission budget, 16 CG iterations per round",
                  "rates": rows, "closed_loop": run_served_ceiling(a, stream, sem, torch)}

    # ---- the paper's own protocol: GDOF/s against E for N = 4, 6, 8
    sweep_paper = None
    if not a.no_paper_sweep and rank == 0:
        sweep_paper = run_paper_sweep(a, stream, sem, torch)

    # ---- errors against the FP64 oracle on the small workload
    vs_oracle = None
    if rank == 0:
        vs_oracle = run_vs_oracle(a, sem, torch)

    # ---- end to end through the public API, host buffers
    e2e = None
    if not a.no_e2e:
        bh = torch.empty(M.nL, dtype=torch.float64).pin_memory()
        xh = torch.empty(M.nL, dtype=torch.float64).pin_memory()
        bh.copy_(b.cpu())
        sem.update(bh, sem.SEM_ALLOC)
        sem.update(xh, sem.SEM_ALLOC)
        sem.update(bh, sem.SEM_TO)
        M.cg_solve(bh, xh, a.tol, a.maxit)
        sem.update(xh, sem.SEM_FROM)
        sem.sync()
        barrier()
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        e_iters = 0
        for _ in range(a.steps):
            sem.update(bh, sem.SEM_TO)
            it, _ = M.cg_solve(bh, xh, a.tol, a.maxit)
            sem.update(xh, sem.SEM_FROM)
            sem.sync()
            e_iters += it
        t_e2e = time.perf_counter() - t0
        barrier()
        t_e2e, e_dofs = job.aggregate(t_e2e, float(E * N ** 3 * e_iters))
        e2e = {"value": e_dofs / t_e2e / 1e9, "unit": "GDOF/s", "h2d_bytes_per_step": M.nL * 8,
               "d2h_bytes_per_step": M.nL * 8, "ms_per_step": 1e3 * t_e2e / a.steps}
        assert np.allclose(xh.numpy(), x.cpu().numpy(), rtol=0, atol=0)
        sem.update(bh, sem.SEM_FREE)
        sem.update(xh, sem.SEM_FREE)

    cpu = None
    if rank == 0 and world == 1 and not a.no_cpu_baseline:
        cg, times = time_oracle(a, a.cpu_iters)
        cpu = {"value": cg, "unit": "GDOF/s", "cores": 1, "kind": "oracle",
               "sample": f"{a.cpu_iters} FP64 CG iterations of the full E={E}, N={N} problem on one host "
                         f"core (single-threaded C oracle, set-up excluded, {times[0]:.1f} s)"}
        if not a.no_cpu_allcores:
            rep = time_oracle_replicas(a, a.cpu_iters, 1)
            if rep is not None:
                n, t_rep, cores = rep
                cpu["all_cores"] = {
                    "value": n * E * N ** 3 * a.cpu_iters / t_rep[0] / 1e9, "unit": "GDOF/s", "cores": n,
                    "host_cores": cores,
                    "sample": f"the same sample run as {n} independent oracle processes (one problem each, "
                              f"started together, time of the slowest: {t_rep[0]:.1f} s)"}

    if rank == 0:
        # long tables first; the headline figures of every leg last (the
        # tail of the line is what survives truncated records)
        line = {"metric": METRIC, "value": value, "unit": "GDOF/s", "n_gpus": world, "steps": a.steps,
                "warmup": a.warmup, "ms_per_step": t_max / a.steps, "higher_is_better": True,
                "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
                "dtype_note": ("FP64 vectors, recurrences and reductions; the operator kernel the tuner chose "
                               + ("evaluates in 64-bit fixed point (one scale per element)" if v64 == 5
                                  else "evaluates in FP64")),
                "config": config_of(a, world, iters_total // max(a.steps, 1)),
                "autotune": tune, "paper_sweep": sweep_paper, "batched": batched, "serve": served,
                "pcg": pcg, "mixed": mixed, "vs_oracle": vs_oracle,
                "roofline": roofline, "cpu_baseline": cpu, "e2e": e2e, "gpu_launches": launches,
                "clocks": clk.summary(),
                "result": {"rel_res_recursive": rel, "rel_res_true": true_res,
                           "cg_iters_per_solve": iters_total // max(a.steps, 1)},
                "summary": summarize(value, t_max / a.steps, roofline, mixed, batched, served, pcg, vs_oracle)}
        print(json.dumps(line), flush=True)
    M.free()
    torch.cuda.synchronize()
    sem.finalize()
    if world > 1:
        dist.destroy_process_group()


def summarize(value, ms_fp64, roofline, mixed, batched, served, pcg, vs_oracle):
    """The headline figure of every leg in a few keys."""
    s = {"fp64_gdofs": value, "fp64_ms_per_solve": ms_fp64, "fp64_solves_per_s": 1e3 / ms_fp64,
         "operator": roofline.get("kernel"), "operator_bound": roofline.get("bound"),
         "operator_frac": roofline.get("frac")}
    if mixed:
        s.update(mixed_gdofs=mixed["value"], mixed_solves_per_s=mixed["solves_per_s"],
                 mixed_speedup_vs_fp64=mixed["speedup_solves_vs_fp64"], mixed_rel_res_true=mixed["rel_res_true"],
                 mixed_hbm_frac=mixed["roofline"]["frac"])
    if vs_oracle:
        s["err_vs_oracle_E64"] = {k: v["err_vs_oracle_inf"] for k, v in vs_oracle["solves"].items()}
    if batched:
        s["batched_solves_per_s"] = {"fp64": batched["fp64"]["solves_per_s"],
                                     "mixed": batched["mixed_bf16"]["solves_per_s"]}
        if "roofline" in batched["fp64"]:
            s["batched_hbm_frac"] = {"fp64": batched["fp64"]["roofline"]["frac"],
                                     "mixed": batched["mixed_bf16"]["roofline"]["frac"]}
    if served:
        s["served"] = [{"rate": r["rate_req_s"], "p50_ms": r["p50_ms"], "p99_ms": r["p99_ms"],
                        "solves_per_s": r["solves_per_s"]} for r in served["rates"]]
        if served.get("closed_loop"):
            s["served_closed_loop_solves_per_s"] = served["closed_loop"]["solves_per_s"]
    if pcg:
        s["pcg_ms_per_solve"] = pcg["ms_per_solve"]
    return s


def run_vs_oracle(a, sem, torch):
    """The small workload (E = 64, N = 7, jitter seed 1, sine source) solved on
    the GPU to 1e-8 and 1e-10 -- FP64 CG with the tuned operator, FP64 CG
    with the DFMA line kernel, mixed refinement with BF16 and FP32 factors --
    each error stated against the FP64 oracle's solution to 1e-12, which
    tests/golden/make_oracle_cg.py wrote (bench.py does not run the oracle)."""
    import numpy as np
    from paper_2606_12650_gb300 import Mesh
    from paper_2606_12650_gb300.inputs import box_vertices
    try:
        g = np.load(GOLDEN_SMALL)
    except OSError:
        return None
    nx, N = int(g["nx"]), int(g["N"])
    M = Mesh(nx, nx, nx, N, box_vertices(nx, nx, nx, 0.05, seed=int(g["seed"])))
    b = torch.from_numpy(g["b"]).cuda()
    x_ref = g["x"]
    scale = np.abs(x_ref).max()
    out = {"workload": f"box {nx}x{nx}x{nx} (E={nx ** 3}), N={N}, jitter 5% seed {int(g['seed'])}, sine source; "
                       f"oracle CG to {float(g['tol']):g} ({int(g['iters'])} iterations) stored in "
                       "tests/golden/oracle_cg_E64_N7.npz", "solves": {}}
    v64, e64, _ = sem.autotune_get(sem.TUNE_F64, N)
    for tol in (1e-8, 1e-10):
        legs = [("fp64_tuned", None), ("fp64_dfma_lines", (1, 4)), ("mixed_bf16", 1), ("mixed_fp32", 0)]
        for name, how in legs:
            x = torch.empty_like(b)
            if name.startswith("fp64"):
                if how is not None:
                    sem.autotune_set(sem.TUNE_F64, N, *how)
                it, rel = M.cg_solve(b, x, tol, a.maxit)
                sem.autotune_set(sem.TUNE_F64, N, v64, e64)
                info = {"iters": it, "rel_res": rel}
            else:
                inner, outer, rel = M.cg_mixed(b, x, tol, 50, a.inner_tol, a.maxit, how)
                info = {"inner_iters": inner, "outer_iters": outer, "rel_res_true": rel}
            torch.cuda.synchronize()
            info["err_vs_oracle_inf"] = float(np.abs(x.cpu().numpy() - x_ref).max() / scale)
            out["solves"][f"{name}_tol{tol:g}"] = info
    M.free()
    return out


def hbm_peak():
    try:
        with open(PEAKS_FILE) as fh:
            return float(json.load(fh)["hbm_gbs"]), "measured (MEASURED_PEAKS.json)"
    except (OSError, ValueError, KeyError):
        return 6800.0, "fallback (6.8 TB/s)"


def run_mixed(a, M, b, x64, t64_ms, job, stream, sem, torch):
    """Same problem and tolerance through mixed-precision refinement; also a
    1e-10 solve (FP64 CG and mixed) for the error table."""
    E, N = a.nx ** 3, a.N
    world, barrier = job.world, job.barrier
    xm = torch.empty_like(b)
    for _ in range(a.warmup):
        M.cg_mixed(b, xm, a.tol, 50, a.inner_tol, a.maxit, 1)
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    barrier()
    torch.cuda.synchronize()
    inner_tot, outer, res = 0, 0, 0.0
    ev0.record(stream)
    for _ in range(a.steps):
        inner, outer, res = M.cg_mixed(b, xm, a.tol, 50, a.inner_tol, a.maxit, 1)
        inner_tot += inner
    ev1.record(stream)
    torch.cuda.synchronize()
    barrier()
    t_ms, dofs = job.aggregate(ev0.elapsed_time(ev1), float(E * N ** 3 * inner_tot))
    err_vs_fp64 = float((xm - x64).abs().max().item() / x64.abs().max().item())
    true_res = M.true_res(b, xm)
    # inner operator kernel (FP32, BF16 G), timed alone on libsem's stream
    for _ in range(3):
        sem.run("cg_ax32", M.handle, 1)
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    for _ in range(a.ax_reps):
        sem.run("cg_ax32", M.handle, 1)
    e1.record(stream)
    torch.cuda.synchronize()
    ax_ms = e0.elapsed_time(e1) / a.ax_reps
    alg = E * (N + 1) ** 3 * 36   # r, p, d in (FP32); p, w, d out (FP32); 6 BF16 factors
    peak, how = hbm_peak()
    gbs = alg / (ax_ms * 1e-3) / 1e9
    traffic = None
    try:
        with open(TRAFFIC_FILE) as fh:
            t = json.load(fh).get("ax_f32_bf16_cg", {})
        if t.get("source_sha") == source_sha(AX32_SOURCES) and t.get("E") == E and t.get("N") == N:
            traffic = t.get("bytes_per_launch")
    except (OSError, ValueError):
        pass
    # 1e-10: FP64 CG reference and mixed refinement
    x10 = torch.empty_like(b)
    t0 = time.perf_counter()
    it10, _ = M.cg_solve(b, x10, 1e-10, a.maxit)
    t_fp64_10 = time.perf_counter() - t0
    xm10 = torch.empty_like(b)
    t0 = time.perf_counter()
    in10, out10, res10 = M.cg_mixed(b, xm10, 1e-10, 50, a.inner_tol, a.maxit, 1)
    t_mix_10 = time.perf_counter() - t0
    err10 = float((xm10 - x10).abs().max().item() / x10.abs().max().item())
    return {"metric": METRIC, "value": dofs / (t_ms * 1e-3) / 1e9, "unit": "GDOF/s",
            "gdofs_counts": "inner FP32 CG iterations (E N^3 per iteration)",
            "dtype": "f32 inner CG (dots: f32 per block, f64 across blocks), bf16 geometric factors, f64 refinement/alpha/beta",
            "workload": f"same problem, mixed-precision refinement to {a.tol:g} (inner tolerance {a.inner_tol:g})",
            "ms_per_solve": t_ms / a.steps, "solves_per_s": 1e3 * a.steps / t_ms * world,
            "fp64_solves_per_s": 1e3 * a.steps / t64_ms * world,
            "speedup_solves_vs_fp64": t64_ms / t_ms,
            "inner_iters_per_solve": inner_tot // max(a.steps, 1), "outer_iters": outer,
            "rel_res_true": true_res, "err_vs_fp64_cg_inf": err_vs_fp64,
            "roofline": {"bound": "hbm", "achieved": gbs, "peak": peak, "unit": "GB/s", "frac": gbs / peak,
                         "traffic": traffic,
                         "kernel": kernel_label(*sem.autotune_get(sem.TUNE_F32_G16, N)[:2], N, "float", "bf16"),
                         "launch_ms": ax_ms, "alg_bytes_per_launch": alg, "peak_source": how},
            "tol_1e-10": {"fp64_cg_iters": it10, "fp64_ms": 1e3 * t_fp64_10,
                          "mixed_inner_iters": in10, "mixed_outer_iters": out10, "mixed_ms": 1e3 * t_mix_10,
                          "mixed_rel_res_true": res10, "err_vs_fp64_cg_inf": err10}}


def run_batched(a, job, rank, stream, sem, torch):
    """256 independent problems (E log-uniform in [8, 4096] as near-cubic boxes,
    N uniform in {3, 5, 7, 9}, jitter 5 %, random right-hand sides), each CG
    phase of all of them one launch per order: FP64 CG and mixed refinement
    to 1e-8.  Throughput counts every problem's own iterations."""
    import numpy as np
    from paper_2606_12650_gb300 import Batch, Mesh
    from paper_2606_12650_gb300.inputs import batch_specs, box_vertices, normal_field
    from paper_2606_12650_gb300.ranks import rank_seed
    world, barrier = job.world, job.barrier
    specs = batch_specs(a.batch_count, seed=rank_seed(4, rank), e_lo=8, e_hi=4096, orders=(3, 5, 7, 9))
    t0 = time.perf_counter()
    meshes, bs = [], []
    for s in specs:
        jit = 0.05 if min(s["nx"], s["ny"], s["nz"]) > 1 else 0.0
        m = Mesh(s["nx"], s["ny"], s["nz"], s["N"], box_vertices(s["nx"], s["ny"], s["nz"], jit, seed=s["mesh_seed"]))
        f = torch.from_numpy(normal_field(m.nL, s["rhs_seed"])).cuda()
        m.gs(f)
        m.mask(f)
        meshes.append(m)
        bs.append(f)
    # per-order tuner: each order of the mix tuned on its largest problem (FP64
    # and the mixed path's FP32/BF16 operator); the batch takes its operator
    # body and elements per item from the resulting table
    tuned = {}
    saved = {(k, N): sem.autotune_get(k, N) for k in (sem.TUNE_F64, sem.TUNE_F32_G16) for N in range(1, 10)}
    if not a.no_tune:
        for N in sorted({m.N for m in meshes}):
            big = max((m for m in meshes if m.N == N), key=lambda m: m.E)
            tuned[N] = {}
            for kind, name in ((sem.TUNE_F64, "fp64"), (sem.TUNE_F32_G16, "fp32_bf16")):
                big.autotune(kind, reps=5)
                v, e, us = sem.autotune_get(kind, N)
                tuned[N][name] = {"variant": VARIANTS[v], "epb": e, "us": us, "tuned_on_E": big.E}
    B = Batch(meshes)
    b_all = torch.cat(bs)
    del bs
    x_all = torch.empty_like(b_all)
    setup_s = time.perf_counter() - t0
    gdof_per_iter = np.array([m.E * m.N ** 3 for m in meshes], dtype=np.float64)
    nL = np.array([m.nL for m in meshes], dtype=np.float64)
    # algorithmic bytes per local node and CG iteration: FP64 -- operator r, p,
    # x in, p, w, x out, 48 B of factors (96), update r, w in, r out (24);
    # mixed -- FP32 operator likewise with BF16 factors (36), FP32 update (12)
    bytes_per_node_iter = {"fp64": 120.0, "mixed_bf16": 48.0}
    hbm, hbm_how = hbm_peak()
    out = {"workload": f"{len(meshes)} problems, E log-uniform [8, 4096] (near-cubic boxes), N in {{3,5,7,9}}, "
                       f"jitter 5%, random RHS; tol {a.tol:g}; per order one launch per CG phase, the orders in parallel",
           "problems": len(meshes), "local_dofs_total": int(B.nL_total), "tuned_per_order": tuned,
           "E_total": int(sum(m.E for m in meshes)), "setup_s": setup_s}
    for mode, name in ((0, "fp64"), (1, "mixed_bf16")):
        B.solve(b_all, x_all, a.tol, a.maxit, mode, a.inner_tol)    # warm-up (graph capture)
        barrier()
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        its, res = B.solve(b_all, x_all, a.tol, a.maxit, mode, a.inner_tol)
        e1.record(stream)
        torch.cuda.synchronize()
        ms, dofs = job.aggregate(e0.elapsed_time(e1), float((gdof_per_iter * its).sum()))
        out[name] = {"ms": ms, "gdofs": dofs / (ms * 1e-3) / 1e9, "solves_per_s": 1e3 * len(meshes) * world / ms,
                     "iters_total": int(its.sum()), "iters_max": int(its.max()), "max_rel_res": float(res.max())}
        # the roofline summed over the problems: HBM time of each problem's
        # own iterations' algorithmic bytes (inner iterations for mixed; the
        # refinement steps' few FP64 passes not counted), against the batch time
        hbm_ms = float((its * nL).sum()) * bytes_per_node_iter[name] / (hbm * 1e9) * 1e3   # per GPU (replicas)
        out[name]["roofline"] = {"bound": "hbm", "alg_bytes_per_node_iter": bytes_per_node_iter[name],
                                 "hbm_time_ms": hbm_ms, "frac": hbm_ms / ms, "peak_gbs": hbm,
                                 "peak_source": hbm_how}
    out["speedup_mixed_vs_fp64"] = out["fp64"]["ms"] / out["mixed_bf16"]["ms"]
    B.free()
    for (k, N), (v, e, _) in saved.items():      # the later legs use the table tuned on the main problem
        sem.autotune_set(k, N, v, e)
    for m in meshes:
        m.free()
    return out


def run_served_ceiling(a, stream, sem, torch, count=256):
    """The serving ceiling: `count` requests of the served mix (E log-uniform
    [8, 8192], N in {5, 7}) all present at once, solved by the batch engine
    (mixed precision, BF16 factors) closed-loop: no arrivals, no admission."""
    from paper_2606_12650_gb300 import Batch, Mesh
    from paper_2606_12650_gb300.serve import make_requests
    reqs = make_requests(count, seed=5)
    meshes, bs = [], []
    for r in reqs:
        m = Mesh(r["nx"], r["ny"], r["nz"], r["N"], r["verts"])
        f = torch.from_numpy(r["f"]).cuda()
        m.gs(f)
        m.mask(f)
        meshes.append(m)
        bs.append(f)
    B = Batch(meshes)
    b_all = torch.cat(bs)
    del bs
    x_all = torch.empty_like(b_all)
    B.solve(b_all, x_all, a.tol, a.maxit, 1, a.inner_tol)     # warm-up (graph capture)
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    its, res = B.solve(b_all, x_all, a.tol, a.maxit, 1, a.inner_tol)
    e1.record(stream)
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1)
    B.free()
    for m in meshes:
        m.free()
    return {"workload": f"{count} requests of the served mix solved as one batch (mixed, BF16 G), closed loop",
            "ms": ms, "solves_per_s": 1e3 * count / ms, "max_rel_res": float(res.max())}


def run_paper_sweep(a, stream, sem, torch):
    """The paper's Nekbone protocol (Section VIII-B): unpreconditioned CG, N in
    {4, 6, 8}, E = 2^1 .. 2^14 (near-cubic boxes, jitter 5 %, sine source),
    100 iterations timed after 100 warm-up iterations, mean of 5; GDOF/s =
    E N^3 100 / t.  Each timed solve includes its initialisation kernel and
    the host's polling of the stop flag."""
    from paper_2606_12650_gb300 import Mesh
    from paper_2606_12650_gb300.inputs import box_vertices, near_cubic
    out = {"workload": "CG 100 iterations (no tolerance), N in {4,6,8}, E = 2^1..2^14 near-cubic, jitter 5%, "
                       "sine source; 100 warm-up iterations, mean of 5 timed solves", "gdofs": {}, "saturation_E": {}}
    for N in (4, 6, 8):
        row = {}
        for k in range(1, 15):
            E = 2 ** k
            nx, ny, nz = near_cubic(E)
            jit = 0.05 if min(nx, ny, nz) > 1 else 0.0
            M = Mesh(nx, ny, nz, N, box_vertices(nx, ny, nz, jit, seed=1))
            b = torch.empty(M.nL, dtype=torch.float64, device="cuda")
            M.rhs_sin(b)
            x = torch.empty_like(b)
            M.cg_solve(b, x, 0.0, 100)
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            e0.record(stream)
            for _ in range(5):
                M.cg_solve(b, x, 0.0, 100)
            e1.record(stream)
            torch.cuda.synchronize()
            t = e0.elapsed_time(e1) / 5 * 1e-3
            row[E] = E * N ** 3 * 100 / t / 1e9
            M.free()
        out["gdofs"][N] = row
        top = max(row.values())
        out["saturation_E"][N] = min(E for E, g in row.items() if g >= 0.9 * top)
    out["saturation_dofs"] = {N: E * N ** 3 for N, E in out["saturation_E"].items()}
    out["paper_context"] = ("the paper publishes no absolute GDOF/s (its plots are absent); it reports saturation "
                            "at about 4e6 DOFs for N >= 6 on one MI250X GCD, FP64 (Section VIII-B)")
    return out


def main():
    a = parse()
    if a.impl == "reference":
        run_reference(a)
    else:
        run_ours(a)


if __name__ == "__main__":
    main()
