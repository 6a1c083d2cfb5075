#!/usr/bin/env python
"""DDM-GMRES throughput on the 256x256 order-2 square (525,312 complex DOFs,
8x8 subdomains, omega = 40 pi, mu^{-1} piecewise constant on 16x16-cell tiles).

One step = thm_assemble (operators, Dirichlet lifting, block-preconditioner
factorisation) + thm_ddm_solve to a global FP64 true residual of 1e-8, with
mu^{-1} already resident in HBM.  The mesh numbering / subdomain structure is
built once per geometry before the timed region (its time is reported apart).

value = DOF*iterations per second (sum over subdomains and sweeps of n_i times
inner GMRES steps, divided by the step time), summed over ranks; the
time-to-1e-8 of the same steps is reported as time_to_1e8_s.  Under torchrun
(N > 1) every rank solves its own copy (replicas: the path does not shard
across GPUs, see the design notes), so scaling is weak.

--impl reference times the FP64 CPU oracle of the same workload on all host
cores (per step the whole first DDM sweep: the paper's block-preconditioned
GMRES in every subdomain, subdomains dealt to one worker process per core).
"""
from __future__ import annotations

import argparse
import json
import math
import os
import statistics
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

WORKLOAD = "square256_p2"
WORKLOAD_DESC = ("square256_p2: unit square, 256x256 quads, order-2 Nedelec (12 DOFs/quad, "
                 "525,312 complex DOFs), 8x8 subdomains of 32x32 cells, omega=40*pi, kappa=1, "
                 "mu^-1 piecewise constant on 16x16-cell tiles U[0.5,2] (seed 20210525), "
                 "E_inc=(0,exp(-i omega x)) Dirichlet on x=0, impedance elsewhere")
METRIC = "DDM-GMRES DOF*iters/s to a 1e-8 FP64 true residual (time-to-1e-8 beside it)"
UNIT = "DOF*iter/s"


def parse():
    p = argparse.ArgumentParser()
    p.add_argument("--gpus", type=int, default=1)
    p.add_argument("--steps", type=int, default=2)
    p.add_argument("--warmup", type=int, default=3)
    p.add_argument("--impl", default="ours", choices=["ours", "reference"])
    p.add_argument("--mode", default="mixed", choices=["mixed", "fp64"])
    p.add_argument("--fp64-steps", type=int, default=1, help="steps of the plain FP64 form timed beside")
    p.add_argument("--no-cpu-baseline", action="store_true")
    p.add_argument("--ref-subdomains", type=int, default=4, help="subdomains per reference sample")
    p.add_argument("--e2e-steps", type=int, default=1)
    p.add_argument("--full-steps", type=int, default=1,
                   help="steps with the full 2x2 block preconditioner (Section 3.2's alternative) timed beside")
    p.add_argument("--prof-steps", type=int, default=1,
                   help="instrumented steps after the timed region (per-launch CUDA-event timing)")
    p.add_argument("--relax", type=int, default=1, help="inexact-Krylov relaxation of the subdomain tolerance")
    p.add_argument("--batch", type=int, default=0, metavar="K",
                   help="instead of the headline workload: the first K problems of the 512-problem batch "
                        "workload solved as one batch and, for comparison, one by one")
    p.add_argument("--table1", action="store_true",
                   help="instead of the headline workload: block-preconditioned GMRES iteration counts against omega "
                        "on the centre-block square (the paper's Example 1 / Table 1), GPU and oracle")
    p.add_argument("--ncu-sweep", action="store_true",
                   help="assemble the workload and run two DDM sweeps only (bounded case for ncu captures)")
    return p.parse_args()


def ncu_sweep(args):
    """Two sweeps of the bench workload (the first builds the factors): the kernel mix of the timed solve, in a few seconds,
    for ncu.  The interface data are seeded random values, so every
    subdomain's solve is active (with zero interface data only the subdomains
    on the Dirichlet side would have a right-hand side)."""
    import torch
    import paper_2105_11993_gb300 as thm
    import workloads as W
    from paper_2105_11993_gb300 import build
    build.build()
    P = W.config(WORKLOAD)
    mesh = thm.Mesh.from_workload(P.mesh, P.order)
    sysg = thm.System(mesh, torch.tensor(P.mu_inv, device="cuda"), P.omega, P.kappa, P.pol, P.direction)
    gen = torch.Generator(device="cpu").manual_seed(20210525)
    g = (torch.randn(sysg.n_iface, generator=gen, dtype=torch.float64)
         + 1j * torch.randn(sysg.n_iface, generator=gen, dtype=torch.float64)).to("cuda") * 1e-2
    for _ in range(2):
        sysg.sweep(g, True, mode=args.mode)
    torch.cuda.synchronize()
    print("ncu sweep done", flush=True)


# --------------------------------------------------------------------------
# clocks sampled during the timed region
# --------------------------------------------------------------------------
class ClockSampler:
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.gpu = gpu_index
        self.proc = None
        self.lines = []

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--id={self.gpu}", f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
                 "-lms", "200"], stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
        except (FileNotFoundError, OSError):
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
        sm, smax, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            f = [x.strip() for x in ln.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                smax = float(f[2])
            except ValueError:
                continue
            for nm, v in zip(names, f[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(nm)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": smax,
                "reasons": sorted(reasons), "samples": len(sm)}


# --------------------------------------------------------------------------
# dist helpers
# --------------------------------------------------------------------------
def dist_env():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


def init_dist(ws, backend):
    if ws > 1:
        import torch.distributed as dist
        os.environ.setdefault("MASTER_ADDR", "127.0.0.1")
        dist.init_process_group(backend=backend)
        return dist
    return None


def barrier(dist):
    if dist is not None:
        dist.barrier()


def allreduce_max(dist, x):
    if dist is None:
        return x
    import torch
    t = torch.tensor([x], dtype=torch.float64, device="cuda" if torch.cuda.is_available() else "cpu")
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def allreduce_sum(dist, x):
    if dist is None:
        return x
    import torch
    t = torch.tensor([x], dtype=torch.float64, device="cuda" if torch.cuda.is_available() else "cpu")
    dist.all_reduce(t)
    return float(t.item())


# --------------------------------------------------------------------------
# CPU oracle sample (cpu_baseline and --impl reference)
# --------------------------------------------------------------------------
ORACLE_SNIPPET = r"""
import json, os, sys, time, platform
sys.path.insert(0, {root!r})
import numpy as np
import workloads as W
from oracle import ddm
P = W.config({workload!r})
t0 = time.perf_counter()
D = ddm.setup(P)
solve = ddm.subdomain_solver(D, "block_gmres", inner_tol=1e-10, restart=120)
src = ddm.local_sources(D)
setup_s = time.perf_counter() - t0

def rhs_of(i):
    r = src[i]
    return r if np.any(r) else np.ones(len(D.subs[i].free), np.complex128)

def solve_one(i):
    D.stats["inner_iters"] = []
    solve(i, rhs_of(i))
    return len(D.subs[i].free) * D.stats["inner_iters"][-1][1]

def cpu_model():
    try:
        for ln in open("/proc/cpuinfo"):
            if ln.lower().startswith(("model name", "cpu part", "hardware")):
                return ln.split(":", 1)[1].strip()
    except OSError:
        pass
    return platform.processor() or platform.machine()

out = {{"setup_s": setup_s, "nproc": os.cpu_count(), "cpu": cpu_model(), "machine": platform.machine(),
       "n_sub": len(D.subs)}}
# (i) one thread: the first DDM sweep (zero interface data) restricted to a fixed subdomain sample
picks = list(range(0, len(D.subs), max(1, len(D.subs) // {nsub})))[:{nsub}]
single = []
for step in range({steps}):
    t = time.perf_counter()
    di = sum(solve_one(i) for i in picks)
    single.append((time.perf_counter() - t, di))
out["single"] = single
out["picks"] = picks
# (ii) all host cores: the whole first sweep (every subdomain), subdomains
# dealt to a pool of one worker per core.  This process never touches a GPU,
# so the workers are forked and share the set-up.
if {allcore_steps} > 0:
    import multiprocessing as mp
    ncore = os.cpu_count()
    order = sorted(range(len(D.subs)), key=lambda i: -len(D.subs[i].free))
    with mp.get_context("fork").Pool(ncore) as pool:
        pool.map(solve_one, order[:ncore])            # workers up (untimed)
        allc = []
        for step in range({allcore_steps}):
            t = time.perf_counter()
            di = sum(pool.map(solve_one, order, chunksize=1))
            allc.append((time.perf_counter() - t, di))
    out["allcore"] = allc
    out["allcore_workers"] = ncore
print(json.dumps(out))
"""


def run_oracle_sample(steps, nsub, allcore_steps=0):
    env = dict(os.environ)
    for k in ("OMP_NUM_THREADS", "OPENBLAS_NUM_THREADS", "MKL_NUM_THREADS"):
        env[k] = "1"
    code = ORACLE_SNIPPET.format(root=ROOT, workload=WORKLOAD, nsub=nsub, steps=steps,
                                 allcore_steps=allcore_steps)
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, env=env, timeout=1800)
    if r.returncode != 0:
        raise RuntimeError(r.stderr[-2000:])
    return json.loads(r.stdout.strip().splitlines()[-1])


def reference_arm(args):
    """The FP64 oracle on all host cores: each step is the whole first DDM
    sweep of the workload (block-preconditioned GMRES in every subdomain,
    subdomains dealt to one worker per core)."""
    ws, rank, _ = dist_env()
    if rank != 0:
        return
    K, Wm = args.steps, args.warmup
    res = run_oracle_sample(0, args.ref_subdomains, allcore_steps=K + Wm)
    timed = res["allcore"][Wm:]
    t = sum(s for s, _ in timed)
    di = sum(d for _, d in timed)
    value = di / t
    cores = res["allcore_workers"]
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
        "steps": K, "warmup": Wm, "ms_per_step": 1e3 * t / K, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": WORKLOAD_DESC,
                   "mode": f"fp64 oracle (numpy/scipy), {cores} worker processes of 1 thread"},
        "cpu_baseline": {"value": value, "unit": UNIT, "cores": cores, "kind": "oracle",
                         "cpu": res["cpu"], "nproc": res["nproc"],
                         "sample": f"per step: the whole first DDM sweep ({res['n_sub']} "
                                   f"block-preconditioned GMRES subdomain solves, tol 1e-10) over {cores} "
                                   f"forked workers; oracle set-up {res['setup_s']:.1f}s untimed"},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)


# --------------------------------------------------------------------------
# our arm
# --------------------------------------------------------------------------
def bytes_per_launch(sysg, mode, cls):
    import paper_2105_11993_gb300 as thm
    return thm.algorithmic_bytes(sysg, mode, cls)


def batch_arm(args):
    """Batched solve of K independent 2-D problems (sides U{16..128}, omega
    U[2pi,32pi], kappa=1, lognormal mu^{-1}, ceil(n/32)^2 subdomains) against
    a loop of the plain solver over the same problems.  Both stop at rtol 1e-8
    or at the same iteration caps (300 interface steps, 3 refinements); the
    coarsest draws (about one cell per wavelength) may not converge, which the
    line reports."""
    import numpy as np
    import torch
    import paper_2105_11993_gb300 as thm
    import workloads as W
    from paper_2105_11993_gb300 import build
    build.build()
    probs = W.batch_problems(512)[:args.batch]
    kw = dict(mode=args.mode, rtol=1e-8, relax=args.relax, outer_maxit=300, max_refine=3, check=False)
    # timed: assembly, factorisation and solve (time to solution); the
    # meshes (host-side numbering) are built beforehand for both arms
    mesh, _ = thm.Mesh.batch([P.mesh for P in probs], 1)
    mu = np.concatenate([P.mu_inv for P in probs])
    om = np.array([P.omega for P in probs])
    meshes = [thm.Mesh.from_workload(P.mesh, 1) for P in probs]
    wp = W.square_problem(8, 2, 1, 5.0)              # warm-up: module loading, first launches
    thm.System(thm.Mesh.from_workload(wp.mesh, 1), wp.mu_inv, wp.omega, 1.0, wp.pol, wp.direction).solve(**kw)
    torch.cuda.synchronize()
    t = time.perf_counter()
    sb = thm.System(mesh, mu, om, 1.0, probs[0].pol, probs[0].direction)
    _, stb = sb.solve(**kw)
    torch.cuda.synchronize()
    tb = time.perf_counter() - t
    tl, dil, conv = 0.0, 0, 0
    for P, m1 in zip(probs, meshes):
        torch.cuda.synchronize()
        t = time.perf_counter()
        s1 = thm.System(m1, P.mu_inv, P.omega, 1.0, P.pol, P.direction)
        _, st1 = s1.solve(**kw)
        torch.cuda.synchronize()
        tl += time.perf_counter() - t
        dil += st1["dof_iters"]
        conv += st1["status"] == 0
    ppw = [2 * math.pi * P.mesh.shape[0] / P.omega for P in probs]
    line = {"metric": "batched DDM-GMRES solve of independent problems vs a loop of single solves",
            "value": stb["dof_iters"] / tb, "unit": UNIT, "n_gpus": 1, "higher_is_better": True,
            "dtype": "f32 operator/preconditioner/inner Krylov + f64 refinement" if args.mode == "mixed" else "f64",
            "data": "synthetic",
            "config": {"workload": f"first {len(probs)} of the 512-problem batch (seed 20210525)",
                       "n_dof": mesh.info()["n_dof"], "n_sub": mesh.info()["n_sub"],
                       "cells_per_wavelength": [min(ppw), max(ppw)], "caps": "300 interface steps, 3 refinements"},
            "batch": {"seconds": tb, "problems_per_s": len(probs) / tb, "status": stb["status"],
                      "max_rel_residual": stb["rel_residual"], "outer_steps": stb["outer_iters"],
                      "dof_iters": stb["dof_iters"]},
            "loop": {"seconds": tl, "problems_per_s": len(probs) / tl, "converged": conv, "dof_iters": dil,
                     "dof_iters_per_s": dil / tl},
            "speedup_time": tl / tb}
    print(json.dumps(line), flush=True)


TABLE1_OMEGAS = (5.0, 10.0, 20.0, 40.0, 80.0)
TABLE1_PAPER = (43, 49, 33, 32, 28)      # the paper's Table 1, block preconditioner (AMG inside, Xeon 8268)


def table1_arm(args):
    """Iterations of GMRES with the block preconditioner of Eq. 7 (exact P^{-1})
    to a relative 1e-8 on one domain: the unit square, 64x64 order-2 quads,
    a centre block [0.25,0.75]^2 of refractive index 1.516 in air, for the
    omegas of the paper's Table 1.  FP64 and mixed precision on the GPU; the
    FP64 oracle's count (MGS GMRES, sparse LU for P) beside each."""
    import torch
    import paper_2105_11993_gb300 as thm
    import workloads as W
    from paper_2105_11993_gb300 import build
    build.build()
    n = 64
    rows = []
    for om in TABLE1_OMEGAS:
        P = W.block_benchmark(n, 1, 2, om)
        mesh = thm.Mesh.from_workload(P.mesh, P.order)
        row = {"omega": om, "cells_per_wavelength_in_block": 2 * math.pi * n / (om * 1.516)}
        for mode in ("fp64", "mixed"):
            sysg = thm.System(mesh, P.mu_inv, P.omega, P.kappa, P.pol, P.direction, eps=P.eps)
            torch.cuda.synchronize()
            t = time.perf_counter()
            _, st = sysg.solve(mode=mode, rtol=1e-8, inner_tol=1e-8, inner_restart=600, inner_maxit=600,
                               max_refine=1, check=False)
            torch.cuda.synchronize()
            row[mode] = {"gmres_iters": st["inner_iters"], "rel_residual": st["rel_residual"],
                         "seconds": time.perf_counter() - t}
        row["oracle_gmres_iters"] = oracle_table1_count(n, om)
        rows.append(row)
    line = {"metric": "block-preconditioned GMRES iterations to 1e-8 vs omega (Table 1 form)",
            "unit": "iterations", "data": "synthetic",
            "config": {"workload": "block_benchmark: unit square, 64x64 order-2 quads (one domain), centre block "
                                   "[0.25,0.75]^2 with n=1.516 (eps=n^2), mu^-1=1, Dirichlet x=0, impedance elsewhere",
                       "preconditioner": "Eq. 7 with the exact P^-1 (nested dissection)"},
            "rows": rows,
            "paper_table1": {"omega": list(TABLE1_OMEGAS), "iters": list(TABLE1_PAPER),
                             "context": "AMG (MueLu) approximation of P^-1, mesh and order not stated, Xeon 8268"}}
    print(json.dumps(line), flush=True)


def oracle_table1_count(n, omega):
    code = (f"import sys; sys.path.insert(0, {ROOT!r})\n"
            "import workloads as W\nfrom oracle import ddm\n"
            f"P = W.block_benchmark({n}, 1, 2, {omega!r})\nD = ddm.setup(P)\n"
            "s = ddm.subdomain_solver(D, 'block_gmres', inner_tol=1e-8, restart=600, maxiter=600)\n"
            "s(0, ddm.local_sources(D)[0])\nprint(D.stats['inner_iters'][-1][1])\n")
    env = dict(os.environ)
    for k in ("OMP_NUM_THREADS", "OPENBLAS_NUM_THREADS", "MKL_NUM_THREADS"):
        env[k] = "1"
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, env=env, timeout=1200)
    return int(r.stdout.strip().splitlines()[-1]) if r.returncode == 0 else None


def kernel_classes_report(thm, prof, ms_total):
    """Per launch class: launches, average CUDA-event time, share of the step."""
    out = {}
    for c, (n, ms) in prof.items():
        out[thm.K_NAMES[c]] = {"launches": n, "avg_launch_us": 1e3 * ms / max(1, n),
                               "share_of_step": ms / ms_total if ms_total > 0 else None}
    return out


def main():
    args = parse()
    if args.impl == "reference":
        return reference_arm(args)
    if args.ncu_sweep:
        return ncu_sweep(args)
    if args.batch > 0:
        return batch_arm(args)
    if args.table1:
        return table1_arm(args)
    ws, rank, local = dist_env()
    import numpy as np
    import torch

    torch.cuda.set_device(local)
    dist = init_dist(ws, "nccl")
    import paper_2105_11993_gb300 as thm
    import workloads as W
    from paper_2105_11993_gb300 import build
    if rank == 0:
        build.build()
    barrier(dist)
    thm.load()
    P = W.config(WORKLOAD)
    mu_h = np.ascontiguousarray(P.mu_inv)
    mu_d = torch.tensor(mu_h, device="cuda")
    st = torch.cuda.current_stream()

    t = time.perf_counter()
    mesh = thm.Mesh.from_workload(P.mesh, P.order)
    mesh_s = time.perf_counter() - t
    mode = args.mode

    def step(m, relax=None, **kw):
        sysg = thm.System(mesh, mu_d, P.omega, P.kappa, P.pol, P.direction, stream=st)
        u, stats = sysg.solve(mode=m, rtol=1e-8, relax=args.relax if relax is None else relax, **kw)
        return sysg, u, stats

    # warm-up: module loading, first launches
    for _ in range(args.warmup):
        step(mode)
    torch.cuda.synchronize()

    # ---- timed region: plain steps, no per-launch instrumentation ----
    thm.profile_enable(0)
    clk = ClockSampler(local)
    clk.start()
    barrier(dist)
    torch.cuda.synchronize()
    launches0 = thm.kernel_launches()
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    e0.record(st)
    stats_all = []
    for _ in range(args.steps):
        _, _, stats = step(mode)
        stats_all.append(stats)
    e1.record(st)
    torch.cuda.synchronize()
    barrier(dist)
    launches = thm.kernel_launches() - launches0
    clocks = clk.stop()
    ms = e0.elapsed_time(e1)
    ms_max = allreduce_max(dist, ms)

    dof_iters = sum(s["dof_iters"] for s in stats_all)
    total_dof_iters = allreduce_sum(dist, dof_iters)
    value = total_dof_iters / (ms_max / 1e3)
    tt = [s["seconds"] for s in stats_all]

    # ---- instrumented steps (after the timed region): per-class CUDA-event
    # timing of every launch, and the work of the subdomain solves counted on the device ----
    classes = (thm.K_SUBSOLVE, thm.K_PINV, thm.K_SPMV, thm.K_DOTS, thm.K_UPDATE, thm.K_KRYLOV, thm.K_DDM, thm.K_SETUP)
    thm.profile_enable(sum(1 << c for c in classes))
    torch.cuda.synchronize()
    p0 = torch.cuda.Event(enable_timing=True)
    p1 = torch.cuda.Event(enable_timing=True)
    p0.record(st)
    names = {thm.K_PINV: "block-preconditioner applies", thm.K_SPMV: "subdomain operator applies",
             thm.K_DOTS: "Gram-Schmidt dot products", thm.K_UPDATE: "Gram-Schmidt updates"}
    work = {c: 0.0 for c in names}
    pstats = []
    for _ in range(max(1, args.prof_steps)):
        sysg, _, s1 = step(mode)
        pstats.append(s1)
        for c in work:
            work[c] += thm.work_bytes(sysg, mode, c)
    p1.record(st)
    torch.cuda.synchronize()
    prof_ms = p0.elapsed_time(p1)
    prof = {c: thm.profile_read(c) for c in classes}
    thm.profile_enable(0)

    # roofline of the dominant kernel (the subdomain solves of a sweep, one launch)
    peaks = {}
    try:
        peaks = json.load(open(os.path.join(ROOT, "MEASURED_PEAKS.json")))
    except (OSError, ValueError):
        pass
    hbm_peak = peaks.get("hbm_gbs", 6800.0)
    peak_src = "measured" if "hbm_gbs" in peaks else "fallback"
    n_launch, sub_ms = prof[thm.K_SUBSOLVE]
    total_work = sum(work.values())
    achieved = total_work / (sub_ms / 1e3) / 1e9 if n_launch and sub_ms > 0 else None
    roofline = {"kernel": "k_subsolve (subdomain GMRES solves, one launch per sweep)", "bound": "hbm",
                "achieved": achieved, "peak": hbm_peak, "unit": "GB/s",
                "frac": (achieved / hbm_peak) if achieved else None,
                "traffic": None,               # no DRAM counters of a whole solve launch
                "peak_source": peak_src, "launches": n_launch, "avg_launch_us": 1e3 * sub_ms / max(1, n_launch),
                "alg_bytes_processed": total_work,
                "alg_bytes_by_part": {names[c]: work[c] for c in names},
                "achieved_definition": "algorithmic bytes of the Arnoldi steps done (counted on the device: factors, "
                                       "operator, basis vectors read and written) / summed CUDA-event time of its "
                                       f"launches, over {max(1, args.prof_steps)} instrumented step(s) run after the "
                                       "timed region",
                "share_of_step": (sub_ms / prof_ms) if prof_ms > 0 else None,
                "classes": kernel_classes_report(thm, prof, prof_ms),
                "instrumented_ms_per_step": prof_ms / max(1, args.prof_steps),
                "instrumented_time_to_1e8_s": statistics.median(s["seconds"] for s in pstats)}

    # plain FP64 form, timed beside (time-to-1e-8); warmed first (FP64 kernels
    # and factorisation).
    # It runs without the relaxation of the subdomain tolerance (its FP64
    # subdomain solves stop exactly at the relaxed tolerance, which costs the
    # interface GMRES more steps than it saves: 1,000 against 361 measured)
    fp64 = None
    if mode == "mixed" and args.fp64_steps > 0:
        step("fp64", relax=0, outer_maxit=3, max_refine=1, check=False)
        torch.cuda.synchronize()
        f0 = torch.cuda.Event(enable_timing=True)
        f1 = torch.cuda.Event(enable_timing=True)
        f0.record(st)
        fstats = []
        for _ in range(args.fp64_steps):
            _, _, s64 = step("fp64", relax=0)
            fstats.append(s64)
        f1.record(st)
        torch.cuda.synchronize()
        fms = f0.elapsed_time(f1) / args.fp64_steps
        fp64 = {"relax": 0, "ms_per_step": fms, "time_to_1e8_s": statistics.median(s["seconds"] for s in fstats),
                "dof_iters_per_s": sum(s["dof_iters"] for s in fstats) / (fms * args.fp64_steps / 1e3),
                "outer_iters": fstats[-1]["outer_iters"], "inner_iters": fstats[-1]["inner_iters"],
                "sweeps": fstats[-1]["sweeps"], "refine_steps": fstats[-1]["refine_steps"],
                "max_inner_iters": fstats[-1]["max_inner_iters"],
                "rel_residual": fstats[-1]["rel_residual"],
                "mixed_speedup_time_to_1e8": statistics.median(s["seconds"] for s in fstats) / statistics.median(tt)}

    # Section 3.2's alternative preconditioner: the exact inverse of the full
    # 2x2 block operator (T_i^{-1}, complex factors: twice the memory), timed
    # beside the Eq. 7 form on the same workload; warmed first
    full = None
    if mode == "mixed" and args.full_steps > 0:
        step(mode, precond="full", outer_maxit=3, max_refine=1, check=False)
        torch.cuda.synchronize()
        full = {"precond": "full 2x2 block operator, exact inverse (T_i^-1 from complex factors)",
                "eq7_inner_iters": stats_all[-1]["inner_iters"], "eq7_time_to_1e8_s": statistics.median(tt)}
        for rlx in (0, 1):
            g0 = torch.cuda.Event(enable_timing=True)
            g1 = torch.cuda.Event(enable_timing=True)
            g0.record(st)
            gstats = []
            for _ in range(args.full_steps):
                sysf, _, sf = step(mode, relax=rlx, precond="full")
                gstats.append(sf)
            g1.record(st)
            torch.cuda.synchronize()
            t1e8 = statistics.median(s["seconds"] for s in gstats)
            full[f"relax{rlx}"] = {
                "ms_per_step": g0.elapsed_time(g1) / args.full_steps, "time_to_1e8_s": t1e8,
                "outer_iters": gstats[-1]["outer_iters"], "inner_iters": gstats[-1]["inner_iters"],
                "max_inner_iters": gstats[-1]["max_inner_iters"], "sweeps": gstats[-1]["sweeps"],
                "refine_steps": gstats[-1]["refine_steps"], "rel_residual": gstats[-1]["rel_residual"],
                "speedup_time_to_1e8_vs_eq7": statistics.median(tt) / t1e8}
        full["factor_bytes"] = thm.factor_bytes(sysf, "full", mode)
        full["eq7_factor_bytes"] = thm.factor_bytes(sysf, "blockdiag", mode)

    # end to end through the host API: mesh from host arrays, mu^{-1} from
    # pinned host memory, solution copied back to host memory
    mu_pin = torch.tensor(mu_h).pin_memory()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    e2e_di = 0
    for _ in range(args.e2e_steps):
        mesh2 = thm.Mesh.from_workload(P.mesh, P.order)
        s2 = thm.System(mesh2, mu_pin.numpy(), P.omega, P.kappa, P.pol, P.direction, stream=st)
        uh, st2 = s2.solve_host(mode=mode, rtol=1e-8, relax=args.relax)
        e2e_di += st2["dof_iters"]
        del s2, mesh2
    torch.cuda.synchronize()
    e2e_t = time.perf_counter() - t0
    e2e_t = allreduce_max(dist, e2e_t)
    e2e_val = allreduce_sum(dist, e2e_di) / e2e_t if args.e2e_steps > 0 else None

    cpu = None
    if rank == 0 and not args.no_cpu_baseline:
        try:
            res = run_oracle_sample(3, args.ref_subdomains, allcore_steps=3)
            one = statistics.median(d / s for s, d in res["single"])
            allc = statistics.median(d / s for s, d in res["allcore"])
            cpu = {"value": allc, "unit": UNIT, "cores": res["allcore_workers"], "kind": "oracle",
                   "cpu": res["cpu"], "nproc": res["nproc"], "machine": res["machine"],
                   "single_thread": {"value": one, "cores": 1,
                                     "sample": f"block-preconditioned GMRES (tol 1e-10) solves of subdomains "
                                               f"{res['picks']} of the first DDM sweep, median of 3 "
                                               f"({[round(s, 2) for s, _ in res['single']]} s)"},
                   "sample": f"the whole first DDM sweep ({res['n_sub']} block-preconditioned GMRES subdomain "
                             f"solves, tol 1e-10) over {res['allcore_workers']} forked single-thread workers, "
                             f"median of 3 ({[round(s, 2) for s, _ in res['allcore']]} s); oracle set-up "
                             f"{res['setup_s']:.1f}s untimed"}
        except Exception as ex:  # noqa: BLE001
            cpu = {"value": None, "unit": UNIT, "cores": None, "kind": "oracle", "sample": f"failed: {ex}"}

    if rank == 0:
        last = stats_all[-1]
        line = {
            "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": ws if ws > 1 else args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms_max / args.steps,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "f32 operator/preconditioner/inner Krylov + f64 refinement" if mode == "mixed" else "f64",
            "data": "synthetic",
            "config": {"workload": WORKLOAD_DESC, "mode": mode, "parallelism": f"replicas x{max(ws, 1)}",
                       "relax": args.relax,
                       "l2": "no flush: the per-step working set (operators, factors, Krylov bases) "
                             "exceeds the 129 MB L2", "step": "thm_assemble + thm_ddm_solve (rtol 1e-8)",
                       "timed_steps": "no per-launch instrumentation; kernel timing comes from separate "
                                      "instrumented steps after the timed region",
                       "mesh_setup_s": mesh_s},
            "time_to_1e8_s": statistics.median(tt),
            "solve": {"outer_iters": last["outer_iters"], "sweeps": last["sweeps"],
                      "inner_iters": last["inner_iters"], "max_inner_iters": last["max_inner_iters"],
                      "refine_steps": last["refine_steps"], "rel_residual": last["rel_residual"],
                      "dof_iters": last["dof_iters"]},
            "fp64": fp64,
            "full_block_variant": full,
            "roofline": roofline,
            "cpu_baseline": cpu,
            "e2e": {"value": e2e_val, "unit": UNIT, "seconds": e2e_t / max(1, args.e2e_steps),
                    "h2d_bytes_per_step": int(mu_h.nbytes),
                    "d2h_bytes_per_step": int(16 * sysg.n_dof),
                    "includes": "thm_mesh_create from host arrays + thm_assemble from host mu^-1 + "
                                "thm_ddm_solve_host"},
            "gpu_launches": int(launches),
            "clocks": clocks,
        }
        print(json.dumps(line), flush=True)
    if dist is not None:
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
