#!/usr/bin/env python3
"""Benchmark: 2D Euler P2 DG DOF-updates/s with the CSWENO limiter on one GB300.

Workload (default): the 1024 x 1024 four-quadrant Riemann problem on [0,1]^2 (2D Euler,
gamma = 1.4, P2 = 6 modes x 4 variables, FP64 state, outflow boundaries, seed 1904, run to
t = 0.25), one SSP-RK3 step = 3 x (stage, troubled-cell flags + compaction, CSWENO limiter),
replayed from the library's CUDA graph.  The timed window starts at t = 0.05 (--t-start),
reached by the plain method without timing.  DOF-updates/s = cells * modes * vars * steps /
time.

  python bench.py [--gpus N --steps K --warmup W] [--impl reference]

With N > 1 (torchrun, one rank per GPU) every rank advances its own replica of the
workload (independent problems: no collective on the data path) and the value is the sum
over ranks ("scaling": "weak").  ``--impl reference`` times the FP64 CPU oracle on the host
cores instead (bounded samples of the same workload).
"""
from __future__ import annotations

import argparse
import json
import math
import os
import statistics
import subprocess
import sys
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

from paper_1904_11147_gb300 import workloads as W  # noqa: E402

METRIC = "2D Euler P2 DG DOF-updates/s incl. CSWENO; learned vs plain indicator"
UNIT = "DOF-updates/s"
# GB300 FP64 vector peak from unit counts and clock: 2 DFMA lanes per clock per SM x 2 flops
# x 152 SMs x 2.07 GHz (MEASURED_PEAKS.json carries no FP64 figure)
FP64_PEAK_TFLOPS = 2 * 2 * 152 * 2.07e9 / 1e12


# ----------------------------------------------------------------------------- algorithmic work
def stage_flops_per_cell(dim: int, pde: int, N: int, faces_per_cell: float = 2.0) -> dict:
    """FP64 flops of one stage of Eq. (5) per cell, counted from the operations of the split
    stage with every sum in FP64 and every weight applied (FMA = 2; add, multiply, reciprocal,
    square root = 1).  This is the work the rate is quoted on; the kernels need fewer FP64
    instructions for it (sums relative to the outermost weight, the density's volume term
    without quadrature, traces in fixed point on the integer pipes).  The face pass
    (two traces, the local Lax-Friedrichs flux at the N+1 face points, the projection on the
    transverse modes) for `faces_per_cell` faces, and the cell pass (sum-factorised volume
    term over symmetric Gauss pairs, lifting, stage combination averaged over the three
    stages)."""
    assert dim == 2
    V = 1 if pde == 0 else 4
    NP = (N + 1) * (N + 2) // 2
    Q = N + 1
    pairs, mid = Q // 2, Q % 2
    even = lambda lo, hi: sum(1 for t in range(lo, hi + 1) if t % 2 == 0)
    odd = lambda lo, hi: sum(1 for t in range(lo, hi + 1) if t % 2 == 1)

    def eval_gauss():  # doubled values of sum_t e_t psi_t / psi_0 at the Q Gauss points
        per_pair = (1 + 2 * odd(3, N)) + 2 * even(2, N) + 2
        return pairs * per_pair + mid * 2 * even(2, N)

    flux = 18 if pde == 1 else 2  # one state's flux and wave speed
    # face pass, per face (traces over psi_0: the constant term needs no multiplication)
    trace = V * (sum(2 * (N - t) for t in range(N + 1)) + eval_gauss())
    llf = 2 * flux + 1 + 4 * V
    proj = V * (2 * pairs + sum(1 + 2 * (pairs - 1) + (2 if (mid and b % 2 == 0) else 0) for b in range(N + 1)))
    face = 2 * trace + Q * llf + proj
    # cell pass, per cell
    vflux = 18 if pde == 1 else 2
    if pde == 1 and N == 3:  # t_b at one x point at a time (modes in shared memory)
        tb = Q * V * sum(2 * (N - b) for b in range(N + 1))
        cols = Q * V * eval_gauss()
        per_x = 4 * pairs + 2 * N * (1 + 2 * (pairs - 1))
        per_x += 2 * sum(1 for b in range(N) for a in range(1, N - b + 1))
        per_x += 2 * sum(1 for b in range(1, N + 1) for a in range(0, N - b + 1))
        red = Q * V * per_x
    else:
        tb = 0
        for qp in range((Q + 1) // 2):
            single = mid and qp == Q // 2
            for b in range(N + 1):
                tb += V * 2 * even(2, N - b)
                if not single and N - b >= 1:
                    tb += V * (1 + 2 * odd(3, N - b) + 2)
        cols = Q * V * eval_gauss()
        red = 0
        for qx in range(Q):
            is_mid = mid and qx == Q // 2
            r = 4 * pairs  # sums and differences of f and g over the y pairs
            for b in range(N):  # x-derivative column sums and their x weights
                r += 1 + 2 * (pairs - 1) + (2 if (mid and b % 2 == 0) else 0)
                r += 2 * sum(1 for a in range(1, N - b + 1) if not (is_mid and a % 2 == 0))
            for b in range(1, N + 1):  # y-derivative column sums
                r += 1 + 2 * (pairs - 1) + (2 if (mid and b % 2 == 1) else 0)
                r += 2 * sum(1 for a in range(0, N - b + 1) if not (is_mid and a % 2 == 1))
            red += V * r
    ab = [(d - b, b) for d in range(N + 1) for b in range(d + 1)]
    # 2/h and 1/h per direction (2 divisions, 2 multiplications), the lifting coefficients
    # -psi_n(1)/h, then (2/hx) X + (2/hy) Y per mode
    combine = V * sum((3 if (a >= 1 and b >= 1) else 1) for a, b in ab if a >= 1 or b >= 1) + 4 + 2 * (N + 1)
    lift = V * (4 * (N + 1) + 4 * NP)
    rk = V * NP * (2 + 5 + 5) / 3.0
    cell = tb + cols + Q * Q * vflux + red + combine + lift + rk
    return {"face": face, "cell": cell, "total": faces_per_cell * face + cell}


def measured_peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        try:
            return json.load(open(p)), "measured"
        except Exception:
            pass
    return {}, "fallback"


# ----------------------------------------------------------------------------- clocks
class ClockSampler:
    def __init__(self, out_path=None):
        self.proc = None
        self.path = out_path

    def __enter__(self):
        q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "--query-gpu=" + q, "--format=csv,noheader,nounits",
                                          "-lms", "50", "-i", str(int(os.environ.get("LOCAL_RANK", "0")))],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except Exception:
            self.proc = None
        return self

    def __exit__(self, *a):
        self.lines = []
        if self.proc is not None:
            self.proc.terminate()
            try:
                out, _ = self.proc.communicate(timeout=5)
            except Exception:
                self.proc.kill()
                out = ""
            self.lines = [l for l in out.splitlines() if l.strip()]
            if self.path:
                with open(self.path, "w") as f:
                    f.write("\n".join(self.lines) + "\n")

    def summary(self):
        sm, mx, reasons = [], [], set()
        for l in getattr(self, "lines", []):
            parts = [p.strip() for p in l.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                mx.append(float(parts[2]))
            except ValueError:
                continue
            names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
            for n, v in zip(names, parts[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(n)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["unsampled"]}
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(mx), "reasons": sorted(reasons),
                "samples": len(sm)}


# ----------------------------------------------------------------------------- CPU oracle
def _oracle_sample(args):
    """Runs the oracle on one window of the workload (outflow edges): `adv` untimed steps
    from the initial data (the troubled fraction grows from ~10 % to ~30 % over them), then
    `steps` timed steps; returns (dofs * steps, seconds, troubled cells over the timed
    stages, cells * stages)."""
    wl_name, n, y0, x0, win, steps, dt, adv = args
    sys.path.insert(0, ROOT)
    import oracle
    w = W.euler_2d_quadrant(n, 2)
    h = 1.0 / n
    o = oracle.Mesh(2, 1, 2, win, win, box=(x0 * h, (x0 + win) * h, y0 * h, (y0 + win) * h), bc=W.BC_OUTFLOW)
    u = o.project_ic(w.ic, w.params[0])
    for _ in range(adv):
        u, _, _ = o.step(u, dt)
    t0 = time.perf_counter()
    flagged = 0
    for _ in range(steps):
        u, nf, _ = o.step(u, dt)
        flagged += nf
    return win * win * 24 * steps, time.perf_counter() - t0, flagged, 3 * steps * win * win


def cpu_oracle_rate(n, dt, win=48, steps=8, workers=None, pool=None, adv=12):
    """Oracle DOF-updates/s on the host cores: one spawn-started process per core, each on
    its own win x win window of the workload (windows straddle the discontinuities),
    advanced `adv` steps untimed before the timed ones."""
    import multiprocessing as mp
    workers = workers or (pool._processes if pool is not None else (os.cpu_count() or 1))
    rng = np.random.default_rng(0)
    jobs = []
    for i in range(workers):
        y0 = int(np.clip(n // 2 - win // 2 + rng.integers(-win, win), 0, n - win))
        x0 = int(np.clip(n // 2 - win // 2 + rng.integers(-win, win), 0, n - win))
        jobs.append(("quadrant", n, y0, x0, win, steps, dt, adv))
    t0 = time.perf_counter()
    if pool is None:
        with mp.get_context("spawn").Pool(workers) as p:
            res = p.map(_oracle_sample, jobs)
    else:
        res = pool.map(_oracle_sample, jobs)
    wall = time.perf_counter() - t0
    dof = sum(r[0] for r in res)
    busy = max(r[1] for r in res)
    frac = sum(r[2] for r in res) / max(sum(r[3] for r in res), 1)
    return dof / busy, workers, ("%d windows of %dx%d cells of the workload, %d untimed then %d timed steps "
                                 "(%.1f s wall); TVB limited %.1f %% of the cells in the timed steps"
                                 % (workers, win, win, adv, steps, wall, 100 * frac))


# ----------------------------------------------------------------------------- helpers
def dist_init():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    if ws > 1:
        import torch.distributed as dist
        backend = "nccl"
        dist.init_process_group(backend)
        return dist, rank, ws
    return None, 0, 1


def max_over_ranks(dist, x):
    """Largest value over the ranks (the job's time is the slowest rank's)."""
    if dist is None:
        return x
    import torch
    dev = "cuda" if dist.get_backend() == "nccl" else "cpu"
    t = torch.tensor([x], dtype=torch.float64, device=dev)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def aggregate_rate(units_per_rank, steps, ms_max, world):
    """Whole-job throughput of independent replicas: all ranks' units over the slowest
    rank's time."""
    return units_per_rank * steps * world / (ms_max / 1e3)


def barrier(dist):
    if dist is not None:
        dist.barrier()


def launch_ranks(n):
    """Starts n local ranks of this script (one per GPU) through torch.distributed.run on
    127.0.0.1 when no launcher did; returns the launcher's exit status."""
    import socket
    sk = socket.socket()
    sk.bind(("127.0.0.1", 0))
    port = sk.getsockname()[1]
    sk.close()
    cmd = [sys.executable, "-m", "torch.distributed.run", "--nnodes=1", "--nproc-per-node", str(n),
           "--master-addr", "127.0.0.1", "--master-port", str(port), os.path.abspath(__file__)] + sys.argv[1:]
    return subprocess.call(cmd)


def reference_arm(args):
    """The oracle on the host cores, same metric, bounded samples of the same workload."""
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return 0
    n = args.size
    w = W.euler_2d_quadrant(n, 2)
    # the same fixed time step the GPU arm uses (CFL 0.1 at the initial state's speeds)
    import oracle
    rho = [w.params[0][4 * q] for q in range(4)]
    speeds = []
    for q in range(4):
        r, u, v, p = w.params[0][4 * q: 4 * q + 4]
        c = math.sqrt(1.4 * p / r)
        speeds.append((abs(u) + c, abs(v) + c))
    ax, ay = max(s[0] for s in speeds), max(s[1] for s in speeds)
    dt = 0.1 / (ax * n + ay * n)
    del rho, oracle
    import multiprocessing as mp
    vals = []
    t0 = time.perf_counter()
    with mp.get_context("spawn").Pool(os.cpu_count() or 1) as pool:
        for i in range(args.warmup + args.steps):
            rate, cores, sample = cpu_oracle_rate(n, dt, win=48, steps=4, pool=pool)
            if i >= args.warmup:
                vals.append(rate)
    value = float(np.mean(vals))
    T = time.perf_counter() - t0
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup,
            # the time one step of the whole mesh takes at the measured rate (the oracle times
            # windows of it, not the whole mesh)
            "ms_per_step": 1e3 * n * n * 24 / value, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": w.name, "cells": n * n, "dofs": n * n * 24, "dt": dt,
                       "window": "each step: one window of the initial data per host core (the oracle "
                                 "runs the plain method only)",
                       "indicator": "tvb", "limiter": "cswenolimit", "parallelism": "replicas"},
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": cores, "kind": "oracle", "sample": sample},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
            "wall_s": T}
    print(json.dumps(line))
    return 0


# ----------------------------------------------------------------------------- main
def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--size", type=int, default=1024)
    ap.add_argument("--workload", default="quadrant",
                    choices=["quadrant", "burgers_batched", "euler_batched_p3", "double_mach"],
                    help="quadrant: 2D Euler P2 four-quadrant problem (size^2, learned vs plain); "
                         "burgers_batched: 64 2D Burgers P2 instances (64^2..512^2); "
                         "euler_batched_p3: 256 2D Euler P3 four-quadrant instances (128^2..1024^2); "
                         "double_mach: Example 11 at --dmr-size (P2, positivity scaling) run to t = 0.2")
    ap.add_argument("--dmr-size", default="960x240")
    ap.add_argument("--dmr-order", type=int, default=2)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--t-start", type=float, default=0.05,
                    help="time of the 1024^2 quadrant problem (run to 0.25) at which the timed window starts; "
                         "the plain method advances the initial data there, untimed")
    ap.add_argument("--arms", default="both", choices=["both", "plain"],
                    help="plain: time only the TVB indicator (no training; for profiling runs)")
    ap.add_argument("--clocks-out", default=None)
    ap.add_argument("--profile-window", action="store_true",
                    help="bracket every arm's timed steps with cudaProfilerStart/Stop (for "
                         "ncu --profile-from-start off)")
    ap.add_argument("--no-batched", action="store_true",
                    help="leave out the batched Burgers P2 and Euler P3 workloads the default line also times")
    ap.add_argument("--p3-steps", type=int, default=5,
                    help="timed steps of the batched Euler P3 workload in the default line (~1.6 s each)")
    ap.add_argument("--no-judge", action="store_true",
                    help="leave out the learned indicator's accuracy check (half-resolution run to the window)")
    ap.add_argument("--judge-steps", type=int, default=16)
    ap.add_argument("--train-size", type=int, default=256,
                    help="mesh side of the learned indicator's training problems (2D Euler P2)")
    ap.add_argument("--train-steps", type=int, default=320)
    ap.add_argument("--no-autotune", action="store_true",
                    help="keep the library's default launch configuration (split stage, 8 limiter blocks "
                         "per SM), e.g. for a profiler run whose timings would mislead the autotuner")
    args = ap.parse_args()
    args.warmup = max(args.warmup, 3)
    if args.gpus > 1 and "WORLD_SIZE" not in os.environ:
        return launch_ranks(args.gpus)
    if args.impl == "reference":
        return reference_arm(args)

    # the CPU-baseline pool is started (spawn) before the first GPU call
    dist, rank, world = dist_init()
    import torch
    import paper_1904_11147_gb300 as dgl

    local = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(local)
    if args.workload == "double_mach":
        return dmr_arm(args, dist, rank, world, torch, dgl)
    if args.workload != "quadrant":
        return batched_arm(args, dist, rank, world, torch, dgl)
    n = args.size
    w = W.euler_2d_quadrant(n, 2)
    st = torch.cuda.Stream()

    # learned indicator: harvested from the plain method on other seeded problems, trained
    # and calibrated with the library's kernels (untimed)
    from paper_1904_11147_gb300 import train as T
    t_train = time.perf_counter()
    net, tau, tinfo = None, 0.0, {"val_recall": None, "tol": None, "val_predicted": 0, "val_tvb_flagged": 1}
    if args.arms == "both":
        with torch.cuda.stream(st):
            # label: the limiter changes the cell's modes n >= 1 by more than 20 % of its
            # scale; threshold at 95 % recall of such cells on held-out problems; harvested
            # on 256^2 problems over 320 steps (closer to the benchmark's resolution than the
            # library's 96^2 default: recall at the benchmark window 0.59 vs 0.21)
            net, tau, tinfo = T.train_indicator(stream=st, tol=0.2, recall=0.95, n=args.train_size,
                                                steps=args.train_steps)
    st.synchronize()
    t_train = time.perf_counter() - t_train

    snapshot = []

    def make_mesh(learned):
        m = dgl.Mesh(2, W.PDE_EULER, 2, [n], [n], w.box, bc=w.bc, stream=st.cuda_stream)
        if snapshot:
            m.set_modes(snapshot[0])
        else:
            m.project_ic(w.ic, w.params[0])
        if learned:
            m.set_indicator(net, tau)
        return m

    mesh = make_mesh(False)
    ws = mesh.max_wavespeed()[0]
    dt = 0.1 / (ws[0] * n + ws[1] * n)
    # the timed window starts at t_start: the plain method advances the initial data there
    # (untimed).  The fraction of troubled cells grows with time (TVB flags ~4 % of the
    # cells in the first steps, ~34 % at t = 0.05, ~67 % at t = 0.25), so a window at
    # t = 0 would not represent the run.
    n_adv = 2 * int(round(args.t_start / dt / 2))
    t_adv = time.perf_counter()
    with torch.cuda.stream(st):
        for _ in range(n_adv):
            mesh.step(dt)
    st.synchronize()
    t_adv = time.perf_counter() - t_adv
    # stage form and limiter grid, measured here on the window's state (untimed)
    tune = (0, 8, 0) if args.no_autotune else mesh.autotune(dt)
    dofs = mesh.size
    u0 = torch.empty(dofs, dtype=torch.float64, device="cuda")
    mesh.get_modes(u0)
    snapshot.append(u0)
    torch.cuda.synchronize()

    def timed_arm(m, ind, clk_path):
        for _ in range(args.warmup):
            m.step(dt, ind)
        st.synchronize()
        m.flag_statistics(reset=True)
        barrier(dist)
        torch.cuda.synchronize()
        l0 = m.launches
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        with ClockSampler(clk_path) as clk:
            if args.profile_window:
                torch.cuda.profiler.start()
            e0.record(st)
            for _ in range(args.steps):
                m.step(dt, ind)
            e1.record(st)
            e1.synchronize()
            if args.profile_window:
                torch.cuda.profiler.stop()
        ms_ = e0.elapsed_time(e1)
        launches_ = m.launches - l0
        barrier(dist)
        torch.cuda.synchronize()
        ms_ = max_over_ranks(dist, ms_)
        tvbf, limited, passes = m.flag_statistics()
        return ms_, launches_, clk, tvbf / max(passes, 1) / (n * n), limited / max(passes, 1) / (n * n)

    with torch.cuda.stream(st):
        if args.arms == "both":
            ms_plain, _, clk_plain, tvb_frac, lim_plain = timed_arm(mesh, dgl.IND_TVB, None)
            lmesh = make_mesh(True)
            ind_main = dgl.IND_MLP
            ms, launches, clk, _, lim_learned = timed_arm(lmesh, ind_main, args.clocks_out)
            fallbacks, failures = lmesh.positivity_report()
        else:
            ms_plain, launches, clk_plain, tvb_frac, lim_plain = timed_arm(mesh, dgl.IND_TVB, args.clocks_out)
            lmesh, ind_main, ms, clk, lim_learned, fallbacks, failures = mesh, dgl.IND_TVB, ms_plain, clk_plain, lim_plain, 0, 0
        value = aggregate_rate(dofs, args.steps, ms, world)
        value_plain = aggregate_rate(dofs, args.steps, ms_plain, world)
        # the paper's own indicator (KXRCF) on the same workload, for comparison
        kx = pw = None
        if args.arms == "both":
            kmesh = make_mesh(False)
            ms_kx, _, _, _, lim_kx = timed_arm(kmesh, dgl.IND_KXRCF, None)
            kx = {"value": aggregate_rate(dofs, args.steps, ms_kx, world), "ms_per_step": ms_kx / args.steps,
                  "limited_fraction": lim_kx}
            kmesh.close()
            # the parent WENO limiter (full-width stencil) on the TVB flags, for comparison
            pmesh = make_mesh(False)
            pmesh.set_limiter(dgl.LIM_PARENT)
            ms_pw, _, _, _, lim_pw = timed_arm(pmesh, dgl.IND_TVB, None)
            pw = {"value": aggregate_rate(dofs, args.steps, ms_pw, world), "ms_per_step": ms_pw / args.steps,
                  "limited_fraction": lim_pw}
            pmesh.close()

        # ------------------------------------------------------------ dominant kernel alone
        mesh.set_modes(u0)
        mesh.step(dt)
        st.synchronize()
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        kst = []
        for _ in range(max(3, min(args.steps, 10))):
            for s in (1, 2, 3):
                ev[0].record(st)
                mesh.rk_stage(s, dt)
                ev[1].record(st)
                ev[1].synchronize()
                kst.append(ev[0].elapsed_time(ev[1]))
        stage_ms = float(np.mean(kst))

        # ------------------------------------------------------------ end to end (host buffers)
        host_in = torch.empty(dofs, dtype=torch.float64, pin_memory=True)
        host_out = torch.empty(dofs, dtype=torch.float64, pin_memory=True)
        host_in.copy_(u0.cpu())
        for _ in range(2):
            lmesh.set_modes(host_in)
            lmesh.step(dt, ind_main)
            lmesh.get_modes(host_out)
        barrier(dist)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        e2 = torch.cuda.Event(enable_timing=True)
        e3 = torch.cuda.Event(enable_timing=True)
        e2.record(st)
        k_e2e = max(3, args.steps // 2)
        for _ in range(k_e2e):
            lmesh.set_modes(host_in)
            lmesh.step(dt, ind_main)
            lmesh.get_modes(host_out)
        e3.record(st)
        e3.synchronize()
        e2e_ms = max(e2.elapsed_time(e3), (time.perf_counter() - t0) * 1e3)
        e2e_ms = max_over_ranks(dist, e2e_ms)
    e2e_value = dofs * k_e2e * world / (e2e_ms / 1e3)
    flagged = lim_learned

    # ------------------------------------------------------------ accuracy of the learned run (untimed)
    judge = missed = None
    if args.arms == "both" and rank == 0 and not args.no_judge:
        with torch.cuda.stream(st):
            judge = judge_learned(dgl, torch, st, w, n, dt, n_adv, u0, mesh, net, tau, args.judge_steps)
            missed = missed_shocks(dgl, torch, st, lmesh, u0, dt, tinfo["tol"] or 0.2)
        st.synchronize()
    mesh.close()
    lmesh.close()
    del u0, snapshot[:]
    torch.cuda.synchronize()
    torch.cuda.empty_cache()

    # ------------------------------------------------------------ batched workloads
    batched = {}
    if not args.no_batched:
        batched["burgers_batched"] = run_batched("burgers_batched", args, dist, rank, world, torch, dgl,
                                                 args.steps, learned=False)
        batched["euler_batched_p3"] = run_batched("euler_batched_p3", args, dist, rank, world, torch, dgl,
                                                  min(args.steps, args.p3_steps), learned=args.arms == "both")

    if rank != 0:
        if dist is not None:
            dist.destroy_process_group()
        return 0
    peaks, src = measured_peaks()
    fp64_peak = float(peaks.get("fp64_tflops", FP64_PEAK_TFLOPS))
    peak_note = ("FP64 from unit counts and clock: 2 DFMA/clk/SM x 2 flop x 152 SMs x 2.07 GHz = %.3f TFLOP/s "
                 "(an FMA microbenchmark on this pool reached 1.20)" % FP64_PEAK_TFLOPS)
    fl = stage_flops_per_cell(2, 1, 2, faces_per_cell=((n + 1) * n * 2) / (n * n))
    flops_cell = fl["total"]
    achieved = flops_cell * n * n / (stage_ms / 1e3) / 1e12
    traffic = None
    tpath = os.path.join(ROOT, "profiles", "stage_traffic.json")
    if os.path.exists(tpath):
        try:
            tr = json.load(open(tpath))
            if tr.get("kernel_hash") == kernel_hash():
                traffic = tr["bytes_per_launch"]
        except Exception:
            traffic = None
    cpu_line = None
    if world == 1 and not args.no_cpu_baseline:
        rate, cores, sample = cpu_oracle_rate(n, dt, win=64, steps=24)
        cpu_line = {"value": rate, "unit": UNIT, "cores": cores, "kind": "oracle", "sample": sample}
    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": ms / args.steps, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": w.name, "cells": n * n, "dofs": dofs, "dt": dt,
                   "window": "%d steps after %d warm-up steps from t = %.4g (%d untimed plain steps, %.0f s)"
                             % (args.steps, args.warmup, n_adv * dt, n_adv, t_adv),
                   "indicator": "learned (TVB-gated MLP)" if args.arms == "both" else "tvb",
                   "training": "%d^2 four-quadrant problems, %d steps, label tolerance 0.2, 95 %% recall"
                               % (args.train_size, args.train_steps),
                   "tvb_M": 0.01, "limiter": "cswenolimit", "graph": True,
                   "autotuned": {"stage_form": "split" if tune[0] == 0 else "fused", "stage_tile_rows": tune[0],
                                 "limiter_blocks_per_sm": tune[1], "stage_persistent_queue": bool(tune[2])},
                   "l2": "state (3 x %.0f MB) larger than L2" % (dofs * 8 / 1e6),
                   "parallelism": "replicas" if world > 1 else "single"},
        "learned": {"value": value, "ms_per_step": ms / args.steps, "limited_fraction": lim_learned, "tau": tau,
                    "positivity_fallbacks": fallbacks, "positivity_failures": failures,
                    "train_s": t_train, "val_recall": tinfo["val_recall"], "label_tol": tinfo["tol"],
                    "val_kept_of_tvb": tinfo["val_predicted"] / max(tinfo["val_tvb_flagged"], 1)},
        "plain": {"value": value_plain, "ms_per_step": ms_plain / args.steps, "limited_fraction": lim_plain,
                  "tvb_flagged_fraction": tvb_frac},
        "learned_over_plain": value / value_plain,
        "judge": judge,
        "missed_shocks": missed,
        "kxrcf": kx,
        "parent_weno": pw,
        "roofline": {"bound": "alu", "kernel": "k_face2 + k_cell2 <Euler,P2> (one stage)", "achieved": achieved,
                     "peak": fp64_peak,
                     "unit": "TFLOP/s", "frac": achieved / fp64_peak, "traffic": traffic,
                     "flops_per_cell": flops_cell, "flops_per_face": fl["face"], "flops_cell_pass": fl["cell"],
                     "launch_ms": stage_ms, "peak_source": src if "fp64_tflops" in peaks else peak_note},
        "hbm_fraction": dofs * 64 / (ms / args.steps / 1e3) / 1e9 / float(peaks.get("hbm_gbs", 6800.0)),
        "hbm_peak_source": "measured" if "hbm_gbs" in peaks else "fallback 6800 GB/s",
        "cpu_baseline": cpu_line,
        "e2e": {"value": e2e_value, "unit": UNIT, "h2d_bytes_per_step": dofs * 8, "d2h_bytes_per_step": dofs * 8},
        "gpu_launches": launches,
        "clocks": clk.summary(),
        "clocks_plain_arm": clk_plain.summary(),
    }
    line.update(batched)
    print(json.dumps(line))
    if dist is not None:
        dist.destroy_process_group()
    return 0


def partition_instances(cells, world):
    """Splits the instances of a batch over `world` ranks: largest first, each to the rank
    with the fewest cells so far (ties to the lower rank).  Every instance lands on exactly
    one rank, and a rank's load exceeds the mean load by less than the largest instance.
    Returns one sorted index list per rank."""
    order = sorted(range(len(cells)), key=lambda i: (-cells[i], i))
    load = [0] * world
    parts = [[] for _ in range(world)]
    for i in order:
        r = min(range(world), key=lambda k: (load[k], k))
        parts[r].append(i)
        load[r] += cells[i]
    return [sorted(p) for p in parts]


def subset_workload(w, idx):
    """The instances idx of a batched workload, as a workload of its own."""
    import dataclasses
    return dataclasses.replace(w, nx=[w.nx[i] for i in idx], ny=[w.ny[i] for i in idx],
                               box=[w.box[i] for i in idx], params=[w.params[i] for i in idx])


def sum_over_ranks(dist, x):
    if dist is None:
        return x
    import torch
    dev = "cuda" if dist.get_backend() == "nccl" else "cpu"
    t = torch.tensor([x], dtype=torch.float64, device=dev)
    dist.all_reduce(t, op=dist.ReduceOp.SUM)
    return float(t.item())


def run_batched(which, args, dist, rank, world, torch, dgl, steps, clocks_out=None, learned=True):
    """Batched workloads: many uneven instances in one mesh, per-instance time steps (CFL
    0.1), steps replayed from the CUDA graph; with several ranks the instances are split
    over them (partition_instances) and each rank advances its own share, no collective on
    the data path.  Burgers: the plain TVB indicator, time steps fixed at the initial state.
    Euler P3: the learned indicator (trained here on P3 four-quadrant problems with the
    label tolerance 0.2 and 95 % recall, untimed) with its plain-indicator fallback, next to
    the plain TVB arm; both with the positivity-preserving scaling after every stage and
    each step's per-instance time step from the wave speeds at the scaling's check points
    (random P3 four-quadrant problems lose positivity without both); that update is timed.
    Returns a dict for the JSON line (rank 0) with the job's DOF count."""
    euler = which != "burgers_batched"
    w_all = W.euler_2d_batched() if euler else W.burgers_2d_batched()
    mine = partition_instances([a * b for a, b in zip(w_all.nx, w_all.ny)], world)[rank]
    if not mine:
        raise RuntimeError("more ranks (%d) than instances (%d)" % (world, w_all.n_inst))
    w = subset_workload(w_all, mine)
    st = torch.cuda.Stream()
    net, tau, tinfo, t_train = None, 0.0, {}, 0.0
    if euler and learned:
        from paper_1904_11147_gb300 import train as T
        t0 = time.perf_counter()
        with torch.cuda.stream(st):
            net, tau, tinfo = T.train_indicator(N=w.N, positivity=True, stream=st, tol=0.2, recall=0.95)
        st.synchronize()
        t_train = time.perf_counter() - t0

    def make_mesh():
        m = dgl.Mesh(2, w.pde, w.N, w.nx, w.ny, w.box, bc=w.bc, stream=st.cuda_stream)
        m.project_ic(w.ic, w.params)
        if euler:
            m.set_positivity(True)
        return m

    m = make_mesh()
    ws = m.max_wavespeed()
    hx = np.array([(b[1] - b[0]) / nx for b, nx in zip(w.box, w.nx)])
    hy = np.array([(b[3] - b[2]) / ny for b, ny in zip(w.box, w.ny)])
    dts = 0.1 / (ws[:, 0] / hx + ws[:, 1] / hy)
    m.set_dt(dts)
    tune = (0, 8, 0) if args.no_autotune else m.autotune(float(dts.min()))
    m.set_dt(dts)
    dofs = m.size
    dofs_job = sum_over_ranks(dist, float(dofs))

    def one_step(mm, ind):
        if euler:  # CFL 0.1 on the check-point wave speeds of the step's starting state
            sp = mm.max_wavespeed(points=True)
            mm.set_dt(0.1 / np.maximum(sp[:, 0] / hx + sp[:, 1] / hy, 1e-300))
        mm.step(0.0, ind)

    def timed(mm, ind, clk_path):
        with torch.cuda.stream(st):
            for _ in range(args.warmup):
                one_step(mm, ind)
            st.synchronize()
            mm.flag_statistics(reset=True)
            mm.positivity_counts(reset=True)
            barrier(dist)
            torch.cuda.synchronize()
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            l0 = mm.launches
            with ClockSampler(clk_path) as clk:
                t0 = time.perf_counter()
                e0.record(st)
                for _ in range(steps):
                    one_step(mm, ind)
                e1.record(st)
                e1.synchronize()
                wall = (time.perf_counter() - t0) * 1e3
            ms_ = max_over_ranks(dist, max(e0.elapsed_time(e1), wall if euler else 0.0))
            launches_ = mm.launches - l0
        tvbf, limited, passes = mm.flag_statistics()
        # instances whose state is no longer finite (checked on the device, per instance)
        u = torch.empty(dofs, dtype=torch.float64, device="cuda")
        mm.get_modes(u)
        per = dofs // w.cells
        bad, off = 0, 0
        for nx, ny in zip(w.nx, w.ny):
            bad += not bool(torch.isfinite(u[off * per:(off + nx * ny) * per]).all())
            off += nx * ny
        del u
        info = {"value": dofs_job * steps / (ms_ / 1e3), "ms_per_step": ms_ / steps,
                "limited_fraction": sum_over_ranks(dist, limited / max(passes, 1)) / w_all.cells,
                "tvb_flagged_fraction": sum_over_ranks(dist, tvbf / max(passes, 1)) / w_all.cells,
                "nonfinite_instances": int(sum_over_ranks(dist, bad)), "gpu_launches": launches_,
                "clocks": clk.summary()}
        if euler:
            a, b = mm.positivity_counts()
            info["positivity_scaled_cells"], info["inadmissible_means"] = int(sum_over_ranks(dist, a)), \
                int(sum_over_ranks(dist, b))
        return ms_, info

    ms_plain, plain = timed(m, dgl.IND_TVB, None if net is not None else clocks_out)
    out = {"workload": w_all.name, "instances": w_all.n_inst, "cells": w_all.cells, "dofs": dofs_job,
           "steps": steps, "warmup": args.warmup,
           "indicator": "learned (TVB-gated MLP)" if net is not None else "tvb",
           "positivity_scaling": euler,
           "time_step": "per step from check-point wave speeds (CFL 0.1), timed" if euler
           else "fixed at the initial state (CFL 0.1)",
           "window": "the first steps after t = 0",
           "autotuned": {"stage_form": "split" if tune[0] == 0 else "fused", "stage_tile_rows": tune[0],
                         "limiter_blocks_per_sm": tune[1], "stage_persistent_queue": bool(tune[2])},
           "l2": "state (3 x %.0f MB) larger than L2" % (dofs * 8 / 1e6),
           "parallelism": ("instances split over %d ranks" % world) if world > 1 else "single",
           "scaling": "strong", "plain": plain, "value": plain["value"], "ms_per_step": plain["ms_per_step"],
           "gpu_launches": plain["gpu_launches"], "clocks": plain["clocks"]}
    if net is not None:
        m.close()  # the full batch is ~20 GB per state copy: one mesh at a time
        torch.cuda.synchronize()
        lm = make_mesh()
        lm.set_dt(dts)
        lm.set_indicator(net, tau)
        ms, info = timed(lm, dgl.IND_MLP, clocks_out)
        fb, fails = lm.positivity_report()
        info["positivity_fallbacks"], info["positivity_failures"] = int(sum_over_ranks(dist, fb)), \
            int(sum_over_ranks(dist, fails))
        info.update({"tau": tau, "train_s": t_train, "val_recall": tinfo.get("val_recall"),
                     "label_tol": tinfo.get("tol"),
                     "val_kept_of_tvb": tinfo.get("val_predicted", 0) / max(tinfo.get("val_tvb_flagged", 1), 1)})
        lm.close()
        out.update({"learned": info, "learned_over_plain": info["value"] / plain["value"], "value": info["value"],
                    "ms_per_step": info["ms_per_step"], "gpu_launches": info["gpu_launches"],
                    "clocks": info["clocks"]})
    else:
        m.close()
    torch.cuda.synchronize()
    return out


def batched_arm(args, dist, rank, world, torch, dgl):
    """--workload burgers_batched / euler_batched_p3: one JSON line for that workload."""
    r = run_batched(args.workload, args, dist, rank, world, torch, dgl, args.steps, args.clocks_out,
                    learned=args.arms == "both")
    if rank != 0:
        return 0
    cfg = {k: r[k] for k in ("workload", "instances", "cells", "dofs", "indicator", "positivity_scaling",
                             "time_step", "window", "autotuned", "l2", "parallelism")}
    cfg.update({"limiter": "cswenolimit", "graph": True, "per_instance_dt": True})
    line = {"metric": METRIC, "value": r["value"], "unit": UNIT, "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": r["ms_per_step"], "higher_is_better": True, "scaling": "strong",
            "vs_baseline": None, "dtype": "f64", "data": "synthetic", "config": cfg, "plain": r["plain"],
            "gpu_launches": r["gpu_launches"], "clocks": r["clocks"]}
    if "learned" in r:
        line["learned"] = r["learned"]
        line["learned_over_plain"] = r["learned_over_plain"]
    print(json.dumps(line))
    return 0


def judge_learned(dgl, torch, st, w, n, dt, n_adv, u0, fine, net, tau, J):
    """The learned indicator's accuracy at the benchmark's window, at half resolution: the
    (n/2)^2 problem of the same seed runs the plain method to the window's start (n_adv / 2
    steps of 2 dt), then J more steps with the plain and with the learned indicator; the
    reference is the benchmark's own n^2 plain run from the window's start (u0) over 2 J
    steps of dt, averaged onto the coarse cells.  Returns the density L1 errors (mean
    absolute error of the cell means) and their ratio."""
    nc = n // 2
    cm = dgl.Mesh(2, W.PDE_EULER, 2, [nc], [nc], w.box, bc=w.bc, stream=st.cuda_stream)
    cm.project_ic(w.ic, w.params[0])
    dtc = 2.0 * dt
    for _ in range(n_adv // 2):
        cm.step(dtc)
    uc0 = torch.empty(cm.size, dtype=torch.float64, device="cuda")
    cm.get_modes(uc0)

    def rho_means(m, cells):
        u = torch.empty(m.size, dtype=torch.float64, device="cuda")
        m.get_modes(u)
        return (u.view(cells, 4, 6)[:, 0, 0] * 0.5).double()

    for _ in range(J):
        cm.step(dtc)
    r_plain = rho_means(cm, nc * nc)
    cm.set_modes(uc0)
    cm.set_indicator(net, tau)
    cm.flag_statistics(reset=True)
    for _ in range(J):
        cm.step(dtc, dgl.IND_MLP)
    r_learned = rho_means(cm, nc * nc)
    tvbf, limited, passes = cm.flag_statistics()
    fb, fails = cm.positivity_report()
    cm.close()
    fine.set_modes(u0)
    for _ in range(2 * J):
        fine.step(dt)
    rf = rho_means(fine, n * n).view(n, n)
    ref = 0.25 * (rf[0::2, 0::2] + rf[1::2, 0::2] + rf[0::2, 1::2] + rf[1::2, 1::2]).reshape(-1)
    e_plain = float((r_plain - ref).abs().mean())
    e_learned = float((r_learned - ref).abs().mean())
    return {"l1_rho_learned": e_learned, "l1_rho_plain": e_plain, "l1_rho_vs_plain": e_learned / e_plain,
            "coarse": "%dx%d" % (nc, nc), "reference": "%dx%d plain (the benchmark mesh)" % (n, n),
            "steps": J, "t_end": (n_adv + 2 * J) * dt, "coarse_limited_fraction": limited / max(passes, 1) / nc ** 2,
            "coarse_tvb_flagged_fraction": tvbf / max(passes, 1) / nc ** 2, "coarse_positivity_fallbacks": fb,
            "coarse_positivity_failures": fails}


def missed_shocks(dgl, torch, st, lm, u0, dt, tol, samples=4, every=5):
    """Cells the network skips although the limiter would change them by more than the
    label tolerance (relative change of the modes n >= 1, the training label), on the
    benchmark mesh: from the window's start, every `every` learned steps the first stage
    of the next step is flagged by the learned indicator and harvested (TVB flags and the
    limiter's change); the state then resumes unchanged."""
    n = lm.cells
    F = dgl.n_features(2, W.PDE_EULER, 2)
    X = torch.empty(n, F, dtype=torch.float32, device="cuda")
    fl = torch.empty(n, dtype=torch.uint8, device="cuda")
    ch = torch.empty(n, dtype=torch.float32, device="cuda")
    saved = torch.empty(lm.size, dtype=torch.float64, device="cuda")
    lm.set_modes(u0)
    missed = labelled = kept_total = tvb_total = 0
    for _ in range(samples):
        for _ in range(every):
            lm.step(dt, dgl.IND_MLP)
        lm.get_modes(saved)
        lm.rk_stage(1, dt)
        kept, _, _ = lm.flag_cells(dgl.IND_MLP, 0.01, want=True)
        lm.harvest(X, fl, ch)
        tvb = fl.cpu().numpy() == 1
        lab = tvb & (ch.cpu().numpy() > tol)
        missed += int((lab & (kept == 0)).sum())
        labelled += int(lab.sum())
        kept_total += int(kept.sum())
        tvb_total += int(tvb.sum())
        lm.set_modes(saved)
    return {"cells": missed, "labelled": labelled, "recall": 1.0 - missed / max(labelled, 1), "label_tol": tol,
            "kept": kept_total, "tvb_flagged": tvb_total, "samples": samples,
            "how": "first stage after every %d learned steps from the window's start" % every}


def dmr_arm(args, dist, rank, world, torch, dgl):
    """Example 11, double Mach reflection: the whole run to t = 0.2 (TVB indicator, CSWENO,
    positivity-preserving scaling after every stage; each step's time step from the
    check-point wave speeds at CFL 0.1, as Zhang and Shu's condition asks), timed with CUDA
    events around the whole loop including the time-step updates.  With several ranks every
    rank runs its own replica."""
    nx, ny = (int(v) for v in args.dmr_size.split("x"))
    N = args.dmr_order
    w = W.double_mach(nx, ny, N)
    st = torch.cuda.Stream()
    g = dgl.Mesh(2, W.PDE_EULER, N, [nx], [ny], w.box, bc=W.BC_DMR, stream=st.cuda_stream)
    g.set_boundary_data(w.params[0])
    g.project_ic(W.IC_DMR, [w.params[0]])
    g.positivity_limit()  # the projected oblique shock has non-admissible points; the scaling fixes them
    g.set_positivity(True)
    h = 4.0 / nx
    torch.cuda.synchronize()
    barrier(dist)
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    t, steps = 0.0, 0
    l0 = g.launches
    with torch.cuda.stream(st), ClockSampler(args.clocks_out) as clk:
        g.flag_statistics(reset=True)
        t0 = time.perf_counter()
        e0.record(st)
        while t < w.t_end - 1e-12:
            sp = g.max_wavespeed(points=True)[0]
            dt = min(0.1 / (sp[0] / h + sp[1] / h), w.t_end - t)
            g.step(dt)
            t += dt
            steps += 1
        e1.record(st)
        e1.synchronize()
        wall = time.perf_counter() - t0
    ms = max_over_ranks(dist, max(e0.elapsed_time(e1), wall * 1e3))
    tvbf, limited, passes = g.flag_statistics()
    changed, bad = g.positivity_counts()
    u = g.get_modes()
    rho = u[:, 0, 0] * 0.5
    if rank != 0:
        return 0
    dofs = g.size
    value = dofs * steps * world / (ms / 1e3)
    line = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": steps, "warmup": 0,
            "ms_per_step": ms / steps, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "f64", "data": "synthetic",
            "config": {"workload": w.name, "cells": nx * ny, "dofs": dofs, "t_end": w.t_end, "indicator": "tvb",
                       "limiter": "cswenolimit", "positivity_scaling": True,
                       "time_step": "per step from check-point wave speeds (CFL 0.1), timed", "graph": True,
                       "parallelism": "replicas" if world > 1 else "single"},
            "limited_fraction": limited / max(passes, 1) / (nx * ny), "positivity_scaled_cells": changed,
            "inadmissible_means": bad, "finite": bool(np.isfinite(u).all()),
            "density_range": [float(rho.min()), float(rho.max())], "gpu_launches": g.launches - l0,
            "clocks": clk.summary()}
    print(json.dumps(line))
    return 0


def kernel_hash():
    import hashlib
    h = hashlib.sha1()
    for f in ("dg_stage2.cu", "dg_weno.cuh", "dg_common.cuh", "dg_shared.cuh"):
        h.update(open(os.path.join(ROOT, "paper_1904_11147_gb300", "csrc", f), "rb").read())
    return h.hexdigest()[:12]


if __name__ == "__main__":
    sys.exit(main())
