#!/usr/bin/env python
"""Benchmark of the FP64 BSSN RK4 hot path on one GB300 (or N replicas).

Metric: FP64 point-updates per second, counted as interior points x RK4
substeps (4 per step) x steps, summed over ranks.  A "step" is one classic
RK4 step of the whole hot path (RHS + dissipation + radiation and parity
boundary conditions + det enforcement, fused RK update) over the workload;
the Hamiltonian constraint is evaluated every `h_every` steps as the
workload prescribes.

Default workload: head-on Brill-Lindquist binary (bare masses 0.5+0.5 at
z = +-0.5), SinhCylindrical (rho_max = z_max = 300, w = 0.2), 256x2x512
interior points, 2000 RK4 steps at CFL 0.5, H every 100 steps.  Inputs are
synthetic closed-form initial data generated on the GPU.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]

N > 1 runs under torch.distributed.run, one independent replica per GPU
(the simulations do not exchange data: weak scaling, no collective on the
data path).  --impl reference times the CPU oracle (plain C, OpenMP over the
host cores) on full RK4 steps of the same workload (a bounded number of them).

At one GPU the default line also carries the two modes against plain
one-run-per-launch on the same GPU, each with its own clock record:
  "batched": the batched workload's seeded runs (64 head-on binaries of
    N_rho 64..256; 100 of its 500 steps each), one nr_batch against one grid at
    a time, final states compared bitwise;
  "served": the served workload's seeded Poisson stream (16 requests of
    1e5..4e6 points, to t = 2M at 80 arrivals per minute, which overloads the
    GPU as the configured 64 requests to t = 50M at 20 per minute do), the
    SRPT server against a plain FIFO queue of single-grid runs, p50/p99/mean
    time to completion of both, final states compared by digest.
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

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

from paper_2505_00097_gb300 import workloads as W  # noqa: E402

METRIC = "BSSN FP64 point-updates/s (RK4 substeps)"
UNIT = "point-updates/s"

# FP64 operations (FMA = 2) per interior point of one RHS evaluation (nr_rhs: the k_d1 pre-pass and k_rhs) that the
# compiled kernels issue, by workload (the kernel variant it runs): (DADD + DMUL + 2 DFMA) / interior points in one
# ncu capture of that workload's nr_rhs.  This is the work of the FP64 pipe; the advection + dissipation sums and
# most first and mixed differences run on the integer pipe and are not in it.  Head-on 256x2x512: k_rhs 162 / 294 / 701,
# k_d1 10.1 / 0 / 5.0; 8th order: 210 / 315 / 748, 20.3 / 5.1 / 15.2.  Large 3D, counted on 96x48x96: k_rhs 228 / 375 / 993
# and 293 / 409 / 1059; k_d1 takes five of eleven differences in FP64, 3 instructions (4 FLOP) or 8 (11) each, for
# 22.46 and 22.93 stored differences per point at 384x192x384.
F_PIPE = {"headon": 1878.2, "headon8": 2076.9, "large3d": 2629.8, "large3d8": 2934.7}
# F_PIPE over twice those instructions: the fraction of the FLOP peak that a fully busy FP64 pipe reaches with this mix (a
# DADD or DMUL takes an FMA's issue slot for 1 FLOP)
PIPE_CEILING = {"headon": 0.8012, "headon8": 0.7905, "large3d": 0.8084, "large3d8": 0.7956}
# The operations of the algorithm as the point code's source has them (add + mul + div + 2 fma, a host census that a
# test recomputes), with the first and mixed differences counted as FP64 sums and the advection + dissipation
# sums not counted: a rate of useful work, part of which is not the FP64 pipe's
F_ALG = {"headon": 2071.3, "large3d": 2963.8, "headon8": 2513.9, "large3d8": 3749.2}
# the same without the k_d1 pre-pass
KERNEL_CENSUS = {"headon": 2027, "headon8": 2391, "large3d": 2874, "large3d8": 3497}
# F_ALG over twice its operations (k_d1 + k_rhs)
MIX_CEILING = {"headon": 0.7827, "headon8": 0.7667, "large3d": 0.7923, "large3d8": 0.7710}
# DRAM bytes (read + write) of the k_d1 and k_rhs launches of one nr_rhs in that capture; for the large 3D grids the
# capture's bytes per interior point at 96x48x96 (6208.0 and 6770.5, mostly register-spill lines)
# times the 28,311,552 points of the full grid
TRAFFIC = {"headon": 24031744 + 87040 + 307848704 + 731901184,
           "headon8": 24973824 + 117248 + 328414464 + 809833216,
           "large3d": round(6208.0 * 28311552), "large3d8": round(6770.5 * 28311552)}
# FP64 operations (add + mul + div) per interior point of one RHS evaluation as the oracle's counting
# build counts them: the plain coordinate-basis evaluation of the same discretisation with generic index
# loops and the reference metric evaluated at every point -- the work of the method evaluated plainly.
# Achieved against it (frac_method) can exceed 1: the kernels compute the same discrete right-hand side
# with about a tenth of those operations
F_METHOD = {"headon": 28967, "headon8": 49631, "large3d": 28970, "large3d8": 49634}
# The diagnostics per interior point of one call, by workload: what the FP64 pipe executes, from an ncu capture of those
# kernels on the head-on state (k_ham 100 / 214 / 458 DADD / DMUL / DFMA, k_mom 26 / 144 / 220, k_psi4 460 / 434 / 1016);
# absent: not captured
DIAG_PIPE = {"headon": {"hamiltonian": 1230.0, "momentum": 610.0, "psi4": 2926.0}}
# the operations of the algorithm: the constraints' point code by a host census that a test recomputes (FMA = 2, one
# division, the square root of |M| not counted; their first and mixed differences counted as FP64 sums, which the
# kernels take on the integer pipe), psi4 as captured
DIAG_FLOPS = {"headon": {"hamiltonian": 1767.0, "momentum": 737.0, "psi4": 2926.0}}
# the census alone
DIAG_CENSUS = {"headon": {"hamiltonian": 1767, "momentum": 737}}
# psi4 modes on the workload's extraction sphere: l <= 8, Gauss-Legendre x uniform nodes
PSI4_LMAX, PSI4_NTHETA, PSI4_NPHI = 8, 24, 48
# FP64 pipe of one SM: 2 DFMA per clock (ncu peak_sustained of
# sm__sass_thread_inst_executed_op_dfma_pred_on), i.e. 4 FLOP per clock
FP64_FLOP_PER_CLK_SM = 4.0
# algorithmic DRAM bytes per interior point of one RHS evaluation (the nr_rhs the roofline times):
# the 24 gridfunctions read once and the 24 right-hand sides written once
B_ALG_RHS = 2 * 24 * 8


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=2000)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--workload", choices=["headon", "headon8", "single_puncture", "large3d", "large3d8", "batch",
                                           "served", "part"],
                    default="headon")
    ap.add_argument("--batch-runs", type=int, default=64)
    ap.add_argument("--parts", default="1,1,4",
                    help="--workload part: partitions per axis of the head-on grid (the chare decomposition)")
    ap.add_argument("--batch-steps", type=int, default=100,
                    help="RK4 steps per run of the batched comparison in the default line (500 in the workload)")
    ap.add_argument("--no-batched", action="store_true", help="skip the batched-vs-plain comparison")
    ap.add_argument("--no-served", action="store_true", help="skip the served-vs-plain comparison")
    ap.add_argument("--line-served-requests", type=int, default=16,
                    help="requests of the served-vs-plain comparison in the default line")
    ap.add_argument("--served-requests", type=int, default=24)
    ap.add_argument("--served-tfinal", type=float, default=2.0)
    ap.add_argument("--served-rate", type=float, default=80.0,
                    help="mean arrivals per minute of the served stream (80 at t_final 2M overloads the GPU as the "
                         "served configuration's 20 per minute at 50M does)")
    ap.add_argument("--served-policy", choices=("srpt", "fifo"), default="srpt")
    ap.add_argument("--served-arms", default="",
                    help="comma list of server arms of --workload served among srpt, fifo, srpt_cap (default: the "
                         "policy and the other one); the plain queue always runs")
    ap.add_argument("--served-starve-s", type=float, default=0.0,
                    help="starvation cap of the srpt_cap arm, seconds")
    ap.add_argument("--served-cap", type=int, default=1000000,
                    help="interior points advanced together by the served arm (0: no cap)")
    ap.add_argument("--profile", choices=("rhs", "diagnostics"), default=None,
                    help="for profiler captures: one nr_rhs (k_d1 + k_rhs) of the workload's initial state, or one "
                         "call each of the constraint and psi4 diagnostics after 4 steps; no timing, no JSON line")
    ap.add_argument("--profile-grid", default="",
                    help="with --profile: interior points as N0,N1,N2 instead of the workload's (a smaller grid of "
                         "the same kernel)")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-diagnostics", action="store_true")
    ap.add_argument("--diag-reps", type=int, default=10)
    ap.add_argument("--cpu-seconds", type=float, default=15.0)
    return ap.parse_args()


def workload(name: str) -> dict:
    return {"headon": W.config_headon, "single_puncture": W.config_single_puncture,
            "large3d": W.config_large3d, "headon8": W.config_headon8, "large3d8": W.config_large3d8}[name]()


def config_of(spec: dict, extra: dict | None = None) -> dict:
    c = {
        "workload": spec["name"],
        "coords": ["SinhSpherical", "SinhCylindrical", "Spherical"][spec["coords"]],
        "grid_interior": list(spec["N"]),
        "ghost_zones": spec["NG"],
        "steps_in_config": spec["steps"],
        "h_every": spec["h_every"],
        "fd_order": 2 * (spec["NG"] - 1),
        "ko_sigma": spec["ko_sigma"] if not isinstance(spec["ko_sigma"], (list, tuple)) or len(set(spec["ko_sigma"])) > 2
        else {"metric": spec["ko_sigma"][0], "gauge": spec["ko_sigma"][17]},
        "cfl": spec["cfl"],
        "integrator": "SSPRK3" if spec.get("integrator", "rk4") == "ssprk3" else "RK4",
        "l2_policy": "inputs larger than L2 (4 resident 24-gridfunction sets)",
    }
    if extra:
        c.update(extra)
    return c


# ------------------------------------------------------------------ dist


def dist_env():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return world, rank, local


def dist_init(world: int, use_cuda: bool):
    if world <= 1:
        return None
    import torch.distributed as dist

    dist.init_process_group(backend="nccl" if use_cuda else "gloo")
    return dist


def reduce_max(dist, x: float, device=None) -> float:
    """max of a float over ranks (identity without a process group)"""
    if dist is None:
        return x
    import torch

    t = torch.tensor([x], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def reduce_sum(dist, x: float, device=None) -> float:
    if dist is None:
        return x
    import torch

    t = torch.tensor([x], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.SUM)
    return float(t.item())


# ---------------------------------------------------------------- clocks


class ClockSampler:
    """nvidia-smi samples (200 ms) of the benchmarked GPU during the timed region."""

    FIELDS = ("uuid,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap,utilization.gpu")

    def __init__(self, uuid: str | None):
        self.uuid = uuid
        self.proc = None
        self.path = None

    def start(self):
        try:
            fd, self.path = tempfile.mkstemp(suffix=".csv")
            os.close(fd)
            self.f = open(self.path, "w")
            self.proc = subprocess.Popen(["nvidia-smi", f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
                                          "-lms", "200"], stdout=self.f, stderr=subprocess.DEVNULL)
        except (OSError, FileNotFoundError):
            self.proc = None

    def stop(self) -> dict | None:
        if self.proc is None:
            return None
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        self.f.close()
        rows = []
        for line in open(self.path):
            parts = [p.strip() for p in line.split(",")]
            if len(parts) < 9:
                continue
            if self.uuid and self.uuid not in parts[0]:
                continue
            rows.append(parts)
        os.unlink(self.path)
        if not rows:
            return None

        def num(s):
            try:
                return float(s)
            except ValueError:
                return None

        sm = [num(r[1]) for r in rows if num(r[1]) is not None]
        mx = [num(r[2]) for r in rows if num(r[2]) is not None]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for r in rows for i in range(4) if r[5 + i].lower() == "active"})
        pw = [num(r[3]) for r in rows if num(r[3]) is not None]
        ut = [num(r[9]) for r in rows if len(r) > 9 and num(r[9]) is not None]
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": reasons, "samples": len(rows), "power_w_max": max(pw) if pw else None,
                "gpu_busy_pct_mean": statistics.mean(ut) if ut else None}


def gpu_uuid(local: int) -> str | None:
    try:
        import torch

        return str(torch.cuda.get_device_properties(local).uuid)
    except Exception:
        return None


# ------------------------------------------------------------- CPU oracle


def oracle_threads() -> int:
    return len(os.sched_getaffinity(0)) if hasattr(os, "sched_getaffinity") else os.cpu_count()


def cpu_baseline(spec: dict, seconds: float) -> dict:
    """The oracle as it stands, on the host cores: time steps of the workload (its integrator) until
    `seconds` pass."""
    from oracle.oracle import Oracle

    o = Oracle(dict(spec, nthreads=0))
    y = o.brill_lindquist(spec["masses"], spec["positions"], spec["perturb_amp"], spec["seed"])
    dt = o.dt()
    ssp = spec.get("integrator", "rk4") == "ssprk3"
    steps = 0
    t0 = time.perf_counter()
    while True:
        (o.ssprk3 if ssp else o.rk4)(y, dt, 1)
        steps += 1
        if time.perf_counter() - t0 >= seconds:
            break
    el = time.perf_counter() - t0
    pts = math.prod(spec["N"])
    out = {"value": pts * (3 if ssp else 4) * steps / el, "unit": UNIT, "cores": oracle_threads(), "kind": "oracle",
           "sample": f"first {steps} {'SSPRK3' if ssp else 'RK4'} steps of {spec['name']} (full grid), {el:.1f} s"}
    if pts <= 4_000_000:
        # the diagnostics on the evolved state, one call each (wall ms on the same cores)
        diag = {}
        for name, fn in (("hamiltonian", lambda: o.hamiltonian(y)), ("momentum", lambda: o.momentum(y)),
                         ("psi4", lambda: o.psi4(y))):
            t0 = time.perf_counter()
            r = fn()
            diag[name + "_ms"] = 1e3 * (time.perf_counter() - t0)
        R = spec.get("psi4_radius")
        if R:
            t0 = time.perf_counter()
            o.psi4_modes(r[0], R, PSI4_NTHETA, PSI4_NPHI, PSI4_LMAX)
            diag["psi4_modes_ms"] = 1e3 * (time.perf_counter() - t0)
        out["diagnostics"] = diag
    return out


def run_reference(args, spec):
    """--impl reference: the CPU oracle on the host cores, timing the same work as a step of the
    GPU arm -- full steps of the workload's integrator on the whole grid (right-hand side,
    dissipation, radiation and parity boundary conditions, the update and det enforcement, with
    the Hamiltonian constraint every h_every steps).  When the requested K + W steps would not fit
    about 150 s, the run is a bounded sample: one warm-up step and as many timed steps as fit."""
    from oracle.oracle import Oracle

    o = Oracle(dict(spec, nthreads=0))
    y = o.brill_lindquist(spec["masses"], spec["positions"], spec["perturb_amp"], spec["seed"])
    dt = o.dt()
    ssp = spec.get("integrator", "rk4") == "ssprk3"
    step = o.ssprk3 if ssp else o.rk4
    h_every = int(spec["h_every"])
    done = 0

    def one():
        nonlocal done
        step(y, dt, 1)
        done += 1
        if h_every and done % h_every == 0:
            o.hamiltonian(y)

    t0 = time.perf_counter()
    one()
    t_step = time.perf_counter() - t0
    budget = 150.0
    if (args.steps + args.warmup) * t_step <= budget:
        warm, steps, bounded = args.warmup, args.steps, False
        for _ in range(warm - 1):
            one()
    else:
        warm, steps, bounded = 1, int(max(1, min(args.steps, (budget - t_step) // t_step))), True
    t0 = time.perf_counter()
    for _ in range(steps):
        one()
    el = time.perf_counter() - t0
    pts = math.prod(spec["N"])
    sub = 3 if ssp else 4
    value = pts * sub * steps / el
    sample = (f"{steps} full {'SSPRK3' if ssp else 'RK4'} steps of {spec['name']} (whole grid, H every {h_every}) "
              f"after {warm} warm-up step(s)" + (f"; bounded sample of the {args.steps} steps asked for" if bounded
                                                 else ""))
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
        "steps": steps, "warmup": warm, "ms_per_step": 1e3 * el / steps, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic (Brill-Lindquist closed form)",
        "config": config_of(spec, {"parallelism": "replicas x1", "dt": dt}),
        "cpu_baseline": {"value": value, "unit": UNIT, "cores": oracle_threads(), "kind": "oracle", "sample": sample},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)


# -------------------------------------------------------------- GPU arm


def run_ours(args, spec, world, rank, local):
    import numpy as np
    import torch

    from paper_2505_00097_gb300 import binding as B

    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    dist = dist_init(world, True)
    B.lib()
    g = B.Grid(spec, device=local)
    g.set_brill_lindquist(spec["masses"], spec["positions"], spec["perturb_amp"], spec["seed"])
    dt = g.dt_cfl
    pts = g.interior
    h_every = int(spec["h_every"])
    stream = torch.cuda.current_stream(dev)   # the library's stream is the legacy stream of this device
    ssp = spec.get("integrator", "rk4") == "ssprk3"
    substeps = 3 if ssp else 4
    step = g.ssprk3_step if ssp else g.rk4_step
    per_step = g.info.launches_per_ssprk3_step if ssp else g.info.launches_per_step
    # k_ham + k_ham_reduce, after a step also the azimuthal ghost refresh (if the grid has one)
    per_h = 2 + int(g.info.n_inner > g.info.n_inner_stencil)

    def run_steps(n, start):
        launches = 0
        for s in range(n):
            step(dt, 1)
            launches += per_step
            if h_every and (start + s + 1) % h_every == 0:
                g.hamiltonian()
                launches += per_h
        return launches

    # warm-up (graph capture happens on the first step)
    run_steps(args.warmup, 0)
    torch.cuda.synchronize()
    uuid = gpu_uuid(local)
    clocks = ClockSampler(uuid)
    if dist is not None:
        dist.barrier()
    torch.cuda.synchronize()
    clocks.start()
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    launches = run_steps(args.steps, args.warmup)
    e1.record(stream)
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1)
    ck = clocks.stop()
    if dist is not None:
        dist.barrier()
    ms_max = reduce_max(dist, ms, dev)
    g.check_finite()
    value = world * pts * substeps * args.steps / (ms_max * 1e-3)

    # dominant kernels: one RHS evaluation (k_d1 + k_rhs), timed alone with CUDA events on the same stream
    T = g.T
    ybuf = torch.empty(24 * T, dtype=torch.float64, device=dev)
    obuf = torch.empty_like(ybuf)
    g.get_state(ybuf, False)
    for _ in range(3):
        g.rhs(ybuf, obuf)
    nrep = 20
    r0 = torch.cuda.Event(enable_timing=True)
    r1 = torch.cuda.Event(enable_timing=True)
    r0.record(stream)
    for _ in range(nrep):
        g.rhs(ybuf, obuf)
    r1.record(stream)
    torch.cuda.synchronize()
    rhs_ms = r0.elapsed_time(r1) / nrep
    del ybuf, obuf
    diag = None if args.no_diagnostics else diagnostics(g, spec, stream, args.workload, args.diag_reps)
    probe = B.fp64_peak(local)
    n_sm = torch.cuda.get_device_properties(local).multi_processor_count
    mhz = (ck or {}).get("sm_mhz") or (ck or {}).get("sm_max_mhz") or 2070.0
    peak = FP64_FLOP_PER_CLK_SM * n_sm * mhz * 1e6
    roof = {"bound": "alu", "kernel": "k_d1 + k_rhs (one FP64 BSSN RHS evaluation + KO + upwind, nr_rhs)",
            "unit": "TFLOP/s",
            "peak": peak / 1e12,
            "peak_source": f"derived: 2 DFMA/clk/SM x {n_sm} SMs x {mhz:.0f} MHz (median SM clock in the timed region)",
            "probe_tflops": probe / 1e12, "launch_ms": rhs_ms, "points_per_launch": pts,
            "traffic": TRAFFIC.get(args.workload), "traffic_algorithmic": B_ALG_RHS * pts,
            "traffic_source": "ncu dram__bytes_read.sum + dram__bytes_write.sum of one nr_rhs (k_d1 + k_rhs); "
                              "the excess over the algorithmic bytes is register-spill lines evicted to DRAM"}
    f_pipe = F_PIPE.get(args.workload)
    if f_pipe:
        f_alg = F_ALG[args.workload]
        ach = f_pipe * pts / (rhs_ms * 1e-3)
        roof.update(achieved=ach / 1e12, frac=ach / peak, flops_per_point=f_pipe,
                    flops_source="the compiled kernels' DADD + DMUL + 2 DFMA per interior point (ncu); the advection + "
                                 "dissipation sums and most first and mixed differences run on the integer pipe and "
                                 "are not counted",
                    mix_ceiling=PIPE_CEILING[args.workload], flops_per_point_algorithm=f_alg,
                    achieved_algorithm=f_alg * pts / (rhs_ms * 1e-3) / 1e12,
                    algorithm_source="FP64 operations per interior point in the kernels' source (host census), the "
                                     "first and mixed differences counted as FP64 sums")
    else:
        roof.update(achieved=None, frac=None, flops_per_point=None)
    f_method = F_METHOD.get(args.workload)
    if f_method:
        am = f_method * pts / (rhs_ms * 1e-3)
        roof.update(flops_per_point_method=f_method, achieved_method=am / 1e12, frac_method=am / peak,
                    method_source="the oracle's counting build: add + mul + div per interior point of the plain "
                                  "coordinate-basis right-hand side")

    # end to end through the C ABI with host buffers: every step uploads the state from
    # pinned host memory, advances it, and reads the new state back.  The headline uses the
    # compact state (interior + pure outer points; inner ghosts are parity copies rebuilt on
    # upload); the full padded array is timed too.
    e2e = None
    if not args.no_e2e:
        n_e2e = min(args.steps, 100)

        def e2e_run(npts, put, get, start):
            host_in = torch.empty(24 * npts, dtype=torch.float64).pin_memory()
            host_out = torch.empty(24 * npts, dtype=torch.float64).pin_memory()
            get(host_in.data_ptr(), True)
            if dist is not None:
                dist.barrier()
            t0 = time.perf_counter()
            for s in range(n_e2e):
                put(host_in.data_ptr(), True)
                run_steps(1, start + s)
                get(host_out.data_ptr(), True)
                host_in, host_out = host_out, host_in
            torch.cuda.synchronize()
            el = reduce_max(dist, time.perf_counter() - t0, dev)
            return world * pts * substeps * n_e2e / el, 24 * npts * 8

        nc = g.info.n_state_points
        stepper = "nr_ssprk3_step" if ssp else "nr_rk4_step"
        integ = "ssprk3" if ssp else "rk4"

        def io_run(start):
            """nr_step_io: the compact state in from pinned host memory, one step, the new compact
            state written to pinned host memory by the step's last stage"""
            host_in = torch.empty(24 * nc, dtype=torch.float64).pin_memory()
            host_out = torch.empty(24 * nc, dtype=torch.float64).pin_memory()
            g.get_state_compact(host_in.data_ptr(), True)
            if dist is not None:
                dist.barrier()
            t0 = time.perf_counter()
            for s in range(n_e2e):
                g.step_io(dt, 1, host_in.data_ptr(), host_out.data_ptr(), integ)
                if h_every and (start + s + 1) % h_every == 0:
                    g.hamiltonian()
                host_in, host_out = host_out, host_in
            torch.cuda.synchronize()
            el = reduce_max(dist, time.perf_counter() - t0, dev)
            return world * pts * substeps * n_e2e / el, 24 * nc * 8

        v, nbytes = io_run(args.warmup + args.steps)
        vc, _ = e2e_run(nc, g.set_state_compact, g.get_state_compact, args.warmup + args.steps + n_e2e)
        vf, fbytes = e2e_run(T, g.set_state, g.get_state, args.warmup + args.steps + 2 * n_e2e)
        e2e = {"value": v, "unit": UNIT, "h2d_bytes_per_step": nbytes, "d2h_bytes_per_step": nbytes, "steps": n_e2e,
               "path": f"nr_step_io per step: compact state ({nc} interior + pure outer points of {T}) uploaded from "
                       f"pinned host memory, one {integ.upper()} step, the new compact state stored to pinned host "
                       "memory by the step's last stage",
               "separate_calls": {"value": vc, "h2d_bytes_per_step": nbytes, "d2h_bytes_per_step": nbytes,
                                  "path": f"nr_set_state_compact + {stepper} + nr_get_state_compact per step"},
               "full_state": {"value": vf, "h2d_bytes_per_step": fbytes, "d2h_bytes_per_step": fbytes,
                              "path": f"nr_set_state(pinned host) + {stepper} + nr_get_state(pinned host) per step"}}

    # the two modes against plain one-run-per-launch on the same GPU (one replica only: the
    # comparisons are per GPU and hold the device for a minute or two)
    modes = {}
    if world == 1 and args.workload == "headon":
        if not args.no_batched:
            modes["batched"] = batch_compare(local, args.batch_runs, args.batch_steps)
        if not args.no_served:
            modes["served"] = served_compare(local, args.line_served_requests, args.served_tfinal,
                                             args.served_rate, ("srpt",), args.served_cap)

    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        cpu = cpu_baseline(spec, args.cpu_seconds)

    if rank == 0:
        line = {
            "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": ms_max / args.steps, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64", "data": "synthetic (Brill-Lindquist closed form on the GPU)",
            "config": config_of(spec, {"parallelism": f"replicas x{world}", "dt": dt}),
            "roofline": roof, "cpu_baseline": cpu, "e2e": e2e, "gpu_launches": launches, "clocks": ck,
        }
        if diag is not None:
            line["diagnostics"] = diag
        line.update(modes)
        print(json.dumps(line), flush=True)
    if dist is not None:
        dist.barrier()
        dist.destroy_process_group()
    g.close()


def diagnostics(g, spec, stream, wl: str, nrep: int) -> dict:
    """Device time per call of the constraint and waveform diagnostics on the evolved state
    (CUDA events on the library's stream, no norm read-back), and the wall time of one
    psi4 mode decomposition (host set-up, sampling, reduction, copy back)."""
    import torch

    T, pts = g.T, g.interior
    dev = torch.device("cuda", torch.cuda.current_device())
    H = torch.empty(T, dtype=torch.float64, device=dev)
    M = torch.empty(3 * T, dtype=torch.float64, device=dev)
    P4 = torch.empty(2 * T, dtype=torch.float64, device=dev)
    calls = {"hamiltonian": (lambda: g.hamiltonian(None, H, norms=False), "nr_hamiltonian: k_ham + k_ham_reduce"),
             "momentum": (lambda: g.momentum(None, M, norms=False), "nr_momentum: k_mom + k_ham_reduce"),
             "psi4": (lambda: g.psi4(P4), "nr_psi4: k_psi4 + k_psi4_ghosts")}
    out = {}
    for name, (fn, what) in calls.items():
        fn()
        torch.cuda.synchronize()
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        for _ in range(nrep):
            fn()
        e1.record(stream)
        torch.cuda.synchronize()
        ms = e0.elapsed_time(e1) / nrep
        d = {"launches": what, "device_ms": ms, "points_per_s": pts / (ms * 1e-3)}
        f = DIAG_PIPE.get(wl, {}).get(name)
        if f:
            d.update(flops_per_point=f, achieved_tflops=f * pts / (ms * 1e-3) / 1e12,
                     flops_per_point_algorithm=DIAG_FLOPS[wl][name])
        out[name] = d
    R = spec.get("psi4_radius")
    if R:
        g.psi4_modes(R, PSI4_NTHETA, PSI4_NPHI, PSI4_LMAX)
        t0 = time.perf_counter()
        for _ in range(nrep):
            c = g.psi4_modes(R, PSI4_NTHETA, PSI4_NPHI, PSI4_LMAX)
        out["psi4_modes"] = {"launches": "nr_psi4_modes: k_psi4 + k_psi4_ghosts + k_sphere_sample + k_sphere_modes",
                             "wall_ms": (time.perf_counter() - t0) * 1e3 / nrep, "radius": R, "lmax": PSI4_LMAX,
                             "nodes": [PSI4_NTHETA, PSI4_NPHI], "abs_C2m": [float(abs(v)) for v in c[:5]]}
    del H, M, P4
    return out


# ------------------------------------------------------- batched / served


def batch_compare(local: int, n_runs: int, steps: int, warm: int = 3) -> dict:
    """The batched workload's runs (seeded: q ~ U[1,4], d ~ U[0.5,2], N_rho in {64, ..., 256}), each
    advanced `steps` RK4 steps twice on the same GPU: plain, one grid at a time with its own
    nr_rk4_step graph, and batched, one nr_batch (one launch per substage over the tiles of all
    grids, autotuned tile).  CUDA-event times of both; every final state compared bitwise."""
    import torch

    from paper_2505_00097_gb300 import binding as B

    dev = torch.device("cuda", local)
    runs = W.config_batch(n_runs=n_runs, steps=steps)
    grids = [B.Grid(s, device=local) for s in runs]
    for g, s in zip(grids, runs):
        g.set_brill_lindquist(s["masses"], s["positions"])
    dts = [g.dt_cfl for g in grids]
    pts = sum(g.interior for g in grids)
    init = []
    for g in grids:
        t = torch.empty(24 * g.T, dtype=torch.float64, device=dev)
        g.get_state(t, False)
        init.append(t)

    def reset():
        for g, t in zip(grids, init):
            g.set_state(t, False)

    ev = lambda: torch.cuda.Event(enable_timing=True)  # noqa: E731
    for g, dt in zip(grids, dts):       # warm-up (the first step captures each grid's graph)
        g.rk4_step(dt, warm)
    reset()
    torch.cuda.synchronize()
    clocks_plain = ClockSampler(gpu_uuid(local))
    clocks_plain.start()
    a0, a1 = ev(), ev()
    a0.record()
    for g, dt in zip(grids, dts):
        g.rk4_step(dt, steps)
    a1.record()
    torch.cuda.synchronize()
    ck_plain = clocks_plain.stop()
    t_plain = a0.elapsed_time(a1) * 1e-3
    plain_final = []
    for g in grids:
        t = torch.empty(24 * g.T, dtype=torch.float64, device=dev)
        g.get_state(t, False)
        plain_final.append(t)
    reset()
    batch = B.Batch(grids)
    tx, ty, tune_ms = batch.autotune(dts)
    batch.rk4_step(dts, warm)           # warm-up (the first step captures the graph)
    reset()
    clocks = ClockSampler(gpu_uuid(local))
    torch.cuda.synchronize()
    clocks.start()
    b0, b1 = ev(), ev()
    b0.record()
    batch.rk4_step(dts, steps)
    b1.record()
    torch.cuda.synchronize()
    ck = clocks.stop()
    t_batch = b0.elapsed_time(b1) * 1e-3
    same = True
    for g, ref in zip(grids, plain_final):
        t = torch.empty(24 * g.T, dtype=torch.float64, device=dev)
        g.get_state(t, False)
        same = same and bool(torch.equal(t, ref))
    batch.close()
    for g in grids:
        g.close()
    del init, plain_final
    value, plain_value = pts * 4 * steps / t_batch, pts * 4 * steps / t_plain
    return {"value": value, "plain_value": plain_value, "ratio": value / plain_value, "unit": UNIT,
            "bitwise_equal_to_plain": same, "runs": len(runs), "interior_points": pts,
            "grid_sizes_rho": sorted({s["N"][0] for s in runs}), "steps_per_run": steps,
            "steps_in_config": 500, "tile": f"{tx}x{ty}", "autotune_stage_ms": tune_ms,
            "seconds": {"batched": t_batch, "plain": t_plain},
            "mode": "batched: one nr_batch, one launch per RK4 substage over all grids (CUDA graph); plain: one "
                    "grid at a time, nr_rk4_step graph per grid; CUDA-event times, inputs resident in HBM",
            "equality": "every grid's full final state compared with torch.equal", "clocks": ck,
            "clocks_plain": ck_plain}


def served_compare(local: int, n_requests: int, t_final: float, rate: float, policies=("srpt",),
                   cap: int = 1000000, starve_s: float = 0.0) -> dict:
    """A seeded Poisson stream of single-puncture and head-on requests of 1e5..4e6 points (the served
    workload's generator), served as it arrives (wall clock) by nr_server with each policy in
    `policies` (continuous batching under an 80 GB budget, points cap `cap`) and by a plain FIFO queue
    of single-grid runs, one at a time.  Each arm ends every request with its Hamiltonian-constraint
    norms, a NaN/Inf check and the 64-bit digest of its final state; the digests are compared.
    Policy "srpt_cap": SRPT with the starvation cap starve_s (requests submitted longer ago go first)."""
    from paper_2505_00097_gb300 import binding as B

    reqs = W.config_served(n_requests=n_requests, t_final=t_final, rate_per_min=rate)

    def serve(mode: str):
        batched = mode != "plain"
        clocks = ClockSampler(gpu_uuid(local))
        clocks.start()
        start = time.perf_counter()
        done, arrive, submitted, digest = {}, {}, [], {}
        host_s = {"admit_s": 0.0, "retire_s": 0.0}
        upd = 0.0
        if batched:
            srv = B.Server(80 * 10 ** 9, 64, device=local)
            srv.set_tile(16, 8)
            srv.set_prefetch(4)
            srv.set_policy("srpt" if mode == "srpt_cap" else mode, cap)
            if mode == "srpt_cap":
                srv.set_starvation_cap(starve_s)
        queue = []
        nxt = 0
        while len(done) < len(reqs):
            now = time.perf_counter() - start
            while nxt < len(reqs) and reqs[nxt]["arrival_s"] <= now:
                r = reqs[nxt]
                if batched:
                    rid = srv.submit(r, r["t_final"], keep_digest=True)
                    submitted.append((rid, nxt))
                else:
                    queue.append(nxt)
                arrive[nxt] = reqs[nxt]["arrival_s"]
                nxt += 1
            if batched:
                nrun, nq = srv.advance(5)
                for rid, k in submitted:
                    if k in done:
                        continue
                    info = srv.poll(rid)
                    if info["status"] in (2, 3):
                        done[k] = time.perf_counter() - start
                        n = reqs[k]["N"]
                        upd += 4.0 * info["steps_done"] * n[0] * n[1] * n[2]
                        digest[k] = srv.fetch_digest(rid) if info["status"] == 2 else None
                idle = nrun == 0 and nq == 0
            else:
                idle = not queue
                if queue:
                    k = queue.pop(0)
                    t0 = time.perf_counter()
                    g = B.Grid(reqs[k], device=local)
                    g.set_brill_lindquist(reqs[k]["masses"], reqs[k]["positions"])
                    host_s["admit_s"] += time.perf_counter() - t0
                    steps = max(1, int(math.ceil(reqs[k]["t_final"] / g.dt_cfl - 1e-9)))
                    g.rk4_step(g.dt_cfl, steps)
                    g.sync()
                    t0 = time.perf_counter()
                    g.hamiltonian()
                    digest[k] = g.digest()
                    g.check_finite()
                    g.close()
                    host_s["retire_s"] += time.perf_counter() - t0
                    done[k] = time.perf_counter() - start
                    upd += 4.0 * steps * g.interior
            if idle and nxt < len(reqs):
                time.sleep(max(0.0, min(0.05, reqs[nxt]["arrival_s"] - (time.perf_counter() - start))))
        makespan = time.perf_counter() - start
        ck = clocks.stop()
        stats = None
        if batched:
            stats = srv.stats()
            srv.close()
        ttc = sorted(done[k] - arrive[k] for k in done)
        q = lambda p: ttc[min(len(ttc) - 1, int(round(p * (len(ttc) - 1))))]  # noqa: E731
        r = {"value": upd / makespan, "p50_ttc_s": q(0.5), "p99_ttc_s": q(0.99),
             "mean_ttc_s": sum(ttc) / len(ttc), "makespan_s": makespan, "clocks": ck}
        if stats:
            r["server_stats"] = stats
        else:
            r["host_s"] = host_s
        return r, digest

    arms = {}
    digests = {}
    for pol in policies:
        arms[pol], digests[pol] = serve(pol)
    plain, dplain = serve("plain")
    out = {"unit": UNIT, "requests": len(reqs), "t_final": t_final, "rate_per_min": rate, "starvation_cap_s": starve_s,
           "points_range": [1e5, 4e6], "hbm_budget_gb": 80, "max_batch_points": cap,
           "plain": plain, "plain_value": plain["value"],
           "mode": "nr_server continuous batching (requests admitted as they arrive, one nr_batch per kind of "
                   "request) against a plain FIFO queue of single-grid nr_rk4_step runs; wall-clock makespan "
                   "and time to completion",
           "equality": "64-bit digest (nr_state_digest) of every request's final state, served vs plain"}
    for pol in policies:
        a = arms[pol]
        same = all(digests[pol].get(k) is not None and digests[pol].get(k) == dplain.get(k) for k in dplain)
        out[pol] = dict(a, ratio=a["value"] / plain["value"], bitwise_equal_to_plain=same)
    head = policies[0]
    out.update(policy=head, value=arms[head]["value"], ratio=out[head]["ratio"],
               bitwise_equal_to_plain=out[head]["bitwise_equal_to_plain"],
               p50_ttc_s=arms[head]["p50_ttc_s"], p99_ttc_s=arms[head]["p99_ttc_s"],
               mean_ttc_s=arms[head]["mean_ttc_s"], clocks=arms[head]["clocks"])
    return out


def run_batch(args, world, rank, local):
    """--workload batch: the batched runs (batch_compare) as the line's headline."""
    import torch

    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    dist = dist_init(world, True)
    r = batch_compare(local, args.batch_runs, args.steps, max(3, args.warmup))
    t_batch = reduce_max(dist, r["seconds"]["batched"], dev)
    t_plain = reduce_max(dist, r["seconds"]["plain"], dev)
    n, pts = r["steps_per_run"], r["interior_points"]
    if rank == 0:
        line = {
            "metric": METRIC, "value": world * pts * 4 * n / t_batch, "unit": UNIT, "n_gpus": world, "steps": n,
            "warmup": max(3, args.warmup), "ms_per_step": 1e3 * t_batch / n, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic (Brill-Lindquist head-on binaries, seeded)",
            "config": {"workload": f"batch_{r['runs']}_headon_sinhcyl", "runs": r["runs"], "interior_points": pts,
                       "grid_sizes_rho": r["grid_sizes_rho"], "steps_per_run": n, "tile": r["tile"],
                       "autotune_stage_ms": r["autotune_stage_ms"]},
            "plain": {"value": world * pts * 4 * n / t_plain, "unit": UNIT,
                      "mode": "one grid at a time, nr_rk4_step graph per grid"},
            "speedup_vs_plain": t_plain / t_batch, "bitwise_equal_to_plain": r["bitwise_equal_to_plain"],
            "clocks": r["clocks"],
        }
        print(json.dumps(line), flush=True)


def run_served(args, world, rank, local):
    """--workload served: the served stream (served_compare) under both policies and the plain queue."""
    import torch

    torch.cuda.set_device(local)
    pols = tuple(a for a in args.served_arms.split(",") if a) if args.served_arms else \
        (args.served_policy, other_name(args.served_policy))
    r = served_compare(local, args.served_requests, args.served_tfinal, args.served_rate, pols, args.served_cap,
                       args.served_starve_s)
    line = {
        "metric": METRIC, "value": r["value"], "unit": UNIT, "n_gpus": 1, "steps": None, "warmup": 0,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
        "data": "synthetic (seeded Poisson request stream)",
        "config": {"workload": f"served_{r['requests']}_requests", "rate_per_min": args.served_rate,
                   "t_final": args.served_tfinal, "points_range": [1e5, 4e6], "hbm_budget_gb": 80,
                   "policy": pols[0], "max_batch_points": args.served_cap, "starvation_cap_s": args.served_starve_s},
        "served": r[pols[0]], **{f"served_{p}": r[p] for p in pols[1:]}, "plain_fifo": r["plain"],
        "speedup_vs_plain": r["ratio"], "bitwise_equal_to_plain": r["bitwise_equal_to_plain"],
        "p50_ttc_vs_plain": r["p50_ttc_s"] / r["plain"]["p50_ttc_s"],
    }
    print(json.dumps(line), flush=True)


def run_part(args, world, rank, local):
    """--workload part: the head-on grid cut into partitions (the chare decomposition of Sec. 3: per substage
    each partition's points, then inner-boundary messages and face-by-face halos) against the whole grid,
    the same steps on the same GPU; CUDA-event times; final states compared by digest."""
    import torch

    from paper_2505_00097_gb300 import binding as B

    torch.cuda.set_device(local)
    spec = W.config_headon()
    parts = tuple(int(v) for v in args.parts.split(","))
    n = args.steps
    warm = max(3, args.warmup)
    ev = lambda: torch.cuda.Event(enable_timing=True)  # noqa: E731
    g = B.Grid(spec, device=local)
    g.set_brill_lindquist(spec["masses"], spec["positions"])
    pg = B.PartGrid(spec, parts, device=local)
    pg.set_brill_lindquist(spec["masses"], spec["positions"])
    dt = g.dt_cfl
    g.rk4_step(dt, warm)
    pg.rk4_step(dt, warm)
    torch.cuda.synchronize()
    a0, a1 = ev(), ev()
    a0.record()
    g.rk4_step(dt, n)
    a1.record()
    torch.cuda.synchronize()
    clocks = ClockSampler(gpu_uuid(local))
    clocks.start()
    b0, b1 = ev(), ev()
    b0.record()
    pg.rk4_step(dt, n)
    b1.record()
    torch.cuda.synchronize()
    ck = clocks.stop()
    t_whole, t_part = a0.elapsed_time(a1) * 1e-3, b0.elapsed_time(b1) * 1e-3
    same = pg.digest() == g.digest()
    pts = g.interior
    line = {
        "metric": METRIC, "value": pts * 4 * n / t_part, "unit": UNIT, "n_gpus": 1, "steps": n, "warmup": warm,
        "ms_per_step": 1e3 * t_part / n, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "f64", "data": "synthetic (Brill-Lindquist closed form on the GPU)",
        "config": {"workload": f"headon_sinhcyl_256x2x512_in_{parts[0]}x{parts[1]}x{parts[2]}_partitions",
                   "parts": list(parts), "messages_per_substage": pg.messages},
        "whole_grid": {"value": pts * 4 * n / t_whole, "ms_per_step": 1e3 * t_whole / n},
        "exchange_overhead": t_part / t_whole - 1.0, "bitwise_equal_to_whole_grid": same, "clocks": ck,
        "note": "all partitions on one GPU: every message is a device-local copy",
    }
    print(json.dumps(line), flush=True)
    pg.close()
    g.close()


def other_name(policy: str) -> str:
    return "fifo" if policy == "srpt" else "srpt"


def run_profile(args):
    """--profile: the launches a profiler capture looks at, on cuda:0, nothing timed."""
    import torch

    from paper_2505_00097_gb300 import binding as B

    spec = workload(args.workload)
    if args.profile_grid:
        spec["N"] = tuple(int(v) for v in args.profile_grid.split(","))
    g = B.Grid(spec)
    g.set_brill_lindquist(spec["masses"], spec["positions"], spec["perturb_amp"], spec["seed"])
    if args.profile == "rhs":
        y = torch.empty(24 * g.T, dtype=torch.float64, device="cuda")
        o = torch.empty_like(y)
        g.get_state(y, False)
        g.rhs(y, o)
    else:
        g.rk4_step(g.dt_cfl, 4)
        g.hamiltonian(None, torch.empty(g.T, dtype=torch.float64, device="cuda"), norms=False)
        g.momentum(None, torch.empty(3 * g.T, dtype=torch.float64, device="cuda"), norms=False)
        g.psi4(torch.empty(2 * g.T, dtype=torch.float64, device="cuda"))
    torch.cuda.synchronize()
    print(f"profile {args.profile}: {spec['name']} interior {g.interior}", flush=True)
    g.close()


def main():
    args = parse()
    world, rank, local = dist_env()
    if args.profile:
        run_profile(args)
        return
    if args.workload == "batch":
        if args.steps == 2000:
            args.steps = 100
        run_batch(args, world, rank, local)
        return
    if args.workload == "served":
        if rank == 0:
            run_served(args, world, rank, local)
        return
    if args.workload == "part":
        if args.steps == 2000:
            args.steps = 200
        if rank == 0:
            run_part(args, world, rank, local)
        return
    spec = workload(args.workload)
    if args.impl == "reference":
        if rank != 0:
            return
        run_reference(args, spec)
        return
    run_ours(args, spec, world, rank, local)


if __name__ == "__main__":
    main()
