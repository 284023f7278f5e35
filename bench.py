#!/usr/bin/env python
"""Benchmark: matrix-free operator apply throughput (GDoF/s) with its roofline, and the time of the
implicit heat-step solve in fp64 vs mixed fp32/fp64 precision.

One step = one application of the implicit heat-step operator (rho c_p / dt) M + K(k(T^n)) with
k(T) = k0 (1 + 0.5 T / T_b), Q2 on a uniform 128^3 mesh of the 600 um box (257^3 = 16,974,593
DoFs, Dirichlet bottom face), in fp64: gather, Gauss-point values and gradients, conductivity from
the interpolated previous temperature, integration and scatter-add, all in the library's CUDA
kernels.  Inputs are resident in HBM; L2 is flushed between timed steps.

The same JSON line carries the other workloads of the run (each measured once, bounded): the fp32
and double-float applies and the laser-driven heat-step solve (fp64 CG vs fp32-inner defect
correction) on the same mesh; the Oseen Q2/Q1 operator on 64^3 (applies, FGMRES solve, interface
source loads); the adaptive-octree reinitialisation with 8 right-hand sides per launch; the 16^3
Helmholtz Jacobi-CG in a CUDA graph; the heat-step adjoint gradient on 64^3; the Q3/Q4 applies;
one melt-pool algorithm step; and the oracle on the host cores.

    python bench.py [--steps K] [--warmup W] [--impl ours|reference] [--quick] [--suite]
    python bench.py --probe WORKLOAD [ARGS...]     build one workload, apply it a few times (for ncu)
Under torchrun (N > 1) every rank runs an independent replica on its own GPU.
"""
import argparse
import hashlib
import json
import os
import statistics
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "GDoF/s of matrix-free operator apply & %HBM roofline; CG solve time FP64 vs mixed"
WORKLOAD = "heat_laser_q2_128"
HBM_FALLBACK_GBS = 6800.0
FP64_PEAK_TFLOPS = 1.25      # GB300 FP64 (vector and tensor) rate of the profiling recipe's table
# Algorithmic flops of one scalar Q2 heat-cell apply as the kernel performs it (FMA = 2), lines in
# difference form and Gauss weights inside the transposes.  Value lines 27 x 9 = 243, the mass term
# 27, derivative lines 27 x 8 = 216, the products with the coefficient 81, derivative transposes in x
# and y 18 x 12 = 216, the combined z transposes 9 x 19 = 171, value transposes in x and y 18 x 9 = 162:
# 1116 with k tabulated per Gauss point.  With k evaluated in the kernel, the nodal T^n is swept to the
# Gauss points (243) and k0 + s T applied (27 x 2): 1413.
HEAT_FLOPS_PER_CELL = {"tabulated": 1116, "inkernel": 1413}
# The double-float kernel evaluates the same cell operator in pairs of fp32 (tabulated w h k): per
# cell 6525 fp32 instructions, 7335 flops with an FMA counted as two (a pair product is 1 FMUL + 3
# FFMA, a pair sum 8 FADD, a renormalisation 3 FADD, a power of two 2 FMUL): value lines 27 x 58 / 67,
# the mass term 108 / 189, derivative lines 27 x 44, the products with the coefficient 324 / 567,
# derivative transposes 18 x 68, combined z transposes 9 x 113 / 122, value transposes 18 x 52 / 61,
# renormalisations 162.  Its roof is the fp32 pipe: 152 SMs x 128 lanes x 2 flops x 2.07 GHz (the
# profiling recipe's unit count and SM clock).
HEAT_DF64_FLOPS_PER_CELL = 7335
HEAT_DF64_INSTRUCTIONS_PER_CELL = 6525
FP32_PEAK_TFLOPS = 152 * 128 * 2 * 2.07e9 / 1e12
# Algorithmic HBM bytes of one heat apply: read u, write v, read the nodal T^n (3 words per DoF).
HEAT_WORDS_PER_DOF = 3
# Algorithmic flops of one Oseen Q2/Q1 cell apply as each kernel variant performs it.
# Gauss-point loop outside, on Gauss-point coefficients with the weight and the powers of h folded
# in (w h^2 rho beta tabulated, so the value terms are multiply-adds only): value sweeps 3 x 270,
# 27 points x 159 (pressure 15, 9 gradients 39, value terms 24, symmetric stress 15 with 2 mu formed
# once, 3 test accumulations 48, continuity 18), nodal pressure and continuity scaling 16,
# integration sweeps 3 x 270 = 5929.
# Component loop outside: pressure at the Gauss points and its test terms 891, three velocity
# components x (value sweeps 270 + 27 points x 80) = 7290, integration sweeps and scaling 899.
OSEEN_FLOPS_PER_CELL = {"component-outer": 891 + 7290 + 899, "qpoint-outer": 810 + 27 * 159 + 16 + 810}
# Algorithmic HBM bytes of one fp64 Oseen apply: read u, write v (16 B per DoF), the nodal
# level set and convection field the coefficients come from (4 x 8 B per velocity node).
OSEEN_BYTES_PER_VEL_NODE = 4 * 8


def max_over_ranks(seconds, dist=None, device="cpu"):
    """The slowest rank's timed-region duration (every rank calls this)."""
    if dist is None:
        return seconds
    import torch
    t = torch.tensor([seconds], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def whole_job_rate(units_per_rank, steps, world, seconds):
    """Whole-job throughput in G units/s: every rank processes units_per_rank per step
    (independent replicas, weak scaling), timed by the slowest rank."""
    return units_per_rank * steps * world / seconds / 1e9


def measured_peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            return json.load(f)
    except Exception:
        return {}


class ClockSampler:
    """Samples nvidia-smi SM clocks and throttle reasons every 50 ms while running (the timed
    region starts after the first sample has arrived)."""
    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index):
        self.index, self.rows, self.proc = index, [], None

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--id={self.index}", f"--query-gpu={self.Q}",
                                          "--format=csv,noheader,nounits", "-lms", "50"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
            t0 = time.time()
            while not self.rows and time.time() - t0 < 3.0:
                time.sleep(0.01)
        except Exception:
            self.proc = None
        return self

    def _read(self):
        for line in self.proc.stdout:
            self.rows.append([x.strip() for x in line.split(",")])

    def __exit__(self, *a):
        if self.proc:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except Exception:
                self.proc.kill()

    def summary(self):
        sm = [float(r[1]) for r in self.rows if len(r) >= 9 and r[1].replace(".", "").isdigit()]
        mx = [float(r[2]) for r in self.rows if len(r) >= 9 and r[2].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for r in self.rows if len(r) >= 9 for i in range(4) if r[5 + i] == "Active"})
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": reasons, "samples": len(self.rows)}


KERNEL_SOURCES = ("apply_f64.cu", "apply_f32.cu", "apply_df64.cu", "apply_df64_uniform.cu", "df_pairs.cuh",
                  "apply_kernels.cuh", "cellops.cuh", "scalar_local.cuh", "lines.cuh", "df64.cuh")


def kernel_hash():
    h = hashlib.sha256()
    for f in KERNEL_SOURCES:
        with open(os.path.join(ROOT, "paper_2501_18781_gb300", "csrc", f), "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()[:16]


def ncu_traffic(key):
    """DRAM bytes per launch of the dominant kernel from the committed ncu summary, if it was
    taken on the current kernel source (else None).  key: workload/arithmetic."""
    p = os.path.join(ROOT, "profiles", "dram_traffic.txt")
    if not os.path.exists(p):
        return None
    kh = kernel_hash()
    for line in open(p):
        parts = line.split()
        if len(parts) >= 3 and not line.startswith("#") and parts[0] == key and parts[1] == kh:
            return float(parts[2])
    return None


# ----------------------------------------------------------------------------- workload builders

def build_heat(ctx, n=128, autotune=True, coef_mode=None):
    """The implicit heat-step operator of the 128^3 laser workload: Q2 on the 600 um box, Dirichlet
    bottom face, k(T^n) from the seeded hot-spot temperature.  Returns (op, map, T^n tensor)."""
    import torch
    import synthetic as syn
    from paper_2501_18781_gb300 import DofMap, Mesh, Operator
    wl = syn.scaled(syn.HEAT_LASER, n)
    p = wl.params
    m = DofMap(Mesh.uniform(ctx, n, wl.lo, wl.hi), 2, 1 << 4)
    x = m.coords()
    T_prev = torch.tensor(syn.heat_initial_temperature(*x.T, p["laser"]["radius"], wl.hi[2]), device="cuda")
    kw = {} if coef_mode is None else {"coef_mode": coef_mode}
    op = Operator(ctx, "heat", [m], rhocp=p["rhocp"], dt=p["dt"], k0=p["k0"], t_boil=p["t_boil"], **kw)
    op.set_field("t_prev", T_prev)
    if autotune:
        op.autotune()   # set-up: coefficient mode, launch shape, fp64 vs double-float
    return op, m, T_prev


def heat_step_rhs(ctx, m, T_prev, n=128):
    """Right-hand side of the laser-driven heat step for theta = T - T_ref: (rho c_p / dt) M theta^n +
    the top-face load of eq. (laser_gauss) (200 W, 50 um), Dirichlet rows 0.  The mass term is the
    library's apply of the same map's heat operator with k0 = 0, the laser load its mf_laser_load."""
    import torch
    import synthetic as syn
    from paper_2501_18781_gb300 import Operator
    wl = syn.scaled(syn.HEAT_LASER, n)
    p = wl.params
    mass = Operator(ctx, "heat", [m], rhocp=p["rhocp"], dt=p["dt"], k0=0.0, t_boil=p["t_boil"], coef_mode=1)
    mass.set_field("t_prev", T_prev)
    theta = T_prev - p["t_ref"]
    lz = p["laser"]
    b = mass.apply(theta) + mass.laser_load(lz["power"], lz["radius"], lz["x0"], lz["y0"], lz["absorptivity"])
    d = torch.tensor(m.export(cell_map=False, constraints=False, coords=False)["dirichlet"], device="cuda")
    b[d] = 0.0
    return b


def build_oseen(ctx, n=64):
    import numpy as np
    import torch
    import synthetic as syn
    from paper_2501_18781_gb300 import DofMap, Mesh, Operator
    wl = syn.scaled(syn.OSEEN_INTERFACE, n)
    p = wl.params
    mesh = Mesh.uniform(ctx, n, wl.lo, wl.hi)
    mu, mp = DofMap(mesh, 2, 0b011111), DofMap(mesh, 1, 0)
    x = mu.coords()
    t1, t2 = syn.wavy_plane_phases(wl.seed)
    phi = syn.initial_level_set(syn.wavy_plane_distance(*x.T, t1, t2), wl.eps)
    beta = np.array(syn.convection_field(*x.T, wl.seed, wl.lo, wl.hi))
    sigma = 1.0 / (p["dt_cfl"] * wl.h)
    op = Operator(ctx, "oseen", [mu, mp], sigma=sigma, rho_l=p["rho_l"], rho_g=p["rho_g"], mu_l=p["mu_l"],
                  mu_g=p["mu_g"], eps=wl.eps)
    op.set_field("phi", torch.tensor(phi, device="cuda"))
    op.set_field("beta", torch.tensor(beta.ravel(), device="cuda"))
    op.autotune()   # set-up: picks the fp64 kernel variant (component- or Gauss-point-outer)
    return op, mu, mp, mesh


def build_reinit_octree(ctx, base=None, levels=None, autotune=True):
    """The adaptive-octree reinitialisation workload: base^3 + levels band refinement around the
    seeded deformed sphere, Q2 with hanging-node constraints."""
    import torch
    import synthetic as syn
    from paper_2501_18781_gb300 import DofMap, Mesh, Operator
    wl = syn.REINIT_OCTREE
    base = base or wl.n
    levels = wl.levels if levels is None else levels
    eps = 2.0 / (base << levels)
    d = lambda X, Y, Z: syn.deformed_sphere_distance(X, Y, Z, wl.seed)
    leaves = syn.refine_band_leaves(base, levels, d, eps)
    m = DofMap(Mesh.octree(ctx, base, levels, leaves), 2, 0)
    x = m.coords()
    phi = torch.tensor(syn.initial_level_set(syn.deformed_sphere_distance(*x.T, wl.seed), eps), device="cuda")
    op = Operator(ctx, "reinit", [m], eps=eps, dtau=0.5 / (base << levels))
    op.set_field("phi", phi)
    op._keep = phi
    if autotune:
        op.autotune()
    return op, m


# ----------------------------------------------------------------------------- timing helpers

def time_apply(op, src, dst, steps, warmup, flush, arith=None):
    import torch
    for _ in range(warmup):
        op.apply(src, dst, arith=arith)
    torch.cuda.synchronize()
    times = []
    for _ in range(steps):
        flush.zero_()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        op.apply(src, dst, arith=arith)
        e1.record()
        e1.synchronize()
        times.append(e0.elapsed_time(e1) / 1e3)
    return times


def _event_ms(fn, reps=5, flush=None):
    import torch
    fn()
    torch.cuda.synchronize()
    ts = []
    for _ in range(reps):
        if flush is not None:
            flush.zero_()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        fn()
        e1.record()
        e1.synchronize()
        ts.append(e0.elapsed_time(e1))
    return statistics.median(ts)


def _apply_rates(op, n, nrhs, flush, reps=5, words=None):
    """G DoF.RHS/s of the fp64, double-float and fp32 applies; with ``words`` (vector words per DoF
    and right-hand side, fields per DoF) also the fraction of the measured HBM peak."""
    import torch
    import synthetic as syn
    u = torch.tensor(syn.uniform_pm1(1, n * nrhs), device="cuda")
    u32 = u.float()
    v, v32 = torch.empty_like(u), torch.empty_like(u32)
    hbm = measured_peaks().get("hbm_gbs", HBM_FALLBACK_GBS)
    out = {}
    for name, fn, wb in (("f64", lambda: op.apply(u, v, nrhs=nrhs), 8),
                         ("df64", lambda: op.apply(u, v, nrhs=nrhs, arith="df64"), 8),
                         ("f32", lambda: op.apply(u32, v32, nrhs=nrhs), 4)):
        ms = _event_ms(fn, reps, flush)
        out[name] = {"ms": ms, "gdofs": n * nrhs / ms / 1e6, "variant": op.variant}
        if words is not None:
            b = (words[0] * nrhs + words[1]) * wb * n
            out[name]["hbm_frac"] = b / (ms * 1e-3) / 1e9 / hbm
            out[name]["bytes_per_launch"] = b
    return out


def _packed_rates(op, n, nrhs, flush, reps=5):
    """G DoF.RHS/s of the packed 16-bit applies (fp32 vectors, pairs of right-hand sides per thread)."""
    import torch
    import synthetic as syn
    u = torch.tensor(syn.uniform_pm1(1, n * nrhs), device="cuda").float()
    v = torch.empty_like(u)
    out = {}
    for arith in ("f16", "bf16"):
        ms = _event_ms(lambda: op.apply(u, v, nrhs=nrhs, arith=arith), reps, flush)
        out[arith] = {"ms": ms, "gdofs": n * nrhs / ms / 1e6, "variant": op.variant}
    return out


def _timed_solve(op, b, reps=1, **kw):
    """Set-up + warm-up solve, then the median of reps timed solves (host clock, synchronised)."""
    import torch
    op.solve(b, **kw)
    torch.cuda.synchronize()
    runs = []
    for _ in range(reps):
        t0 = time.perf_counter()
        _, info = op.solve(b, **kw)
        torch.cuda.synchronize()
        runs.append((time.perf_counter() - t0, info))
    sec, info = sorted(runs, key=lambda r: r[0])[len(runs) // 2]
    return {"seconds": sec, "iterations": info["iterations"], "outer": info["outer_iterations"],
            "rel_residual": info["rel_residual"], "status": info["status"]}


def e2e_applies(op, src, steps, arith=None):
    """Seconds for `steps` end-to-end applies (pinned host input -> device -> apply -> pinned host
    output), pipelined and serial.  Pipelined: copies on two non-blocking streams and the apply on the
    library's stream, ordered by events, with two device input and output buffers, so the upload of
    step k+1 and the download of step k-1 overlap the apply of step k."""
    import torch
    n = src.numel()
    hsrc = torch.empty(n, dtype=src.dtype, pin_memory=True)
    hsrc.copy_(src.cpu())
    hdst = [torch.empty(n, dtype=src.dtype, pin_memory=True) for _ in range(2)]
    dsrc = [torch.empty_like(src) for _ in range(2)]
    ddst = [torch.empty_like(src) for _ in range(2)]
    comp = torch.cuda.current_stream()
    up, down = torch.cuda.Stream(), torch.cuda.Stream()
    ev = lambda: torch.cuda.Event()
    in_ready, in_free = [ev(), ev()], [ev(), ev()]
    out_ready, out_free = [ev(), ev()], [ev(), ev()]
    for e in in_free + out_free:
        e.record(comp)

    def run(k_steps):
        for k in range(k_steps):
            b = k % 2
            with torch.cuda.stream(up):
                up.wait_event(in_free[b])
                dsrc[b].copy_(hsrc, non_blocking=True)
                in_ready[b].record(up)
            comp.wait_event(in_ready[b])
            comp.wait_event(out_free[b])
            op.apply(dsrc[b], ddst[b], arith=arith)
            in_free[b].record(comp)
            out_ready[b].record(comp)
            with torch.cuda.stream(down):
                down.wait_event(out_ready[b])
                hdst[b].copy_(ddst[b], non_blocking=True)
                out_free[b].record(down)

    run(4)
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(up)
    run(steps)
    for s_ in (comp, up):
        down.wait_stream(s_)
    e1.record(down)
    e1.synchronize()
    piped = e0.elapsed_time(e1) / 1e3
    # the same steps one after another on one stream
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    for _ in range(steps):
        dsrc[0].copy_(hsrc, non_blocking=True)
        op.apply(dsrc[0], ddst[0], arith=arith)
        hdst[0].copy_(ddst[0], non_blocking=True)
    e1.record()
    e1.synchronize()
    return piped, e0.elapsed_time(e1) / 1e3


# ----------------------------------------------------------------------------- sub-measurements

HEAT_SOLVERS = {"fp64": dict(solver="cg", precond="chebyshev"),
                "mixed": dict(solver="defect_correction", precond="chebyshev", inner_tol=1e-4, inner_maxit=100),
                # the same two with every fp64-accurate operator apply in double-float on the fp32 pipes
                "fp64_df64_applies": dict(solver="cg", precond="chebyshev", fp64_arith="df64"),
                "mixed_df64_outer": dict(solver="defect_correction", precond="chebyshev", inner_tol=1e-4,
                                         inner_maxit=100, fp64_arith="df64")}


def heat_solve_comparison(ctx, op, m, T_prev, n=128):
    """The implicit heat step on n^3 Q2 cells to 1e-10: fp64 CG with Chebyshev(4)-Jacobi vs fp32 inner
    CG (same preconditioner in fp32) inside fp64 defect correction.  Right-hand side: the laser load
    and (rho c_p / dt) M theta^n; also a seeded uniform right-hand side as a second case."""
    import torch
    import synthetic as syn
    out = {"workload": f"heat_laser_q2_{n}", "n_dofs": m.n_dofs, "tol": 1e-10}
    b = heat_step_rhs(ctx, m, T_prev, n)
    for name, kw in HEAT_SOLVERS.items():
        out[name] = _timed_solve(op, b, tol=1e-10, use_graph=True, **kw)
    out["speedup_mixed_over_fp64"] = out["fp64"]["seconds"] / out["mixed"]["seconds"]
    out["speedup_df64_applies_over_fp64"] = out["fp64"]["seconds"] / out["fp64_df64_applies"]["seconds"]
    br = torch.tensor(syn.uniform_pm1(1, m.n_dofs), device="cuda")
    br[torch.tensor(m.export(cell_map=False, constraints=False, coords=False)["dirichlet"], device="cuda")] = 0
    rnd = {name: _timed_solve(op, br, tol=1e-10, use_graph=True, **kw) for name, kw in HEAT_SOLVERS.items()}
    rnd["speedup_mixed_over_fp64"] = rnd["fp64"]["seconds"] / rnd["mixed"]["seconds"]
    out["random_rhs"] = rnd
    # the same solves on the sample the host oracle solves (cpu_baseline.heat_solve): same matrix,
    # same right-hand side, for a same-size comparison
    ops, ms, _ = build_heat(ctx, CPU_SAMPLE_N)
    d = ms.export(cell_map=False, constraints=False, coords=False)["dirichlet"].astype(bool)
    bs = torch.tensor(sample_heat_rhs(ms.n_dofs, d), device="cuda")
    out[f"sample_{CPU_SAMPLE_N}"] = {name: _timed_solve(ops, bs, tol=1e-10, use_graph=True, **HEAT_SOLVERS[name])
                                     for name in ("fp64", "mixed")}
    return out


def oseen_workload(ctx, flush, n=64, solve=True):
    """The Oseen Q2/Q1 operator on n^3: fp64 / double-float / fp32 applies with the FP64-pipe and HBM
    rooflines of the fp64 kernel, the FGMRES solve, and the interface source loads."""
    op, mu, mp, mesh = build_oseen(ctx, n)
    rates = _apply_rates(op, op.n, 1, flush, reps=10)
    ncells = mu.n_cells
    flops = OSEEN_FLOPS_PER_CELL["qpoint-outer" if "qpoint-outer" in rates["f64"]["variant"] else "component-outer"] * ncells
    hbm = measured_peaks().get("hbm_gbs", HBM_FALLBACK_GBS)
    alg = 16 * op.n + OSEEN_BYTES_PER_VEL_NODE * mu.n_dofs
    s64 = rates["f64"]["ms"] * 1e-3
    out = {"workload": f"oseen_q2q1_interface_{n}", "n_dofs": op.n, "cells": ncells, "apply": rates,
           "roofline_f64": {"bound": "alu", "achieved": flops / s64 / 1e12, "peak": FP64_PEAK_TFLOPS,
                            "unit": "TFLOP/s", "frac": flops / s64 / 1e12 / FP64_PEAK_TFLOPS,
                            "flops_per_launch": flops},
           "hbm_f64": {"achieved": alg / s64 / 1e9, "peak": hbm, "unit": "GB/s", "frac": alg / s64 / 1e9 / hbm,
                       "bytes_per_launch": alg},
           "hbm_f32": {"bytes_per_launch": alg // 2,
                       "frac": alg / 2 / (rates["f32"]["ms"] * 1e-3) / 1e9 / hbm}}
    out["interface_sources"] = interface_sources_timing(ctx, op, mu, flush)
    if solve:
        out["solve"] = oseen_solve(ctx, op, mu, mp)
    return out


def reinit_octree_workload(ctx, flush, solves=True):
    """Adaptive octree (base 32^3 + 3 levels, ~12.3M Q2 DoFs with hanging nodes), 8 right-hand sides
    per launch: fp64 / double-float / fp32 batched and single applies with the fraction of HBM of the
    algorithmic bytes (per right-hand side u read and v written, plus the nodal level set once:
    136N bytes in fp64, 72N in fp32), and the 8-RHS mixed-precision solve to 1e-10."""
    import numpy as np
    import torch
    import synthetic as syn
    wl = syn.REINIT_OCTREE
    op, m = build_reinit_octree(ctx)
    r = {"workload": wl.name, "n_dofs": m.n_dofs, "cells": m.n_cells, "hanging_nodes": m.n_constraints,
         "nrhs": wl.nrhs,
         "apply_batched": _apply_rates(op, m.n_dofs, wl.nrhs, flush, reps=3, words=(2, 1)),
         "apply_single": _apply_rates(op, m.n_dofs, 1, flush, reps=3, words=(2, 1))}
    if solves:
        B = torch.tensor(np.concatenate([syn.uniform_pm1(s, m.n_dofs) for s in range(1, wl.nrhs + 1)]), device="cuda")
        r["mixed_solve_8rhs"] = _timed_solve(op, B, nrhs=wl.nrhs, solver="defect_correction", precond="chebyshev",
                                             tol=1e-10, use_graph=True)
    return r


def helmholtz_workload(ctx):
    """Helmholtz 16^3 (35,937 DoFs, L2-resident: launch-latency bound): apply rates and the Jacobi-CG
    solve to 1e-10, launched directly and with the iteration body replayed as a CUDA graph."""
    import torch
    import synthetic as syn
    from paper_2501_18781_gb300 import DofMap, Mesh, Operator
    wl = syn.HELMHOLTZ_SPHERE
    p = wl.params
    m = DofMap(Mesh.uniform(ctx, wl.n, wl.lo, wl.hi), 2, 0)
    x = m.coords()
    phi = syn.initial_level_set(syn.sphere_distance(*x.T), wl.eps)
    op = Operator(ctx, "helmholtz", [m], mass_coef=p["mass"], a_liquid=p["a_liquid"], a_gas=p["a_gas"])
    op.set_field("phi", torch.tensor(phi, device="cuda"))
    op.autotune()
    b = torch.tensor(syn.uniform_pm1(1, m.n_dofs), device="cuda")
    r = {"workload": wl.name, "n_dofs": m.n_dofs, "apply": _apply_rates(op, m.n_dofs, 1, None, reps=20)}
    for g in (False, True):
        r["cg_jacobi_graph" if g else "cg_jacobi"] = _timed_solve(op, b, reps=3, solver="cg", precond="jacobi",
                                                                  tol=1e-10, use_graph=g)
    return r


def heat_adjoint_workload(ctx, flush):
    """Heat-step adjoint on 64^3 (2,146,689 DoFs): forward GMRES, adjoint GMRES with the transposed
    convection, the four laser-parameter gradients and dJ/dk_q; fp64 to 1e-10."""
    import numpy as np
    import torch
    import synthetic as syn
    from paper_2501_18781_gb300 import DofMap, Mesh, Operator
    wl = syn.HEAT_ADJOINT
    p = wl.params
    m = DofMap(Mesh.uniform(ctx, wl.n, wl.lo, wl.hi), 2, 1 << 4)
    x = m.coords()
    beta = np.array(syn.convection_field(*x.T, wl.seed, wl.lo, wl.hi))
    kq = syn.kq_field(m.n_cells * 27, wl.seed, p["k0"])
    op = Operator(ctx, "heat", [m], rhocp=p["rhocp"], dt=p["dt"], k0=p["k0"], t_boil=p["t_boil"])
    keep = [torch.tensor(beta.ravel(), device="cuda"), torch.tensor(kq, device="cuda")]
    op.set_field("beta", keep[0])
    op.set_field("k_qpoint", keep[1])
    ztop = wl.hi[2]
    lz = p["laser"]
    th_prev = syn.heat_initial_temperature(*x.T, lz["radius"], ztop) - p["t_ref"]
    target = syn.heat_target_temperature(*x.T, ztop, wl.seed + 4) - p["t_ref"]
    tp, tt = torch.tensor(th_prev, device="cuda"), torch.tensor(target, device="cuda")
    lzt = (lz["power"], lz["radius"], lz["x0"], lz["y0"], lz["absorptivity"])
    kw = dict(solver="gmres", precond="jacobi", tol=1e-10, restart=50)
    op.heat_step_gradient(lzt, tp, tt, p["box_half"], p["box_depth"], **kw)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    J, g, gk, _, _ = op.heat_step_gradient(lzt, tp, tt, p["box_half"], p["box_depth"], **kw)
    torch.cuda.synchronize()
    sec = time.perf_counter() - t0
    # the same with the forward and adjoint GMRES applies in double-float (the convective operator
    # and its transpose on the fp32 pipes); J and the gradients agree to the solves' tolerance
    kwd = dict(kw, fp64_arith="df64")
    op.heat_step_gradient(lzt, tp, tt, p["box_half"], p["box_depth"], **kwd)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    Jd, gd, _, _, _ = op.heat_step_gradient(lzt, tp, tt, p["box_half"], p["box_depth"], **kwd)
    torch.cuda.synchronize()
    secd = time.perf_counter() - t0
    # mixed precision: defect correction with fp32 inner GMRES on the operator and on its
    # transpose, the outer residuals in double-float
    kwm = dict(solver="defect_correction", precond="jacobi", tol=1e-10, restart=30, maxit=50, fp64_arith="df64")
    op.heat_step_gradient(lzt, tp, tt, p["box_half"], p["box_depth"], **kwm)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    Jm, gm, _, _, _ = op.heat_step_gradient(lzt, tp, tt, p["box_half"], p["box_depth"], **kwm)
    torch.cuda.synchronize()
    secm = time.perf_counter() - t0
    return {"workload": wl.name, "n_dofs": m.n_dofs, "gradient_seconds": sec,
            "gradient_seconds_df64_applies": secd, "gradient_seconds_mixed": secm, "J": J, "dJ_dlaser": g,
            "J_rel_diff_df64_applies": abs(Jd - J) / abs(J) if J else 0.0,
            "J_rel_diff_mixed": abs(Jm - J) / abs(J) if J else 0.0,
            "dJ_dlaser_max_rel_diff_mixed": max(abs(a - b) for a, b in zip(gm, g)) / max(abs(v) for v in g),
            "apply": _apply_rates(op, m.n_dofs, 1, flush)}


def oseen_solve(ctx, op, mu, mp):
    """The Oseen saddle-point solve to 1e-10: flexible GMRES(50) with the block upper-triangular
    preconditioner (fp32 inner applies), a seeded right-hand side with zero Dirichlet rows."""
    import numpy as np
    import torch
    import synthetic as syn
    b = syn.uniform_pm1(1, op.n)
    d = mu.export(cell_map=False, constraints=False, coords=False)["dirichlet"]
    b[np.concatenate([np.tile(d, 3), np.zeros(mp.n_dofs, bool)])] = 0
    bt = torch.tensor(b, device="cuda")
    kw = dict(solver="gmres", precond="block_triangular", restart=50, maxit=400, tol=1e-10, velocity_steps=10,
              schur_tol=0.1, schur_maxit=30)
    out = {"solver": "fgmres(50) + block-triangular (fp32 inner)", "tol": 1e-10}
    for key, graph, ar in (("seconds_direct", False, "f64"), ("seconds", True, "f64"), ("seconds_df64_outer", True, "df64")):
        op.solve(bt, use_graph=graph, fp64_arith=ar, **kw)         # set-up + warm-up
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        _, info2 = op.solve(bt, use_graph=graph, fp64_arith=ar, **kw)
        torch.cuda.synchronize()
        out[key] = time.perf_counter() - t0
        if ar == "f64":
            info = info2
        else:
            out["df64_outer"] = {"iterations": info2["iterations"], "rel_residual": info2["rel_residual"],
                                 "status": info2["status"]}
    out.update(iterations=info["iterations"], rel_residual=info["rel_residual"], status=info["status"],
               preconditioner="replayed CUDA graph", schur_steps_per_call=info["inner_steps"] / info["iterations"])
    return out


def meltpool_oseen(ctx, n, flush, darcy_c=None):
    """The Oseen workload with the melt-pool terms switched on (three-phase rho/mu, Darcy damping,
    trace-corrected stress) and a hot spot across the interface.  The paper damps with C = 1e12
    kg/(m^3 s) at a time step of 0.01 us (rho_l / dt = 4.1e11): C / (rho_l sigma) = 2.45.  The
    unit-cube workload has sigma = 1/dt = 2n, so C is scaled to keep that ratio (C = 1e12 * 1e-8 *
    sigma); the unscaled 1e12 makes even a direct solve stall at a 1e-7 relative residual here.
    Solid below T_s far from the spot.  fp64 and fp32 apply rates and the FGMRES solve to 1e-10 with
    the interface source loads as right-hand side."""
    import numpy as np
    import torch
    import synthetic as syn
    from paper_2501_18781_gb300 import DofMap, Mesh, Operator
    from paper_2501_18781_gb300._lib import MF_OSEEN_DARCY, MF_OSEEN_THREE_PHASE, MF_OSEEN_TRACE_CORRECTION
    wl = syn.scaled(syn.OSEEN_INTERFACE, n)
    p = wl.params
    mesh = Mesh.uniform(ctx, n, wl.lo, wl.hi)
    mu, mp = DofMap(mesh, 2, 0b011111), DofMap(mesh, 1, 0)
    x = mu.coords()
    t1, t2 = syn.wavy_plane_phases(wl.seed)
    phi = syn.initial_level_set(syn.wavy_plane_distance(*x.T, t1, t2), wl.eps)
    beta = np.array(syn.convection_field(*x.T, wl.seed, wl.lo, wl.hi))
    T = syn.interface_temperature(*x.T, t_base=1500.0)
    sigma = 1.0 / (p["dt_cfl"] * wl.h)
    if darcy_c is None:
        darcy_c = 1e12 * 1e-8 * sigma
    op = Operator(ctx, "oseen", [mu, mp], sigma=sigma, rho_l=p["rho_l"], rho_g=p["rho_g"],
                  mu_l=p["mu_l"], mu_g=p["mu_g"], eps=wl.eps, rho_s=p["rho_l"], mu_s=p["mu_l"], t_solidus=1933.0,
                  t_liquidus=2200.0, darcy_c=darcy_c, darcy_b=1.0,
                  oseen_flags=MF_OSEEN_THREE_PHASE | MF_OSEEN_DARCY | MF_OSEEN_TRACE_CORRECTION)
    fields = [torch.tensor(phi, device="cuda"), torch.tensor(beta.ravel(), device="cuda"), torch.tensor(T, device="cuda")]
    op.set_field("phi", fields[0])
    op.set_field("beta", fields[1])
    op.set_field("t_prev", fields[2])
    u = torch.tensor(syn.uniform_pm1(1, op.n), device="cuda")
    v = torch.empty_like(u)
    u32, v32 = u.float(), torch.empty(op.n, dtype=torch.float32, device="cuda")
    ms64 = _event_ms(lambda: op.apply(u, v), 10, flush)
    msdf = _event_ms(lambda: op.apply(u, v, arith="df64"), 10, flush)
    ms32 = _event_ms(lambda: op.apply(u32, v32), 10, flush)
    # right-hand side: the interface loads of this temperature field (hybrid recoil force in the
    # momentum rows, evaporative dilation in the continuity rows)
    ev, ti = syn.EVAPORATION, syn.TI64
    src = op.interface_sources(fields[2], ev["p_amb"], ev["h_v"], ev["molar_mass"], ev["t_boil"],
                               ti["rho_l"] * ti["cp_l"], ti["rho_g"] * ti["cp_g"], outputs=("u", "p"))
    bt = torch.cat([src["u"], src["p"]])
    kw = dict(solver="gmres", precond="block_triangular", restart=50, maxit=400, tol=1e-10, use_graph=True)
    op.solve(bt, **kw)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    _, info = op.solve(bt, **kw)
    torch.cuda.synchronize()
    sec = time.perf_counter() - t0
    # the same with the outer applies in double-float
    kwd = dict(kw, fp64_arith="df64")
    op.solve(bt, **kwd)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    _, infod = op.solve(bt, **kwd)
    torch.cuda.synchronize()
    return {"workload": f"oseen_meltpool_{n}", "variant": op.variant, "darcy_c": darcy_c,
            "apply_f64": {"ms": ms64, "gdofs": op.n / ms64 / 1e6}, "apply_df64": {"ms": msdf, "gdofs": op.n / msdf / 1e6},
            "apply_f32": {"ms": ms32, "gdofs": op.n / ms32 / 1e6},
            "solve": {"seconds": sec, "iterations": info["iterations"],
                      "rel_residual": info["rel_residual"], "status": info["status"]},
            "solve_df64_outer": {"seconds": time.perf_counter() - t0, "iterations": infod["iterations"],
                                 "rel_residual": infod["rel_residual"], "status": infod["status"]}}


def build_meltpool_step(ctx, n=64):
    """The melt-pool step workload on the 600 um box (n^3 cells): maps, the seeded state (fp64
    device tensors) and the MeltPoolStep with every term switched on."""
    import numpy as np
    import torch
    import synthetic as syn
    from paper_2501_18781_gb300 import DofMap, MeltPoolStep, Mesh
    from paper_2501_18781_gb300._lib import MF_OSEEN_DARCY, MF_OSEEN_THREE_PHASE, MF_OSEEN_TRACE_CORRECTION
    wl = syn.scaled(syn.MELTPOOL_STEP, n)
    p, ti, ev = wl.params, syn.TI64, syn.EVAPORATION
    mesh = Mesh.uniform(ctx, n, wl.lo, wl.hi)
    maps = [DofMap(mesh, 2, 0b011111), DofMap(mesh, 1, 0), DofMap(mesh, 2, 0), DofMap(mesh, 2, 1 << 4)]
    x = maps[0].coords()
    state = {k: torch.tensor(np.ascontiguousarray(v.ravel()), device="cuda")
             for k, v in syn.meltpool_state(*x.T, wl.seed, wl.lo, wl.hi, wl.eps, u_max=p["u_max"]).items()}
    sol, dar, st = p["solid"], p["darcy"], p["surface_tension"]
    step = MeltPoolStep(
        ctx, maps,
        evaporation=dict(mass_flux="knight", p_ambient=ev["p_amb"], latent_heat=ev["h_v"], molar_mass=ev["molar_mass"],
                         t_boil=ev["t_boil"], sticking=ev["sticking"], gas_constant=8.314),
        laser=p["laser"], gravity=p["gravity"], dt=p["dt"], eps=wl.eps, rho_l=ti["rho_l"], rho_g=ti["rho_g"],
        mu_l=ti["mu_l"], mu_g=ti["mu_g"], rhocp_l=ti["rho_l"] * ti["cp_l"], rhocp_g=ti["rho_g"] * ti["cp_g"],
        k_l=ti["k_l"], k_g=ti["k_g"], oseen_flags=MF_OSEEN_THREE_PHASE | MF_OSEEN_DARCY | MF_OSEEN_TRACE_CORRECTION,
        rho_s=sol["rho_s"], mu_s=sol["mu_s"], t_solidus=sol["t_solidus"], t_liquidus=sol["t_liquidus"],
        darcy_c=dar["C"], darcy_b=dar["b"], alpha0=st["alpha0"], alpha1=st["alpha1"], t_alpha=st["t_alpha"],
        alpha_res=st["alpha_res"], reinit_steps=p["reinit_steps"], dtau=p["dtau_cells"] * wl.h, tol=p["tol"],
        flow_tol=p["flow_tol"], maxit=500, reinit_mixed=p["reinit_mixed"], flow_velocity_steps=p["flow_velocity_steps"],
        flow_schur_maxit=p["flow_schur_maxit"], flow_schur_tol=p["flow_schur_tol"])
    return wl, maps, state, step


def meltpool_step(ctx, n=64, reps=3):
    """One step of the melt-pool algorithm on the 600 um box (64^3 cells: 2.1M Q2 nodes per field,
    6.7M velocity-pressure DoFs): predictors, level-set advection (GMRES) with the variant-1
    transport velocity, 2 reinitialisation steps (CG), two-phase heat with laser and evaporative
    cooling (GMRES), melt-pool Navier-Stokes with surface tension, recoil and Darcy damping
    (FGMRES, block-triangular).  The same state is advanced reps times after one warm-up step."""
    import torch
    wl, maps, state, step = build_meltpool_step(ctx, n)
    p = wl.params
    step.advance(state)
    torch.cuda.synchronize()
    runs = []
    for _ in range(reps):
        t0 = time.perf_counter()
        _, info = step.advance(state)
        torch.cuda.synchronize()
        runs.append((time.perf_counter() - t0, info))
    wall, info = sorted(runs, key=lambda r: r[0])[len(runs) // 2]
    nu, npr = maps[0].n_dofs, maps[1].n_dofs
    return {"workload": wl.name, "n_u": nu, "n_p": npr, "unknowns_per_step": 5 * nu + npr, "ms_per_step": wall * 1e3,
            "stage_seconds": dict(zip(("advection", "reinit", "heat", "flow", "total"), info["seconds"])),
            "iterations": {k: info[k + "_iterations"] for k in ("advection", "reinit", "heat", "flow")},
            "rel_residuals": {k: info[k + "_residual"] for k in ("advection", "reinit", "heat", "flow")},
            "status": info["status"], "tol": p["tol"], "flow_tol": p["flow_tol"]}


def qk_flops_per_cell(k):
    """Sum-factorised Q_k Helmholtz apply, P = k + 1: 3 interpolation sweeps, 3 collocation
    derivatives, 3 transposed derivatives and 3 transposed sweeps of P^4 multiply-adds each, and
    about 10 flops per Gauss point for the pointwise work."""
    P = k + 1
    return 2 * 12 * P ** 4 + 10 * P ** 3


def helmholtz_qk(ctx, flush, solves=False):
    """Q3 on 64^3 and Q4 on 48^3 cells (193^3 = 7,189,057 DoFs each), the sphere coefficient
    a = 1 + 999 H(phi): fp64 and fp32 applies with the L2 flushed; with ``solves`` also the Q3
    solve comparison."""
    import torch
    import synthetic as syn
    from paper_2501_18781_gb300 import DofMap, Mesh, Operator
    out = {}
    for k, n in ((3, 64), (4, 48)):
        m = DofMap(Mesh.uniform(ctx, n), k, 0)
        eps = 1.0 / (2 * n)
        phi = torch.tensor(syn.initial_level_set(syn.sphere_distance(*m.coords().T), eps), device="cuda")
        op = Operator(ctx, "helmholtz", [m], mass_coef=1.0, a_liquid=1000.0, a_gas=1.0, eps=eps)
        op.set_field("phi", phi)
        fl = qk_flops_per_cell(k) * m.n_cells
        r = {"cells": m.n_cells, "n_dofs": m.n_dofs, "flops_per_cell": qk_flops_per_cell(k)}
        for dt in (torch.float64, torch.float32):
            u = torch.tensor(syn.uniform_pm1(1, m.n_dofs), device="cuda").to(dt)
            v = torch.empty_like(u)
            op.apply(u, v)
            ms = _event_ms(lambda: op.apply(u, v), 10, flush)
            r["f64" if dt == torch.float64 else "f32"] = {"ms": ms, "gdofs": m.n_dofs / ms / 1e6,
                                                          "tflops": fl / ms / 1e9, "variant": op.variant}
        r["f64"]["frac_of_fp64_peak"] = r["f64"]["tflops"] / FP64_PEAK_TFLOPS
        if k == 3:
            # the tensor-core kernel: 2 dense products of 2 x 64 x 256 flops per cell, three split terms
            u = torch.tensor(syn.uniform_pm1(1, m.n_dofs), device="cuda").float()
            v = torch.empty_like(u)
            op.apply(u, v, arith="tc")
            ms = _event_ms(lambda: op.apply(u, v, arith="tc"), 10, flush)
            dense = 3 * 2 * 2 * 64 * 256 * m.n_cells
            r["tc_bf16x3"] = {"ms": ms, "gdofs": m.n_dofs / ms / 1e6, "tensor_tflops": dense / ms / 1e9,
                              "sum_factorised_tflops_equiv": fl / ms / 1e9, "variant": op.variant}
        if k == 3 and solves:
            # solves to 1e-10: fp64 Jacobi-CG; defect correction with fp32 Chebyshev-CG inner solves on
            # the CUDA cores or on the tensor cores
            b = torch.tensor(syn.uniform_pm1(2, m.n_dofs), device="cuda")
            # (this contrast-1000 problem needs ~1750 Jacobi-CG iterations in fp64: the inner solves get
            # room to reach their 1e-4)
            runs = {"fp64_cg_jacobi": dict(solver="cg", precond="jacobi"),
                    "mixed_inner_f32": dict(solver="defect_correction", precond="chebyshev", inner_arith="f32",
                                            inner_maxit=3000),
                    "mixed_inner_tensor_cores": dict(solver="defect_correction", precond="chebyshev",
                                                     inner_arith="tc", inner_maxit=3000)}
            r["solve"] = {}
            for name, kw in runs.items():
                op.solve(b, tol=1e-10, **kw)
                torch.cuda.synchronize()
                t0 = time.perf_counter()
                _, info = op.solve(b, tol=1e-10, **kw)
                torch.cuda.synchronize()
                r["solve"][name] = {"seconds": time.perf_counter() - t0, "iterations": info["iterations"],
                                    "outer": info["outer_iterations"], "rel_residual": info["rel_residual"],
                                    "status": info["status"]}
        out[f"q{k}"] = r
    return out


def interface_sources_timing(ctx, op, mu, flush, reps=10):
    """The fused interface-source kernel (evaporative dilation, cooling and hybrid recoil loads)
    on the Oseen mesh, Knight's mass flux, a hot spot across the interface."""
    import torch
    import synthetic as syn
    ev, ti = syn.EVAPORATION, syn.TI64
    T = torch.tensor(syn.interface_temperature(*mu.coords().T), device="cuda")
    args = (T, ev["p_amb"], ev["h_v"], ev["molar_mass"], ev["t_boil"], ti["rho_l"] * ti["cp_l"], ti["rho_g"] * ti["cp_g"])
    op.interface_sources(*args)
    ms = _event_ms(lambda: op.interface_sources(*args), reps, flush)
    return {"ms": ms, "cells_per_s": mu.n_cells / ms * 1e3, "gdofs": op.n / ms / 1e6,
            "outputs": "recoil force (3 n_u), dilation (n_p), cooling (n_u)"}




# ----------------------------------------------------------------------------- the oracle on the host

CPU_SAMPLE_N = 32   # 32^3 cells of the heat workload: 274,625 DoFs, 16.6M nonzeros (past the host caches)


def _oracle_heat_matrix(n, with_map=False):
    """The oracle's assembled heat-step matrix of the headline workload on an n^3 mesh (the same
    recipe: 600 um box, Dirichlet bottom, k(T^n) from the seeded hot spot)."""
    import synthetic as syn
    from oracle import assemble as asm
    from oracle import mesh as omesh
    wl = syn.scaled(syn.HEAT_LASER, n)
    p = wl.params
    dm = omesh.uniform_dofmap(n, wl.lo, wl.hi, 2, 1 << 4)
    T = syn.heat_initial_temperature(*dm.dof_coords().T, p["laser"]["radius"], wl.hi[2])
    A = asm.heat_matrix(dm, p["rhocp"], p["dt"], p["k0"], p["t_boil"], T_prev=T)
    return (A, wl.name, dm) if with_map else (A, wl.name)


def sample_heat_rhs(n_dofs, dirichlet):
    """The seeded uniform right-hand side of the heat-step sample solves, zero on Dirichlet rows (the
    same vector on the host and on the GPU)."""
    import synthetic as syn
    b = syn.uniform_pm1(1, n_dofs)
    b[dirichlet] = 0.0
    return b


def cpu_oracle_heat_solve(n=CPU_SAMPLE_N):
    """The oracle's fp64 CG with Chebyshev(4)-Jacobi (lambda_max from 20 Lanczos steps, x 1.1, on
    [lambda_max / 30, lambda_max]) to 1e-10 on the n^3 instance of the heat step (one host core,
    scipy's CSR product): the CPU side of the headline solve, at the sample size the oracle assembles
    in about a second."""
    import synthetic as syn
    from oracle import krylov
    t0 = time.perf_counter()
    A, name, dm = _oracle_heat_matrix(n, with_map=True)
    t_asm = time.perf_counter() - t0
    b = sample_heat_rhs(dm.n_dofs, dm.dirichlet)
    op = lambda v: A @ v
    t0 = time.perf_counter()
    diag = A.diagonal()
    lmax = 1.1 * krylov.lanczos_lambda_max(op, diag, syn.uniform_pm1(9, dm.n_dofs), steps=20)
    _, its, res = krylov.cg(op, b, krylov.chebyshev(op, diag, lmax / 30.0, lmax, 4), tol=1e-10)
    return {"workload": name, "n_dofs": dm.n_dofs, "cores": 1, "assembly_seconds": t_asm,
            "seconds": time.perf_counter() - t0, "cg_iterations": its, "rel_residual": res,
            "solver": "fp64 CG + Chebyshev(4)-Jacobi, Lanczos set-up included"}


def _spmv_worker(args):
    """One host process: the rows [r0, r1) of the oracle's CSR matrix applied repeatedly for a fixed
    wall-clock window; returns the rows processed."""
    import numpy as np
    import scipy.sparse as sp
    data, indices, indptr, shape, u, window = args
    A = sp.csr_matrix((data, indices, indptr), shape=shape)
    u = np.asarray(u)
    A @ u
    reps, t0 = 0, time.perf_counter()
    while time.perf_counter() - t0 < window:
        A @ u
        reps += 1
    return shape[0] * reps, time.perf_counter() - t0


def _host_cpu():
    model = None
    try:
        out = subprocess.run(["lscpu"], capture_output=True, text=True, timeout=10).stdout
        for line in out.splitlines():
            if line.lower().startswith("model name"):
                model = line.split(":", 1)[1].strip()
                break
    except Exception:
        pass
    return {"os_cpu_count": os.cpu_count(), "model": model}


def cpu_oracle_baseline(n=CPU_SAMPLE_N, window=4.0):
    """The oracle as it stands (assembled CSR from full-quadrature element matrices, scipy's
    one-thread CSR product) applying the headline operator on an n^3 sample: one host core, and all
    host cores as row blocks in a pool of spawned processes (each applies its block for the same
    wall-clock window; the rate is the rows processed by all over the window)."""
    import multiprocessing as mp
    import numpy as np
    import synthetic as syn
    t0 = time.perf_counter()
    A, name = _oracle_heat_matrix(n)
    t_asm = time.perf_counter() - t0
    u = syn.uniform_pm1(1, A.shape[0])
    one = _spmv_worker((A.data, A.indices, A.indptr, A.shape, u, window))
    cores = os.cpu_count() or 1
    bounds = np.linspace(0, A.shape[0], cores + 1).astype(np.int64)
    jobs = []
    for i in range(cores):
        B = A[bounds[i]:bounds[i + 1]]
        jobs.append((B.data, B.indices, B.indptr, B.shape, u, window))
    with mp.get_context("spawn").Pool(cores) as pool:
        res = pool.map(_spmv_worker, jobs)
    all_rate = sum(r[0] for r in res) / max(r[1] for r in res) / 1e9
    return {"value": all_rate, "unit": "GDoF/s", "cores": cores, "kind": "oracle",
            "sample": f"{name} ({A.shape[0]} DoFs, {A.nnz} nonzeros): assembled-CSR SpMV, {cores} processes x "
                      f"{window:.0f} s row blocks (assembly {t_asm:.1f} s untimed)",
            "value_1core": one[0] / one[1] / 1e9, "host": _host_cpu()}


def cpu_oracle_helmholtz_cg():
    """The oracle's Jacobi-CG to 1e-10 on the Helmholtz 16^3 workload (35,937 DoFs, one core): the
    CPU side of the graph-CG measurement."""
    import synthetic as syn
    from oracle import assemble as asm
    from oracle import krylov
    from oracle import mesh as omesh
    wl = syn.HELMHOLTZ_SPHERE
    p = wl.params
    t0 = time.perf_counter()
    dm = omesh.uniform_dofmap(wl.n, wl.lo, wl.hi, 2)
    phi = syn.initial_level_set(syn.sphere_distance(*dm.dof_coords().T), wl.eps)
    A = asm.helmholtz_matrix(dm, phi, p["mass"], p["a_liquid"], p["a_gas"])
    t_asm = time.perf_counter() - t0
    b = syn.uniform_pm1(1, dm.n_dofs)
    t0 = time.perf_counter()
    _, its, res = krylov.cg(lambda v: A @ v, b, krylov.jacobi(A.diagonal()), tol=1e-10)
    return {"workload": wl.name, "n_dofs": dm.n_dofs, "cores": 1, "assembly_seconds": t_asm,
            "cg_jacobi_seconds": time.perf_counter() - t0, "cg_iterations": its, "rel_residual": res}


def reference_arm(args, rank, world):
    """The oracle timed on the host cores on this arm's metric: each step one assembled-CSR product
    of the headline heat operator on a 32^3 sample (assembly untimed), as the oracle stands (one core)."""
    out = {"impl": "reference", "metric": METRIC, "unit": "GDoF/s", "n_gpus": world, "steps": args.steps,
           "warmup": args.warmup, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
           "dtype": "f64", "data": "synthetic"}
    if rank != 0:
        return None
    import synthetic as syn
    A, name = _oracle_heat_matrix(CPU_SAMPLE_N)
    u = syn.uniform_pm1(1, A.shape[0])
    for _ in range(args.warmup):
        A @ u
    t0 = time.perf_counter()
    for _ in range(args.steps):
        A @ u
    dt = time.perf_counter() - t0
    val = A.shape[0] * args.steps / dt / 1e9
    out.update(value=val, ms_per_step=dt / args.steps * 1e3,
               config={"workload": WORKLOAD, "sample": name, "n_dofs": int(A.shape[0]),
                       "note": f"oracle: assembled-CSR SpMV of a {CPU_SAMPLE_N}^3 instance (assembly untimed)"},
               cpu_baseline={"value": val, "unit": "GDoF/s", "cores": 1, "kind": "oracle",
                             "sample": f"{name}: assembled CSR SpMV, {args.steps} steps", "host": _host_cpu()},
               e2e={"value": val, "unit": "GDoF/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0})
    return out


# ----------------------------------------------------------------------------- profiler probe

def probe(argv):
    """Build one workload and apply its operator a few times, for profilers such as ncu:
        heat [n] [f32|f64|df64] [inkernel|tabulated]
        oseen [n] [f32|f64|df64]
        reinit [base] [levels] [f32|f64|df64] [nrhs]
        oseen_solve [n] [maxit]
        heat_solve [n] [fp64|mixed|fp64_df64_applies|mixed_df64_outer]
        heat_adjoint [n] [f64|df64] [forward|transpose]
        helmholtz_qk [k] [n] [f32|f64|tc]
        meltpool_step [n]
    Inputs come from the seeded generators; every apply runs in libmfgb."""
    import numpy as np
    import torch
    import synthetic as syn
    from paper_2501_18781_gb300 import Context, DofMap, Mesh, Operator, build_library
    build_library()
    ctx = Context(0)
    kind = argv[0] if argv else "heat"

    def run(op, n, prec, nrhs=1, reps=4):
        u = torch.tensor(syn.uniform_pm1(1, n * nrhs), device="cuda")
        if prec in ("f32", "tc"):
            u = u.float()
        v = torch.empty_like(u)
        for _ in range(reps):
            op.apply(u, v, nrhs=nrhs, arith=prec if prec in ("df64", "tc") else None)
        torch.cuda.synchronize()
        print(op.variant, n, "x", nrhs)

    if kind == "heat":
        n = int(argv[1]) if len(argv) > 1 else 128
        prec = argv[2] if len(argv) > 2 else "f32"
        mode = None if len(argv) <= 3 else (0 if argv[3] == "inkernel" else 1)
        op, m, _ = build_heat(ctx, n, autotune=mode is None, coef_mode=mode)
        run(op, m.n_dofs, prec)
    elif kind in ("oseen", "oseen_solve"):
        n = int(argv[1]) if len(argv) > 1 else 64
        op, mu, mp, _ = build_oseen(ctx, n)
        if kind == "oseen":
            run(op, op.n, argv[2] if len(argv) > 2 else "f64")
        else:
            # flexible GMRES with the block-triangular preconditioner, capped at maxit iterations
            maxit = int(argv[2]) if len(argv) > 2 else 400
            b = syn.uniform_pm1(1, op.n)
            d = mu.export(cell_map=False, constraints=False, coords=False)["dirichlet"]
            b[np.concatenate([np.tile(d, 3), np.zeros(mp.n_dofs, bool)])] = 0
            bt = torch.tensor(b, device="cuda")
            for _ in range(2):
                _, info = op.solve(bt, solver="gmres", precond="block_triangular", maxit=maxit, tol=1e-10)
            torch.cuda.synchronize()
            print(op.variant, n, info)
    elif kind == "heat_adjoint":
        # the convective heat operator of the adjoint workload (nodal beta, k per Gauss point)
        n = int(argv[1]) if len(argv) > 1 else 64
        prec = argv[2] if len(argv) > 2 else "df64"
        tr = len(argv) > 3 and argv[3] == "transpose"
        wl = syn.scaled(syn.HEAT_ADJOINT, n)
        p = wl.params
        m = DofMap(Mesh.uniform(ctx, n, wl.lo, wl.hi), 2, 1 << 4)
        x = m.coords()
        op = Operator(ctx, "heat", [m], rhocp=p["rhocp"], dt=p["dt"], k0=p["k0"], t_boil=p["t_boil"])
        keep = [torch.tensor(np.array(syn.convection_field(*x.T, wl.seed, wl.lo, wl.hi)).ravel(), device="cuda"),
                torch.tensor(syn.kq_field(m.n_cells * 27, wl.seed, p["k0"]), device="cuda")]
        op.set_field("beta", keep[0])
        op.set_field("k_qpoint", keep[1])
        u = torch.tensor(syn.uniform_pm1(1, m.n_dofs), device="cuda")
        if prec == "f32":
            u = u.float()
        v = torch.empty_like(u)
        for _ in range(4):
            op.apply(u, v, transpose=tr, arith="df64" if prec == "df64" else None)
        torch.cuda.synchronize()
        print(op.variant, m.n_dofs)
    elif kind == "heat_solve":
        # the heat-step solve the bench times (laser right-hand side, tolerance 1e-10, graph replay),
        # once to set up and once more
        n = int(argv[1]) if len(argv) > 1 else 128
        op, m, T_prev = build_heat(ctx, n)
        b = heat_step_rhs(ctx, m, T_prev, n)
        kw = HEAT_SOLVERS[argv[2] if len(argv) > 2 else "mixed"]
        op.solve(b, tol=1e-10, use_graph=True, **kw)
        torch.cuda.synchronize()
        torch.cuda.nvtx.range_push("timed_solve")   # for ncu --nvtx-include timed_solve/
        _, info = op.solve(b, tol=1e-10, use_graph=True, **kw)
        torch.cuda.synchronize()
        torch.cuda.nvtx.range_pop()
        print(op.variant, n, info)
    elif kind == "meltpool_step":
        # one melt-pool algorithm step after a warm-up step, inside the NVTX range "timed_step"
        n = int(argv[1]) if len(argv) > 1 else 64
        _, _, state, step = build_meltpool_step(ctx, n)
        step.advance(state)
        torch.cuda.synchronize()
        torch.cuda.nvtx.range_push("timed_step")   # for ncu --nvtx-include timed_step/
        _, info = step.advance(state)
        torch.cuda.synchronize()
        torch.cuda.nvtx.range_pop()
        print(n, {k: info[k] for k in ("seconds", "advection_iterations", "reinit_iterations", "heat_iterations",
                                       "flow_iterations", "status")})
    elif kind == "helmholtz_qk":
        k = int(argv[1]) if len(argv) > 1 else 3
        n = int(argv[2]) if len(argv) > 2 else 64
        m = DofMap(Mesh.uniform(ctx, n), k, 0)
        eps = 1.0 / (2 * n)
        phi = syn.initial_level_set(syn.sphere_distance(*m.coords().T), eps)
        op = Operator(ctx, "helmholtz", [m], mass_coef=1.0, a_liquid=1000.0, a_gas=1.0, eps=eps)
        op.set_field("phi", torch.tensor(phi, device="cuda"))
        run(op, m.n_dofs, argv[3] if len(argv) > 3 else "f32")
    elif kind == "reinit":
        base = int(argv[1]) if len(argv) > 1 else 16
        levels = int(argv[2]) if len(argv) > 2 else 3
        op, m = build_reinit_octree(ctx, base, levels, autotune=False)
        run(op, m.n_dofs, argv[3] if len(argv) > 3 else "f32", int(argv[4]) if len(argv) > 4 else 1)
    else:
        raise SystemExit(f"unknown workload {kind}")


# ----------------------------------------------------------------------------- main

def main():
    if len(sys.argv) > 1 and sys.argv[1] == "--probe":
        probe(sys.argv[2:])
        return
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=400)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--quick", action="store_true", help="the headline workload only")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--suite", action="store_true", help="also the melt-pool Oseen operator and the Q3 solves")
    ap.add_argument("--n", type=int, default=128)
    args = ap.parse_args()
    args.warmup = max(args.warmup, 3)

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if args.impl == "reference":
        out = reference_arm(args, rank, world)
        if out is not None:
            print(json.dumps(out))
        return

    # the oracle's host baseline first: its process pool is spawned before any GPU work
    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline and not args.quick:
        cpu = cpu_oracle_baseline()
        cpu["helmholtz_16_cg"] = cpu_oracle_helmholtz_cg()
        cpu["heat_solve"] = cpu_oracle_heat_solve()

    import torch
    torch.cuda.set_device(local)
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))

    from paper_2501_18781_gb300 import Context, build_library
    import synthetic as syn
    build_library()
    ctx = Context(local)
    op, m, T_prev = build_heat(ctx, args.n)
    n, ncells = op.n, m.n_cells
    src = torch.tensor(syn.uniform_pm1(1, n), device="cuda")
    dst = torch.empty_like(src)
    flush = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")   # > 129 MB L2

    # warm-up and set-up (Gauss-point coefficient tables) outside the timed region; the fp64-accurate
    # apply runs in the arithmetic measured faster here: the fp64 pipes or double-float pairs on the
    # fp32 pipes (both meet the same 1e-12 parity bar)
    pick = {}
    for arith in (None, "df64"):
        for _ in range(args.warmup):
            op.apply(src, dst, arith=arith)
        pick[arith] = statistics.median(time_apply(op, src, dst, 5, 0, flush, arith=arith))
    arith = min(pick, key=pick.get)
    torch.cuda.synchronize()
    if dist:
        dist.barrier()
    torch.cuda.synchronize()
    l0 = ctx.launch_count()
    with ClockSampler(local) as clocks:
        times = time_apply(op, src, dst, args.steps, 0, flush, arith=arith)
    launches = ctx.launch_count() - l0
    variant = op.variant
    total = max_over_ranks(sum(times), dist, "cuda")
    value = whole_job_rate(n, args.steps, world, total)
    mean = total / args.steps

    # end to end through the public API: every step copies its input from pinned host memory to the
    # device, applies the operator and copies the result back to pinned host memory
    e2e_t, e2e_serial_t = e2e_applies(op, src, args.steps, arith)
    e2e_t = max_over_ranks(e2e_t, dist, "cuda")
    e2e = {"value": n * args.steps * world / e2e_t / 1e9, "unit": "GDoF/s",
           "h2d_bytes_per_step": n * 8, "d2h_bytes_per_step": n * 8,
           "pipelined": "the host-to-device copy of step k+1 and the device-to-host copy of step k-1 run on two "
                        "copy streams while step k's apply runs (double-buffered device vectors, event-ordered)",
           "serial_value": n * args.steps * world / max_over_ranks(e2e_serial_t, dist, "cuda") / 1e9}

    peaks = measured_peaks()
    hbm = peaks.get("hbm_gbs", HBM_FALLBACK_GBS)
    if arith == "df64":
        flops = HEAT_DF64_FLOPS_PER_CELL * ncells
        peak, peak_src, key = FP32_PEAK_TFLOPS, "GB300 fp32 pipe: 152 SMs x 128 lanes x 2 x 2.07 GHz (recipe)", "df64"
    else:
        flops = HEAT_FLOPS_PER_CELL["inkernel" if "/inkernel" in variant else "tabulated"] * ncells
        peak, peak_src, key = FP64_PEAK_TFLOPS, "GB300 FP64 rate of the profiling recipe", "f64"
    alg_bytes = HEAT_WORDS_PER_DOF * 8 * n
    achieved = flops / mean / 1e12
    out = {
        "metric": METRIC, "value": value, "unit": "GDoF/s", "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": mean * 1e3, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "df64" if arith == "df64" else "f64", "data": "synthetic",
        "config": {"workload": f"heat_laser_q2_{args.n}", "n_dofs": n, "cells": ncells, "element": "Q2",
                   "arithmetic": ("double-float: fp64 vectors, pairs of fp32 in the kernel" if arith == "df64"
                                  else "fp64") + " (the faster of the two in warm-up; both pass the 1e-12 bar)",
                   "operator": "(rho c_p / dt) M + K(k(T^n)), k = k0 (1 + 0.5 T / T_b), Dirichlet bottom",
                   "parallelism": "replicas" if world > 1 else "single",
                   "l2": "flushed between timed steps (256 MB write); vectors of 136 MB exceed L2",
                   "variant": variant},
        "roofline": {"bound": "alu", "achieved": achieved, "peak": peak, "unit": "TFLOP/s",
                     "frac": achieved / peak, "traffic": ncu_traffic(f"heat_laser_q2_{args.n}/{key}"),
                     "flops_per_launch": flops, "peak_source": peak_src},
        "hbm_roofline": {"achieved": alg_bytes / mean / 1e9, "peak": hbm, "unit": "GB/s",
                         "frac": alg_bytes / mean / 1e9 / hbm, "bytes_per_launch": alg_bytes,
                         "peak_source": "MEASURED_PEAKS.json (of measured)" if "hbm_gbs" in peaks else "fallback"},
        "e2e": e2e, "gpu_launches": launches, "clocks": clocks.summary(),
    }
    if arith == "df64":
        # the pair arithmetic is mostly additions, which fill an fp32-pipe issue slot for one flop:
        # the same work as a fraction of the pipe's instruction rate (one per lane per clock)
        out["roofline"]["issue_frac"] = HEAT_DF64_INSTRUCTIONS_PER_CELL * ncells / mean / 1e12 / (FP32_PEAK_TFLOPS / 2)
        out["roofline"]["fp32_instructions_per_launch"] = HEAT_DF64_INSTRUCTIONS_PER_CELL * ncells
    # the same operator in fp32 (the arithmetic of the mixed solver's inner applies) and in
    # double-float, with their HBM fractions
    src32, dst32 = src.float(), torch.empty(n, dtype=torch.float32, device="cuda")
    t32 = time_apply(op, src32, dst32, max(5, args.steps // 2), 3, flush)
    ms32 = sum(t32) / len(t32) * 1e3
    out["fp32_apply"] = {"value": n / ms32 / 1e6, "unit": "GDoF/s", "ms_per_step": ms32, "variant": op.variant,
                         "hbm_roofline": {"bytes_per_launch": alg_bytes // 2,
                                          "frac": alg_bytes / 2 / (ms32 * 1e-3) / 1e9 / hbm, "peak": hbm},
                         "traffic": ncu_traffic(f"heat_laser_q2_{args.n}/f32")}
    for name, ar in (("f64_apply", None), ("df64_apply", "df64")):
        tt = time_apply(op, src, dst, max(5, args.steps // 2), 3, flush, arith=ar)
        ms = sum(tt) / len(tt) * 1e3
        out[name] = {"value": n / ms / 1e6, "unit": "GDoF/s", "ms_per_step": ms, "variant": op.variant}
        if ar == "df64":
            out[name]["note"] = "fp64 vectors, double-float cell arithmetic on the fp32 pipes"
            out[name]["roofline"] = {"bound": "alu", "unit": "TFLOP/s", "peak": FP32_PEAK_TFLOPS,
                                     "achieved": HEAT_DF64_FLOPS_PER_CELL * ncells / ms / 1e9,
                                     "frac": HEAT_DF64_FLOPS_PER_CELL * ncells / ms / 1e9 / FP32_PEAK_TFLOPS,
                                     "issue_frac": HEAT_DF64_INSTRUCTIONS_PER_CELL * ncells / ms / 1e9 /
                                                   (FP32_PEAK_TFLOPS / 2)}
        else:
            fl = HEAT_FLOPS_PER_CELL["inkernel" if "/inkernel" in op.variant else "tabulated"] * ncells
            out[name]["roofline"] = {"bound": "alu", "unit": "TFLOP/s", "peak": FP64_PEAK_TFLOPS,
                                     "achieved": fl / ms / 1e9, "frac": fl / ms / 1e9 / FP64_PEAK_TFLOPS}
    if rank == 0 and not args.quick:
        out["solve"] = heat_solve_comparison(ctx, op, m, T_prev, args.n)
        del op, m, T_prev, src, dst, src32, dst32
        torch.cuda.empty_cache()
        w = out["workloads"] = {}
        w["oseen_q2q1_interface_64"] = oseen_workload(ctx, flush)
        w["reinit_octree_q2_32_l3"] = reinit_octree_workload(ctx, flush)
        w["helmholtz_sphere_q2_16"] = helmholtz_workload(ctx)
        w["heat_adjoint_q2_64"] = heat_adjoint_workload(ctx, flush)
        w["helmholtz_qk"] = helmholtz_qk(ctx, flush, solves=args.suite)
        w["meltpool_step"] = meltpool_step(ctx, 64, reps=2)
        if args.suite:
            w["oseen_meltpool"] = meltpool_oseen(ctx, 64, flush)
    if cpu is not None:
        out["cpu_baseline"] = cpu
    if rank == 0:
        print(json.dumps(out))
    if dist:
        dist.barrier()
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
