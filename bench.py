#!/usr/bin/env python
"""Throughput of the GB300 DG2 flood solver (cell-updates per second).

Workload: the synthetic floodplain, 2000 x 1000 cells at dx = 2 m (fBm terrain,
Hurst 0.8, 3 m relief, incised sinuous channel, triangular 20 m^3/s inflow
hydrograph peaking at 1 h on a 40 m west-edge segment, Manning 0.035 / 0.05,
transmissive east/south/north edges), started with 1 m of water in the channel
and run to t = 1 h (the hydrograph peak) once by the FP32 DG2-NL path; every
variant then times its steps from that saved state.  A step is one full RK2 time step (friction,
[local limiting], both stages with fluxes, operators, wet-dry treatment,
Courant reduction, time/ledger update) through the C ABI.

The ensemble variant runs 256 members of log-uniform sizes (18.6 M cells) from
dry to t = 1 h in FP32 with one set of launches per step, after the tile-shape
autotuner.  The adjoint variant times the gauge-misfit gradient (Manning field
and 64 inflow knots) of 4000 FP64 DG2-NL steps on 512 x 512 cells with 64
checkpoints against the misfit alone (the adjoint/forward time ratio).

One line of JSON on rank 0.  With --impl reference the CPU oracle is timed
instead (a bounded 500 x 250 sample of the same workload recipe).
"""
import argparse
import json
import os
import subprocess
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "DG2 cell-updates/s (FP64, FP32) & % HBM roofline; adjoint/forward time ratio"
NX, NY, DX = 2000, 1000, 2.0
SPIN_T = 3600.0          # floodplain spin-up (s of simulated time): the hydrograph peak
URBAN_SPIN_T = 30.0      # urban spin-up (s): 600 steps at dt_max 0.05 s
# Unique bytes each kernel must move per cell: the planes it must read and write once.
BYTES_PER_CELL = {
    "fp64": {"friction": 16 * 8, "stage1": {"nl": 21 * 8, "ll": 27 * 8},
             "stage2": {"nl": 30 * 8, "ll": 30 * 8}},
    # FP32 free-surface form: 10 state planes (eta0 as hi + lo), 2 face-topography planes,
    # Manning n; friction is fused into the stages (stage 1 applies it to the U^n it reads),
    # so it moves no bytes of its own.  Stage 1 reads U^n, the beds and n and writes U1 and
    # Q (DG2-LL: the limited slopes; DG2-NL: U^n's discharge modes after friction); stage 2
    # reads U1, the beds, U^n's depth planes and Q (DG2-LL also U^n's average discharges and
    # n, whose friction it recomputes) and writes U^n+1.
    "fp32": {"friction": 0, "stage1": {"nl": (10 + 2 + 1 + 16) * 4, "ll": (10 + 2 + 1 + 16) * 4},
             "stage2": {"nl": (10 + 4 + 6 + 2 + 10) * 4, "ll": (10 + 4 + 6 + 1 + 2 + 10) * 4}},
}
KERNELS = ["friction", "stage1", "stage2"]
# Algorithmic FP64 operations per wet cell (add, mul, div, sqrt, cbrt each one), each
# face flux counted once: measured with oracle/opcount.cpp (friction 111, spatial
# operator 381, limiter 83 per cell; RK combination 18 / 27; Courant rate 8), plus the
# 4 multiplications of the default face revision's thin-limit thresholds.
FLOPS_PER_WET_CELL = {"friction": 111, "stage1": {"nl": 403, "ll": 486},
                      "stage2": {"nl": 420, "ll": 503}}
# DRAM bytes (read + write) per launch of a variant's dominant kernel from one ncu
# capture (summarised in the named profile), valid only for the device sources it
# was taken with: the key is a hash of the stage kernels' sources
# (STAGE_SOURCES), and the roofline's traffic is null once they change.
TRAFFIC = {
    ("fp64_ll", "stage2"): (19_392_256, "fcc4a955a03cdd80",
                            "profiles/stage_kernel_fp64_ll_floodplain2000x1000_t3600.md"),
    ("fp32_ll", "stage1"): (15_138_816, "fcc4a955a03cdd80",
                            "profiles/ens_stage_kernel_fp32_ll_floodplain2000x1000_t3600.md"),
    ("fp32_nl_flooded", "stage1"): (193_274_624, "fcc4a955a03cdd80",
                                    "profiles/ens_stage_kernel_fp32_nl_flooded2000x1000.md"),
}
# FP64 issue rate of GB300 by ncu's peak_sustained (2 DFMA per SM per cycle), used only
# if the live measurement below cannot run
FP64_PEAK_DERIVED = 152 * 2 * 2 * 2.07
FP64_PEAK_REPS, FP64_PEAK_ITERS = 30, 16384


def fp64_peak(B, local):
    """FP64 FMA throughput measured on this GPU (dg2_fp64_fma_peak: independent DFMA
    chains on every SM, CUDA-event timed), median of back-to-back runs over about a
    second, with the SM clock sampled meanwhile."""
    clk = ClockSampler(local)
    clk.start()
    runs = [B.dg2_fp64_fma_peak(4, FP64_PEAK_ITERS)[0] for _ in range(FP64_PEAK_REPS)]
    c = clk.stop()
    return {"gflops": float(np.median(runs)), "max_gflops": float(np.max(runs)),
            "runs": FP64_PEAK_REPS, "clocks": c,
            "how": "dg2_fp64_fma_peak: 4 x 256 threads per SM, 8 independent DFMA chains of "
                   f"{FP64_PEAK_ITERS} per thread, 2 FLOP per FMA, median of "
                   f"{FP64_PEAK_REPS} back-to-back runs"}


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=1000)
    ap.add_argument("--warmup", type=int, default=10)
    ap.add_argument("--impl", default="gb300", choices=["gb300", "reference"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--only", default="", help="comma-separated variant keys (profiling)")
    ap.add_argument("--state-cache", default="",
                    help="npz file holding the spun-up floodplain state: loaded if present, "
                         "else written (lets a profiler run skip the spin-up launches)")
    return ap.parse_args()


def dist_setup(n):
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("gloo")
    return rank, world, local


def barrier(world):
    if world > 1:
        import torch.distributed as dist
        dist.barrier()


def max_over_ranks(x, world):
    if world == 1:
        return x
    import torch
    import torch.distributed as dist
    t = torch.tensor([x], dtype=torch.float64)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


class ClockSampler:
    """nvidia-smi clock / throttle sampling during the timed region."""
    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index):
        self.gpu = gpu_index
        self.proc = None
        self.rows = []

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.gpu), f"--query-gpu={self.Q}", "--format=csv,noheader,nounits",
                 "-lms", "100"], stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except (FileNotFoundError, OSError):
            self.proc = None

    def stop(self):
        if not self.proc:
            return None
        self.proc.terminate()
        try:
            out, _ = self.proc.communicate(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
            out, _ = self.proc.communicate()
        sm, mx, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in out.strip().splitlines():
            f = [x.strip() for x in line.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                mx = float(f[2])
            except ValueError:
                continue
            for nm, v in zip(names, f[5:9]):
                if v.lower() == "active":
                    reasons.add(nm)
        if not sm:
            return None
        return {"sm_mhz": float(np.median(sm)), "sm_max_mhz": mx, "reasons": sorted(reasons),
                "samples": len(sm)}


def workload(nx=NX, ny=NY, dx=DX):
    from paper_2010_02003_gb300 import inputs
    return inputs.floodplain(nx=nx, ny=ny, dx=dx, initial="channel")


def peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            return json.load(f), "measured"
    except (OSError, ValueError):
        return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0}, "fallback"


# The sources the solver's stage kernels are compiled from (the adjoint, the
# no-allocation mass and the FP64 peak probe are separate kernels in files of
# their own and do not enter the hash).
STAGE_SOURCES = ("dg2_api.cu", "dg2_device.cuh", "dg2_ens.cu", "dg2_fs32.cuh",
                 "dg2_fs32_staged.cuh", "dg2_fv.cuh", "dg2_internal.h")


def device_src_hash():
    import hashlib
    h = hashlib.sha256()
    d = os.path.join(ROOT, "paper_2010_02003_gb300", "csrc")
    for f in sorted(STAGE_SOURCES):
        h.update(f.encode())
        with open(os.path.join(d, f), "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()[:16]


def traffic_of(key, kernel):
    """(bytes per launch, profile) if the capture matches the current device sources."""
    t = TRAFFIC.get((key, kernel))
    if t is None or t[1] != device_src_hash():
        return None, None
    return t[0], t[2]


def spun_up(B, case, t_spin, variant=0):
    """State of `case` at t_spin, from its initial state, by the FP32 path's run_to
    (input preparation: not timed)."""
    s = B.solver_from_case(case, variant=variant, precision=1)
    n = s.run_to(t_spin)
    st, t = s.state(), s.time()[0]
    s.close()
    return st, t, n


def kernel_roofline(run, prec, var, cells, peak_gbs, peak_src, key="", fp64=None):
    """Roofline of the dominant kernel of one timed run (live CUDA-event timing).
    FP64: FP64-pipe bound, algorithmic FLOPs per wet cell; FP32: HBM bound, unique
    bytes per cell of the tiles the kernels computed (counted on the device; dry
    tiles are exact fixed points and are skipped)."""
    kms = run["kernel_ms"] / max(run["timed"], 1)
    dom = int(np.argmax(kms))
    names = {"friction": "friction", "stage1": "stage 1", "stage2": "stage 2"}
    kname = f"{prec} {var.upper()} {names[KERNELS[dom]]}"
    kernel_ms = {n: float(k) for n, k in zip(KERNELS, kms)}
    traffic, prof = traffic_of(key, KERNELS[dom])
    if prec == "fp64":
        tab = FLOPS_PER_WET_CELL[KERNELS[dom]]
        per_cell = tab if dom == 0 else tab[var]
        wet = run["wet_fraction"] * cells
        achieved = per_cell * wet / (kms[dom] * 1e-3) / 1e9
        if fp64:
            peak, src = fp64["gflops"], "measured on this GPU (" + fp64["how"] + ")"
        else:
            peak, src = FP64_PEAK_DERIVED, "derived: 152 SMs x 2 DFMA/clk x 2 FLOP x 2.07 GHz"
        return {"bound": "alu", "kernel": kname, "achieved": achieved, "peak": peak,
                "unit": "GFLOP/s", "frac": achieved / peak, "traffic": traffic,
                "traffic_profile": prof, "peak_source": src,
                "flops_per_wet_cell": per_cell, "wet_cells": wet, "kernel_ms": kernel_ms}
    tab = BYTES_PER_CELL[prec][KERNELS[dom]]
    per_cell = tab if dom == 0 else tab[var]
    act = run["active_cells"]
    achieved = per_cell * act / (kms[dom] * 1e-3) / 1e9
    return {"bound": "hbm", "kernel": kname, "achieved": achieved, "peak": peak_gbs,
            "unit": "GB/s", "frac": achieved / peak_gbs, "traffic": traffic,
            "traffic_profile": prof, "peak_source": peak_src,
            "bytes_per_cell": per_cell, "active_cells": act, "kernel_ms": kernel_ms}


def time_variant(B, torch, case, variant, steps, warmup, timing=True, precision=0, start=None,
                 wetdry=0):
    """Device-timed steps of one variant, from `start` = (planes, t), or after running
    the solver itself to t = `start` (a number; untimed spin-up), or from the case's
    initial state (None)."""
    s = B.solver_from_case(case, variant=variant, precision=precision, wetdry=wetdry)
    if isinstance(start, tuple):
        s.set_state(start[0], start[1])
    elif start is not None:
        s.run_to(float(start))
    st = s.stream
    for _ in range(warmup):
        s.step(-1.0)
    torch.cuda.synchronize()
    st0 = s.state()
    wet = float((st0[0] > 1e-5).mean())
    if timing:
        B.dg2_enable_kernel_timing(s.ctx, True)
    tiles0 = s.tile_stats()[3]
    l0 = s.launches()
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    ev0.record(st)
    for _ in range(steps):
        s.step(-1.0)
    ev1.record(st)
    torch.cuda.synchronize()
    ms = ev0.elapsed_time(ev1)
    launches = s.launches() - l0
    kt, n = B.dg2_kernel_times(s.ctx) if timing else (np.zeros(3), 0)
    tiles = s.tile_stats()[3] - tiles0
    t_sim, _ = s.time()
    finite = bool(np.isfinite(s.state()).all())
    return {"solver": s, "ms": ms, "launches": launches, "kernel_ms": kt, "timed": n,
            "wet_fraction": wet,
            "active_cells": int(np.prod(s.tile_shape())) * tiles / max(steps, 1),
            "t_sim": t_sim, "finite": finite}


def e2e_run(B, torch, case, variant, steps, start):
    """Same steps through the public API with host buffers: the start state goes up
    from pinned host memory, the final state and the mass come back, all timed."""
    s = B.solver_from_case(case, variant=variant)
    nx, ny = case.nx, case.ny
    pin_in = torch.empty((9, ny, nx), dtype=torch.float64, pin_memory=True).numpy()
    pin_out = torch.empty((9, ny, nx), dtype=torch.float64, pin_memory=True).numpy()
    pin_in[...] = start[0]
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    B.dg2_set_state(s.ctx, pin_in, start[1])
    for _ in range(steps):
        s.step(-1.0)
    B.dg2_get_state(s.ctx, nx, ny, out=pin_out)
    mass, ledger = s.mass()
    dt_s = time.perf_counter() - t0
    return dt_s, pin_in.nbytes, pin_out.nbytes + 16


CPU_STEPS = 20            # oracle steps timed from the GPU's saved state
CPU_SERIAL_BUDGET_S = 30.0


def _oracle_from(case, start, threads, limiter=True):
    import oracle
    o = oracle.Oracle(case.nx, case.ny, case.dx, case.dy, cfl=case.cfl, limiter=limiter,
                      bc=case.bc, dt_max=case.dt_max, threads=threads)
    o.set_dem(case.z_corner, case.manning, case.n_uniform, case.eta_corner)
    for f in case.inflows:
        o.add_inflow(f.edge, f.s0, f.length, f.t_knots, f.q_knots)
    o.set_state(start[0], start[1])
    return o


def cpu_baseline(case, start, steps=CPU_STEPS):
    """The oracle (FP64 DG2-LL, default face revision) on the GPU's own workload: the
    full floodplain grid from the same saved t = 1 h state the GPU variants step from,
    `steps` Courant steps on every host core (the oracle's OpenMP build: rows in
    parallel, bit-identical to the serial build) and on one core (the serial build,
    stopped after CPU_SERIAL_BUDGET_S if slower).  Every cell counts, as on the GPU."""
    import oracle
    cores = os.cpu_count() or 1
    o = _oracle_from(case, start, threads=True)
    used = oracle.set_threads(cores)
    t0 = time.perf_counter()
    for _ in range(steps):
        o.step()
    el_all = time.perf_counter() - t0
    o1 = _oracle_from(case, start, threads=False)
    n1, t0 = 0, time.perf_counter()
    while n1 < steps and time.perf_counter() - t0 < CPU_SERIAL_BUDGET_S:
        o1.step()
        n1 += 1
    el_1 = time.perf_counter() - t0
    cells = case.nx * case.ny
    return {"value": cells * steps / el_all, "unit": "cell-updates/s", "cores": used,
            "kind": "oracle",
            "value_1core": cells * n1 / el_1,
            "sample": f"{steps} DG2-LL steps of the full {case.nx}x{case.ny} floodplain from the "
                      f"same saved t = {start[1]:.0f} s state the GPU times ({el_all:.1f} s on "
                      f"{used} threads); one core: {n1} steps in {el_1:.1f} s"}


def run_reference(args, rank, world):
    if rank != 0:
        return
    small = workload(500, 250)
    import oracle
    o = oracle.Oracle(small.nx, small.ny, small.dx, small.dy, cfl=small.cfl, limiter=True, bc=small.bc,
                      threads=True)
    cores = oracle.set_threads(os.cpu_count() or 1)
    o.set_dem(small.z_corner, small.manning, small.n_uniform, small.eta_corner)
    for f in small.inflows:
        o.add_inflow(f.edge, f.s0, f.length, f.t_knots, f.q_knots)
    for _ in range(args.warmup):
        o.step()
    t0 = time.perf_counter()
    for _ in range(args.steps):
        o.step()
    el = time.perf_counter() - t0
    v = small.nx * small.ny * args.steps / el
    line = {"impl": "reference", "metric": METRIC, "value": v, "unit": "cell-updates/s",
            "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": 1e3 * el / args.steps, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": "floodplain 500x250 dx=2 m (bounded sample of the 2000x1000 "
                                   "floodplain recipe), DG2-LL, FP64 CPU oracle"},
            "cpu_baseline": {"value": v, "unit": "cell-updates/s", "cores": cores, "kind": "oracle",
                             "sample": f"{args.steps} DG2-LL steps on a 500x250 floodplain (same "
                                       f"recipe, channel start), OpenMP build on {cores} threads"},
            "e2e": {"value": v, "unit": "cell-updates/s", "h2d_bytes_per_step": 0,
                    "d2h_bytes_per_step": 0}}
    print(json.dumps(line))


VARIANTS = [
    # key, workload, variant, precision[, face revision: 1 = as printed in Sec. 2.1.2]
    ("fp64_ll", "floodplain", 1, 0),
    ("fp64_ll_printed", "floodplain", 1, 0, 1),
    ("fp64_nl", "floodplain", 0, 0),
    ("fp32_ll", "floodplain", 1, 1),
    ("fp32_nl", "floodplain", 0, 1),
    ("fp64_nl_flooded", "flooded", 0, 0),
    ("fp32_nl_flooded", "flooded", 0, 1),
    ("fp32_ll_flooded", "flooded", 1, 1),
    ("fp32_nl_urban", "urban", 0, 1),      # 8192 x 8192, rain + point inflow, 500 steps
]
URBAN_STEPS = 500
ENS_MEMBERS, ENS_T_END = 256, 3600.0
ENS_SEQ_SAMPLE, ENS_SEQ_T = 16, 300.0


def ensemble_variant(B, torch, inputs, n=ENS_MEMBERS, t_end=ENS_T_END):
    """The ensemble recipe: n floodplain members of log-uniform sizes, each with its own
    roughness, inflow and Courant step, FP32 DG2-NL, run from dry to t_end in one set of
    launches per step (CUDA graphs), tile shape chosen by the autotuner first.  Timed
    with CUDA events on the ensemble's stream; cell-updates count every cell of every
    member for each of its own steps."""
    cases = inputs.ensemble(n=n)
    mem = [B.solver_from_case(c, variant=B.DG2_NL, precision=B.DG2_FP32) for c in cases]
    ens = B.Ensemble(mem)
    st = ens.stream
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    shape = ens.autotune(t_end, 16)
    torch.cuda.synchronize()
    tune_s = time.perf_counter() - t0
    steps0 = [m.steps() for m in mem]
    tiles0 = [m.tile_stats()[3] for m in mem]
    l0 = ens.launches()
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    ev0.record(st)
    nsteps = ens.run_to(t_end)
    ev1.record(st)
    torch.cuda.synchronize()
    ms = ev0.elapsed_time(ev1)
    upd = sum(c.nx * c.ny * (m.steps() - a) for c, m, a in zip(cases, mem, steps0))
    tiles = sum(m.tile_stats()[3] - a for m, a in zip(mem, tiles0))
    cells = sum(c.nx * c.ny for c in cases)
    wet = sum(float((m.state()[0] > 1e-5).sum()) for m in mem) / cells
    out = {"value": upd / (ms * 1e-3), "unit": "cell-updates/s", "members": n, "cells": cells,
           "t_end_s": t_end, "ensemble_steps": nsteps, "member_cell_updates": upd,
           "ms_total": ms, "ms_per_step": ms / max(nsteps, 1), "tile_shape": list(shape),
           "autotune_ms_per_step": [float(x) for x in ens.tune_times()],
           "autotune_s": tune_s, "launches": ens.launches() - l0,
           "computed_cells": tiles * shape[0] * shape[1], "wet_fraction_end": wet}
    # whole-step HBM figure: unique bytes of both stages per computed cell
    per_cell = sum(v if isinstance(v, int) else v["nl"] for v in BYTES_PER_CELL["fp32"].values())
    out["step_bytes_per_s"] = per_cell * out["computed_cells"] / (ms * 1e-3)
    ens.close()
    for m in mem:
        m.close()
    # the same kind of members one after another through the single-problem path
    seq = inputs.ensemble(n=ENS_SEQ_SAMPLE)
    sol = [B.solver_from_case(c, variant=B.DG2_NL, precision=B.DG2_FP32) for c in seq]
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for s_ in sol:
        s_.run_to(ENS_SEQ_T)
    torch.cuda.synchronize()
    seq_s = time.perf_counter() - t0
    seq_upd = sum(c.nx * c.ny * s_.steps() for c, s_ in zip(seq, sol))
    out["sequential"] = {"members": ENS_SEQ_SAMPLE, "t_end_s": ENS_SEQ_T,
                         "value": seq_upd / seq_s, "unit": "cell-updates/s",
                         "how": "dg2_run_to on each member in turn (host wall clock)"}
    for s_ in sol:
        s_.close()
    return out


ADJ_N, ADJ_STEPS, ADJ_SNAP, ADJ_KNOTS = 512, 4000, 64, 64


def adjoint_variant(B, torch, inputs, steps=ADJ_STEPS, precision=0, ref=None):
    """Discrete adjoint on the calibration recipe: the 512 x 512 floodplain terrain
    (dx 2 m, seed 2014) under a gently tilted free surface (every cell wet: the
    channel start's thin films make the step map chaotic, and its exact derivative
    over 4000 steps grows like its round-off amplification), whose truth is the
    generator's two-zone Manning field and triangular inflow; step sizes frozen from
    a Courant-step run of the truth; 8 gauges sampled every 10 s; misfit against the
    truth's depths at Manning 0.04 everywhere and the inflow's 64 knots at 0.8 x
    truth.  Times the
    misfit alone (forward) and misfit + gradient (forward, checkpointed reverse)
    with CUDA events on the adjoint's stream; the plain FP64 DG2-NL solver doing the
    same steps is timed beside it.  precision 1: the FP32-storage adjoint (FP32 state,
    checkpoints and adjoint fields, FP64 arithmetic), whose gradient is compared with
    the FP64 run's (`ref`)."""
    case = inputs.flooded_plain(ADJ_N, ADJ_N, 2.0, seed=2014)
    s = B.solver_from_case(case, variant=B.DG2_NL, precision=B.DG2_FP64)
    init = s.state()
    dts = np.array([s.step(-1.0, want_dt=True) for _ in range(steps)])
    # the plain solver over the same steps (forced dt), device-timed
    s.set_state(init, 0.0)
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    ev0.record(s.stream)
    for dt in dts:
        s.step(float(dt))
    ev1.record(s.stream)
    torch.cuda.synchronize()
    plain_ms = ev0.elapsed_time(ev1)
    s.close()
    t = np.cumsum(dts)
    samples = [int(np.argmax(t >= m)) + 1 for m in np.arange(10.0, t[-1], 10.0)]
    # 64 knots over the run carrying the truth hydrograph
    f = case.inflows[0]
    tk = np.linspace(0.0, float(t[-1]), ADJ_KNOTS)
    q_true = np.interp(tk, f.t_knots, f.q_knots)
    f.t_knots, f.q_knots = tk, q_true
    truth = B.Adjoint(case, nsnap=ADJ_SNAP, max_steps=steps)
    truth.set_schedule(dts, samples, np.zeros((len(samples), truth.ngauge)))
    _, h_true = truth.forward()
    truth.close()
    a = B.Adjoint(case, nsnap=ADJ_SNAP, max_steps=steps, precision=precision)
    a.set_schedule(dts, samples, h_true)
    man0 = np.full((case.ny, case.nx), 0.04)
    a.set_params(man0, 0.8 * q_true)
    st = a.stream
    torch.cuda.synchronize()
    ev0.record(st)
    J, _ = a.forward()
    ev1.record(st)
    torch.cuda.synchronize()
    fwd_ms = ev0.elapsed_time(ev1)
    f0, r0 = a.counts()
    ev0.record(st)
    J2, gn, gq = a.gradient()
    ev1.record(st)
    torch.cuda.synchronize()
    grad_ms = ev0.elapsed_time(ev1)
    f1, r1 = a.counts()
    a.close()
    out_ref = {}
    if ref is not None:
        out_ref = {"misfit_vs_fp64": abs(J - ref["misfit"]) / ref["misfit"],
                   "grad_manning_vs_fp64": float(np.abs(gn - ref["gn"]).max() /
                                                 np.abs(ref["gn"]).max()),
                   "grad_knots_vs_fp64": float(np.abs(gq - ref["gq"]).max() /
                                               np.abs(ref["gq"]).max())}
    return {**out_ref, "precision": "fp32 storage, fp64 arithmetic" if precision else "fp64",
            "gn": gn, "gq": gq,
            "cells": case.nx * case.ny, "steps": steps, "t_end_s": float(t[-1]),
            "samples": len(samples), "gauges": 8, "knots": ADJ_KNOTS, "checkpoints": ADJ_SNAP,
            "misfit": J, "forward_ms": fwd_ms, "gradient_ms": grad_ms,
            "value": grad_ms / fwd_ms, "unit": "adjoint/forward time ratio",
            "vs_plain_fp64_nl": grad_ms / plain_ms, "plain_fp64_nl_ms": plain_ms,
            "forward_steps_in_gradient": f1 - f0, "reverse_steps": r1 - r0,
            "grad_manning_norm": float(np.linalg.norm(gn)),
            "grad_knots_norm": float(np.linalg.norm(gq))}


SCHEME_WINDOW_S = 120.0   # simulated seconds each scheme runs in the cost comparison
FV_CFL = 0.5              # the Courant bound of the FV schemes' positivity (Sec. 2.2.2)


def timed_window(B, torch, cs, start, kw, span):
    """One scheme's dg2_run_to over `span` simulated seconds from `start` (planes, time),
    timed with CUDA events after 3 warm-up steps."""
    planes, t0 = start[0].copy(), start[1]
    if "scheme" in kw:
        planes[[1, 2, 4, 5, 7, 8]] = 0.0      # the FV schemes hold averages only
    s = B.solver_from_case(cs, **kw)
    try:
        s.set_state(planes, t0)
        for _ in range(3):
            s.step(-1.0)
        t_a = s.time()[0]
        n0, l0 = s.steps(), s.launches()
        ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        ev0.record(s.stream)
        s.run_to(t_a + span)
        ev1.record(s.stream)
        torch.cuda.synchronize()
        ms = ev0.elapsed_time(ev1)
        n = s.steps() - n0
        return {"ms": ms, "steps": n, "ms_per_step": ms / max(n, 1),
                "ms_per_simulated_s": ms / span, "window_s": span, "cells": cs.nx * cs.ny,
                "dx_m": cs.dx, "cfl": kw.get("cfl", cs.cfl), "launches": s.launches() - l0,
                "t_reached": s.time()[0] - t_a}
    finally:
        s.close()
        torch.cuda.empty_cache()


def scheme_cost_variant(B, torch, case, start, coarse_case, coarse_start,
                        window=SCHEME_WINDOW_S):
    """Run-time cost of the schemes over the same simulated window from the same
    state (the GB300 counterpart of the paper's Table 3): DG2-NL, DG2-LL, MUSCL-FV2
    and FV1 in FP64 at 2 m, and DG2-NL on the twice-coarser 4 m grid of the same
    recipe.  Each run is one dg2_run_to (CUDA graphs, own Courant steps), timed
    with CUDA events after 3 warm-up steps.

    MUSCL-FV2 beside the banks can leave the scheme's bounds (a film between two cells
    of opposite discharge); when it does is a matter of rounding.  Its run alone is then
    taken again over half the window: `failed` lists what ended so, and the schemes it is
    divided by are timed over its window too.  Any other scheme's error is the bench's."""
    plan = {"dg2_nl": (case, start, {"variant": B.DG2_NL}),
            "dg2_ll": (case, start, {"variant": B.DG2_LL}),
            "fv2": (case, start, {"scheme": B.DG2_SCHEME_FV2, "cfl": FV_CFL}),
            "fv1": (case, start, {"scheme": B.DG2_SCHEME_FV1, "cfl": FV_CFL}),
            "dg2_nl_4m": (coarse_case, coarse_start, {"variant": B.DG2_NL})}
    runs, failed = {}, []
    for name, what in plan.items():
        span = window
        while name not in runs:
            try:
                runs[name] = timed_window(B, torch, *what, span)
            except B.Dg2Error as e:
                if name != "fv2" or e.code != B.DG2_E_NONFINITE or span < window / 16:
                    raise
                failed.append({"run": name, "window_s": span, "error": str(e)})
                span /= 2
    span = runs["fv2"]["window_s"]

    def r(a, b):
        if runs[b]["window_s"] != runs[a]["window_s"]:
            key = f"{b}_{span:g}s"
            if key not in runs:
                runs[key] = timed_window(B, torch, *plan[b], span)
            b = key
        return runs[a]["ms_per_simulated_s"] / runs[b]["ms_per_simulated_s"]

    ratios = {"dg2_ll/dg2_nl": r("dg2_ll", "dg2_nl"), "fv2/dg2_nl": r("fv2", "dg2_nl"),
              "fv1/dg2_nl": r("fv1", "dg2_nl"), "fv2_2m/dg2_nl_4m": r("fv2", "dg2_nl_4m")}
    short = "" if span == window else f" (fv2 and its ratios: {span:g} s)"
    return {"workload": f"floodplain from t = {start[1]:.0f} s, {window:.0f} s of simulated time"
                        f"{short}, FP64 (DG2 at Cr 0.33, FV at Cr 0.5)",
            "runs": runs, "failed": failed, "time_ratios": ratios}


def main():
    args = parse()
    rank, world, local = dist_setup(args.gpus)
    if args.impl == "reference":
        run_reference(args, rank, world)
        return
    import torch
    from paper_2010_02003_gb300 import binding as B, build as build_mod, inputs
    if not os.path.exists(B.LIB_PATH):
        build_mod.build()
    torch.cuda.set_device(local)
    only = set(args.only.split(",")) if args.only else None
    cases = {"floodplain": workload(), "flooded": inputs.flooded_plain(NX, NY, DX)}
    starts = {"flooded": None}
    if args.state_cache and os.path.exists(args.state_cache):
        z = np.load(args.state_cache)
        st, t, nspin = z["planes"], float(z["t"]), int(z["steps"])
    else:
        st, t, nspin = spun_up(B, cases["floodplain"], SPIN_T)
        if args.state_cache:
            np.savez(args.state_cache, planes=st, t=t, steps=nspin)
    starts["floodplain"] = (st, t)
    if not only or any(k.endswith("urban") for k in only):
        cases["urban"] = inputs.urban()
        starts["urban"] = URBAN_SPIN_T
    cells = NX * NY
    warmup = max(3, args.warmup)
    pk, pk_src = peaks()

    fp64 = None
    try:
        fp64 = fp64_peak(B, local)
    except Exception as e:  # noqa: BLE001 -- reported, the derived peak is used instead
        print(f"FP64 peak measurement failed: {e}", file=sys.stderr)

    results = {}
    clocks = None
    for key, wl, var, prec, *rest in VARIANTS:
        wd = rest[0] if rest else 0
        if only and key not in only:
            continue
        barrier(world)
        clk = ClockSampler(local) if key == "fp64_ll" else None
        if clk:
            clk.start()
        case = cases[wl]
        ncell = case.nx * case.ny
        nsteps = URBAN_STEPS if (wl == "urban" and args.steps >= 50) else args.steps
        run = time_variant(B, torch, case, var, nsteps, warmup, precision=prec, start=starts[wl],
                           wetdry=wd)
        if clk:
            clocks = clk.stop()
        ms = max_over_ranks(run["ms"], world)
        run["value"] = world * ncell * nsteps / (ms * 1e-3)
        run["ms_max"] = ms
        run["steps"] = nsteps
        run["cells"] = ncell
        run["roofline"] = kernel_roofline(run, "fp32" if prec else "fp64", "ll" if var else "nl",
                                          ncell, pk["hbm_gbs"], pk_src, key, fp64)
        run.pop("solver").close()
        results[key] = run
        torch.cuda.empty_cache()

    adj = adj32 = None
    if not only or "fp64_nl_adjoint" in only or "fp32_nl_adjoint" in only:
        barrier(world)
        adj = adjoint_variant(B, torch, inputs)
        torch.cuda.empty_cache()
        if not only or "fp32_nl_adjoint" in only:
            adj32 = adjoint_variant(B, torch, inputs, precision=1, ref=adj)
            torch.cuda.empty_cache()
        for r in (adj, adj32):
            if r is not None:
                r.pop("gn")
                r.pop("gq")

    schemes = None
    if not only or "fp64_schemes" in only:
        barrier(world)
        coarse = workload(NX // 2, NY // 2, 2 * DX)
        cst, ct, _ = spun_up(B, coarse, SPIN_T)
        schemes = scheme_cost_variant(B, torch, cases["floodplain"], starts["floodplain"],
                                      coarse, (cst, ct))

    ens = None
    if not only or "fp32_nl_ensemble" in only:
        barrier(world)
        ens = ensemble_variant(B, torch, inputs)
        if "fp64_nl" in results:
            ens["vs_fp64_single_nl"] = ens["value"] / results["fp64_nl"]["value"]
        torch.cuda.empty_cache()

    if not results:
        if rank == 0:
            extra = {k: v for k, v in (("fp32_nl_ensemble", ens), ("fp64_nl_adjoint", adj),
                                       ("fp32_nl_adjoint", adj32), ("fp64_schemes", schemes))
                     if v}
            print(json.dumps({"metric": METRIC, "variants": extra}))
        return
    head = "fp64_ll" if "fp64_ll" in results else next(iter(results))
    hd = results[head]
    e2e = None
    if not only or "fp64_ll" in only:
        e2e_s, h2d, d2h = e2e_run(B, torch, cases["floodplain"], B.DG2_LL, args.steps,
                                  starts["floodplain"])
        e2e = {"value": world * cells * args.steps / max_over_ranks(e2e_s, world),
               "unit": "cell-updates/s", "h2d_bytes_per_step": h2d / args.steps,
               "d2h_bytes_per_step": d2h / args.steps}

    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        cpu = cpu_baseline(cases["floodplain"], starts["floodplain"])
    if rank == 0:
        variants = {k: {"value": r["value"], "ms_per_step": r["ms_max"] / r["steps"],
                        "steps": r["steps"], "cells": r["cells"],
                        "wet_fraction": r["wet_fraction"], "finite": r["finite"],
                        "roofline": r["roofline"]}
                    for k, r in results.items() if k != head}
        if ens is not None:
            variants["fp32_nl_ensemble"] = ens
        if adj is not None:
            variants["fp64_nl_adjoint"] = adj
        if adj32 is not None:
            variants["fp32_nl_adjoint"] = adj32
        if schemes is not None:
            variants["fp64_schemes"] = schemes
        line = {"metric": METRIC, "value": hd["value"], "unit": "cell-updates/s", "n_gpus": world,
                "steps": hd["steps"], "warmup": warmup, "ms_per_step": hd["ms_max"] / hd["steps"],
                "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
                "dtype": "f64" if head.startswith("fp64") else "f32", "data": "synthetic",
                "config": {"workload": "floodplain 2000x1000 dx=2 m from t=1 h (channel start run to "
                                       "the hydrograph peak), DG2-LL, FP64, default face revision "
                                       "(positivity-consistent revision of partially wet cells, a "
                                       "repair of Sec. 2.1.2's; the printed revision is variant "
                                       "fp64_ll_printed)"
                           if head == "fp64_ll" else head,
                           "variant": head, "cells": cells, "t_start_s": SPIN_T,
                           "spin_up_steps": nspin,
                           "wet_fraction": hd["wet_fraction"],
                           "l2": "inputs larger than L2 (state 2 x 145 MB)",
                           "parallelism": f"replicas x{world}"},
                "variants": variants,
                "gpu_launches": int(hd["launches"]), "roofline": hd["roofline"], "e2e": e2e,
                "cpu_baseline": cpu, "clocks": clocks, "fp64_peak": fp64}
        print(json.dumps(line))
    if world > 1:
        import torch.distributed as dist
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
