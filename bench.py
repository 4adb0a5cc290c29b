#!/usr/bin/env python
"""Benchmark: cell-stage updates/s of the fused HWENO-U stage on 2D Euler 2048^2.

Workload: 2D Euler (gamma = 1.4) on [0,1]^2, 2048 x 2048 cells, 3 moments per component,
seeded 4-quadrant Riemann data (rho, p in [0.1, 2], u, v in [-1, 1]) with an isentropic
vortex (seed 0 + rank), transmissive boundaries, CFL 0.6.  One bench step = one modified
SSP-RK3 time step (dt kernel + three fused stage kernels) over the whole grid; value =
cells * 3 * steps / seconds, timed with CUDA events on the engine's stream.

Arms:
  default            this library (FP64 path is the headline; the FP32-bulk/FP64-weights path
                     is reported alongside with its L1/Linf deviation from the FP64 path)
  --impl reference   the FP64 CPU oracle (a deliberately slow, serial C program) on bounded
                     windows of the same workload, on the host cores
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

N_DEFAULT = 2048
METRIC = "cell-stage updates/s (2D Euler 2048^2, FP32 vs FP64 at stated L1 err); p50/p99 solve"
UNIT = "cell-stage/s"
# Algorithmic FP64 flops per cell-stage of 2D Euler with the characteristic decomposition:
# the oracle's exact count (oracle/flop_count.cpp; tests/test_oracle_flops.py re-derives
# these numbers): the distinct data-dependent additions, subtractions, multiplications,
# divisions and square roots on which a stage's outputs depend, plus the wave speeds of every
# output cell.  Stage 1: 10052 + 26; stages 2 and 3: 10088 + 26 (their convex combination).
ORACLE_FLOPS_STAGE1 = 10078.0
ORACLE_FLOPS_STEP_MEAN = (10078.0 + 2 * 10114.0) / 3.0
# FP64 / FP32 FMA rates used when the library's probe (hweno_fma_peak) cannot run; the probe
# measured 1.19 TFLOP/s FP64 and 74 TFLOP/s FP32 on a GB300 (FMA = 2 flops).
FP64_PEAK_TFLOPS_FALLBACK = 1.19
FP32_PEAK_TFLOPS_FALLBACK = 74.2
# FP64 arithmetic the fused 2D Euler characteristic kernel executes per cell-stage, from the
# ncu thread-instruction counts of one 2048^2 launch in its default geometry (96 x 2 tiles, 22
# bands of 94 columns in 152 segments of 297 band-rows;
# profiles/instruction_counts.md) per updated cell less the 2.5 % of
# redundant ring-cell reconstruction: operations (DFMA + DMUL + DADD) of stage 1, the timed
# launch, 2371 -> 2313 (2337 in stages 2 and 3).  The FP64
# pipe executes one such operation per lane per clock, so its operation rate is half the FMA
# flop rate.
FP64_OPS_PER_CELL_STAGE = 2313.0
# DRAM bytes read + written by the same launch (ncu)
FP64_STAGE_DRAM_BYTES = 499.4e6 + 662.5e6
# FP64 pipe utilisation of the same launch (% of peak sustained, active cycles)
FP64_PIPE_UTIL_NCU = 0.930
# FP32-bulk kernel (same workload, ncu): FP64 arithmetic operations per cell-stage (832 per
# updated cell in its default geometry, 96 x 2 tiles, less 2.5 % ring redundancy; stages 2 and
# 3), FP32 flops, and the DRAM bytes of a stage 1 launch
FP32BULK_FP64_OPS_PER_CELL_STAGE = 812.0
FP32BULK_FP32_FLOPS_PER_CELL_STAGE = 3960.0
FP32BULK_STAGE_DRAM_BYTES = 522.9e6 + 688.4e6
ALGO_BYTES_PER_CELL_STAGE = 277.3   # 12 values read + 12 written (+8 V-hat, stage mean), FP64


def _dist_env():
    return int(os.environ.get("RANK", "0")), int(os.environ.get("WORLD_SIZE", "1")), \
        int(os.environ.get("LOCAL_RANK", "0"))


def max_over_ranks(x: float, world: int, device=None) -> float:
    """The largest value of x over all ranks (the job's time is its slowest rank's); one
    all-reduce, on a CUDA tensor under NCCL or a CPU tensor under gloo."""
    if world <= 1:
        return float(x)
    import torch
    import torch.distributed as dist
    t = torch.tensor([float(x)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def replica_throughput(units_per_rank: float, ms_max: float, world: int) -> float:
    """Weak scaling over independent replicas: every rank processes units_per_rank units in
    its own time; the job's throughput is all units over the slowest rank's time."""
    return world * units_per_rank / (ms_max / 1e3)


def _workload_config(n, extra=None):
    cfg = {"workload": f"2D Euler quadrant+vortex {n}x{n}, 3 moments x 4 components, "
                       f"transmissive, CFL 0.6, SSP-RK3 step = 3 fused stages",
           "cells": n * n, "global_batch": 1, "seq_len": n * n, "parallelism": "replicas",
           "l2": (f"inputs larger than L2 (state {n * n * 96 / 1e6:.0f} MB per buffer), no flush"
                  if n * n * 96 > 129e6 else
                  f"state {n * n * 96 / 1e6:.0f} MB per buffer fits in L2; no flush (the stage "
                  f"kernel is FP64-bound, not memory-bound)")}
    if extra:
        cfg.update(extra)
    return cfg


class ClockSampler:
    """nvidia-smi sampling of SM clocks and throttle reasons during the timed region."""

    def __init__(self, index: int = 0):
        self.index = index
        self.proc = None

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.index),
                 "--query-gpu=clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.hw_slowdown,"
                 "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
                 "clocks_event_reasons.sw_power_cap", "--format=csv,noheader,nounits", "-lms", "200"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except OSError:
            self.proc = None
        return self

    def __exit__(self, *a):
        self.out = ""
        if self.proc:
            self.proc.terminate()
            try:
                self.out, _ = self.proc.communicate(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()
                self.out, _ = self.proc.communicate()

    def summary(self):
        sm, mx, reasons = [], 0.0, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in (getattr(self, "out", "") or "").splitlines():
            f = [x.strip() for x in line.split(",")]
            if len(f) < 7:
                continue
            try:
                sm.append(float(f[0]))
                mx = max(mx, float(f[1]))
            except ValueError:
                continue
            for nm, v in zip(names, f[3:7]):
                if v.lower() == "active":
                    reasons.add(nm)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": mx or None,
                "reasons": sorted(reasons), "samples": len(sm)}


# ------------------------------------------------------------------------------------------
def _host_threads() -> int:
    return max(1, os.cpu_count() or 1)


def run_reference(args):
    """The FP64 oracle on the host cores: each step = one full SSP-RK3 step of the OpenMP
    build (all host cores) on a window of the same seeded 2048^2 state."""
    rank, world, _ = _dist_env()
    if rank != 0:
        return
    import oracle as O
    from paper_2402_03074_gb300 import inputs as I
    win = args.ref_window
    threads = O.threads_available(_host_threads())
    w = I.quadrant_vortex_2d(0, args.n, window=((args.n - win) // 2, (args.n - win) // 2, win, win))
    op = O.Problem(dim=2, eq=O.EULER, nx=w.nx, ny=w.ny, x0=w.x0, x1=w.x1, y0=w.y0, y1=w.y1,
                   bc=w.bc, cfl=0.6)
    U = w.U0.copy()
    t = 0.0
    for _ in range(args.warmup):
        U, t, _, _ = O.step(op, U, t, threads=threads)
    t0 = time.perf_counter()
    for _ in range(args.steps):
        U, t, _, _ = O.step(op, U, t, threads=threads)
    el = time.perf_counter() - t0
    cs = w.nx * w.ny * 3 * args.steps
    val = cs / el
    sample = (f"{args.steps} SSP-RK3 steps of the FP64 C oracle (OpenMP over rows, {threads} "
              f"threads) on the central {win}x{win} window of the seeded {args.n}^2 state "
              f"(same cell size)")
    line = {"metric": METRIC, "value": val, "unit": UNIT, "impl": "reference", "n_gpus": 0,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * el / args.steps,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic (seeded)", "config": _workload_config(args.n),
            "cpu_baseline": {"value": val, "unit": UNIT, "cores": threads, "kind": "oracle",
                             "sample": sample},
            "e2e": {"value": val, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line))


def cpu_baseline(n, seconds_target, c4):
    """The oracle on the host cores: (1) the serial build on one core, SSP-RK3 steps of the
    central 128^2 window of the seeded n^2 state for about seconds_target; (2) the OpenMP
    build on all host cores, the 200-step run of the same generator at c4["n"]^2 (seed 0),
    which is also the reference of the GPU results in c4 (L1 / Linf of the cell averages,
    relative to the mean |average| of each component)."""
    import oracle as O
    from paper_2402_03074_gb300 import inputs as I
    win = 128
    w = I.quadrant_vortex_2d(0, n, window=((n - win) // 2, (n - win) // 2, win, win))
    op = O.Problem(dim=2, eq=O.EULER, nx=w.nx, ny=w.ny, x0=w.x0, x1=w.x1, y0=w.y0, y1=w.y1,
                   bc=w.bc, cfl=0.6)
    U, t, steps = w.U0.copy(), 0.0, 0
    t0 = time.perf_counter()
    while time.perf_counter() - t0 < seconds_target:
        U, t, _, _ = O.step(op, U, t)
        steps += 1
    el = time.perf_counter() - t0
    serial = {"value": win * win * 3 * steps / el, "unit": UNIT, "cores": 1, "kind": "oracle",
              "sample": f"{steps} SSP-RK3 steps of the serial FP64 C oracle on the central "
                        f"{win}x{win} window of the seeded {n}^2 state ({el:.1f} s)"}
    if c4 is None:
        return serial
    threads = O.threads_available(_host_threads())
    m = c4["n"]
    w4 = I.quadrant_vortex_2d(0, m)
    op4 = O.Problem(dim=2, eq=O.EULER, nx=m, ny=m, x0=w4.x0, x1=w4.x1, y0=w4.y0, y1=w4.y1,
                    bc=w4.bc, cfl=0.6)
    t0 = time.perf_counter()
    ref, tref, ns, st = O.run(op4, w4.U0, max_steps=c4["steps"], threads=threads)
    el4 = time.perf_counter() - t0
    scale = np.abs(ref[:, 0]).mean(axis=(1, 2))[:, None, None]
    errs = {}
    for name in ("fp64", "mixed32"):
        d = np.abs(c4[name][:, 0] - ref[:, 0]) / scale
        errs[name] = {"l1": float(d.mean()), "linf": float(d.max())}
    c4_report = {"workload": f"2D Euler quadrant+vortex {m}x{m} (seed 0), {ns} SSP-RK3 steps "
                             f"(CFL 0.6) from identical inputs",
                 "oracle_t": tref, "gpu_t": c4["t"], "fp64_vs_oracle": errs["fp64"],
                 "mixed32_vs_oracle": errs["mixed32"],
                 "note": "L1 / Linf of the cell averages against the FP64 oracle, relative to "
                         "the mean |average| of each component"}
    return {"value": m * m * 3 * ns / el4, "unit": UNIT, "cores": threads, "kind": "oracle",
            "sample": f"{ns} SSP-RK3 steps of the FP64 C oracle (OpenMP over rows, {threads} "
                      f"threads) at {m}^2, the same generator ({el4:.1f} s)",
            "serial": serial, "c4_vs_oracle": c4_report}


# ------------------------------------------------------------------------------------------
def run_ours(args):
    import torch

    rank, world, local = _dist_env()
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", init_method="env://")
        torch.cuda.set_device(local)
    dev = local if world > 1 else 0
    torch.cuda.set_device(dev)
    from paper_2402_03074_gb300 import build as B
    B.build()
    from paper_2402_03074_gb300 import _binding as H
    from paper_2402_03074_gb300 import inputs as I

    n = args.n
    w = I.quadrant_vortex_2d(rank, n)
    U0 = w.U0
    peaks = measure_peaks(H, dev)
    eng = H.hweno_create(device=dev)
    stream = torch.cuda.ExternalStream(H.hweno_engine_stream(eng))

    def barrier():
        torch.cuda.synchronize()
        if world > 1:
            import torch.distributed as dist
            dist.barrier()

    def prob(precision):
        return H.make_problem(dim=2, equation=H.HWENO_EULER, nx=n, ny=n, x0=0.0, x1=1.0, y0=0.0,
                              y1=1.0, bc=w.bc, cfl=0.6, precision=precision)

    def timed_steps(precision, steps, warmup):
        sid = H.hweno_open(eng, prob(precision), U0)
        H.hweno_advance(eng, sid, math.inf, max_steps=warmup)
        barrier()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        H.hweno_advance(eng, sid, math.inf, max_steps=steps)
        e1.record(stream)
        e1.synchronize()
        ms = e0.elapsed_time(e1)
        barrier()
        out = np.empty_like(U0)
        H.hweno_get_state(eng, sid, out)
        H.hweno_close(eng, sid)
        return ms, out

    # launch-geometry autotuner (before any timing, like compilation): the tile shape of the
    # 2D stage kernel for this grid in both precisions, kept in the process's tuning table
    # and used by every later launch of such a problem
    tiles = {}
    if args.tuning_file:
        tiles = {"loaded": args.tuning_file, "entries": H.hweno_tuning_load(args.tuning_file)}
    elif not args.no_autotune:
        for name, prec in (("fp64", H.HWENO_FP64), ("mixed32", H.HWENO_MIXED32)):
            r, b, ms = H.hweno_autotune(eng, prob(prec), U0)
            tq = H.hweno_tuning_query(prob(prec)) or {}
            tiles[name] = {"rows": r, "bands": b, "width": tq.get("width", 0), "stage_ms": ms}
        if args.save_tuning:
            H.hweno_tuning_save(args.save_tuning)

    # headline: FP64 path
    with ClockSampler(dev) as clk:
        ms64, out64 = timed_steps(H.HWENO_FP64, args.steps, args.warmup)
    ms64 = max_over_ranks(ms64, world, device="cuda")
    cell_stages = n * n * 3 * args.steps
    value = replica_throughput(cell_stages, ms64, world)

    # the fused stage kernel alone: per-launch duration from events on its stream
    d = torch.device("cuda", dev)

    def stage_kernel_ms(p):
        Ud = torch.from_numpy(U0).to(d)
        Uo = torch.empty_like(Ud)
        Vh = torch.zeros((4, 2, n, n), dtype=torch.float64, device=d)
        a_in = torch.zeros(2, dtype=torch.float64, device=d)
        H.hweno_alpha_device(p, Ud, a_in, torch.cuda.current_stream().cuda_stream)
        a_out = torch.zeros(2, dtype=torch.float64, device=d)
        torch.cuda.synchronize()
        dtv = 0.6 / ((a_in[0] + a_in[1]).item() * n)
        dtt = torch.tensor([dtv], dtype=torch.float64, device=d)
        st = torch.zeros(1, dtype=torch.int32, device=d)
        ks = torch.cuda.Stream(device=d)
        times = []
        with torch.cuda.stream(ks):
            for rep in range(args.kernel_reps + 1):
                e0 = torch.cuda.Event(enable_timing=True)
                e1 = torch.cuda.Event(enable_timing=True)
                e0.record(ks)
                H.hweno_stage_device(p, 1, Ud, Ud, Vh, Uo, a_in, a_out, dtt, st, ks.cuda_stream)
                e1.record(ks)
                e1.synchronize()
                if rep > 0:
                    times.append(e0.elapsed_time(e1))
        del Ud, Uo, Vh
        return statistics.mean(times)

    p64 = prob(H.HWENO_FP64)
    k_ms = stage_kernel_ms(p64)

    # FP32-bulk / FP64-weights path on identical inputs
    mixed = None
    if not args.no_mixed:
        ms32, out32 = timed_steps(H.HWENO_MIXED32, args.steps, args.warmup)
        diff = np.abs(out32[:, 0] - out64[:, 0])
        scale = np.abs(out64[:, 0]).mean(axis=(1, 2))[:, None, None]
        k32_ms = stage_kernel_ms(prob(H.HWENO_MIXED32))
        ops32 = FP32BULK_FP64_OPS_PER_CELL_STAGE * n * n / (k32_ms / 1e3) / 1e12
        pipe64 = peaks["fp64_tflops"] / 2.0
        mixed = {"value": world * cell_stages / (ms32 / 1e3), "unit": UNIT, "dtype": "f32+f64",
                 "ms_per_step": ms32 / args.steps,
                 "roofline": {"bound": "alu (FP64 share)", "unit": "TOP/s (FP64 operations)",
                              "kernel_ms": k32_ms, "achieved": ops32, "peak": pipe64,
                              "frac": ops32 / pipe64,
                              "fp64_ops_per_cell_stage": FP32BULK_FP64_OPS_PER_CELL_STAGE,
                              "fp32_tflops": FP32BULK_FP32_FLOPS_PER_CELL_STAGE * n * n /
                                             (k32_ms / 1e3) / 1e12,
                              "fp32_peak_tflops": peaks["fp32_tflops"],
                              "traffic": FP32BULK_STAGE_DRAM_BYTES if n == 2048 else None,
                              "peak_note": "FP64 pipe operation rate = half the FMA flop rate "
                                           "measured by hweno_fma_peak in this run"},
                 "l1_vs_fp64": float((diff / scale).mean()),
                 "linf_vs_fp64": float((diff / scale).max()),
                 "error_note": "relative to the mean |average| of each component, after the "
                               "timed steps from identical inputs; FP64 path = oracle to 1e-12"}

    longr = None
    if args.long_steps > 0:
        longr = long_runs(H, I, eng, stream, U0, w.bc, n, args.long_steps,
                          autotune=not args.no_autotune)

    # end to end through the C ABI with host buffers: per step H2D of the state from pinned
    # memory, one step, D2H of the new state
    e2e = None
    if not args.no_e2e:
        pin = torch.empty(U0.shape, dtype=torch.float64, pin_memory=True).numpy()
        pin[...] = U0
        sid = H.hweno_open(eng, p64, pin)
        tsim = 0.0

        def e2e_step(tsim):
            H.hweno_set_state(eng, sid, pin, tsim)
            H.hweno_step(eng, sid)
            return H.hweno_get_state(eng, sid, pin)[1]
        tsim = e2e_step(tsim)   # untimed: the first pass through each entry point
        torch.cuda.synchronize()
        barrier()
        t0 = time.perf_counter()
        for _ in range(args.e2e_steps):
            tsim = e2e_step(tsim)
        torch.cuda.synchronize()
        el = time.perf_counter() - t0
        H.hweno_close(eng, sid)
        e2e = {"value": world * n * n * 3 * args.e2e_steps / el, "unit": UNIT,
               "h2d_bytes_per_step": int(U0.nbytes), "d2h_bytes_per_step": int(U0.nbytes),
               "steps": args.e2e_steps}
    # the 200-step C4 run at a size the OpenMP oracle finishes in seconds (the oracle's side
    # runs in the cpu_baseline leg, after every GPU measurement)
    c4small = None
    if world == 1 and not args.no_cpu_baseline and args.c4_oracle_n > 0:
        m = args.c4_oracle_n
        w4 = I.quadrant_vortex_2d(0, m)
        c4small = {"n": m, "steps": args.c4_oracle_steps}
        for name, prec in (("fp64", H.HWENO_FP64), ("mixed32", H.HWENO_MIXED32)):
            p = H.make_problem(dim=2, equation=H.HWENO_EULER, nx=m, ny=m, x0=w4.x0, x1=w4.x1,
                               y0=w4.y0, y1=w4.y1, bc=w4.bc, cfl=0.6, precision=prec)
            sid = H.hweno_open(eng, p, w4.U0)
            H.hweno_advance(eng, sid, math.inf, max_steps=args.c4_oracle_steps)
            c4small[name], tt = H.hweno_get_state(eng, sid, np.empty_like(w4.U0))
            H.hweno_close(eng, sid)
            if name == "fp64":
                c4small["t"] = tt
    c1 = c1_timing(H, I, eng, stream) if not args.no_c1 else None
    H.hweno_destroy(eng)

    served = served_small = None
    budget = 150 * 10**9  # the served configuration's HBM admission budget
    factory = lambda: H.hweno_create(device=dev, hbm_budget_bytes=budget)  # noqa: E731
    if not args.no_served:
        served = served_stream(H, I, factory, args.served_m, args.served_rate,
                               [int(g) for g in args.served_grids.split(",")],
                               args.served_tlo, args.served_thi, seed=rank)
    if not args.no_served_small:
        served_small = served_stream(H, I, factory, args.served_m, args.served_rate,
                                     [128, 256, 384, 512], 0.02, 0.05, seed=rank)
    tubes = None
    if not args.no_tubes:
        tubes = tubes_1d(H, I, lambda: H.hweno_create(device=dev), args.tubes, args.tubes_n,
                         args.tubes_t, autotune=not args.no_autotune)

    if rank != 0:
        return
    # ALU roofline of the FP64 stage kernel: the oracle's algorithmic FP64 flops of the timed
    # launch (stage 1) per second against the FP64 FMA flop rate measured in this run; the
    # FP64-pipe view beside it counts the operations the kernel itself executes (ncu)
    tflops = ORACLE_FLOPS_STAGE1 * n * n / (k_ms / 1e3) / 1e12
    ops = FP64_OPS_PER_CELL_STAGE * n * n / (k_ms / 1e3) / 1e12
    roofline = {"bound": "alu", "unit": "TFLOP/s (FP64)", "achieved": tflops,
                "peak": peaks["fp64_tflops"], "frac": tflops / peaks["fp64_tflops"],
                "traffic": FP64_STAGE_DRAM_BYTES if n == 2048 else None,
                "kernel": "stage2d_kernel<EULER, characteristic, double>",
                "kernel_ms": k_ms, "flops_per_cell_stage": ORACLE_FLOPS_STAGE1,
                "flops_note": "the oracle's exact count for stage 1 (distinct data-dependent "
                              "FP64 operations its outputs depend on, plus the output wave "
                              "speeds); the kernel needs fewer: FMAs, shared subexpressions",
                "peak_note": peaks["source"],
                "fp64_pipe": {"unit": "TOP/s (FP64 operations the kernel executes)",
                              "ops_per_cell_stage": FP64_OPS_PER_CELL_STAGE,
                              "achieved": ops, "peak": peaks["fp64_tflops"] / 2.0,
                              "frac": ops / (peaks["fp64_tflops"] / 2.0),
                              "ncu_pipe_util": FP64_PIPE_UTIL_NCU},
                "hbm_GBps": ALGO_BYTES_PER_CELL_STAGE * n * n / (k_ms / 1e3) / 1e9,
                "hbm_frac": ALGO_BYTES_PER_CELL_STAGE * n * n / (k_ms / 1e3) / 1e9 /
                            peaks["hbm_gbs"] if peaks.get("hbm_gbs") else None}
    # launches in the timed region: hweno_advance replays a captured graph of four steps (dt +
    # three stage kernels each), ceil(K / 4) times for K steps; the steps past the limit in the
    # last replay launch and return at once
    line = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": ms64 / args.steps, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic (seeded)",
            "config": _workload_config(n, {"tile_shape": tiles or "default"}),
            "gpu_launches": 16 * math.ceil(args.steps / 4),
            "clocks": clk.summary(), "roofline": roofline, "mixed32": mixed, "e2e": e2e,
            "served": served, "served_small": served_small, "tubes_1d": tubes,
            "long_runs": longr, "c1_advection": c1, "peaks_measured": peaks}
    if world == 1 and not args.no_cpu_baseline:
        line["cpu_baseline"] = cpu_baseline(n, args.cpu_seconds, c4small)
    print(json.dumps(line))


def c1_timing(H, I, eng, stream, reps=3):
    """Linear advection u_t + u_x = 0, u0 = 0.5 + sin(pi x) on [0, 2], N = 200, CFL 0.6, T = 2
    (334 steps, the last one clipped): microseconds per SSP-RK3 step through hweno_advance
    (graph replays of four steps, the host reading the step scalars between replays), CUDA
    events on the engine's stream, best of `reps` runs after one untimed one; and the error of
    the result against the exact translated solution."""
    import torch
    w = I.advection_sine_1d(200)
    p = H.make_problem(dim=1, equation=H.HWENO_ADVECTION, nx=200, x0=0.0, x1=2.0, ax=1.0,
                       cfl=0.6)
    best, steps, out = float("inf"), 0, None
    for rep in range(reps + 1):
        sid = H.hweno_open(eng, p, w.U0)
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        steps = H.hweno_advance(eng, sid, 2.0)
        e1.record(stream)
        e1.synchronize()
        out, _ = H.hweno_get_state(eng, sid, np.empty_like(w.U0))
        H.hweno_close(eng, sid)
        if rep > 0:
            best = min(best, e0.elapsed_time(e1))
    e = np.abs(out[0, 0] - I.advection_exact_1d(200, 2.0)[0, 0])
    return {"workload": "1D linear advection, u0 = 0.5 + sin(pi x) on [0, 2], N = 200, periodic, "
                        "CFL 0.6, T = 2", "steps": steps, "us_per_step": best * 1e3 / steps,
            "l1_vs_exact": float(e.mean()), "linf_vs_exact": float(e.max())}


def measure_peaks(H, dev):
    """FP64 and FP32 FMA rates of this GPU from the library's FMA-chain probe, and its HBM
    copy bandwidth (bytes read + written by a 2 GiB device-to-device copy, best of five)."""
    import torch
    out = {}
    try:
        out["fp64_tflops"] = H.hweno_fma_peak(dev, True) / 1e12
        out["fp32_tflops"] = H.hweno_fma_peak(dev, False) / 1e12
        out["source"] = "FMA rates measured in this run by hweno_fma_peak (FMA chains on every SM)"
    except Exception as e:   # the probe failed: use an earlier measurement and say so
        out["fp64_tflops"] = FP64_PEAK_TFLOPS_FALLBACK
        out["fp32_tflops"] = FP32_PEAK_TFLOPS_FALLBACK
        out["source"] = f"earlier FMA-chain measurement (probe failed: {e})"
    a = torch.empty(2 ** 28, dtype=torch.float64, device=torch.device("cuda", dev))
    b = torch.empty_like(a)
    a.fill_(1.0)
    best = float("inf")
    for rep in range(6):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        b.copy_(a)
        e1.record()
        e1.synchronize()
        if rep > 0:
            best = min(best, e0.elapsed_time(e1))
    out["hbm_gbs"] = 2.0 * a.numel() * 8 / (best / 1e3) / 1e9
    del a, b
    return out


def served_stream(H, I, eng_factory, m, rate, grids, t_lo, t_hi, seed=0):
    """Seeded Poisson stream of 2D Euler solves served by continuous batching, and the same
    requests through the plain per-solve FP64 loop.  Returns the report dict."""
    rng = np.random.default_rng(seed)
    arrive = np.cumsum(rng.exponential(1.0 / rate, size=m))
    ns = rng.choice(grids, size=m)
    Ts = rng.uniform(t_lo, t_hi, size=m)
    kinds = rng.integers(0, 2, size=m)         # 0 quadrant Riemann + vortex, 1 periodic vortex
    precs = rng.integers(0, 2, size=m)         # 0 FP64, 1 FP32 bulk / FP64 weights
    reqs = []
    for q in range(m):
        n = int(ns[q])
        w = I.quadrant_vortex_2d(seed + 100 + q, n) if kinds[q] == 0 else I.vortex_periodic_2d(n)
        p = H.make_problem(dim=2, equation=H.HWENO_EULER, nx=n, ny=n, x0=w.x0, x1=w.x1, y0=w.y0,
                           y1=w.y1, bc=w.bc, cfl=0.6, t_end=float(Ts[q]),
                           precision=H.HWENO_MIXED32 if precs[q] else H.HWENO_FP64)
        reqs.append((w, p))

    def stats(fin, t0):
        tts = np.array([fin[q] - (t0 + arrive[q]) for q in range(m)])
        span = max(fin.values()) - (t0 + arrive[0])
        return {"solves_per_s": m / span, "p50_s": float(np.percentile(tts, 50)),
                "p99_s": float(np.percentile(tts, 99)), "makespan_s": span}

    # continuous batching
    eng = eng_factory()
    t0 = time.perf_counter()
    submitted, live, fin, cell_stages = 0, {}, {}, 0
    while len(fin) < m:
        now = time.perf_counter() - t0
        while submitted < m and arrive[submitted] <= now:
            w, p = reqs[submitted]
            live[H.hweno_submit(eng, p, w.U0)] = submitted
            submitted += 1
        if not live:
            time.sleep(max(0.0, min(0.01, arrive[submitted] - now)))
            continue
        H.hweno_serve(eng, 8)
        for tk in list(live):
            q = live[tk]
            out = np.empty(reqs[q][0].U0.shape)
            rc, info = H.hweno_poll(eng, tk, out)
            if rc == H.HWENO_OK:
                fin[q] = time.perf_counter()
                cell_stages += reqs[q][1].nx * reqs[q][1].ny * 3 * info.steps
                del live[tk]
    H.hweno_destroy(eng)
    served = stats(fin, t0)
    served["cell_stages_per_s"] = cell_stages / served["makespan_s"]

    # plain per-solve FP64 loop, same requests and arrival times
    eng = eng_factory()
    t0 = time.perf_counter()
    fin = {}
    for q in range(m):
        now = time.perf_counter() - t0
        if arrive[q] > now:
            time.sleep(arrive[q] - now)
        w, p = reqs[q]
        p.precision = H.HWENO_FP64
        sid = H.hweno_open(eng, p, w.U0)
        H.hweno_advance(eng, sid, p.t_end)
        H.hweno_get_state(eng, sid, np.empty_like(w.U0))
        H.hweno_close(eng, sid)
        fin[q] = time.perf_counter()
    H.hweno_destroy(eng)
    plain = stats(fin, t0)
    return {"requests": m, "rate_per_s": rate, "grids": [int(g) for g in grids],
            "hbm_budget_bytes": 150 * 10**9,
            "t_end_range": [t_lo, t_hi], "mixed_fraction": float(precs.mean()),
            "served": served, "plain_fp64_loop": plain,
            "speedup_solves_per_s": served["solves_per_s"] / plain["solves_per_s"]}


def long_runs(H, I, eng, stream, U0, bc, n, steps, autotune=True):
    """The long 2D Euler runs: `steps` FP64 steps of the 1024^2 quadrant + vortex state (seed
    1) with its conservation drift (transmissive: the net boundary flux), and `steps` steps of
    the n^2 state in FP64 and in the FP32-bulk path from identical inputs, with the L1 / Linf
    deviation of the FP32-bulk result (relative to the mean |average| of each component).  The
    FP64 GPU path stands in for the FP64 oracle here (they agree within 1e-12 per stage; the
    serial oracle would need hours for these runs)."""
    import torch

    def run(p, U):
        sid = H.hweno_open(eng, p, U)
        S0, A0 = H.hweno_conservation(eng, sid, 4)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        H.hweno_advance(eng, sid, math.inf, max_steps=steps)
        e1.record(stream)
        e1.synchronize()
        ms = e0.elapsed_time(e1)
        S1, _ = H.hweno_conservation(eng, sid, 4)
        out, t = H.hweno_get_state(eng, sid, np.empty_like(U))
        H.hweno_close(eng, sid)
        return out, t, ms, float((np.abs(S1 - S0) / A0).max())

    w3 = I.quadrant_vortex_2d(1, 1024)
    p3 = H.make_problem(dim=2, equation=H.HWENO_EULER, nx=1024, ny=1024, bc=w3.bc, cfl=0.6)
    if autotune:
        H.hweno_autotune(eng, p3, w3.U0)
    _, t3, ms3, drift3 = run(p3, w3.U0)
    res = {"c3": {"workload": f"2D Euler quadrant+vortex 1024x1024 (seed 1), FP64, {steps} steps",
                  "cell_stages_per_s": 1024 * 1024 * 3 * steps / (ms3 / 1e3), "t": t3,
                  "conservation_drift": drift3}}
    rec = {}
    for name, prec in (("fp64", H.HWENO_FP64), ("mixed32", H.HWENO_MIXED32)):
        p = H.make_problem(dim=2, equation=H.HWENO_EULER, nx=n, ny=n, bc=bc, cfl=0.6,
                           precision=prec)
        rec[name] = run(p, U0)
    diff = np.abs(rec["mixed32"][0][:, 0] - rec["fp64"][0][:, 0])
    scale = np.abs(rec["fp64"][0][:, 0]).mean(axis=(1, 2))[:, None, None]
    res["c4"] = {"workload": f"2D Euler quadrant+vortex {n}x{n} (seed 0), {steps} steps, FP64 and "
                             f"FP32-bulk from identical inputs",
                 "fp64_cell_stages_per_s": n * n * 3 * steps / (rec["fp64"][2] / 1e3),
                 "mixed32_cell_stages_per_s": n * n * 3 * steps / (rec["mixed32"][2] / 1e3),
                 "t_fp64": rec["fp64"][1], "t_mixed32": rec["mixed32"][1],
                 "l1_mixed32_vs_fp64": float((diff / scale).mean()),
                 "linf_mixed32_vs_fp64": float((diff / scale).max())}
    return res


def tubes_1d(H, I, eng_factory, tubes, n, t_end, autotune=True):
    """1D Euler shock tubes (seeds 0..tubes-1, n cells, to t_end): one tube alone in the
    default 1D layout and, after the autotuner has picked the block width and threads per
    cell for this grid, in the tuned one (microseconds per step, host clock around
    hweno_advance); every tube through the plain per-solve FP64 loop (one graph-replayed step
    sequence per tube, one after the other, tuned layout), and all tubes at once through the
    served path (one persistent launch per stage over the blocks of every tube, one thread per
    cell).  Returns the report dict."""
    ws = [I.shock_tube_1d(sd, n=n, t_end=t_end) for sd in range(tubes)]
    probs = [H.make_problem(dim=1, equation=H.HWENO_EULER, nx=n, x0=w.x0, x1=w.x1, bc=w.bc,
                            cfl=0.6, t_end=t_end) for w in ws]
    eng = eng_factory()

    def one_tube():
        sid = H.hweno_open(eng, probs[0], ws[0].U0)
        t0 = time.perf_counter()
        st = H.hweno_advance(eng, sid, t_end)
        el = time.perf_counter() - t0
        out, _ = H.hweno_get_state(eng, sid, np.empty_like(ws[0].U0))
        H.hweno_close(eng, sid)
        return 1e6 * el / st, out
    runs = [one_tube() for _ in range(2)]
    single = {"default_layout_us_per_step": min(r[0] for r in runs)}
    tube0_default = runs[0][1]
    if autotune:
        width, lanes, ms = H.hweno_autotune(eng, probs[0], ws[0].U0)
        single["tuned_layout"] = {"block_width": width, "threads_per_cell": lanes,
                                  "stage_us": 1e3 * ms}
        single["tuned_layout_us_per_step"] = min(one_tube()[0] for _ in range(2))
    plain_out, steps = [], 0
    t0 = time.perf_counter()
    for w, p in zip(ws, probs):
        sid = H.hweno_open(eng, p, w.U0)
        steps += H.hweno_advance(eng, sid, t_end)
        out, _ = H.hweno_get_state(eng, sid, np.empty_like(w.U0))
        H.hweno_close(eng, sid)
        plain_out.append(out)
    el_plain = time.perf_counter() - t0
    H.hweno_destroy(eng)
    eng = eng_factory()
    t0 = time.perf_counter()
    tks = [H.hweno_submit(eng, p, w.U0) for w, p in zip(ws, probs)]
    done, served_out, steps_b = {}, {}, 0
    while len(done) < len(tks):
        H.hweno_serve(eng, 64)
        for q, tk in enumerate(tks):
            if q in done:
                continue
            out = np.empty_like(ws[q].U0)
            rc, info = H.hweno_poll(eng, tk, out)
            if rc == H.HWENO_OK:
                done[q] = info.steps
                served_out[q] = out
    el_b = time.perf_counter() - t0
    H.hweno_destroy(eng)
    steps_b = sum(done.values())
    diff = 0.0
    for q, w in enumerate(ws):
        S = np.abs(w.U0[:, 0]).max(axis=(1, 2)).reshape(-1, 1, 1, 1)
        diff = max(diff, float((np.abs(served_out[q] - plain_out[q]) /
                                np.maximum(np.abs(plain_out[q]), S)).max()))
    S0 = np.abs(ws[0].U0[:, 0]).max(axis=(1, 2)).reshape(-1, 1, 1, 1)
    same_layout = float((np.abs(served_out[0] - tube0_default) /
                         np.maximum(np.abs(tube0_default), S0)).max())
    cs = lambda st: st * n * 3
    return {"workload": f"{tubes} seeded 1D Euler shock tubes, {n} cells each, T = {t_end}",
            "single_tube": single,
            "steps": steps, "plain_fp64_loop": {"seconds": el_plain,
                                                "cell_stages_per_s": cs(steps) / el_plain},
            "batched": {"seconds": el_b, "cell_stages_per_s": cs(steps_b) / el_b},
            "speedup": el_plain / el_b, "max_rel_diff_batched_vs_plain": diff,
            "tube0_batched_vs_plain_same_layout": same_layout,
            "diff_note": "the batched path and the default single-solve layout run the same "
                         "operations (bitwise equal in FP64, whatever the threads per cell)",
            "same_steps": steps_b == steps}


def run_paper_tables(args):
    """The paper's accuracy examples at their finest mesh (240 cells per direction) to their end
    times at CFL 0.6, FP64: GPU wall time per run (host clock, state upload to result
    download) and L1 / Linf error of the cell averages against the exact solution, next to
    the paper's serial CPU time of the same mesh (Tables 3.1, 3.3, 3.4, 3.6; context only: the
    paper does not state its time step or time unit)."""
    import torch
    from paper_2402_03074_gb300 import build as B
    B.build()
    from paper_2402_03074_gb300 import _binding as H
    from paper_2402_03074_gb300 import inputs as I
    n = 240
    cases = [
        ("Table 3.1, 1D Burgers", I.burgers_sine_1d(n), H.HWENO_BURGERS,
         lambda t: I.burgers_exact_1d(n, t), 1.56e-01),
        ("Table 3.3, 1D Euler", I.euler_density_wave_1d(n), H.HWENO_EULER,
         lambda t: I.euler_density_wave_exact_1d(n, t), 1.34e01),
        ("Table 3.4, 2D Burgers", I.burgers_sine_2d(n), H.HWENO_BURGERS,
         lambda t: I.burgers_exact_2d(n, t), 3.69e02),
        # the wavenumber whose errors Table 3.6 prints: sin(pi (x + y) / 2), not the
        # sin(pi (x + y)) of the example's text
        ("Table 3.6, 2D Euler", I.euler_density_wave_2d(n, k=0.5), H.HWENO_EULER,
         lambda t: I.euler_density_wave_exact_2d(n, t, k=0.5), 2.14e05),
    ]
    eng = H.hweno_create()
    for name, w, eq, exact, paper_s in cases:
        p = H.make_problem(dim=w.dim, equation=eq, nx=w.nx, ny=w.ny, x0=w.x0, x1=w.x1,
                           y0=w.y0, y1=w.y1, bc=w.bc, cfl=0.6)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        sid = H.hweno_open(eng, p, w.U0)
        steps = H.hweno_advance(eng, sid, w.t_end)
        out, t = H.hweno_get_state(eng, sid, np.empty_like(w.U0))
        el = time.perf_counter() - t0
        H.hweno_close(eng, sid)
        e = np.abs(out[0, 0] - exact(w.t_end)[0, 0])
        print(json.dumps({"case": name, "mesh": n, "t_end": w.t_end, "steps": steps,
                          "gpu_seconds": el, "l1": float(e.mean()), "linf": float(e.max()),
                          "paper_cpu_time": paper_s}), flush=True)
    H.hweno_destroy(eng)


def run_dt_sweep(args):
    """Time-step dependence of the paper's 2D accuracy examples (Tables 3.4-3.6), FP64: the
    error against the exact solution of Example 3.3 (2D Burgers, T = 0.5/pi) and Example 3.4
    (2D Euler density wave, T = 2, at the printed wavenumber and at half of it) at 40^2,
    80^2, 120^2, for dt = c dx with c in {0.1, 0.02, 0.005} and for the CFL 0.6 rule, with the
    scale-invariant weights (Eq. 2.22) and the linear weights; for Euler at the printed
    wavenumber also the original weights and the component-wise reconstruction.  One JSON line
    per run, beside the printed values."""
    from paper_2402_03074_gb300 import build as B
    B.build()
    from paper_2402_03074_gb300 import _binding as H
    from paper_2402_03074_gb300 import inputs as I
    with open(os.path.join(ROOT, "tests", "golden", "paper_tables.json")) as f:
        tables = json.load(f)
    eng = H.hweno_create()
    variants = {"scale-invariant": (H.HWENO_W_SCALE_INVARIANT, 1),
                "linear": (H.HWENO_W_LINEAR, 1),
                "original": (H.HWENO_W_ORIGINAL, 1),
                "scale-invariant, component-wise": (H.HWENO_W_SCALE_INVARIANT, 0)}
    cases = [("Table 3.4, 2D Burgers", H.HWENO_BURGERS, n, I.burgers_sine_2d(n),
              lambda n, t: I.burgers_exact_2d(n, t), "table_3_4_burgers_2d",
              ("scale-invariant", "linear")) for n in (40, 80, 120)]
    # Example 3.4 at the printed wavenumber sin(pi (x + y)) and at sin(pi (x + y) / 2), whose
    # errors Table 3.6 prints
    for kk in (1.0, 0.5):
        cases += [(f"Table 3.6, 2D Euler, k = {kk}", H.HWENO_EULER, n,
                   I.euler_density_wave_2d(n, k=kk),
                   lambda n, t, kk=kk: I.euler_density_wave_exact_2d(n, t, k=kk),
                   "table_3_6_euler_2d", tuple(variants) if kk == 1.0 else
                   ("scale-invariant", "linear")) for n in (40, 80, 120)]
    for name, eq, n, w, exact, key, names in cases:
        ex = exact(n, w.t_end)
        printed = tables[key].get(str(n))
        for c in ("cfl0.6", 0.1, 0.02, 0.005):
            for vname in names:
                wm, ch = variants[vname]
                p = H.make_problem(dim=2, equation=eq, nx=n, ny=n, x0=w.x0, x1=w.x1, y0=w.y0,
                                   y1=w.y1, bc=w.bc, cfl=0.6, weights=wm, characteristic=ch,
                                   dt_fixed=0.0 if c == "cfl0.6" else c * (w.x1 - w.x0) / n)
                sid = H.hweno_open(eng, p, w.U0)
                steps = H.hweno_advance(eng, sid, w.t_end)
                out, t = H.hweno_get_state(eng, sid, np.empty_like(w.U0))
                H.hweno_close(eng, sid)
                e = np.abs(out[0, 0] - ex[0, 0])
                rec = {"case": name, "mesh": n, "dt": c if c == "cfl0.6" else f"{c} dx",
                       "weights": vname, "steps": steps, "l1": float(e.mean()),
                       "linf": float(e.max()), "paper_l1": printed["l1"],
                       "paper_linf": printed["linf"]}
                if eq == H.HWENO_BURGERS:
                    ev = np.abs(out[0, 1] - ex[0, 1])
                    rec["first_moment_l1"] = float(ev.mean())
                    rec["first_moment_linf"] = float(ev.max())
                print(json.dumps(rec), flush=True)
    H.hweno_destroy(eng)


def run_sweep(args):
    """Convergence of the FP64 and FP32-bulk paths on the periodic isentropic vortex
    (rho = p = 1, u = v = 1 plus the vortex, [0,1]^2, T = 0.05) against the exact translated
    solution, N = 128 .. 2048; dt = 0.6 dx / 4 (N0 / N)^(2/3) so that the RK3 error does not
    mask fifth order (the paper fixes only CFL 0.6)."""
    import torch
    from paper_2402_03074_gb300 import build as B
    B.build()
    from paper_2402_03074_gb300 import _binding as H
    from paper_2402_03074_gb300 import inputs as I
    T = args.sweep_T
    sizes = [int(x) for x in args.sweep_sizes.split(",")]
    eng = H.hweno_create()
    rows = []
    for n in sizes:
        w = I.vortex_periodic_2d(n, t_end=T)
        ex = I.vortex_periodic_exact_2d(n, T)
        dt = 0.6 / n / 4.0 * (sizes[0] / n) ** (2.0 / 3.0)
        rec = {"n": n}
        for name, prec in (("fp64", H.HWENO_FP64), ("mixed32", H.HWENO_MIXED32)):
            p = H.make_problem(dim=2, equation=H.HWENO_EULER, nx=n, ny=n, x0=0, x1=1, y0=0, y1=1,
                               dt_fixed=dt, precision=prec)
            sid = H.hweno_open(eng, p, w.U0)
            t0 = time.perf_counter()
            steps = H.hweno_advance(eng, sid, T)
            el = time.perf_counter() - t0
            out, t = H.hweno_get_state(eng, sid, np.empty_like(w.U0))
            H.hweno_close(eng, sid)
            e = np.abs(out[0, 0] - ex[0, 0])
            rec[name] = {"l1": float(e.mean()), "linf": float(e.max()), "steps": steps,
                         "seconds": el}
        rows.append(rec)
        print(json.dumps(rec), flush=True)
    H.hweno_destroy(eng)
    for a, b in zip(rows, rows[1:]):
        r = math.log(b["n"] / a["n"])
        print(json.dumps({"n": [a["n"], b["n"]],
                          "order_l1_fp64": math.log(a["fp64"]["l1"] / b["fp64"]["l1"]) / r,
                          "order_l1_mixed32": math.log(a["mixed32"]["l1"] / b["mixed32"]["l1"]) / r}))


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--n", type=int, default=N_DEFAULT)
    ap.add_argument("--kernel-reps", type=int, default=5)
    ap.add_argument("--e2e-steps", type=int, default=10)
    ap.add_argument("--cpu-seconds", type=float, default=15.0)
    ap.add_argument("--ref-window", type=int, default=512)
    ap.add_argument("--c4-oracle-n", type=int, default=256,
                    help="grid of the 200-step GPU-vs-oracle comparison in cpu_baseline (0: skip)")
    ap.add_argument("--c4-oracle-steps", type=int, default=200)
    ap.add_argument("--no-c1", action="store_true")
    ap.add_argument("--no-mixed", action="store_true")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-served", action="store_true")
    ap.add_argument("--no-tubes", action="store_true")
    ap.add_argument("--no-autotune", action="store_true",
                    help="use the default launch geometry instead of the autotuned one")
    ap.add_argument("--save-tuning", default="", help="write the autotuned table to this file")
    ap.add_argument("--tuning-file", default="",
                    help="load the tuning table from this file instead of autotuning")
    ap.add_argument("--long-steps", type=int, default=200,
                    help="steps of the long 1024^2 / 2048^2 runs (0: skip them)")
    ap.add_argument("--tubes", type=int, default=16)
    ap.add_argument("--tubes-n", type=int, default=4000)
    ap.add_argument("--tubes-t", type=float, default=1.5)
    ap.add_argument("--served-m", type=int, default=16)
    ap.add_argument("--served-rate", type=float, default=50.0,
                    help="Poisson arrival rate of the served stream, requests/s")
    ap.add_argument("--served-grids", default="128,256,384,512,768,1024")
    ap.add_argument("--served-tlo", type=float, default=0.1)
    ap.add_argument("--served-thi", type=float, default=0.3)
    ap.add_argument("--no-served-small", action="store_true",
                    help="skip the short stream (grids to 512^2, T in [0.02, 0.05])")
    ap.add_argument("--sweep", action="store_true", help="precision / convergence study")
    ap.add_argument("--dt-sweep", action="store_true",
                    help="time-step dependence of the 2D accuracy examples (Tables 3.4-3.6)")
    ap.add_argument("--paper-tables", action="store_true",
                    help="the paper's accuracy examples at 240 cells per direction")
    ap.add_argument("--sweep-sizes", default="128,256,512,1024,2048")
    ap.add_argument("--sweep-T", type=float, default=0.05)
    args = ap.parse_args()
    if args.warmup < 3:
        args.warmup = 3
    if args.sweep:
        run_sweep(args)
    elif args.dt_sweep:
        run_dt_sweep(args)
    elif args.paper_tables:
        run_paper_tables(args)
    elif args.impl == "reference":
        run_reference(args)
    else:
        run_ours(args)


if __name__ == "__main__":
    main()
