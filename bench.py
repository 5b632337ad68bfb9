#!/usr/bin/env python3
"""Benchmark: FP64 cell-updates/s of the ALE-WENO hot path on GB300.

Workload: the large single instance of the 1D shallow-water dam break with a dry region
(N = 2^20 cells on [0, 10], h = 2 / 0.5 / 0 on [0,5) / [5,8) / [8,10], hu = 0,
b = 0.8 exp(-5 (x-5)^2), transmissive, mesh velocity = Gaussian-smoothed fluid velocity
(sigma 8 cells), CFL 0.08). A step is one full SSP-RK3 step (mesh velocity, three
reconstruction + limiter + wave-speed reduction stages, three flux + source + update stages).
A cell-update is one cell advanced by one step.

python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]
Multi-GPU (torchrun): every rank advances an independent replica (weak scaling, no
collective on the data path); the timing is the max over ranks.
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

N_CELLS = 1 << 20
WORKLOAD = "dam_break_dry: N=2^20 cells on [0,10], FP64, transmissive, dry region, Gaussian fluid-driven mesh, CFL 0.08"
METRIC = "cell-updates/s FP64 (fwd, plain single instance)"
UNIT = "cell-updates/s"
FP64_PEAK_TFLOPS = 152 * 2 * 2 * 2.070e9 / 1e12  # SMs x DFMA/clk x 2 flop x max SM clock
# DRAM bytes (read + write) of a k_recon launch on this workload, averaged over the three
# stages, from one ncu capture of the current kernels (128-cell tiles, staged by bulk copies): stage 1
# reads the cached reciprocals of the widths, 4 values per cell (75.6 + 70.6 MB), stage 2 writes them
# (42.5 + 136.6 MB), stage 3 does neither (42.0 + 75.1 MB).
RECON_DRAM_BYTES = (75_617_280 + 70_609_920 + 42_510_848 + 136_626_176 + 42_032_640 + 75_084_800) // 3
# Fraction of cycles the FP64 pipe was busy during the same k_recon launches (ncu
# sm__pipe_fp64_cycles_active, the three stages): the kernel is bound by FP64 instruction issue.
RECON_FP64_PIPE_ACTIVE = (0.8253 + 0.8498 + 0.8584) / 3
# FP64 FLOP equivalents per cell the same launches executed (ncu dadd + dmul + 2 dfma
# instructions over the 2^20 cells; stages 1, 2, 3): what the hardware did, beside the method's
# count and that of the closed-form per-cell functions.
RECON_EXECUTED_FLOPS = (95.8 + 123.4 + 123.4) / 3
# The source term's mesh-only part in the method figures: the interpolant's width ratios in
# closed form (6 products and the cell's reciprocal width), as the paper's construction needs
# them. The closed-form per-cell functions spend more there (the six entries of the antisymmetric
# source form, counted in their own figures) to spend less on the state arithmetic.
METHOD_SOURCE_GEOM_FLOPS = 7.0
# The method's FP64 operations per cell, counted by the CPU oracle on an operation-counting
# scalar type (oracle.count_step; tests/test_bench_contract.py recounts them): the arithmetic on
# state-dependent values of one stage's reconstruction + limiter, and of one whole SSP-RK3 step,
# on the initial state of this workload (2^20 cells) and, cell-weighted, of the first 16
# instances of the batched workload. The oracle builds the mesh-only coefficients by Gaussian
# elimination, which is not a figure of the method; the method figures add the kernels'
# closed-form count of that mesh-only part in every stage (no reuse across stages). The kernels reach the same results
# with fewer operations, so this count times the rate can pass the hardware's peak: it is reported as
# method_count (a multiple of the peak), and is no roofline.
ORACLE_RECON_FLOPS = 318.60
ORACLE_STEP_FLOPS = 1891.80
ORACLE_BATCH_STEP_FLOPS = 1893.17
# The same counts for the scheme variants on the dam-break workload (reconstruction, step).
ORACLE_VARIANT_FLOPS = {"nonwb": (583.01, 2613.02), "special": (366.61, 1780.82)}
# DRAM bytes per k_update launch (stages 1, 2, 3: 193.0 + 47.5, 201.4 + 82.7, 226.5 + 56.4 MB), the
# fraction of cycles its FP64 pipe was busy and the FP64 FLOP equivalents per cell it executed
# (ncu, the same capture as for k_recon above; 128-thread update blocks, 127-cell tiles).
UPDATE_DRAM_BYTES = (192_998_656 + 47_543_040 + 201_380_352 + 82_679_808 + 226_542_848 + 56_431_360) // 3
UPDATE_FP64_PIPE_ACTIVE = (0.8680 + 0.8670 + 0.8604) / 3
UPDATE_EXECUTED_FLOPS = (106.2 + 124.3 + 127.3) / 3
# FP64 pipe instructions per cell and launch (ncu sm__inst_executed_pipe_fp64 x 32 lanes over the cells; stages 1, 2, 3), the
# roofline numerators: every kernel is bound by their issue, one warp instruction per 64 cycles and sub-partition,
# which a fused multiply-add fills with two FLOPs. By scheme (2^18-cell dam break for the variants, 2^18-cell bump):
# (reconstruction, update).
RECON_INSTR = (81.3 + 85.4 + 85.4) / 3
UPDATE_INSTR = (73.6 + 92.7 + 93.7) / 3
VARIANT_INSTR = {"nonwb": ((82.8 + 91.1 + 91.1) / 3, (71.6 + 90.7 + 91.7) / 3),
                 "special": ((96.2 + 100.3 + 100.3) / 3, (110.9 + 108.9 + 105.8) / 3),
                 "bump": ((75.8 + 89.9 + 89.9) / 3, (73.6 + 94.7 + 91.7) / 3)}
MESH_INSTR = 13.8  # the fluid-driven mesh's filter
BATCH_STEP_INSTR = (79.7 + 83.5 + 83.5) + (75.8 + 94.3 + 95.3)
# A gradient's forward steps and its reverse of a step (65536-cell basin).
BASIN_STEP_INSTR = (78.3 + 82.9 + 82.8) + (74.6 + 92.8 + 93.8)
REVERSE_STEP_INSTR = 224.4 + 234.0 + 248.9


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=300)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-batched", action="store_true")
    ap.add_argument("--batched-steps", type=int, default=20)
    ap.add_argument("--no-adjoint", action="store_true")
    ap.add_argument("--adjoint-steps", type=int, default=4000)
    ap.add_argument("--batched-adjoint-steps", type=int, default=256)
    ap.add_argument("--no-batched-adjoint", action="store_true")
    ap.add_argument("--no-variants", action="store_true")
    ap.add_argument("--variant-steps", type=int, default=100)
    ap.add_argument("--no-loop-baseline", action="store_true",
                    help="skip the per-instance launch-loop comparisons of the batched sections (profiling runs)")
    return ap.parse_args()


def dist_env():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    return int(os.environ.get("RANK", "0")), int(os.environ.get("LOCAL_RANK", "0")), ws


class ClockSampler:
    """nvidia-smi samples of SM clock and throttle reasons during the timed region."""

    Q = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,clocks_event_reasons.hw_slowdown,"
         "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
         "clocks_event_reasons.sw_power_cap")

    def __init__(self, index):
        self.index = index
        self.proc = None
        self.lines = []

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.index), f"--query-gpu={self.Q}",
                                          "--format=csv,noheader,nounits", "-lms", "100"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.thread = threading.Thread(target=self._read, daemon=True)
            self.thread.start()
        except OSError:
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
        self.thread.join(timeout=2)
        sm, smax, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for l in self.lines:
            f = [x.strip() for x in l.split(",")]
            if len(f) < 8:
                continue
            try:
                sm.append(float(f[0]))
                smax.append(float(f[1]))
            except ValueError:
                continue
            for n, v in zip(names, f[4:8]):
                if v.lower().startswith("active"):
                    reasons.add(n)
        return {"sm_mhz": float(np.median(sm)) if sm else None, "sm_max_mhz": max(smax) if smax else None,
                "reasons": sorted(reasons), "samples": len(sm)}


def problem():
    from paper_2208_06588_gb300 import workloads as W
    return W.dam_break_dry(N=N_CELLS)


def config_of(pr):
    from paper_2208_06588_gb300 import binding as B
    return B.make_config(g=pr.g, cfl=pr.cfl, eps_weno=pr.eps_weno, gauss_sigma=pr.gauss_sigma,
                         gauss_half=pr.gauss_half, bc=pr.bc, mesh=pr.mesh)


def op_counts(pr):
    """FP64 operations per cell of the reconstruction and update kernels, counted by running the
    closed-form per-cell code (swale_cell.cuh) on a host counting type over a sample of cells."""
    from paper_2208_06588_gb300 import opcount
    return opcount.count_stage(pr.E, pr.hu, pr.b, pr.J, bc=pr.bc, sample=1 << 16)


def fp64_roofline(flops_per_cell_step, cell_steps_per_s, scope,
                  basis="FP64 instructions issued per cell-step (ncu), two FLOPs of the peak each", method_flops=None):
    """Whole-job FP64 roofline: FLOPs of a cell-step times the measured cell-steps per second,
    against the FP64 peak. Every kernel of the step is FP64-pipe bound (DRAM below 25 %), so this
    is the slower of the two rooflines. Callers pass twice the FP64 instructions that the kernels issue, so frac is the
    share of the pipe's issue slots; method_flops: the method's operations (the oracle's count, see ORACLE_STEP_FLOPS), reported
    beside it as a multiple of the peak."""
    achieved = flops_per_cell_step * cell_steps_per_s / 1e12
    out = {"bound": "alu", "scope": scope, "achieved": achieved, "peak": FP64_PEAK_TFLOPS, "unit": "TFLOP/s",
           "frac": achieved / FP64_PEAK_TFLOPS, "flops_per_cell_step": flops_per_cell_step, "basis": basis}
    if method_flops is not None:
        out["method_count"] = {"flops_per_cell_step": method_flops,
                               "times_peak": method_flops * cell_steps_per_s / 1e12 / FP64_PEAK_TFLOPS}
    return out


def method_step_flops(oc, oracle_step=ORACLE_STEP_FLOPS):
    """The method's FLOPs per cell-update: the oracle's count of the step's state arithmetic plus
    the mesh-only geometry of all three stages (reconstruction and source), in closed form."""
    return oracle_step + 3.0 * (oc["geom_flops"] + METHOD_SOURCE_GEOM_FLOPS)


def gradient_step_flops(nsteps, ckpt_every, tape):
    """Twice the FP64 instructions per cell and step of a gradient: the forward run, the recomputes (a step's segment once
    unless it is one of the last two, and the step itself once more without the tape) and the reverse."""
    nseg = -(-nsteps // ckpt_every)
    kept = nsteps - max(0, nseg - (1 if nseg == 1 else 2)) * ckpt_every
    runs = 2.0 - kept / nsteps + (0.0 if tape else 1.0)
    return 2.0 * (runs * BASIN_STEP_INSTR + REVERSE_STEP_INSTR)


def cpu_oracle_rate(n_cells, steps):
    """The CPU oracle as it stands, single thread, on a sample of the same workload."""
    import oracle
    from paper_2208_06588_gb300 import workloads as W
    pr = W.dam_break_dry(N=n_cells)
    st = oracle.State(pr.E, pr.hu, pr.b, pr.J, pr.x)
    P = oracle.Params(g=pr.g, cfl=pr.cfl, bc=pr.bc, mesh=pr.mesh, gauss_sigma=pr.gauss_sigma,
                      gauss_half=pr.gauss_half)
    oracle.lib()
    t0 = time.perf_counter()
    r = oracle.run(P, st, pr.profile, nsteps=steps)
    dt = time.perf_counter() - t0
    return n_cells * r["steps"] / dt, dt


def _oracle_instance(job):
    """One batched instance advanced by the CPU oracle (runs in a spawned worker process)."""
    import oracle
    x, E, hu, b, prof, cfl, steps = job
    st = oracle.State(E, hu, b, np.diff(x), x)
    P = oracle.Params(cfl=cfl, bc="reflective", mesh="profile", mesh_T=1.0)
    return oracle.run(P, st, prof, nsteps=steps)["steps"] * E.size


def cpu_oracle_small_rates():
    """The CPU oracle, one thread, 10 steps of the small periodic instance (N = 200) and of the
    65536-cell Gaussian basin of the adjoint case."""
    import oracle
    from paper_2208_06588_gb300 import workloads as W
    out = {}
    for name, pr in (("smooth_periodic_200", W.smooth_periodic(200)), ("gaussian_basin_65536", W.gaussian_basin())):
        P = oracle.Params(g=pr.g, cfl=pr.cfl, eps_weno=pr.eps_weno, mesh_T=pr.mesh_T, bc=pr.bc, mesh=pr.mesh,
                          dt_fixed=pr.dt_fixed)
        st = oracle.State(pr.E, pr.hu, pr.b, pr.J, pr.x)
        t0 = time.perf_counter()
        r = oracle.run(P, st, pr.profile, nsteps=10)
        el = time.perf_counter() - t0
        out[name] = {"value": pr.N * r["steps"] / el, "unit": UNIT, "cores": 1, "kind": "oracle",
                     "sample": f"{r['steps']} steps, {el:.2f} s"}
    return out


def cpu_oracle_batched_rate(n_inst=1024, steps=5):
    """The CPU oracle as it stands on the batched workload's first n_inst instances, one
    instance per task over a spawned process pool with one worker per available core."""
    import multiprocessing as mp
    from paper_2208_06588_gb300 import workloads as W
    bt = W.many_basins(B=4096)
    jobs = []
    for i in range(n_inst):
        pr = bt.instance(i)
        jobs.append((pr.x, pr.E, pr.hu, pr.b, pr.profile, pr.cfl, steps))
    cores = len(os.sched_getaffinity(0)) if hasattr(os, "sched_getaffinity") else os.cpu_count()
    with mp.get_context("spawn").Pool(cores) as pool:
        pool.map(_oracle_instance, jobs[:cores])  # start-up and library load outside the timing
        t0 = time.perf_counter()
        done = sum(pool.map(_oracle_instance, jobs, chunksize=1))
        el = time.perf_counter() - t0
    cells = int(bt.off[n_inst])
    return {"value": done / el, "unit": UNIT, "cores": cores, "kind": "oracle",
            "sample": f"{steps} SSP-RK3 steps of the first {n_inst} instances of the batched workload ({cells} cells, "
                      f"{el:.1f} s), one instance per task on {cores} worker processes"}


def bench_batched(args, stream, dev, rank=0, ws=1):
    """Batched forward: 4096 instances, 256..16384 cells each, one launch per kernel per stage for
    all instances (autotuned tile sizes), against the plain per-instance launch loop on the same
    512-instance subset. With several ranks each takes a contiguous, cell-balanced share of the
    instances (no data exchange); the time is the max over ranks."""
    import torch
    from paper_2208_06588_gb300 import binding as B
    from paper_2208_06588_gb300 import shard
    from paper_2208_06588_gb300 import workloads as W
    bt_all = W.many_basins(B=4096)
    bt = shard.subset(bt_all, *shard.partition(bt_all.off, ws, rank)) if ws > 1 else bt_all
    cfg = B.make_config(g=bt.g, eps_weno=bt.eps_weno, mesh_T=bt.mesh_T, bc=bt.bc, mesh=bt.mesh, cfl=0.6)
    s = B.Solver(cfg, stream.cuda_stream)
    s.set_batch(bt)
    tiles = B.swale_autotune(s.ctx, 3, autotune_cache())
    B.swale_enqueue(s.ctx, 3)
    stream.synchronize()
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    shard.barrier()
    ev0.record(stream)
    B.swale_enqueue(s.ctx, args.batched_steps)
    ev1.record(stream)
    stream.synchronize()
    ms = shard.max_over_ranks(ev0.elapsed_time(ev1), dev)
    bits = s.status()[0]
    s.close()
    ntot = int(bt_all.off[-1])
    out = {"workload": "many_basins: 4096 instances, N_i ~ U{256..16384} (sum %d cells), reflective, sine mesh "
                       "motion A ~ U[0,0.05], CFL 0.6 / 0.08 (dry)" % ntot,
           "value": ntot * args.batched_steps / (ms * 1e-3), "unit": UNIT, "steps": args.batched_steps,
           "ms_per_step": ms / args.batched_steps, "tiles": list(tiles), "status_bits": bits,
           "parallelism": f"instances sharded over {ws} ranks" if ws > 1 else "single", "scaling": "weak"}
    from paper_2208_06588_gb300 import opcount
    pr0 = bt_all.instance(0)
    oc0 = opcount.count_stage(pr0.E, pr0.hu, pr0.b, pr0.J, bc=pr0.bc, sample=1 << 13)
    out["roofline"] = fp64_roofline(2.0 * BATCH_STEP_INSTR, out["value"], "whole step, all kernels",
                                    method_flops=method_step_flops(oc0, ORACLE_BATCH_STEP_FLOPS))
    if args.no_loop_baseline:
        return out
    # Same work, batched vs one context per instance (launches per instance and step).
    sub = 512
    sb = W.Batch(name="subset", off=bt.off[:sub + 1].copy(), x=bt.x[:int(bt.off[sub]) + sub],
                 h=bt.h[:int(bt.off[sub])], hu=bt.hu[:int(bt.off[sub])], b=bt.b[:int(bt.off[sub])],
                 E=bt.E[:int(bt.off[sub])], profile=bt.profile[:int(bt.off[sub]) + sub], cfl=bt.cfl[:sub])
    nsub = int(sb.off[-1])
    ksub = 24  # three 8-step graphs, batched and per instance alike
    s = B.Solver(cfg, stream.cuda_stream)
    s.set_batch(sb)
    B.swale_set_tiles(s.ctx, *tiles)
    B.swale_enqueue(s.ctx, 2)
    stream.synchronize()
    ev0.record(stream)
    B.swale_enqueue(s.ctx, ksub)
    ev1.record(stream)
    stream.synchronize()
    ms_b = ev0.elapsed_time(ev1)
    s.close()
    solvers = []
    for i in range(sub):
        pr = sb.instance(i)
        c = B.make_config(g=pr.g, eps_weno=pr.eps_weno, mesh_T=pr.mesh_T, bc=pr.bc, mesh=pr.mesh, cfl=pr.cfl)
        si = B.Solver(c, stream.cuda_stream)
        si.set_problem(pr.x, pr.E, pr.hu, pr.b, pr.profile, q0_is_eta=True)
        B.swale_enqueue(si.ctx, 2)
        solvers.append(si)
    for si in solvers:  # each context captures its own 8-step graph before the timing
        B.swale_enqueue(si.ctx, 8)
    stream.synchronize()
    ev0.record(stream)
    for si in solvers:  # every instance replays its own step graphs, one instance after the other
        B.swale_enqueue(si.ctx, ksub)
    ev1.record(stream)
    stream.synchronize()
    ms_l = ev0.elapsed_time(ev1)
    for si in solvers:
        si.close()
    out["vs_per_instance_loop"] = {"instances": sub, "cells": nsub, "steps": ksub,
                                   "batched": nsub * ksub / (ms_b * 1e-3),
                                   "per_instance_loop": nsub * ksub / (ms_l * 1e-3),
                                   "speedup": ms_l / ms_b,
                                   "loop": "one context per instance, swale_enqueue(ctx_i, steps) in turn "
                                           "(each replays its own 8-step CUDA graphs)"}
    return out


def autotune_cache():
    cache = os.path.join(os.path.expanduser("~"), ".cache", "swale_autotune.jsonl")
    os.makedirs(os.path.dirname(cache), exist_ok=True)
    return cache


def _events():
    import torch
    return torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)


def _timed(stream, fn):
    ev0, ev1 = _events()
    stream.synchronize()
    ev0.record(stream)
    fn()
    ev1.record(stream)
    stream.synchronize()
    return ev0.elapsed_time(ev1)


def bench_adjoint(args, stream, dev=None, ws=1):
    """Gradient of the gauge misfit (16 gauges) of the 65536-cell Gaussian basin over
    args.adjoint_steps steps, checkpoints every 64 steps: one swale_adjoint call with host
    observations and host gradients, against the forward alone over the same steps."""
    import torch
    from paper_2208_06588_gb300 import binding as B
    from paper_2208_06588_gb300 import workloads as W
    from paper_2208_06588_gb300 import shard
    K, C = args.adjoint_steps, 64
    gp = W.gauge_problem(N=65536, nsteps=K, G=16)
    pr = gp.problem
    N, G = pr.N, gp.gauges.size
    cfg = B.make_config(g=pr.g, cfl=pr.cfl, eps_weno=pr.eps_weno, mesh_T=pr.mesh_T, bc=pr.bc, mesh=pr.mesh,
                        dt_fixed=pr.dt_fixed)
    free0 = torch.cuda.mem_get_info()[0]
    s = B.Solver(cfg, stream.cuda_stream)
    s.set_problem(pr.x, pr.E, pr.hu, pr.b, pr.profile, q0_is_eta=True)
    stream.synchronize()
    state_bytes = free0 - torch.cuda.mem_get_info()[0]
    B.swale_enqueue(s.ctx, 16)
    s.set_problem(pr.x, pr.E, pr.hu, pr.b, pr.profile, q0_is_eta=True)
    ms_fwd = _timed(stream, lambda: B.swale_enqueue(s.ctx, K))
    J, gE, gM, gB = np.zeros(1), np.zeros(N), np.zeros(N), np.zeros(N)
    obs = np.ascontiguousarray(gp.h_obs)
    s.set_problem(pr.x, pr.E, pr.hu, pr.b, pr.profile, q0_is_eta=True)
    B.swale_adjoint(s.ctx, min(K, 32), 8, G, gp.gauges, obs, J, gE, gM, gB)  # warm-up
    s.set_problem(pr.x, pr.E, pr.hu, pr.b, pr.profile, q0_is_eta=True)
    shard.barrier()
    ms = shard.max_over_ranks(_timed(stream, lambda: B.swale_adjoint(s.ctx, K, C, G, gp.gauges, obs, J, gE, gM, gB)),
                              dev)
    bits = s.status()[0]
    # The same gradient with the tape (swale_set_adjoint_tape): every step run twice, not three
    # times, for about 81 doubles per cell and step of two segments.
    B.swale_set_adjoint_tape(s.ctx, 1)
    s.set_problem(pr.x, pr.E, pr.hu, pr.b, pr.profile, q0_is_eta=True)
    Jt, gEt = np.zeros(1), np.zeros(N)
    ms_t = shard.max_over_ranks(_timed(stream, lambda: B.swale_adjoint(s.ctx, K, C, G, gp.gauges, obs, Jt, gEt, None,
                                                                       None)), dev)
    s.close()
    adj_bytes = B.swale_adjoint_bytes(1, N, K, C, G)
    tape = {"ms_per_gradient": ms_t, "value": ws * N * K / (ms_t * 1e-3), "ckpt_every": C,
            "adjoint_scratch_bytes": int(B.swale_adjoint_bytes(1, N, K, C, G, tape=1)),
            "grad_eta_rel_diff": float(np.abs(gEt - gE).max() / np.abs(gE).max()),
            "roofline": fp64_roofline(gradient_step_flops(K, C, True), ws * N * K / (ms_t * 1e-3),
                                      "whole gradient: up to 2 forward steps + reverse sweep per step")}
    return {"workload": f"gaussian_basin N={N} [0,1] reflective, 4 Gaussian bumps, eta0 from 32 Gaussian basis "
                        f"functions, sine mesh motion A=0.02, fixed dt; {K} SSP-RK3 steps; 16 gauges",
            "metric": "cell-updates/s FP64 (forward + adjoint)", "unit": UNIT,
            "value": ws * N * K / (ms * 1e-3), "gradients_per_s": ws * 1e3 / ms, "ms_per_gradient": ms,
            "parallelism": f"replicas x{ws}" if ws > 1 else "single",
            "ckpt_every": C, "forward_only_ms": ms_fwd, "adjoint_over_forward": ms / ms_fwd,
            "forward_only_value": N * K / (ms_fwd * 1e-3),
            "peak_device_bytes": int(state_bytes + adj_bytes), "adjoint_scratch_bytes": int(adj_bytes),
            "J": float(J[0]), "grad_norms": [float(np.linalg.norm(v)) for v in (gE, gM, gB)], "status_bits": bits,
            "call": "swale_adjoint (host gauges, observations and gradients)", "mode": "recompute inside each step",
            "tape_mode": tape,
            "roofline": fp64_roofline(gradient_step_flops(K, C, False), ws * N * K / (ms * 1e-3),
                                      "whole gradient: up to 3 forward steps + reverse sweep per step")}


def bench_batched_adjoint(args, stream, dev=None, rank=0, ws=1):
    """Batched gradients: 512 Gaussian basins (N_i ~ U{1024..32768}, per-instance seeds and CFL
    dt), args.batched_adjoint_steps steps, checkpoints every 64 steps, all instances in the same
    launches; against one swale_adjoint call per instance on a 32-instance subset."""
    import torch
    from paper_2208_06588_gb300 import binding as B
    from paper_2208_06588_gb300 import workloads as W
    from paper_2208_06588_gb300 import shard
    K, C, G = args.batched_adjoint_steps, 64, 16
    gb = W.many_gauge_basins(B=512, nsteps=K, G=G)
    Nt_all, B_all = int(gb.batch.off[-1]), gb.batch.B
    if ws > 1:  # a contiguous, cell-balanced share of the instances per rank
        i0, i1 = shard.partition(gb.batch.off, ws, rank)
        gb = W.GaugeBatch(batch=shard.subset(gb.batch, i0, i1), gauges=gb.gauges[i0 * G:i1 * G],
                          h_obs=np.ascontiguousarray(gb.h_obs[:, i0:i1, :]), nsteps=K)
    bt = gb.batch
    Nt = int(bt.off[-1])
    cfg = B.make_config(g=bt.g, eps_weno=bt.eps_weno, mesh_T=bt.mesh_T, bc=bt.bc, mesh=bt.mesh, cfl=0.6)
    free0 = torch.cuda.mem_get_info()[0]
    s = B.Solver(cfg, stream.cuda_stream)
    s.set_batch(bt)
    stream.synchronize()
    state_bytes = free0 - torch.cuda.mem_get_info()[0]
    B.swale_set_tiles(s.ctx, 128, 128, 0, 0)
    B.swale_enqueue(s.ctx, 4)
    s.set_batch(bt)
    ms_fwd = _timed(stream, lambda: B.swale_enqueue(s.ctx, K))
    s.set_batch(bt)
    J, gE, gM, gB = np.zeros(bt.B), np.zeros(Nt), np.zeros(Nt), np.zeros(Nt)
    obs = np.ascontiguousarray(gb.h_obs)
    B.swale_adjoint(s.ctx, 8, 4, G, gb.gauges, obs, J, gE, gM, gB)  # warm-up
    s.set_batch(bt)
    shard.barrier()
    ms = shard.max_over_ranks(_timed(stream, lambda: B.swale_adjoint(s.ctx, K, C, G, gb.gauges, obs, J, gE, gM, gB)),
                              dev)
    bits = s.status()[0]
    # With the tape (swale_set_adjoint_tape): the checkpoint interval that needs the least memory
    # for the full 2000 steps, if that fits in 80 % of the free HBM.
    tape = None
    free_now = torch.cuda.mem_get_info()[0]
    cands = sorted((B.swale_adjoint_bytes(bt.B, Nt, 2000, c, G, tape=1), c) for c in (8, 16, 32, 64))
    if cands[0][0] <= 0.8 * free_now:
        Ct = cands[0][1]
        B.swale_set_adjoint_tape(s.ctx, 1)
        s.set_batch(bt)
        shard.barrier()
        try:
            ms_t = shard.max_over_ranks(_timed(stream, lambda: B.swale_adjoint(s.ctx, K, Ct, G, gb.gauges, obs, J, gE,
                                                                               gM, gB)), dev)
            tape = {"ms": ms_t, "value": Nt_all * K / (ms_t * 1e-3), "gradients_per_s": B_all * 1e3 / ms_t,
                    "ckpt_every": Ct, "adjoint_over_forward": ms_t / ms_fwd,
                    "peak_device_bytes": int(state_bytes + B.swale_adjoint_bytes(bt.B, Nt, K, Ct, G, tape=1)),
                    "peak_device_bytes_2000_steps": int(state_bytes + cands[0][0]),
                    "roofline": fp64_roofline(gradient_step_flops(K, Ct, True), Nt_all * K / (ms_t * 1e-3),
                                              "whole gradient: up to 2 forward steps + reverse sweep per step")}
        except B.SwaleError as err:
            tape = {"unavailable": str(err)}
        B.swale_set_adjoint_tape(s.ctx, 0)
    s.close()
    adj_bytes = B.swale_adjoint_bytes(bt.B, Nt, K, C, G)
    full_bytes = B.swale_adjoint_bytes(bt.B, Nt, 2000, C, G)
    out = {"workload": f"many_gauge_basins: 512 instances, N_i ~ U{{1024..32768}} (sum {Nt} cells), per-instance "
                       f"seeds, CFL 0.6 dt per instance, 16 gauges each; {K} steps timed (of 2000 in the full "
                       f"case; the cost per step does not depend on the step count)",
           "metric": "cell-updates/s FP64 (forward + adjoint)", "unit": UNIT,
           "value": Nt_all * K / (ms * 1e-3), "gradients_per_s": B_all * 1e3 / ms, "steps": K, "ckpt_every": C,
           "parallelism": f"instances sharded over {ws} ranks" if ws > 1 else "single",
           "forward_only_value": Nt * K / (ms_fwd * 1e-3), "adjoint_over_forward": ms / ms_fwd,
           "peak_device_bytes": int(state_bytes + adj_bytes), "peak_device_bytes_2000_steps": int(state_bytes + full_bytes),
           "status_bits": bits,
           "roofline": fp64_roofline(gradient_step_flops(K, C, False), Nt_all * K / (ms * 1e-3),
                                     "whole gradient: up to 3 forward steps + reverse sweep per step"),
           "mode": "recompute inside each step", "tape_mode": tape}
    if args.no_loop_baseline:
        return out
    # One swale_adjoint per instance on a subset, same steps, against the batch of the subset.
    sub, Ks = 32, min(K, 64)
    sb = W.Batch(name="subset", off=bt.off[:sub + 1].copy(), x=bt.x[:int(bt.off[sub]) + sub],
                 h=bt.h[:int(bt.off[sub])], hu=bt.hu[:int(bt.off[sub])], b=bt.b[:int(bt.off[sub])],
                 E=bt.E[:int(bt.off[sub])], profile=bt.profile[:int(bt.off[sub]) + sub], cfl=bt.cfl[:sub])
    ns = int(sb.off[-1])
    gx = np.ascontiguousarray(gb.gauges[:sub * G])
    ob = np.ascontiguousarray(gb.h_obs[:Ks, :sub, :])
    s = B.Solver(cfg, stream.cuda_stream)
    s.set_batch(sb)
    Jb, g1, g2, g3 = np.zeros(sub), np.zeros(ns), np.zeros(ns), np.zeros(ns)
    ms_b = _timed(stream, lambda: B.swale_adjoint(s.ctx, Ks, C, G, gx, ob, Jb, g1, g2, g3))
    s.close()
    solvers = []
    for i in range(sub):
        pr = sb.instance(i)
        si = B.Solver(cfg, stream.cuda_stream)
        si.set_problem(pr.x, pr.E, pr.hu, pr.b, pr.profile, q0_is_eta=True)
        solvers.append((si, pr.N, np.ascontiguousarray(gx[i * G:(i + 1) * G]),
                        np.ascontiguousarray(ob[:, i, :])))

    def loop():
        for si, n, gxi, obi in solvers:
            Ji, a, b_, c = np.zeros(1), np.zeros(n), np.zeros(n), np.zeros(n)
            B.swale_adjoint(si.ctx, Ks, C, G, gxi, obi, Ji, a, b_, c)

    ms_l = _timed(stream, loop)
    for si, *_ in solvers:
        si.close()
    out["vs_per_instance_loop"] = {"instances": sub, "cells": ns, "steps": Ks, "batched": ns * Ks / (ms_b * 1e-3),
                                   "per_instance_loop": ns * Ks / (ms_l * 1e-3), "speedup": ms_l / ms_b}
    return out


def bench_variant(args, stream, pr, scheme="hydrostatic", bottom=None):
    """One single-instance workload with a scheme variant: K graph-replayed steps timed with CUDA
    events, then K steps with per-kernel events for the roofline of the dominant kernel."""
    import torch
    from paper_2208_06588_gb300 import binding as B
    from paper_2208_06588_gb300 import opcount
    K = args.variant_steps
    cfg = B.make_config(g=pr.g, cfl=pr.cfl, eps_weno=pr.eps_weno, mesh_T=pr.mesh_T, gauss_sigma=pr.gauss_sigma,
                        gauss_half=pr.gauss_half, bc=pr.bc, mesh=pr.mesh, scheme=scheme)
    ctx = B.swale_create(cfg, stream.cuda_stream)
    B.swale_set_problem(ctx, pr.N, pr.x, pr.E, pr.hu, pr.b, pr.profile, 1)
    if bottom is not None:
        B.swale_set_bottom_function(ctx, *bottom)
    B.swale_enqueue(ctx, args.warmup)
    ms = _timed(stream, lambda: B.swale_enqueue(ctx, K))
    B.swale_set_timing(ctx, True)
    B.swale_enqueue(ctx, K)
    fam = B.swale_get_timing(ctx)
    B.swale_set_timing(ctx, False)
    bits, steps, _ = B.swale_get_status(ctx)
    B.swale_destroy(ctx)
    oc = opcount.count_stage(pr.E, pr.hu, pr.b, pr.J, bc=pr.bc, sample=1 << 16, scheme=scheme)
    dom = "reconstruction" if fam["reconstruction"][0] >= fam["update"][0] else "update"
    o_rec, o_step = ORACLE_VARIANT_FLOPS.get(scheme, (ORACLE_RECON_FLOPS, ORACLE_STEP_FLOPS))
    fl = (o_rec + oc["geom_flops"]) if dom == "reconstruction" else (o_step - 3.0 * o_rec) / 3.0 + METHOD_SOURCE_GEOM_FLOPS
    instr = VARIANT_INSTR.get(scheme, VARIANT_INSTR["bump"])[0 if dom == "reconstruction" else 1]
    ms_dom, n_dom = fam[dom]
    per_s = pr.N / (ms_dom / n_dom * 1e-3)
    roof = fp64_roofline(2.0 * instr, per_s, "dominant kernel, per launch", method_flops=fl)
    return {"value": pr.N * K / (ms * 1e-3), "unit": UNIT, "steps": K, "ms_per_step": ms / K, "status_bits": bits,
            "roofline": {**roof, "kernel": dom, "avg_launch_ms": ms_dom / n_dom},
            "fp64_flops_per_cell_stage": {"recon": oc["recon_flops"], "update": oc["update_flops"]}}


def bench_variants(args, stream):
    """The scheme variants beside the default one, at 2^20 cells: the non-well-balanced scheme
    (characteristic reconstruction, plain LF flux) and the special source-term scheme on the
    dam-break workload, and the L2-projection bottom on the dam break over a rectangular bump
    with the bump-aligned mesh."""
    from paper_2208_06588_gb300 import workloads as W
    out = {}
    pr = problem()
    r = bench_variant(args, stream, pr, scheme="nonwb")
    r["workload"] = WORKLOAD + "; non-well-balanced scheme (Eq. se2D / s2D)"
    out["nonwb_dam_break"] = r
    r = bench_variant(args, stream, pr, scheme="special")
    r["workload"] = WORKLOAD + "; special source-term scheme (Eq. special2D)"
    out["special_dam_break"] = r
    pr = W.bump_dam_break(N=N_CELLS)
    r = bench_variant(args, stream, pr, bottom=pr.meta["bottom"])
    r["workload"] = ("bump_dam_break: N=2^20 cells on [0,1500], b = 8 on [562.5,937.5], eta = 20 / 15, transmissive, "
                     "bump-aligned motion (Eq. wangge3, T = 60), L2-projection bottom (Eq. baverage), CFL 0.6")
    out["l2_bottom_bump_dam_break"] = r
    return out


def run_reference(args):
    """Reference arm: the CPU oracle (plain C++ FP64, one thread) on the same workload as the GPU
    arm, every step one SSP-RK3 step of all 2^20 cells (about 2-4 s per step on one core)."""
    rank, _, ws = dist_env()
    if rank != 0:
        return
    import oracle
    pr = problem()
    st = oracle.State(pr.E, pr.hu, pr.b, pr.J, pr.x)
    P = oracle.Params(g=pr.g, cfl=pr.cfl, bc=pr.bc, mesh=pr.mesh, gauss_sigma=pr.gauss_sigma,
                      gauss_half=pr.gauss_half)
    oracle.run(P, st, pr.profile, nsteps=max(args.warmup, 0))
    t0 = time.perf_counter()
    r = oracle.run(P, st, pr.profile, nsteps=args.steps)
    el = time.perf_counter() - t0
    v = pr.N * r["steps"] / el
    sample = (f"{args.steps} SSP-RK3 steps of the full 2^20-cell workload after {args.warmup} warm-up steps "
              f"({el:.1f} s, one thread)")
    out = {"impl": "reference", "metric": METRIC, "value": v, "unit": UNIT, "n_gpus": args.gpus,
           "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * el / max(r["steps"], 1),
           "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
           "data": "synthetic", "config": run_config(pr.N, ws),
           "cpu_baseline": {"value": v, "unit": UNIT, "cores": 1, "kind": "oracle", "sample": sample},
           "e2e": {"value": v, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
           "status": r["status"]}
    print(json.dumps(out), flush=True)


def run_config(N, ws):
    """The workload as both arms name it in their JSON line."""
    return {"workload": WORKLOAD, "cells": N, "parallelism": f"replicas x{ws}" if ws > 1 else "single",
            "l2": "working set ~230 MB per stage > 126 MB L2 (no flush needed)"}


def summary(out):
    """Compact figures of every section, placed last in the JSON line so that a captured tail of
    the output keeps them."""
    r3 = lambda v: None if v is None else float(f"{v:.4g}")
    sm = {"fwd_2p20": {"value": r3(out["value"]), "ms_per_step": r3(out["ms_per_step"]),
                       "frac": r3(out["roofline"]["frac"]), "step_frac": r3(out["step_roofline"]["frac"]),
                       "e2e": r3(out["e2e"]["value"])}}
    b = out.get("batched")
    if b:
        sm["batched_fwd"] = {"value": r3(b["value"]), "ms_per_step": r3(b["ms_per_step"]),
                             "frac": r3(b["roofline"]["frac"]),
                             "speedup_vs_loop": r3(b.get("vs_per_instance_loop", {}).get("speedup"))}
    a = out.get("adjoint")
    if a:
        sm["adjoint"] = {"value": r3(a["value"]), "ms_per_gradient": r3(a["ms_per_gradient"]),
                         "frac": r3(a["roofline"]["frac"]), "tape_value": r3(a["tape_mode"]["value"])}
    a = out.get("batched_adjoint")
    if a:
        t = a.get("tape_mode") or {}
        sm["batched_adjoint"] = {"value": r3(a["value"]), "gradients_per_s": r3(a["gradients_per_s"]),
                                 "frac": r3(a["roofline"]["frac"]), "tape_value": r3(t.get("value")),
                                 "tape_gradients_per_s": r3(t.get("gradients_per_s")),
                                 "speedup_vs_loop": r3(a.get("vs_per_instance_loop", {}).get("speedup"))}
    v = out.get("variants")
    if v:
        sm["variants"] = {k: r3(x["value"]) for k, x in v.items()}
    return sm


def main():
    args = parse()
    if args.impl == "reference":
        run_reference(args)
        return
    rank, local, ws = dist_env()
    import torch
    import torch.distributed as dist
    if ws > 1:
        torch.cuda.set_device(local)
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    dev = torch.device("cuda", local if ws > 1 else 0)
    torch.cuda.set_device(dev)
    from paper_2208_06588_gb300 import binding as B
    B.lib()
    pr = problem()
    N = pr.N
    stream = torch.cuda.Stream(device=dev)
    ctx = B.swale_create(config_of(pr), stream.cuda_stream)
    B.swale_set_problem(ctx, N, pr.x, pr.E, pr.hu, pr.b, None, 1)
    # Tile sizes from the library's autotuner (cached per device and problem shape; the state is
    # restored after the trial steps).
    tiles = B.swale_autotune(ctx, 3, autotune_cache())

    def barrier():
        if ws > 1:
            dist.barrier()

    # Warm-up (also instantiates the step graph).
    B.swale_enqueue(ctx, args.warmup)
    stream.synchronize()
    # ---- device-timed region: K steps replayed as CUDA graphs ----
    barrier()
    torch.cuda.synchronize()
    clocks = ClockSampler(torch.cuda.current_device())
    clocks.start()
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    ev0.record(stream)
    B.swale_enqueue(ctx, args.steps)
    ev1.record(stream)
    stream.synchronize()
    torch.cuda.synchronize()
    barrier()
    ms = ev0.elapsed_time(ev1)
    # ---- per-kernel durations: K more steps with CUDA events around every launch (no graphs) ----
    B.swale_set_timing(ctx, True)
    B.swale_enqueue(ctx, args.steps)
    fam = B.swale_get_timing(ctx)
    B.swale_set_timing(ctx, False)
    clk = clocks.stop()
    bits, steps_done, last_dt = B.swale_get_status(ctx)
    B.swale_destroy(ctx)
    if ws > 1:
        t = torch.tensor([ms], device=dev, dtype=torch.float64)
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
        ms = float(t.item())
    value = ws * N * args.steps / (ms * 1e-3)
    launches = sum(n for _, n in fam.values())  # the same kernels as the graph-replayed timed region

    # ---- end-to-end through the public C ABI with host buffers ----
    pin = {k: torch.from_numpy(np.ascontiguousarray(v)).pin_memory()
           for k, v in (("x", pr.x), ("E", pr.E), ("hu", pr.hu), ("b", pr.b))}
    outs = {k: torch.empty(n, dtype=torch.float64).pin_memory()
            for k, n in (("eta", N), ("hu", N), ("b", N), ("x", N + 1), ("t", 1))}
    barrier()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    ctx2 = B.swale_create(config_of(pr), stream.cuda_stream)
    B.swale_set_problem(ctx2, N, pin["x"], pin["E"], pin["hu"], pin["b"], None, 1)
    B.swale_set_tiles(ctx2, *tiles)
    B.swale_advance(ctx2, args.steps)
    B.swale_get_state(ctx2, None, outs["hu"], outs["b"], outs["eta"], outs["x"], outs["t"])
    e2e_s = time.perf_counter() - t0
    B.swale_destroy(ctx2)
    if ws > 1:
        t = torch.tensor([e2e_s], device=dev, dtype=torch.float64)
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
        e2e_s = float(t.item())
    h2d = sum(v.numel() * 8 for v in pin.values())
    d2h = sum(v.numel() * 8 for v in outs.values())
    e2e = {"value": ws * N * args.steps / e2e_s, "unit": UNIT, "h2d_bytes_per_step": h2d / args.steps,
           "d2h_bytes_per_step": d2h / args.steps,
           "call": "swale_create + swale_set_problem(host) + swale_set_tiles + swale_advance(K) + "
                   "swale_get_state(host) + destroy"}

    # ---- batched and adjoint sections (every rank: sharded batches, replicated single instance) ----
    batched = None
    if not args.no_batched:
        batched = bench_batched(args, stream, dev, rank, ws)
    adjoint = batched_adjoint = None
    if not args.no_adjoint:
        adjoint = bench_adjoint(args, stream, dev, ws)
        if not args.no_batched_adjoint:
            batched_adjoint = bench_batched_adjoint(args, stream, dev, rank, ws)

    variants = None
    if not args.no_variants:
        variants = bench_variants(args, stream)

    if rank != 0:
        if ws > 1:
            dist.destroy_process_group()
        return

    # ---- roofline of the dominant kernel (FP64 ALU bound) ----
    oc = op_counts(pr)
    ms_rec, n_rec = fam["reconstruction"]
    ms_upd, n_upd = fam["update"]
    dom = "reconstruction" if ms_rec >= ms_upd else "update"
    # The method's count per cell and launch (oracle count + mesh-only geometry of the stage).
    method_recon = ORACLE_RECON_FLOPS + oc["geom_flops"]
    method_update = (ORACLE_STEP_FLOPS - 3.0 * ORACLE_RECON_FLOPS) / 3.0 + METHOD_SOURCE_GEOM_FLOPS
    flops_cell = method_recon if dom == "reconstruction" else method_update
    instr_cell = RECON_INSTR if dom == "reconstruction" else UPDATE_INSTR
    ms_dom, n_dom = fam[dom]
    per_s = N / (ms_dom / n_dom * 1e-3)
    achieved = 2.0 * instr_cell * per_s / 1e12
    roof = {"bound": "alu", "kernel": f"k_{'recon' if dom == 'reconstruction' else 'update'} (per stage)",
            "achieved": achieved, "peak": FP64_PEAK_TFLOPS, "unit": "TFLOP/s", "frac": achieved / FP64_PEAK_TFLOPS,
            "traffic": RECON_DRAM_BYTES if dom == "reconstruction" else UPDATE_DRAM_BYTES,
            "traffic_unit": "bytes per launch (ncu dram__bytes_read.sum + dram__bytes_write.sum of the kernel, "
                            "N = 2^20, the autotuned tiles, mean of the three stages)",
            "fp64_instructions_per_cell": instr_cell, "cells_per_launch": N,
            "flops_basis": "FP64 instructions issued per cell (ncu), two FLOPs of the peak each: the share of the pipe's "
                           "issue slots",
            "method_count": {"flops_per_cell": flops_cell, "times_peak": flops_cell * per_s / 1e12 / FP64_PEAK_TFLOPS,
                             "source": "the CPU oracle's count of the state arithmetic + the mesh-only geometry in closed "
                                       "form; the kernels reach the same result with fewer operations"},
            "ncu_fp64_pipe_active": RECON_FP64_PIPE_ACTIVE if dom == "reconstruction" else UPDATE_FP64_PIPE_ACTIVE,
            "executed": {"flops_per_cell": RECON_EXECUTED_FLOPS if dom == "reconstruction" else UPDATE_EXECUTED_FLOPS,
                         "frac": (RECON_EXECUTED_FLOPS if dom == "reconstruction" else UPDATE_EXECUTED_FLOPS) * per_s
                         / 1e12 / FP64_PEAK_TFLOPS,
                         "source": "ncu dadd + dmul + 2 dfma per cell of one step's launches of the kernel"},
            "avg_launch_ms": ms_dom / n_dom,
            "peak_source": "FP64 DFMA: 152 SMs x 2 DFMA/clk x 2 flop x 2.07 GHz (measured DFMA chain: 1.195 TFLOP/s)",
            "kernel_ms_share": {k: round(v[0] / max(sum(x[0] for x in fam.values()), 1e-30), 4)
                                for k, v in fam.items()}}

    cpu = None
    if not args.no_cpu_baseline:
        rate, secs = cpu_oracle_rate(N_CELLS, 3)
        cpu = {"value": rate, "unit": UNIT, "cores": 1, "kind": "oracle",
               "sample": f"3 SSP-RK3 steps of the full 2^20-cell workload ({secs:.1f} s, one thread)"}
        if batched is not None:
            batched["cpu_baseline"] = cpu_oracle_batched_rate()
        cpu["other_workloads"] = cpu_oracle_small_rates()

    out = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": ws, "steps": args.steps,
           "warmup": args.warmup, "ms_per_step": ms / args.steps, "higher_is_better": True, "scaling": "weak",
           "vs_baseline": None, "dtype": "f64", "data": "synthetic",
           "config": run_config(N, ws), "tiles": list(tiles),
           "e2e": e2e, "gpu_launches": launches, "clocks": clk, "roofline": roof,
           "step_roofline": fp64_roofline(2.0 * (3.0 * (RECON_INSTR + UPDATE_INSTR) + MESH_INSTR), value,
                                          "whole step, all kernels", method_flops=method_step_flops(oc)),
           "cpu_baseline": cpu,
           "status_bits": bits, "steps_done_device": steps_done, "last_dt": last_dt, "batched": batched,
           "adjoint": adjoint, "batched_adjoint": batched_adjoint, "variants": variants,
           "fp64_ops_per_cell_stage": oc}
    out["summary"] = summary(out)
    print(json.dumps(out), flush=True)
    if ws > 1:
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
