#!/usr/bin/env python
"""Benchmark: Lippmann-Schwinger solves per second on one GB300.

Workload (one "step" = one pass of the whole method over one batch): the
largest configuration that fits one GPU, a 1024 x 1024 grid (h = 5 m,
c0 = 2000 m/s, f = 30 Hz) with a seeded Marmousi-like velocity model
(30-60 smoothed layers, 1500-5500 m/s with depth, 5-10 faults) and 16 point
sources on the top row.  The step builds the Green table and spectrum, the
contrast and the source fields, the randomized HODLR preconditioner
(quadtree 32 x 32 leaves, 10 levels, rank 40 + 10 Gaussian probes, q = 0;
built in FP32 with FP64-accurate sketch QR and truncation, kept as BF16)
with its recursive block inversion, and solves all 16 sources to an FP64
relative residual of 1e-6: FP32 FGMRES(30) with H as right preconditioner
inside FP64 iterative refinement.  Only sources that reach 1e-6 count as
solves.

Multi-GPU (torchrun): every rank solves its own copy of the workload
(independent (source, frequency) problems, no data-path collective); value is
all ranks' solves over the slowest rank's time.

--impl reference times the CPU oracle on a bounded sample of the same workload.
"""
from __future__ import annotations

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

METRIC = "LS solves/sec (src x freq) at rel. residual 1e-6; FFT-operator HBM GB/s vs peak"
WORKLOAD = "marmousi-like-1024x1024-30Hz-16src"
TOL = 1e-6
RANK, OVERSAMPLE, LEVELS, SEED = 40, 10, 10, 1004


def load_peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        with open(p) as f:
            d = json.load(f)
        return d.get("hbm_gbs", 6800.0), "measured"
    return 6800.0, "fallback"


class ClockSampler:
    """nvidia-smi clock and throttle samples during the timed region."""

    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, device_index: int):
        self.dev = device_index
        self.rows = []
        self.proc = None
        self.thread = None

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.dev), f"--query-gpu={self.Q}",
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except (OSError, ValueError):
            self.proc = None
            return

        def rd():
            for line in self.proc.stdout:
                self.rows.append([t.strip() for t in line.split(",")])
        self.thread = threading.Thread(target=rd, daemon=True)
        self.thread.start()

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        if self.thread:
            self.thread.join(timeout=2)
        sm, mx, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for r in self.rows:
            if len(r) < 9:
                continue
            try:
                sm.append(float(r[1]))
                mx = float(r[2])
            except ValueError:
                continue
            for nm, v in zip(names, r[5:9]):
                if v.lower() == "active":
                    reasons.add(nm)
        return {"sm_mhz": float(np.median(sm)) if sm else None, "sm_max_mhz": mx,
                "samples": len(sm), "reasons": sorted(reasons)}


# The kernel family with the largest share of the step's serialised launch
# list (an ncu capture of one step, gpu__time_duration per launch): the truncation's
# eigen-decompositions (FP64 Cholesky factor, one-sided FP32 Jacobi),
# latency-bound; timed live with CUDA events on their launching streams over
# the timed steps, against the algorithmic 36 k^3 real flops per matrix.
DOMINANT = "heev"
DOMINANT_KERNEL = ("heev: eigen-decompositions of the sketches' k x k Gram matrices for the truncation "
                   "(one-sided FP32 Jacobi on the FP64 Cholesky factor; k = 50), 36 k^3 flops each")
# DRAM bytes (read + write) per launch of the dominant family from one ncu
# capture of this workload's step, or None when not captured for this build.
DOMINANT_TRAFFIC_PER_LAUNCH = None
# The largest bandwidth-bound kernel of the H apply's level products: the
# partials of the BF16 H apply (k_lr_partial_ws), timed over whole H applies
# after the timed steps, L2 flushed between applies.
SOLVE_KERNEL = ("k_lr_partial_ws: every level's W^H x partials of the BF16 HODLR apply (tcgen05, warp-specialised "
                "bulk-copy ring), 16 vectors at 1024^2")
# DRAM bytes of one 16-field 1024^2 FP32 RESIDUAL apply (passes k_fa, k_fb,
# k_fc: 381 + 488 + 639 MB), from one ncu capture of a cold apply.
OPERATOR_TRAFFIC = 1.5083e9


def fp32_alu_peak_tflops(sms: int = 152, sm_mhz: float = 2070.0) -> float:
    """Nominal FP32 CUDA-core peak from the SM count and the maximum SM
    clock: SMs x 128 FP32 lanes x 2 flops (fused multiply-add) x clock.
    Only a fallback: the bench divides by the peak that lsw_measure_peak
    measures on the device."""
    return round(sms * 128 * 2 * sm_mhz * 1e6 / 1e12, 1)


def op_bytes_c64(n: int, nsrc: int) -> float:
    """Algorithmic bytes of one batched c64 operator apply (RESIDUAL mode):
    read u and u0, write y (8 B each per cell and source), plus chi (8 B per
    cell, FP64) and the quarter spectrum (8 B per entry) once per batch."""
    nz = nx = int(round(n ** 0.5))
    return 24.0 * n * nsrc + 8.0 * n + 8.0 * (nz + 1) * (nx + 1)


def reduce_over_ranks(ms_local: float, solves_local: float, device):
    """Whole-job timing of the replicas: the slowest rank's time and the sum of
    every rank's converged solves (each rank solves its own copy of the
    workload; these two scalars are the only collectives)."""
    import torch
    import torch.distributed as dist
    t = torch.tensor([ms_local], dtype=torch.float64, device=device)
    c = torch.tensor([float(solves_local)], dtype=torch.float64, device=device)
    if dist.is_available() and dist.is_initialized() and dist.get_world_size() > 1:
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
        dist.all_reduce(c, op=dist.ReduceOp.SUM)
    return float(t.item()), float(c.item())


def hparams(lsw):
    return lsw.HParams(kind=lsw.H_HODLR, prec=lsw.BF16, levels=LEVELS, split=lsw.SPLIT_QUADTREE, rank=RANK,
                       oversample=OVERSAMPLE, q=0, seed=SEED)


def sparams(lsw):
    return lsw.SolveParams(prec=lsw.MIXED, method=lsw.FGMRES, tol=TOL, inner_tol=1e-3, restart=30, max_iter=400,
                           max_outer=8)


def run_ours(args):
    import torch
    import torch.distributed as dist

    from paper_2005_01372_gb300 import lsw, media

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1:
        dist.init_process_group("nccl")
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    stream = torch.cuda.current_stream()

    wl = media.marmousi_1024()
    vel_host = torch.from_numpy(np.ascontiguousarray(wl.velocity.ravel())).pin_memory()
    vel = vel_host.to(dev)
    hp, sp = hparams(lsw), sparams(lsw)
    flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device=dev)   # 256 MiB > L2

    def step(v):
        G = lsw.build_green(wl.nz, wl.nx, wl.h, wl.c0, wl.freq_hz)
        chi = G.contrast(v)
        u0 = G.point_sources(wl.sources, lsw.C128)
        H = lsw.build_hmatrix(G, chi, hp)
        u, infos = lsw.solve_series(G, chi, H, u0, sp=sp)
        return u, infos

    for _ in range(args.warmup):
        step(vel)
    torch.cuda.synchronize()

    # ---- timed region: K steps, inputs resident in HBM, L2 flushed between steps.
    if world > 1:
        dist.barrier()
    torch.cuda.synchronize()
    clocks = ClockSampler(local)
    clocks.start()
    l0 = lsw.launch_count()
    lsw.kernel_timer_start(DOMINANT)
    times, conv, worst, applies = [], 0, 0.0, []
    t_wall = time.perf_counter()
    for _ in range(args.steps):
        flush.zero_()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        u, infos = step(vel)
        e1.record(stream)
        e1.synchronize()
        times.append(e0.elapsed_time(e1))
        ok = [i for i in infos if i.status == 0 and i.rel_residual <= TOL]
        conv += len(ok)
        worst = max(worst, max(i.rel_residual for i in infos))
        # operator applies per source: one per inner iteration, one FP64
        # residual per refinement step plus the initial one
        applies.extend(i.iterations + i.outer + 1 for i in infos)
    torch.cuda.synchronize()
    wall = time.perf_counter() - t_wall
    launches = lsw.launch_count() - l0
    dom_ms, dom_bytes, dom_flops, dom_n = lsw.kernel_timer_read()
    lsw.kernel_timer_stop()
    clk = clocks.stop()
    if world > 1:
        dist.barrier()
    ms_max, solves = reduce_over_ranks(float(np.sum(times)), conv, dev)
    value = solves / (ms_max / 1e3)

    # ---- end to end through the public API with host buffers
    e2e_times = []
    out_host = torch.empty((len(wl.sources), wl.n), dtype=torch.complex128).pin_memory()
    for _ in range(1):
        flush.zero_()
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        v = vel_host.to(dev, non_blocking=True)
        u, infos = step(v)
        out_host.copy_(u, non_blocking=True)
        e1.record(stream)
        e1.synchronize()
        e2e_times.append(e0.elapsed_time(e1))
    e2e_value = sum(1 for i in infos if i.status == 0 and i.rel_residual <= TOL) * world / (
        float(np.mean(e2e_times)) / 1e3)

    # ---- the FFT operator alone (its three passes timed with CUDA events on
    # its stream): the solve's RESIDUAL apply in FP32 on the 16 source
    # fields, with L2 flushed between applies (inside the solves most operator
    # applies are replayed from a CUDA graph, which the family timer does not see)
    G = lsw.build_green(wl.nz, wl.nx, wl.h, wl.c0, wl.freq_hz)
    chi = G.contrast(vel)
    uf = G.point_sources(wl.sources, lsw.C64)
    yf = torch.empty_like(uf)
    lsw.apply_operator(G, chi, uf, uf, lsw.OP_RESIDUAL, y=yf)
    torch.cuda.synchronize()
    lsw.kernel_timer_start("operator_c64")
    for _ in range(20):
        flush.zero_()
        lsw.apply_operator(G, chi, uf, uf, lsw.OP_RESIDUAL, y=yf)
    op_ms, op_bytes, op_flops, op_n = lsw.kernel_timer_read()
    lsw.kernel_timer_stop()
    fp32_peak = lsw.measure_peak(0)

    # ---- the level partials of the H apply, timed over whole applies
    H = lsw.build_hmatrix(G, chi, hp)
    xs = G.point_sources(wl.sources, lsw.C64)
    ys = torch.empty_like(xs)
    lsw.apply_precond(H, xs, ys)
    torch.cuda.synchronize()
    lsw.kernel_timer_start("lr_partial")
    for _ in range(20):
        flush.zero_()
        lsw.apply_precond(H, xs, ys)
    lp_ms, lp_bytes, lp_flops, lp_n = lsw.kernel_timer_read()
    lsw.kernel_timer_stop()
    del H

    peak, peak_kind = load_peaks()
    dom_gbs = dom_bytes / (dom_ms / 1e3) / 1e9 if dom_ms > 0 else 0.0
    dom_tf = dom_flops / (dom_ms / 1e3) / 1e12 if dom_ms > 0 else 0.0
    roof = {"kernel": DOMINANT_KERNEL, "bound": "alu", "achieved": round(dom_tf, 5), "peak": round(fp32_peak, 2),
            "peak_kind": "measured: lsw_measure_peak FP32 FMA probe on this device", "unit": "TFLOP/s",
            "frac": round(dom_tf / fp32_peak, 6) if fp32_peak > 0 else None, "traffic": DOMINANT_TRAFFIC_PER_LAUNCH,
            "launches": int(dom_n), "avg_launch_ms": round(dom_ms / max(1, dom_n), 4),
            "achieved_gbs": round(dom_gbs, 3), "hbm_frac": round(dom_gbs / peak, 6)}
    lp_avg = lp_ms / max(1, lp_n)
    lp_gbs = lp_bytes / (lp_ms / 1e3) / 1e9 if lp_ms > 0 else 0.0
    lp_roof = {"kernel": SOLVE_KERNEL, "bound": "hbm", "achieved": round(lp_gbs, 1), "peak": peak,
               "peak_kind": peak_kind, "unit": "GB/s", "frac": round(lp_gbs / peak, 4) if peak else None,
               "traffic": None, "launches": int(lp_n), "avg_launch_ms": round(lp_avg, 4),
               "algorithmic_bytes_per_launch": round(lp_bytes / max(1, lp_n))}
    op_tf = op_flops / (op_ms / 1e3) / 1e12 if op_ms > 0 else 0.0
    op_gbs = op_bytes / (op_ms / 1e3) / 1e9 if op_ms > 0 else 0.0
    op_avg = op_ms / max(1, op_n)
    op_roof = {"kernel": "FFT operator in FP32, passes k_fa + k_fb + k_fc, RESIDUAL on the 16 source fields at "
                         "1024^2, timed alone with L2 flushed between applies", "bound": "alu",
               "achieved": round(op_tf, 2), "peak": round(fp32_peak, 2),
               "peak_kind": "measured: lsw_measure_peak FP32 FMA probe on this device",
               "unit": "TFLOP/s", "frac": round(op_tf / fp32_peak, 4) if fp32_peak > 0 else None,
               "algorithmic_gbs": round(op_gbs, 1), "hbm_frac": round(op_gbs / peak, 4),
               "hbm_peak": peak, "hbm_peak_kind": peak_kind,
               "dram_traffic_per_apply": OPERATOR_TRAFFIC,
               "dram_gbs": round(OPERATOR_TRAFFIC / (op_avg / 1e3) / 1e9, 1) if OPERATOR_TRAFFIC else None,
               "dram_frac": round(OPERATOR_TRAFFIC / (op_avg / 1e3) / 1e9 / peak, 4) if OPERATOR_TRAFFIC else None,
               "applies": int(op_n), "avg_apply_ms": round(op_avg, 4)}

    if rank == 0:
        line = {"metric": METRIC, "value": round(value, 4), "unit": "solves/s", "n_gpus": world,
                "steps": args.steps, "warmup": args.warmup, "ms_per_step": round(ms_max / args.steps, 3),
                "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "c64+bf16+f64",
                "data": "synthetic",
                "config": {"workload": WORKLOAD, "grid": "1024x1024", "h_m": wl.h, "freq_hz": wl.freq_hz,
                           "sources_per_gpu": len(wl.sources),
                           "preconditioner": f"HODLR quadtree 32x32 leaves, {LEVELS} levels, rank {RANK}+"
                                             f"{OVERSAMPLE}, q=0, FP32 build, BF16 storage",
                           "solver": "FGMRES(30) right-preconditioned, FP64 iterative refinement to 1e-6",
                           "l2": "256 MiB buffer written between timed steps", "parallelism": f"replicas{world}"},
                "solves_converged": int(solves), "max_rel_residual": worst,
                "operator_applies_per_solve": round(float(np.mean(applies)), 1),
                "roofline": roof, "solve_roofline": lp_roof, "operator_roofline": op_roof,
                "e2e": {"value": round(e2e_value, 4), "unit": "solves/s",
                        "h2d_bytes_per_step": int(vel_host.numel() * 8),
                        "d2h_bytes_per_step": int(out_host.numel() * 16)},
                "clocks": clk, "gpu_launches": int(launches), "wall_s": round(wall, 3)}
        if not args.no_cpu_baseline and world == 1:
            line["cpu_baseline"] = cpu_baseline(float(np.mean(applies)))
        print(json.dumps(line), flush=True)
    if world > 1:
        dist.destroy_process_group()


def run_extra(args):
    """Further measured workloads, one JSON line each (not the headline line).

    anomaly-batched: three layered media with Gaussian anomalies (seeds 31,
      32, 33) on 128^2, 256^2, 512^2 (h = 10 m) at 5, 10, ..., 40 Hz with 64
      sources each (1536 solves), solved through lsw_solve_batched (HODLR with
      32 x 32 leaves, rank 20 + 10, FP32; FP32 FGMRES(30) in FP64 refinement
      to 1e-6), four problems at a time; --rank-max R lets a problem that
      does not converge be rebuilt with a doubled rank, up to R.
    layered-salt-256: a 256^2 layered medium with a salt ellipse (h = 10 m,
      15 Hz, 32 sources on the top row), HODLR with 32 x 32 leaves (6 levels),
      rank 20 + 10, FP32, mixed-precision FGMRES(30) to 1e-6; the build is in
      every step.
    marmousi-subset-sweep / salt-subset-sweep: the paper's own experiment
      shapes (Sec. 3.1, 3.2): a 248 x 81 Marmousi-like model at h = 15 m
      embedded in a 256 x 128 grid, or a 700 x 150 salt model at h = 10 m
      embedded in 1024 x 256 (zero contrast outside, which is exact), one
      source in the middle of the top row, the integer frequencies 1..20 Hz
      in ascending order through lsw_solve_sweep: HODLR with 32 x 32 leaves,
      FP32, 10 probes of oversampling, the paper's rank policy (start at 10,
      +10 after a failure within 30 iterations or a solve that needed more
      than 10, at most 50), and the paper's preconditioned series in FP32
      inside FP64 refinement to 1e-6 (--sweep-method fgmres: FGMRES(30)).
    c128-one-at-a-time-1024: the headline 1024^2 workload on the plain FP64
      path: c128 operator, HODLR in FP64 at the same rank, FGMRES(30) in FP64,
      one source per solve call, the build in every step.
    c128-one-at-a-time: the 256^2 salt workload on the plain FP64
      path, one source per solve call: c128 operator, HODLR in FP64, FGMRES(30)
      in FP64; the build is charged once per 32 sources."""
    import torch

    from paper_2005_01372_gb300 import lsw, media

    dev = torch.device("cuda", int(os.environ.get("LOCAL_RANK", "0")))
    torch.cuda.set_device(dev)
    if args.workload == "anomaly-batched":
        groups = []
        for n, seed, levels in ((128, 31, 4), (256, 32, 6), (512, 33, 8)):
            probs = []
            for f in (5.0, 10.0, 15.0, 20.0, 25.0, 30.0, 35.0, 40.0):
                wl = media.layered_anomaly(n, f, 64, seed)
                probs.append({"nz": n, "nx": n, "h": wl.h, "c0": wl.c0, "freq_hz": f, "sources": wl.sources,
                              "velocity": torch.from_numpy(np.ascontiguousarray(wl.velocity.ravel())).to(dev)})
            hp = lsw.HParams(kind=lsw.H_HODLR, prec=lsw.C64, levels=levels, rank=20, oversample=10, seed=1002,
                             rank_max=args.rank_max)
            groups.append((probs, hp))
        sp = lsw.SolveParams(prec=lsw.MIXED, method=lsw.FGMRES, tol=TOL, inner_tol=1e-3, restart=30, max_iter=120,
                             max_outer=8)

        def step():
            ok, total, per = 0, 0, []
            for probs, hp in groups:
                _, infos = lsw.solve_batched(probs, hp, sp, max_concurrent=4)
                for p, inf in zip(probs, infos):
                    good = sum(1 for i in inf if i.status == 0 and i.rel_residual <= TOL)
                    ok += good
                    total += len(inf)
                    per.append(good)
            return ok, total, per
        cfg = {"workload": "layered-anomaly-{128,256,512}^2-5..40Hz-64src-batched", "problems": 24,
               "sources_per_problem": 64,
               "preconditioner": f"HODLR 32x32 leaves, rank 20+10, FP32, rank raised up to {args.rank_max}"
               if args.rank_max > 20 else "HODLR 32x32 leaves, rank 20+10, FP32",
               "solver": "FGMRES(30) in FP64 refinement to 1e-6, lsw_solve_batched, 4 concurrent"}
    elif args.workload == "layered-salt-256":
        wl = media.layered_salt(256, 15.0, 32, 2)
        vel = torch.from_numpy(np.ascontiguousarray(wl.velocity.ravel())).to(dev)
        hp = lsw.HParams(kind=lsw.H_HODLR, prec=lsw.C64, levels=6, split=lsw.SPLIT_QUADTREE, rank=20,
                         oversample=10, q=0, seed=1002)
        sp = lsw.SolveParams(prec=lsw.MIXED, method=lsw.FGMRES, tol=TOL, inner_tol=1e-3, restart=30, max_iter=60,
                             max_outer=8)

        def step():
            G = lsw.build_green(wl.nz, wl.nx, wl.h, wl.c0, wl.freq_hz)
            chi = G.contrast(vel)
            u0 = G.point_sources(wl.sources, lsw.C128)
            H = lsw.build_hmatrix(G, chi, hp)
            _, infos = lsw.solve_series(G, chi, H, u0, sp=sp)
            ok = sum(1 for i in infos if i.status == 0 and i.rel_residual <= TOL)
            return ok, len(infos), None
        cfg = {"workload": "layered-salt-256x256-15Hz-32src", "grid": "256x256", "h_m": 10.0, "freq_hz": 15.0,
               "preconditioner": "HODLR quadtree 32x32 leaves, 6 levels, rank 20+10, q=0, FP32",
               "solver": "FGMRES(30) right-preconditioned, FP64 iterative refinement to 1e-6"}
    elif args.workload in ("marmousi-subset-sweep", "salt-subset-sweep"):
        wl = media.marmousi_subset() if args.workload.startswith("marmousi") else media.salt_subset()
        vel = torch.from_numpy(np.ascontiguousarray(wl.velocity.ravel())).to(dev)
        levels = int(np.log2(wl.n // 1024))
        hp = lsw.HParams(kind=lsw.H_HODLR, prec=lsw.C64, levels=levels, oversample=10, seed=1005)
        pol = lsw.SweepPolicy(rank0=10, rank_step=10, rank_max=50, raise_iters=10)
        m = lsw.FGMRES if args.sweep_method == "fgmres" else lsw.SERIES
        sp = lsw.SolveParams(prec=lsw.MIXED, method=m, tol=TOL, inner_tol=1e-3, restart=30, max_iter=30,
                             max_outer=8)
        freqs = [float(f) for f in range(1, 21)]
        per_f = []

        def step():
            _, info, _ = lsw.solve_sweep(wl.nz, wl.nx, wl.h, wl.c0, vel, freqs, wl.sources, hp, pol, sp)
            per_f[:] = [{"f": i.freq_hz, "rank": i.rank, "builds": i.builds, "iters": i.max_iterations,
                         "status": i.status} for i in info]
            ok = sum(i.converged for i in info)
            return ok, len(freqs) * len(wl.sources), None
        cfg = {"workload": wl.name, "grid": f"{wl.nx}x{wl.nz} (x by z)", "h_m": wl.h, "freqs_hz": "1..20",
               "preconditioner": f"HODLR 32x32 leaves, {levels} levels, FP32, rank 10..50 by the paper's policy",
               "solver": ("FGMRES(30)" if m == lsw.FGMRES else "preconditioned series (<= 30 steps)")
               + " in FP64 refinement to 1e-6, lsw_solve_sweep"}
    elif args.workload == "c128-one-at-a-time-1024":
        wl = media.marmousi_1024()
        vel = torch.from_numpy(np.ascontiguousarray(wl.velocity.ravel())).to(dev)
        hp = lsw.HParams(kind=lsw.H_HODLR, prec=lsw.C128, levels=LEVELS, rank=RANK, oversample=OVERSAMPLE,
                         seed=SEED)
        sp = lsw.SolveParams(prec=lsw.C128, method=lsw.FGMRES, tol=TOL, restart=30, max_iter=1200)

        def step():
            G = lsw.build_green(wl.nz, wl.nx, wl.h, wl.c0, wl.freq_hz)
            chi = G.contrast(vel)
            H = lsw.build_hmatrix(G, chi, hp)
            ok = 0
            for s in wl.sources:
                u0 = G.point_sources([s], lsw.C128)
                _, inf = lsw.solve_series(G, chi, H, u0, sp=sp)
                ok += sum(1 for i in inf if i.status == 0 and i.rel_residual <= TOL)
            return ok, len(wl.sources), None
        cfg = {"workload": WORKLOAD, "path": "c128 operator, FP64 HODLR (rank 40+10), FP64 FGMRES(30), one source "
                                             "per call"}
    else:
        wl = media.layered_salt(256, 15.0, 32, 2)
        vel = torch.from_numpy(np.ascontiguousarray(wl.velocity.ravel())).to(dev)
        hp = lsw.HParams(kind=lsw.H_HODLR, prec=lsw.C128, levels=6, rank=20, oversample=10, seed=1002)
        sp = lsw.SolveParams(prec=lsw.C128, method=lsw.FGMRES, tol=TOL, restart=30, max_iter=300)

        def step():
            G = lsw.build_green(wl.nz, wl.nx, wl.h, wl.c0, wl.freq_hz)
            chi = G.contrast(vel)
            H = lsw.build_hmatrix(G, chi, hp)
            ok = 0
            for s in wl.sources:
                u0 = G.point_sources([s], lsw.C128)
                _, inf = lsw.solve_series(G, chi, H, u0, sp=sp)
                ok += sum(1 for i in inf if i.status == 0 and i.rel_residual <= TOL)
            return ok, len(wl.sources), None
        cfg = {"workload": "layered-salt-256x256-15Hz-32src",
               "path": "c128 operator, FP64 HODLR, FP64 FGMRES(30), one source per call"}
    for _ in range(args.warmup):
        step()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    ok = total = 0
    per = None
    for _ in range(args.steps):
        o, t, per = step()
        ok += o
        total += t
    torch.cuda.synchronize()
    wall = time.perf_counter() - t0
    line = {"metric": METRIC.split(";")[0], "value": round(ok / wall, 3), "unit": "solves/s", "n_gpus": 1,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": round(1e3 * wall / args.steps, 1),
            "higher_is_better": True, "solves_converged": ok, "solves_attempted": total, "config": cfg}
    if per is not None:
        line["converged_per_problem"] = per
    if args.workload.endswith("-sweep"):
        line["per_frequency"] = per_f
    print(json.dumps(line), flush=True)


# Operator applies per solve of the headline workload on the GPU path (inner
# FGMRES iterations + FP64 residuals, mean over the 16 sources), measured by
# this bench on GB300 ("operator_applies_per_solve" of its line).  The
# reference arm, which runs without a GPU, converts its per-apply time to
# solves/s with it.
APPLIES_PER_SOLVE = 300.0


class OracleArm:
    """The CPU oracle, as it stands, on a bounded sample of the workload.

    A complete oracle solve of the 1024^2 workload is out of reach: its
    HODLR preconditioner has 1024 dense leaves of 1024 x 1024 (16 GB in
    complex128) and a recursive inversion of hours.  What the oracle can do
    in bounded time is the part every solve repeats most: one FP64
    application of I - G0 V (RESIDUAL mode, the FFT convolution on the
    zero-padded 2048 x 2048 grid) for one source.  A step times one such
    apply; solves/s = 1 / (applies per solve x seconds per apply), with the
    GPU path's measured applies per solve.  Leaving out the preconditioner's
    build and apply makes this an upper bound on the oracle's solves/s."""

    def __init__(self):
        from oracle import operator as oop
        from paper_2005_01372_gb300 import media

        self.oop = oop
        self.cores = len(os.sched_getaffinity(0))
        self.wl = media.marmousi_1024()
        self.P = oop.Problem.from_workload(self.wl)
        self.u0 = self.P.sources(self.wl.sources[:1])
        self.k = 0

    def step(self):
        t0 = time.perf_counter()
        y = self.oop.apply(self.oop.RESIDUAL, self.P.spec, self.P.chi, self.u0, self.u0, self.P.nz, self.P.nx)
        t = time.perf_counter() - t0
        return t, bool(np.all(np.isfinite(y)))

    def sample_text(self, applies_per_solve: float, n: int):
        return ("same workload; %d FP64 RESIDUAL applies of I - G0 V on one 1024^2 source field (numpy FFT on "
                "the 2048^2 padded grid) timed, scaled by %.1f applies per solve; the oracle's HODLR build and "
                "apply (16 GB of complex128 leaves) are not run, so the value bounds the oracle from above"
                % (n, applies_per_solve))


def cpu_baseline(applies_per_solve: float = APPLIES_PER_SOLVE):
    """A bounded oracle sample (see OracleArm), reported with its sample."""
    arm = OracleArm()
    arm.step()
    ts = [arm.step()[0] for _ in range(3)]
    t_apply = float(np.mean(ts))
    return {"value": round(1.0 / (applies_per_solve * t_apply), 6), "unit": "solves/s", "cores": arm.cores,
            "kind": "oracle", "bound": "upper", "seconds_per_apply": round(t_apply, 4),
            "sample": arm.sample_text(applies_per_solve, len(ts))}


def run_reference(args):
    """The reference arm: the CPU oracle on the host cores (rank 0 only)."""
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    arm = OracleArm()
    for _ in range(args.warmup):
        arm.step()
    times = []
    for _ in range(args.steps):
        t, good = arm.step()
        times.append(t)
    t_apply = float(np.mean(times))
    v = 1.0 / (APPLIES_PER_SOLVE * t_apply)
    line = {"impl": "reference", "metric": METRIC, "value": round(v, 6), "unit": "solves/s", "n_gpus": 1,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": round(1e3 * APPLIES_PER_SOLVE * t_apply, 1),
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "c128", "data": "synthetic",
            "config": {"workload": WORKLOAD, "grid": "1024x1024", "h_m": 5.0, "freq_hz": 30.0,
                       "solver": "oracle FP64 operator applies only (bounded sample)"},
            "cpu_baseline": {"value": round(v, 6), "unit": "solves/s", "cores": arm.cores, "kind": "oracle",
                             "bound": "upper", "sample": arm.sample_text(APPLIES_PER_SOLVE, args.steps)},
            "e2e": {"value": round(v, 6), "unit": "solves/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=2)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--workload", default=WORKLOAD, choices=[WORKLOAD, "layered-salt-256", "anomaly-batched",
                                                              "c128-one-at-a-time", "c128-one-at-a-time-1024",
                                                              "marmousi-subset-sweep", "salt-subset-sweep"],
                    help="the headline workload (default) or a further measured one")
    ap.add_argument("--rank-max", type=int, default=0, help="anomaly-batched: rank adaptation limit (0: off)")
    ap.add_argument("--sweep-method", default="series", choices=["series", "fgmres"],
                    help="*-subset-sweep: the paper's preconditioned series or FGMRES(30)")
    args = ap.parse_args()
    if args.impl == "reference":
        run_reference(args)
    elif args.workload != WORKLOAD:
        run_extra(args)
    else:
        run_ours(args)


if __name__ == "__main__":
    main()
