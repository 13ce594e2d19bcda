#!/usr/bin/env python
"""Benchmark of the batched EFM collision step on GB300.

Workload (one "step"): 4096 spatial cells in 3D, N drawn uniformly from {24, 32, 40, 48}, box
[-8, 8]^3, hard-sphere kernel, angular rank R = 32, FP32 transforms and products; each step is one
forward-Euler update F <- F + dt Q^sigma[F] (dt = 0.01) of every cell with the fused FP64 moment,
entropy and entropy-production reductions, launched through the C ABI (one graph-captured launch
per distinct N).  Inputs are Maxwellians (density U[0.5,2], |u| <= 1, temperature U[0.5,2]) times
(1 + 0.3 sum of 3 Gaussian bumps), renormalised, seed 1234 (+ rank).

Metric: collision evaluations per second counted as cell grid points, sum_cells N^3 per second.
Timing: W warm-up steps, then K steps between CUDA events on the launching stream, bracketed by a
barrier and device synchronisation; max over ranks.  The inputs (about 0.9 GB) exceed the L2.

After the timed steps (N = 1 only) the "surrogate" object compares the learned surrogate with the
plain operator on 16384-cell batches (N = 32, hard-sphere and Maxwell kernels): throughput of both
on the same resident batch, and the accuracy of the band the surrogate path delivers: the guarded
policies (a checker network sends the cells it doubts to the plain operator, Q returned on the
grid) and the audit policies (none; any audited miss sends the whole batch to the plain operator;
more than 5% of audited cells missing does).  --no-surrogate skips it.  The "hbm_kernels" object then times the
library's HBM-bound kernels (moments / entropy and free transport) on resident N = 32 batches
against the measured HBM copy rate; --no-kernels skips it.  The line carries these legs' figures of
merit; their full reports go to standard error.

--impl reference times the FP64 CPU oracle (direct O(R N^6) sum of the paper's operator) on the
host cores, on a bounded sample of the same workload.
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

METRIC = "collision evals/sec (cells×N^d) and HBM GB/s vs roofline; surrogate vs plain"
UNIT = "cell-points/s"
L_BOX = 8.0
R_RANK = 32
DT = 0.01
N_CHOICES = (24, 32, 40, 48)


def workload_config(ncells):
    return {"workload": "batched 3D hard-sphere EFM Euler step: %d cells, N~U{24,32,40,48}, L=8, R=32, "
                        "FP32 transforms, FP64 moments/entropy" % ncells,
            "cells": ncells, "N_choices": list(N_CHOICES), "L": L_BOX, "kernel": "hard_sphere",
            "R": R_RANK, "dt": DT, "launch": "one graph-captured persistent cluster launch per N",
            "l2": "inputs larger than L2 (about 0.9 GB of FP32 cells)"}


# ------------------------------------------------------------------ per-cell work model ------

def n_ops(R=R_RANK):
    """Inverse 3D transforms per cell.  The hard-sphere kernel's R = 2 n_mu n_phi n_c terms share
    n_e = n_mu n_phi first directions; by linearity each e needs two transforms (a_e and the
    weighted sum of its partners), plus one for the loss: 2 n_e + 1 (R = 32 -> 17)."""
    table = {32: (2, 4, 2), 64: (2, 4, 4)}
    nmu, nphi, nc = table[R]
    return 2 * nmu * nphi + 1


def flops_per_cell(N, R=R_RANK):
    """Algorithmic FP32 flops of one collision evaluation of one cell, counted as the work model of
    the hot-path scope: (#transforms) real 3D FFTs at 2.5 M log2 M flops each (M = N^3) plus 2 R M
    for the R-term products, with #transforms = n_mu n_phi (1 + n_c) + 2 for the hard-sphere
    decomposition (a transform per first direction, one per partner direction, the forward
    transform and the loss): 26 for R = 32.  The kernel itself runs fewer transforms (see
    executed_flops_per_cell), so this is the work of the method, not of the implementation."""
    table = {32: (2, 4, 2), 64: (2, 4, 4)}
    nmu, nphi, nc = table[R]
    M = float(N) ** 3
    return (nmu * nphi * (1 + nc) + 2) * 2.5 * M * np.log2(M) + 2.0 * R * M


def executed_flops_per_cell(N, R=R_RANK):
    """The flops the kernel actually executes under the same per-transform count: 1 forward and
    n_ops inverse transforms (partners folded by linearity), the spectral multiply (2 flops per
    half-spectrum complex value) and the accumulate (2 flops per point per op)."""
    M = float(N) ** 3
    ops = n_ops(R)
    return (1 + ops) * 2.5 * M * np.log2(M) + ops * (M + 2.0 * M)


def bytes_per_cell(N):
    """Algorithmic HBM bytes: read F once, write F once (FP32)."""
    return 8.0 * float(N) ** 3


# ------------------------------------------------------------------ clocks -------------------

class ClockSampler:
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index):
        self.index = index
        self.proc = None
        self.lines = []

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.index), "--query-gpu=" + self.FIELDS, "--format=csv,noheader,nounits",
                 "-lms", "200"], stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
        except Exception:
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
        except Exception:
            self.proc.kill()
        sm, smax, reasons = [], [], set()
        names = ("hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap")
        for ln in self.lines:
            parts = [p.strip() for p in ln.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                smax.append(float(parts[2]))
            except ValueError:
                continue
            for nm, v in zip(names, parts[5:9]):
                if v.lower() == "active":
                    reasons.add(nm)
        return {"sm_mhz": float(np.median(sm)) if sm else None, "sm_max_mhz": max(smax) if smax else None,
                "reasons": sorted(reasons), "samples": len(sm)}


# ------------------------------------------------------------------ distributed helpers ------

def dist_setup(args):
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1:
        import torch.distributed as dist
        backend = "nccl" if args.impl == "ours" else "gloo"
        if backend == "nccl":
            import torch
            torch.cuda.set_device(local)
        dist.init_process_group(backend=backend)
    return world, rank, local


def barrier(world):
    if world > 1:
        import torch.distributed as dist
        dist.barrier()


def max_over_ranks(world, x, device=None):
    if world == 1:
        return x
    import torch
    import torch.distributed as dist
    t = torch.tensor([x], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


# ------------------------------------------------------------------ CPU oracle legs ----------

def oracle_cell_seconds(N, seed):
    import oracle
    from paper_1704_07369_gb300 import inputs
    F = inputs.mixture_cell(3, N, L_BOX, seed)
    p = oracle.Params(d=3, N=N, T=L_BOX, kernel=oracle.KERNEL_HARD_SPHERE, R=R_RANK)
    t0 = time.perf_counter()
    oracle.collide(p, F)
    return time.perf_counter() - t0


def mix_rate_from_samples(samples):
    """Cell-points/s of the oracle on the N mix from timed cells, extrapolating the direct sum's
    N^6 cost (fit through the timed sizes) to the untimed sizes."""
    Ns = np.array(sorted(samples))
    ts = np.array([samples[n] for n in Ns])
    if len(Ns) >= 2:
        expo = np.polyfit(np.log(Ns), np.log(ts), 1)[0]
    else:
        expo = 6.0
    t_of = {n: samples.get(n, ts[-1] * (n / Ns[-1]) ** expo) for n in N_CHOICES}
    mean_pts = np.mean([n ** 3 for n in N_CHOICES])
    mean_t = np.mean([t_of[n] for n in N_CHOICES])
    return mean_pts / mean_t, expo, t_of


def cpu_baseline():
    import oracle
    oracle.build()
    samples = {24: oracle_cell_seconds(24, 1234), 32: oracle_cell_seconds(32, 1235)}
    rate, expo, t_of = mix_rate_from_samples(samples)
    return {"value": rate, "unit": UNIT, "cores": oracle.num_threads(), "kind": "oracle",
            "sample": "one full N=24 cell (%.2f s) and one N=32 cell (%.2f s), FP64 direct sum of eq. Qsk "
                      "(O(R N^6)); N=40/48 extrapolated with the fitted cost exponent %.2f" %
                      (samples[24], samples[32], expo)}


def run_reference(args, world, rank):
    if rank != 0:
        return 0
    import oracle
    oracle.build()
    times = []
    for i in range(args.warmup + args.steps):
        dt = oracle_cell_seconds(24, 1234 + i)
        if i >= args.warmup:
            times.append(dt)
    t24 = float(np.mean(times))
    rate, expo, _ = mix_rate_from_samples({24: t24})
    line = {"impl": "reference", "metric": METRIC, "value": rate, "unit": UNIT, "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": t24 * 1e3, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": workload_config(args.cells),
            "cpu_baseline": {"value": rate, "unit": UNIT, "cores": oracle.num_threads(), "kind": "oracle",
                             "sample": "each step: one full N=24 cell of the workload by the FP64 direct sum "
                                       "(eq. Qsk); rate on the N mix extrapolated with cost ~ N^6"},
            "e2e": {"value": rate, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)
    return 0


# ------------------------------------------------------------------ GPU arm -----------------

def run_ours(args, world, rank, local):
    import torch

    import paper_1704_07369_gb300 as ef
    from paper_1704_07369_gb300 import inputs

    device = torch.device("cuda", local)
    torch.cuda.set_device(device)
    ef.build()
    if "EF_AUTOTUNE_CACHE" not in os.environ:
        # plans of the same sizes (the batch and the streamed leg's chunks) share one tuning
        import tempfile
        os.environ["EF_AUTOTUNE_CACHE"] = os.path.join(tempfile.mkdtemp(prefix="ef_tune_"), "tune.txt")
    if args.strong:
        # one global batch, split over the ranks by work (every rank computes the same split)
        from paper_1704_07369_gb300 import shard
        Ns_all = inputs.ragged_sizes(args.cells, seed=1234)
        mine = shard.partition(Ns_all, world)[rank]
        Ns = Ns_all[mine]
        cell_seeds = 1234 + mine
        total_pts_all = float(np.sum(Ns_all.astype(np.float64) ** 3))
    else:
        # weak scaling: a batch of its own per rank
        seed = 1234 + 100003 * rank
        Ns = inputs.ragged_sizes(args.cells, seed=seed)
        cell_seeds = seed + np.arange(len(Ns))
        total_pts_all = None
    offs = np.concatenate([[0], np.cumsum(Ns.astype(np.int64) ** 3)])
    total_pts = int(offs[-1])
    host = torch.empty(total_pts, dtype=torch.float32, pin_memory=True)
    hv = host.numpy()
    for i, n in enumerate(Ns):
        hv[offs[i]:offs[i + 1]] = inputs.mixture_cell(3, int(n), L_BOX, int(cell_seeds[i])).ravel()
    plan = ef.Plan(3, None, L_BOX, ef.EF_KERNEL_HARD_SPHERE, R_RANK, ef.EF_PREC_F32, batched_N=Ns)
    plan.set_graph(True)
    F = host.to(device)
    diag = torch.zeros(args.cells, ef.EF_DIAG_STRIDE, dtype=torch.float64, device=device)
    stream = torch.cuda.Stream(device)
    nlaunch = len(set(int(n) for n in Ns))

    def step():
        plan.euler(F, DT, 1, diag, stream=stream)

    with torch.cuda.stream(stream):
        for _ in range(args.warmup):
            step()
    torch.cuda.synchronize()
    st = plan.status(sync=1, reset=1)
    if st not in (ef.EF_OK,):
        raise RuntimeError("device status %d after warm-up" % st)

    sampler = ClockSampler(local)
    barrier(world)
    torch.cuda.synchronize()
    sampler.start()
    time.sleep(0.3)
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    for _ in range(args.steps):
        step()
    e1.record(stream)
    torch.cuda.synchronize()
    barrier(world)
    ms = e0.elapsed_time(e1)
    clocks = sampler.stop()
    st = plan.status(sync=1, reset=1)
    ms_max = max_over_ranks(world, ms, device)
    step_s = ms_max / 1e3 / args.steps
    pts_per_step = float(total_pts)
    job_pts = total_pts_all if args.strong else pts_per_step * world
    value = job_pts / step_s

    # roofline of the collide kernel (the only kernel in the step): algorithmic FP32 flops per
    # launch over the average launch duration (launches are back to back on the stream)
    flops_step = float(sum(flops_per_cell(int(n)) for n in Ns))
    bytes_step = float(sum(bytes_per_cell(int(n)) for n in Ns))
    per_launch_s = step_s / nlaunch
    sm_clock = 2070.0
    fp32_peak = 152 * 128 * 2 * sm_clock * 1e6 / 1e12       # TFLOP/s at the maximum SM clock
    achieved_tf = flops_step / nlaunch / per_launch_s / 1e12
    peaks_path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    hbm_peak = 6800.0
    hbm_src = "fallback"
    if os.path.exists(peaks_path):
        with open(peaks_path) as f:
            hbm_peak = float(json.load(f).get("hbm_gbs", hbm_peak))
            hbm_src = "measured"
    traffic = None
    tpath = os.path.join(ROOT, "profiles", "traffic.json")
    if os.path.exists(tpath):
        with open(tpath) as f:
            tj = json.load(f)
        if tj.get("kernel_hash") == ef_kernel_hash():
            traffic = tj.get("bytes_per_launch_full_step")
    exec_tf = float(sum(executed_flops_per_cell(int(n)) for n in Ns)) / nlaunch / per_launch_s / 1e12
    roof = {"bound": "alu", "achieved": achieved_tf, "peak": fp32_peak, "unit": "TFLOP/s",
            "frac": achieved_tf / fp32_peak, "traffic": traffic,
            "work_model": "(n_mu n_phi (1 + n_c) + 2) 2.5 M log2 M + 2 R M flops per cell, M = N^3 (26 transforms at R = 32)",
            "executed": {"TFLOP_s": exec_tf, "frac": exec_tf / fp32_peak,
                         "model": "18 transforms per cell actually run (partners folded by linearity)"},
            "peak_source": "FP32 CUDA-core peak from unit counts: 152 SMs x 128 lanes x 2 flop x 2070 MHz",
            "hbm_view": {"achieved_GBps": bytes_step / step_s / 1e9, "peak_GBps": hbm_peak,
                         "frac": bytes_step / step_s / 1e9 / hbm_peak, "peak_source": hbm_src}}

    # end to end through the C ABI with host buffers: every step uploads F from pinned host memory,
    # steps it and downloads F and the diagnostics, through ef_stream_euler_step, which cuts the
    # batch into chunks on their own streams so that the copies overlap other chunks' steps
    e2e = None
    if not args.no_e2e:
        sp = ef.StreamPlan(3, Ns, L_BOX, ef.EF_KERNEL_HARD_SPHERE, R_RANK, ef.EF_PREC_F32, nchunks=args.chunks)
        ehost = host.clone().pin_memory()
        diag_host = torch.empty(diag.shape, dtype=torch.float64, pin_memory=True)
        for _ in range(2):
            sp.euler(ehost, DT, 1, diag_host, stream=stream)
        torch.cuda.synchronize()
        # the raw copy rates of this pinned buffer, outside the timed region (context for the
        # end-to-end time, which they bound from below)
        dcopy = torch.empty(ehost.shape, dtype=ehost.dtype, device=device)
        cev = [torch.cuda.Event(enable_timing=True) for _ in range(3)]
        with torch.cuda.stream(stream):
            dcopy.copy_(ehost, non_blocking=True)
            cev[0].record(stream)
            dcopy.copy_(ehost, non_blocking=True)
            cev[1].record(stream)
            ehost.copy_(dcopy, non_blocking=True)
            cev[2].record(stream)
        torch.cuda.synchronize()
        nbytes = ehost.numel() * ehost.element_size()
        copy_rates = {"h2d_GBps": nbytes / cev[0].elapsed_time(cev[1]) / 1e6,
                      "d2h_GBps": nbytes / cev[1].elapsed_time(cev[2]) / 1e6}
        # both directions at once, as the pipelined step runs them (half the buffer each way)
        half = ehost.numel() // 2
        s2 = torch.cuda.Stream()
        cev[0].record(stream)
        s2.wait_event(cev[0])
        with torch.cuda.stream(stream):
            dcopy[:half].copy_(ehost[:half], non_blocking=True)
        with torch.cuda.stream(s2):
            ehost[half:].copy_(dcopy[half:], non_blocking=True)
        cev[1].record(s2)
        stream.wait_event(cev[1])
        cev[2].record(stream)
        torch.cuda.synchronize()
        copy_rates["both_directions_GBps"] = nbytes / cev[0].elapsed_time(cev[2]) / 1e6
        del dcopy
        barrier(world)
        k = max(1, min(args.steps, 10))
        t0 = torch.cuda.Event(enable_timing=True)
        t1 = torch.cuda.Event(enable_timing=True)
        t0.record(stream)
        h0 = time.perf_counter()
        for _ in range(k):
            sp.euler(ehost, DT, 1, diag_host, stream=stream)
        enqueue_ms = (time.perf_counter() - h0) * 1e3 / k      # host time to issue one step's work
        t1.record(stream)
        torch.cuda.synchronize()
        e2e_ms = max_over_ranks(world, t0.elapsed_time(t1), device) / k
        e2e = {"value": job_pts / (e2e_ms / 1e3), "unit": UNIT,
               "h2d_bytes_per_step": ehost.numel() * 4,
               "d2h_bytes_per_step": ehost.numel() * 4 + diag_host.numel() * 8,
               "ms_per_step": e2e_ms, "chunks": sp.info()["chunks"], "copy_rates_of_the_buffer": copy_rates,
               "host_issue_ms_per_step": enqueue_ms,
               "api": "ef_stream_euler_step (uploads, steps on four compute streams, downloads: overlapped)",
               "status": int(sp.status(sync=1, reset=1))}
        sp.close()

    if rank != 0:
        return 0
    cfg = workload_config(args.cells)
    cfg["shapes"] = [{k: v for k, v in ci.items() if k in ("N", "cells", "cluster", "threads", "prefetch", "tuned_us")}
                     for ci in plan.class_info()]
    line = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": step_s * 1e3, "higher_is_better": True,
            "scaling": "strong" if args.strong else "weak",
            "vs_baseline": None, "dtype": "f32", "data": "synthetic", "config": cfg,
            "cells_per_s": (args.cells if args.strong else args.cells * world) / step_s, "status": int(st), "roofline": roof,
            "clocks": clocks, "e2e": e2e, "gpu_launches": nlaunch * args.steps}
    if not args.no_surrogate and world == 1:
        line["surrogate"] = surrogate_leg(args, device)
    if not args.no_kernels and world == 1:
        line["hbm_kernels"] = hbm_kernels_leg(device)
    if not args.no_precision and world == 1:
        line["precision"] = precision_leg(device)
    if not args.no_cpu_baseline and world == 1:
        line["cpu_baseline"] = cpu_baseline()
    elif not args.no_cpu_baseline:
        line["cpu_baseline"] = None
    short, full = printed_line(line)
    if full:
        print("extra legs in full: " + json.dumps(full), file=sys.stderr, flush=True)
    print(json.dumps(short), flush=True)
    return 0


def printed_line(line):
    """(the line to print, what it leaves out).  The extra legs' reports (surrogate, hbm_kernels, precision) run
    to tens of kilobytes, and a reader that keeps only the end of the output would lose the line they are in: in
    the line each is cut down to its figures of merit, and all of it goes to standard error."""
    short, full = dict(line), {}

    def num(x):
        return float("%.5g" % x) if isinstance(x, float) else x

    def pick(d, keys):
        return {k: num(d[k]) for k in keys if k in d}

    for leg in ("surrogate", "hbm_kernels", "precision"):
        rep = line.get(leg)
        if not isinstance(rep, dict):
            continue
        full[leg] = rep
        if "error" in rep:
            short[leg] = {"error": str(rep["error"])[:200]}
        elif leg == "surrogate":
            short[leg] = {k: dict(pick(r, ("plain_ms",)),
                                  speedup_vs_plain={p: num(v["speedup_vs_plain"]) for p, v in r["policies"].items()})
                          for k, r in rep.get("kernels", {}).items()}
        elif leg == "hbm_kernels":
            short[leg] = {k: num(v["frac_of_measured_hbm"]) for k, v in rep.items() if isinstance(v, dict)}
        else:
            short[leg] = {k: pick(v, ("fp32_ms", "fp64_ms", "fp32_ms_per_step", "fp64_ms_per_step", "gpu_ms_per_eval",
                                      "gpu_ms_per_step", "oracle_ms_per_step")) for k, v in rep.items() if isinstance(v, dict)}
    return short, full


# -------------------------------------------------------------- precision and small configs -

def precision_leg(device):
    """The workloads besides the batched step, each timed on the GPU (CUDA events) and compared with
    the FP64 oracle:
      config 4 (precision study): 256 BKW-family cells, 3D, N = 64, L = 10, hard spheres, R = 64, in
        FP32 and FP64; errors against the oracle at sampled points of two cells (the points where
        |Q| peaks among them), the mass each path puts into Q (exactly zero for the oracle's sum,
        eq. Qsk at k = 0), and the entropy production sum Q ln F per cell, FP32 against FP64 (the
        FP64 path being the one that matches the oracle to 1e-12);
      config 2: one BKW cell (t0 = 5.5), 3D, N = 32, L = 8, Maxwell molecules, R = 32, 200 Euler
        steps in FP64 and FP32: time per step, distance to the BKW solution at the end, FP32
        against FP64; the oracle's time per evaluation measured at N = 16 and extrapolated to
        N = 32 with the direct sum's N^6 cost;
      config 1: the 2D bi-Gaussian, N = 16, L = 8, Maxwell, R = 16, FP64: one evaluation plus 100
        Euler steps, GPU against the oracle step by step (time per step on both)."""
    import torch

    import oracle
    import paper_1704_07369_gb300 as ef
    from paper_1704_07369_gb300 import inputs
    out = {}
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]

    def timed(fn, reps):
        fn()
        torch.cuda.synchronize()
        ev[0].record()
        for _ in range(reps):
            fn()
        ev[1].record()
        torch.cuda.synchronize()
        return ev[0].elapsed_time(ev[1]) / reps

    try:
        oracle.build()
        # ---- config 4
        N, L, R, n = 64, 10.0, 64, 256
        cells = inputs.bkw_family_cells(3, N, L, n, seed=4321)
        c4 = {"workload": "256 BKW-family cells, 3D, N=64, L=10, hard spheres, R=64", "cells": n}
        Q = {}
        for prec, name in ((ef.EF_PREC_F32, "fp32"), (ef.EF_PREC_F64, "fp64")):
            plan = ef.Plan(3, N, L, ef.EF_KERNEL_HARD_SPHERE, R, prec)
            dt = torch.float32 if prec == ef.EF_PREC_F32 else torch.float64
            F = torch.tensor(cells, dtype=dt, device=device)
            Qd = torch.empty_like(F)
            ms = timed(lambda: plan.collide(F, Qd, ncells=n), 3)
            mom = torch.zeros(n, ef.EF_DIAG_STRIDE, dtype=torch.float64, device=device)
            plan.moments(F, Qd, mom, ncells=n)
            torch.cuda.synchronize()
            c4[name + "_ms"] = ms
            c4[name + "_cells_per_s"] = n / ms * 1e3
            c4[name + "_status"] = int(plan.status(sync=1, reset=1))
            h3 = (2 * L / N) ** 3
            mass = mom[:, 0].double().cpu().numpy()
            dmass = Qd.double().sum(dim=(1, 2, 3)).cpu().numpy() * h3
            c4.setdefault("mass_of_Q_rel", {})[name] = float(np.abs(dmass / mass).max())
            Q[name] = (Qd[:2].double().cpu().numpy(), mom[:, 6].cpu().numpy())
            del F, Qd, plan
            torch.cuda.empty_cache()
        p4 = oracle.Params(d=3, N=N, T=L, kernel=oracle.KERNEL_HARD_SPHERE, R=R, J=6)
        err32, err64, npts = 0.0, 0.0, 0
        for i in range(2):
            q32, q64 = Q["fp32"][0][i].ravel(), Q["fp64"][0][i].ravel()
            idx = np.unique(np.concatenate([np.argsort(np.abs(q64))[-8:], np.random.default_rng(i).integers(0, q64.size, 56)]))
            ref = oracle.collide_points_fft(p4, cells[i], idx)
            sc = np.abs(ref).max()
            err32 = max(err32, float(np.abs(q32[idx] - ref).max() / sc))
            err64 = max(err64, float(np.sqrt(((q64[idx] - ref) ** 2).sum() / (ref ** 2).sum())))
            npts += idx.size
        c4["Q_vs_oracle_sampled"] = {"fp32_rel_linf_of_max": err32, "fp64_rel_l2": err64, "points": npts, "cells": 2}
        P32, P64 = Q["fp32"][1], Q["fp64"][1]
        c4["entropy_production_fp32_vs_fp64"] = {"max_rel": float(np.abs((P32 - P64) / P64).max()),
                                                 "same_sign": bool(np.all(np.sign(P32) == np.sign(P64))),
                                                 "all_nonpositive_fp64": bool(np.all(P64 <= 0))}
        out["config4"] = c4
        # ---- config 2
        N, L, R, steps = 32, 8.0, 32, 200
        F0 = inputs.bkw(3, N, L, 5.5)
        c2 = {"workload": "BKW t0=5.5, 3D, N=32, L=8, Maxwell, R=32, 200 Euler steps dt=0.01"}
        fin = {}
        for prec, name in ((ef.EF_PREC_F64, "fp64"), (ef.EF_PREC_F32, "fp32")):
            plan = ef.Plan(3, N, L, ef.EF_KERNEL_MAXWELL, R, prec)
            dt = torch.float32 if prec == ef.EF_PREC_F32 else torch.float64
            F = torch.tensor(F0[None], dtype=dt, device=device)
            torch.cuda.synchronize()
            ev[0].record()
            plan.euler(F, 0.01, nsteps=steps, ncells=1)
            ev[1].record()
            torch.cuda.synchronize()
            c2[name + "_ms_per_step"] = ev[0].elapsed_time(ev[1]) / steps
            c2[name + "_status"] = int(plan.status(sync=1, reset=1))
            fin[name] = F[0].double().cpu().numpy()
        ex = inputs.bkw(3, N, L, 5.5 + steps * 0.01)
        for name in ("fp64", "fp32"):
            c2[name + "_rel_l2_vs_bkw_end"] = float(np.sqrt(((fin[name] - ex) ** 2).sum() / (ex ** 2).sum()))
        c2["fp32_vs_fp64_rel_linf"] = float(np.abs(fin["fp32"] - fin["fp64"]).max() / np.abs(fin["fp64"]).max())
        t0 = time.perf_counter()
        oracle.collide(oracle.Params(d=3, N=16, T=L, kernel=ef.EF_KERNEL_MAXWELL, R=R, J=6), inputs.bkw(3, 16, L, 5.5))
        t16 = time.perf_counter() - t0
        c2["oracle_s_per_eval"] = {"N16_measured": t16, "N32_extrapolated_N6": t16 * 64.0, "cores": oracle.num_threads()}
        out["config2"] = c2
        # ---- config 1
        N, L, R = 16, 8.0, 16
        F0 = inputs.bigauss2d(N, L)
        plan = ef.Plan(2, N, L, ef.EF_KERNEL_MAXWELL, R, ef.EF_PREC_F64)
        F = torch.tensor(F0[None], dtype=torch.float64, device=device)
        Qd = torch.empty_like(F)
        ms_q = timed(lambda: plan.collide(F, Qd, ncells=1), 20)
        torch.cuda.synchronize()
        ev[0].record()
        plan.euler(F, 0.01, nsteps=100, ncells=1)
        ev[1].record()
        torch.cuda.synchronize()
        gpu_step = ev[0].elapsed_time(ev[1]) / 100
        p1 = oracle.Params(d=2, N=N, T=L, kernel=oracle.KERNEL_MAXWELL, R=R)
        t0 = time.perf_counter()
        Fo = oracle.euler(p1, F0, 0.01, steps=100)
        o_step = (time.perf_counter() - t0) / 100 * 1e3
        out["config1"] = {"workload": "2D bi-Gaussian, N=16, L=8, Maxwell, R=16, FP64, 1 evaluation + 100 Euler steps",
                          "gpu_ms_per_eval": ms_q, "gpu_ms_per_step": gpu_step, "oracle_ms_per_step": o_step,
                          "oracle_cores": oracle.num_threads(),
                          "rel_l2_vs_oracle_after_100": float(np.sqrt(((F[0].cpu().numpy() - Fo) ** 2).sum() / (Fo ** 2).sum())),
                          "status": int(plan.status(sync=1, reset=1))}
        return out
    except Exception as exc:          # reported, never fatal to the bench line
        out["error"] = "%s: %s" % (type(exc).__name__, exc)
        return out


# -------------------------------------------------------------- HBM-bound kernels ----------

def _measured_hbm_gbs():
    """The measured HBM copy rate of MEASURED_PEAKS.json (GB/s), else the 6800 GB/s fallback."""
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        with open(path) as f:
            return float(json.load(f).get("hbm_gbs", 6800.0))
    return 6800.0


def hbm_kernels_leg(device):
    """Device time and bandwidth of the library's HBM-bound kernels on resident FP32 N = 32 cells
    (CUDA events, 3 warm-up and 20 timed calls on the current stream; inputs far larger than L2):
    ef_moments_entropy on 16384 cells (F alone, then F and Q) and ef_transport_step on 4096
    cells.  Bytes are the algorithmic ones: each input value read once, each output written once."""
    import torch
    import paper_1704_07369_gb300 as ef
    try:
        peak = _measured_hbm_gbs()
        plan = ef.Plan(3, 32, 8.0, ef.EF_KERNEL_HARD_SPHERE, 32, ef.EF_PREC_F32)
        cell = 32 ** 3
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]

        def timed(fn, reps=20):
            for _ in range(3):
                fn()
            torch.cuda.synchronize()
            ev[0].record()
            for _ in range(reps):
                fn()
            ev[1].record()
            torch.cuda.synchronize()
            return ev[0].elapsed_time(ev[1]) / reps

        out = {}
        n = 16384
        F = torch.rand(n, 32, 32, 32, device=device) + 0.01
        Q = torch.rand_like(F) - 0.5
        mom = torch.zeros(n, ef.EF_DIAG_STRIDE, dtype=torch.float64, device=device)
        for name, q in (("moments_F", None), ("moments_FQ", Q)):
            ms = timed(lambda: plan.moments(F, q, mom, ncells=n))
            by = n * cell * 4 * (1 if q is None else 2) + n * ef.EF_DIAG_STRIDE * 8
            out[name] = {"cells": n, "ms": ms, "GBps": by / ms / 1e6, "frac_of_measured_hbm": by / ms / 1e6 / peak}
        del Q, mom
        n = 4096
        G = torch.empty(n, 32, 32, 32, device=device)
        ms = timed(lambda: plan.transport(F[:n], G, 0.25, 0.01, ncells=n))
        by = 2 * n * cell * 4
        out["transport"] = {"cells": n, "ms": ms, "GBps": by / ms / 1e6, "frac_of_measured_hbm": by / ms / 1e6 / peak}
        out["status"] = int(plan.status(sync=1, reset=1))
        del F, G
        torch.cuda.empty_cache()
        return out
    except Exception as exc:          # reported, never fatal to the bench line
        return {"error": "%s: %s" % (type(exc).__name__, exc)}


# ------------------------------------------------------------------ surrogate leg ----------

SUR_N = 32
SUR_CELLS = 16384
SUR_TRAIN = 204800
SUR_TOL = 1e-3
SUR_AUDIT = 0.02
SUR_BATCH = 512
SUR_HIDDEN = 768            # network width and depth (4 hidden layers)
SUR_LAYERS = 5
SUR_LR = 5e-4
SUR_LR1 = 1e-6
SUR_TARGET = 5.0            # speed-up over the plain operator the budgeted checker threshold is sized for
SUR_BUDGETS = (0.02, 0.04, 0.08)   # fixed budgets reported beside it


def _quantiles(e):
    import torch
    e = e.double()
    return {"mean": float(e.mean()), "p50": float(e.median()), "p90": float(torch.quantile(e, 0.9)),
            "p99": float(torch.quantile(e, 0.99)), "max": float(e.max()),
            "frac_le_tol": float((e <= SUR_TOL).double().mean())}


def surrogate_leg(args, device):
    """Surrogate vs plain on batches of 16384 BKW-family cells (3D, N = 32, L = 8), for the
    hard-sphere and Maxwell kernels: the network (928 -> 768 x 4 -> 926, bf16 weights, FP32
    accumulation) and a checker network of the same shape are trained on 204800 cells generated by
    the library; the checker threshold is calibrated on 16384 held-out cells; then plain-operator
    and surrogate throughput are timed on a third batch.  The guarded policies ("checked_*_to_grid")
    deliver the mean of the two networks, send the cells where they disagree most to the plain
    operator and return Q on the grid; they run without the entropy-production gate (the checker
    gate replaces it, and the band of ln F is half of the feature pass).  The budgeted threshold
    flags a fixed fraction of cells: the largest one that the measured cost of the guarded path
    (a line in the number of flagged cells through the times at the smallest and largest fixed
    budgets) keeps at SUR_TARGET times the plain operator, and fixed fractions beside it.  Every delivered band is
    compared cell by cell with the plain FP32 band (all cells) and the FP64 band (first 1024 cells),
    the grid Q with the plain Q, beside the band's truncation floor.  The other policies return the
    band only; the unaudited one judges no cell and is an upper bound of the speed, not a guarded
    result."""
    import torch

    import paper_1704_07369_gb300 as ef
    from paper_1704_07369_gb300 import inputs
    from paper_1704_07369_gb300 import surrogate as S

    out = {"workload": "3D BKW family (t0~U[0.5,10], rho~U[0.5,2], theta~U[0.5,2], |u|<=1), N=32, L=8, R=32, "
                       "FP32 plain operator vs bf16 MLP surrogate with gates, audit and fallback",
           "cells": SUR_CELLS, "train_cells": SUR_TRAIN, "epochs": args.sur_epochs, "batch": SUR_BATCH,
           "network": "928 -> %d x %d -> 926, ReLU, bf16 weights" % (SUR_HIDDEN, SUR_LAYERS - 1),
           "lr": SUR_LR, "lr_final": SUR_LR1, "tol": SUR_TOL, "inputs": "926 band floats + theta + relative entropy",
           "audit_fraction": SUR_AUDIT, "metric": "band rel-L2 per cell, modes |k|<=6", "kernels": {}}
    F = torch.empty(SUR_CELLS, SUR_N, SUR_N, SUR_N, device=device)
    Q = torch.empty_like(F)
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    for kern, name in ((ef.EF_KERNEL_HARD_SPHERE, "hard_sphere"), (ef.EF_KERNEL_MAXWELL, "maxwell")):
        plan = S.make_plan(kern, N=SUR_N, L=L_BOX)
        t0 = time.perf_counter()
        fF, fQ, fM = S.features_of_family(plan, SUR_TRAIN, seed=1000)
        data_s = time.perf_counter() - t0
        tr = S.Trainer(plan, nhidden=SUR_HIDDEN, nlayers=SUR_LAYERS, batch=SUR_BATCH, max_infer_batch=SUR_CELLS, seed=0)
        t0 = time.perf_counter()
        hist = tr.fit(fF, fQ, fM, epochs=args.sur_epochs, lr0=SUR_LR, lr1=SUR_LR1, warmup=0.05)
        torch.cuda.synchronize()
        train_s = time.perf_counter() - t0
        t0 = time.perf_counter()
        hist_c = tr.fit_checker(epochs=args.sur_epochs, lr0=SUR_LR, lr1=SUR_LR1, warmup=0.05)
        torch.cuda.synchronize()
        train_c_s = time.perf_counter() - t0
        del fF, fQ, fM
        tr._train_set = None
        # the checked policies run without the entropy-production gate (calibration included)
        tr.sur.set_entropy_gate(False)
        inputs.bkw_family_torch(SUR_N, L_BOX, SUR_CELLS, 9_000_000, device=device, out=F)
        # references: plain FP32 band of every cell, FP64 band of the first 1024
        plan.collide(F, Q, ncells=SUR_CELLS)
        ref = torch.zeros(SUR_CELLS, ef.EF_FEATURE_STRIDE, device=device)
        ef.ef_features(plan.handle, Q, ref, SUR_CELLS)
        n64 = 1024
        plan64 = S.make_plan(kern, N=SUR_N, L=L_BOX, prec=ef.EF_PREC_F64)
        F64 = F[:n64].double()
        Q64 = torch.empty_like(F64)
        plan64.collide(F64, Q64, ncells=n64)
        ref64 = torch.zeros(n64, ef.EF_FEATURE_STRIDE, device=device)
        ef.ef_features(plan64.handle, Q64, ref64, n64)
        del F64, Q64

        def timed(fn, reps):
            for i in range(3):
                fn(i)
            torch.cuda.synchronize()
            ev[0].record()
            for i in range(reps):
                fn(100 + i)
            ev[1].record()
            torch.cuda.synchronize()
            return ev[0].elapsed_time(ev[1]) / reps

        reps = max(3, min(args.steps, 10))
        plain_ms = timed(lambda i: plan.collide(F, Q, ncells=SUR_CELLS), reps)
        q = torch.zeros(SUR_CELLS, ef.EF_FEATURE_STRIDE, device=device)
        flags = torch.zeros(SUR_CELLS, dtype=torch.int32, device=device)
        Qg = torch.empty_like(F)
        # the guarded path's cost: its time with no cell flagged, and the plain operator's per cell;
        # the budget that keeps it at SUR_TARGET times the plain operator
        tr.sur.set_checker(tr.checker, 3.0e38)
        noflag_ms = timed(lambda i: tr.sur.infer_ex(F, q, flags, SUR_CELLS, Q=Qg, audit_fraction=0.0, seed=i, tol=SUR_TOL), reps)
        # checker thresholds from a held-out calibration batch (seeds disjoint from training and test)
        def calibrate_budgets(items):
            inputs.bkw_family_torch(SUR_N, L_BOX, SUR_CELLS, 8_000_000, device=device, out=F)
            out_b = {}
            for pname, b in items:
                thr_b, fl_b, _, left_b = tr.calibrate(F, SUR_CELLS, SUR_TOL, budget=max(b, 1.0 / SUR_CELLS))
                out_b[pname] = {"budget": b, "threshold": thr_b, "flagged_fraction": fl_b, "misses_left_unflagged": left_b}
            inputs.bkw_family_torch(SUR_N, L_BOX, SUR_CELLS, 9_000_000, device=device, out=F)
            return out_b

        inputs.bkw_family_torch(SUR_N, L_BOX, SUR_CELLS, 8_000_000, device=device, out=F)
        thr, cal_flagged, cal_miss, _ = tr.calibrate(F, SUR_CELLS, SUR_TOL, margin=0.8)
        cal_b = calibrate_budgets([("checked_budget%g_to_grid" % b, b) for b in SUR_BUDGETS])
        res = {"plain_ms": plain_ms, "plain_cells_per_s": SUR_CELLS / plain_ms * 1e3,
               "train": {"data_s": data_s, "train_s": train_s, "final_loss": hist[-1],
                         "checker_train_s": train_c_s, "checker_final_loss": hist_c[-1]},
               "checker_calibration": {"cells": SUR_CELLS, "misses_in_calibration_set": cal_miss,
                                       "catch_all": {"threshold": thr, "flagged_fraction": cal_flagged, "margin": 0.8},
                                       "budgets": cal_b},
               "policies": {}}
        # the guarded path end to end: checker gate, Q on the grid (band reconstruction where the
        # prediction is delivered, the plain operator's full Q where it is not), no audit; with the
        # threshold that flagged every calibration miss, and with the ones that flag fixed budgets
        proj = torch.empty(n64, SUR_N, SUR_N, SUR_N, device=device)
        ef.ef_features_inverse(plan.handle, ref[:n64], proj, n64)

        def guarded(pname, th):
            tr.sur.set_checker(tr.checker, th)
            ms = timed(lambda i: tr.sur.infer_ex(F, q, flags, SUR_CELLS, Q=Qg, audit_fraction=0.0, seed=i, tol=SUR_TOL), reps)
            f = flags.cpu().numpy()
            e = S.band_rel_l2(q, ref)
            e64 = S.band_rel_l2(q[:n64], ref64)
            # Q on the grid against the plain operator's full Q, and the band's own truncation floor
            # (the plain Q against its projection on the band), per cell over the first 1024 cells
            Qd, Gd, Pd = Q[:n64].double(), Qg[:n64].double(), proj.double()
            nrm = Qd.pow(2).sum(dim=(1, 2, 3)).sqrt()
            full_err = (Gd - Qd).pow(2).sum(dim=(1, 2, 3)).sqrt() / nrm
            floor = (Pd - Qd).pow(2).sum(dim=(1, 2, 3)).sqrt() / nrm
            del Qd, Gd, Pd
            res["policies"][pname] = {
                "audit_fraction": 0.0, "checker_threshold": th, "ms": ms, "cells_per_s": SUR_CELLS / ms * 1e3,
                "speedup_vs_plain": plain_ms / ms, "output": "Q on the grid (N^3 per cell)",
                "checker_flagged": int(((f & 32) != 0).sum()), "gated": int(((f & 1) != 0).sum()),
                "plain_used": int(((f & 8) != 0).sum()),
                "band_rel_l2_vs_fp32_plain": _quantiles(e), "band_rel_l2_vs_fp64_first1024": _quantiles(e64),
                "full_Q_rel_l2_vs_plain_first1024": _quantiles(full_err),
                "band_truncation_floor_first1024": {"p50": float(floor.median()), "max": float(floor.max()),
                                                    "mean": float(floor.mean())}}
            return ms, int(((f & 8) != 0).sum())

        guarded("checked_catch_all_to_grid", thr)
        probe = []
        for k, v in cal_b.items():
            probe.append(guarded(k, v["threshold"]))
        # the guarded path's time as a line in the number of flagged cells, through the fixed budgets
        # that flagged the fewest and the most (the fallback launches add a fixed cost, so the line's
        # intercept lies above the time with no cell flagged), and the budget that keeps the guarded
        # path at SUR_TARGET times the plain operator
        (ms_lo, n_lo), (ms_hi, n_hi) = min(probe, key=lambda t: t[1]), max(probe, key=lambda t: t[1])
        per_flag = max((ms_hi - ms_lo) / max(n_hi - n_lo, 1), plain_ms / SUR_CELLS)
        base_ms = max(noflag_ms, ms_lo - per_flag * n_lo)
        budget_t = max(0.0, (plain_ms / SUR_TARGET - base_ms) / (per_flag * SUR_CELLS))
        res["guarded_cost"] = {"no_cell_flagged_ms": noflag_ms, "with_fallback_base_ms": base_ms,
                               "ms_per_flagged_cell": per_flag, "plain_ms_per_cell_full_batch": plain_ms / SUR_CELLS,
                               "target_speedup": SUR_TARGET, "budget_for_target": budget_t}
        cal_t = calibrate_budgets([("checked_budget_to_grid", budget_t)])
        res["checker_calibration"]["budgets"].update(cal_t)
        guarded("checked_budget_to_grid", cal_t["checked_budget_to_grid"]["threshold"])
        del proj
        del Qg
        tr.sur.set_checker(None, 1.0)
        tr.sur.set_entropy_gate(True)
        # unguarded upper bound (nothing judges the cells) and the audit policies, band output only
        for pname, audit, max_miss in (("no_audit_unjudged", 0.0, 0.0), ("audit_strict", SUR_AUDIT, 0.0),
                                       ("audit_tolerant", SUR_AUDIT, 0.05)):
            tr.sur.set_policy(max_miss_fraction=max_miss)
            ms = timed(lambda i: tr.sur.infer(F, q, flags, SUR_CELLS, audit, i, SUR_TOL), reps)
            # the timed calls again, untimed, to count the draws that sent the batch to the plain operator
            fallbacks = 0
            for i in range(reps):
                tr.sur.infer(F, q, flags, SUR_CELLS, audit, 100 + i, SUR_TOL)
                fallbacks += int(((flags & 16) != 0).any().item())
            f = flags.cpu().numpy()
            e = S.band_rel_l2(q, ref)
            e64 = S.band_rel_l2(q[:n64], ref64)
            res["policies"][pname] = {
                "audit_fraction": audit, "max_miss_fraction": max_miss, "ms": ms,
                "cells_per_s": SUR_CELLS / ms * 1e3, "speedup_vs_plain": plain_ms / ms,
                "gated": int(((f & 1) != 0).sum()), "audited": int(((f & 2) != 0).sum()),
                "audit_misses": int(((f & 4) != 0).sum()), "plain_used": int(((f & 8) != 0).sum()),
                "batch_fallback": bool(((f & 16) != 0).any()), "timed_calls": reps, "batch_fallback_calls": fallbacks,
                "band_rel_l2_vs_fp32_plain": _quantiles(e), "band_rel_l2_vs_fp64_first1024": _quantiles(e64)}
        tr.sur.set_policy(0.0)
        out["kernels"][name] = res
        del tr, plan, plan64, ref, ref64, q, flags
        torch.cuda.empty_cache()
    return out


COLLIDE_SOURCES = ("ef_collide_impl.cuh", "ef_collide_rg.cuh", "ef_collide_tm.cuh", "ef_fft.cuh", "ef_internal.h",
                   "ef_collide_variant.inc", "ef_collide_f32_3d.cu", "ef_collide_rg_f32.cu", "ef_collide_rg_async_f32.cu",
                   "ef_collide_rg_split_f32.cu", "ef_collide_tm_f32.cu",
                   "ef_cluster_launch.h")


def ef_kernel_hash():
    """Hash of the sources that define the FP32 3D collide kernel: the stored DRAM traffic is
    reported only while they are unchanged."""
    import hashlib
    h = hashlib.sha256()
    d = os.path.join(ROOT, "paper_1704_07369_gb300", "csrc")
    for name in COLLIDE_SOURCES:
        with open(os.path.join(d, name), "rb") as f:
            h.update(f.read())
    return h.hexdigest()[:16]


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", choices=("ours", "reference"), default="ours")
    ap.add_argument("--cells", type=int, default=4096)
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-surrogate", action="store_true")
    ap.add_argument("--no-kernels", action="store_true", help="skip the HBM-bound kernels' timings")
    ap.add_argument("--no-precision", action="store_true",
                    help="skip the precision study (N = 64) and the small configurations' timings")
    ap.add_argument("--chunks", type=int, default=32, help="chunks of the streamed end-to-end leg")
    ap.add_argument("--strong", action="store_true",
                    help="split one --cells batch over the ranks (default: a batch per rank)")
    ap.add_argument("--sur-epochs", type=int, default=300)
    args = ap.parse_args()
    args.warmup = max(args.warmup, 3) if args.impl == "ours" else args.warmup
    world, rank, local = dist_setup(args)
    if args.impl == "reference":
        rc = run_reference(args, world, rank)
    else:
        rc = run_ours(args, world, rank, local)
    if world > 1:
        import torch.distributed as dist
        dist.destroy_process_group()
    return rc


if __name__ == "__main__":
    sys.exit(main())
