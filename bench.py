#!/usr/bin/env python
"""Throughput of the wavelet-Sobolev PAT reconstruction on GB300.

One step = one full reconstruction of the 3D 256^3 workload (the largest
single-GPU configuration): constant speed of sound 1500 m/s, order-4
staggered stencil, 800 time samples, 4096 sensors on a Fibonacci sphere,
p0 = a vessel tree plus 5 blobs, 1% noise, separable 3D db4 with 4 levels,
s = 1, alpha = 1e-2 relative to lambda_max of E_s* K* K E_s (estimated by
power iteration before timing), and 30 CG iterations on
(E_s* K* K E_s + alpha I) u = E_s* K* y (plus the right-hand side's K* and
the final E_s u).  Metric: reconstruction iterations per second (one K + one
K* per iteration), whole job.

With N > 1 (torchrun) every rank solves its own independently seeded
instance (weak scaling, no data-path collective).

--workload vessels times the 2D 512 x 512 workload instead: smooth random
speed of sound in [1400, 1600] m/s, order-8 stencil, 1500 time samples, 512
sensors on a circle, db4 with 5 levels; one step = its four reconstructions
(s in {1, 2} x alpha in {1e-3, 1e-2}, 100 CG iterations each) through
pat_solve_multi, two right-hand sides per persistent wave launch.

--workload batch64 times 64 independent reconstructions of uneven size
(n in {128..512}, order 8, 50 CG iterations each) through the batched
engine, one step = one batched solve, beside the same solves one after the
other.

--workload limited times the paper-like limited-view experiment: 512x512
with a 10-cell absorbing layer, 80 sensors along one face, data simulated
on a grid twice as fine, one step = one 15-iteration GMRES reconstruction.

--sweep prints one line per grid of the per-step engines' HBM sweep
(2D 2048^2 .. 16384^2 x orders {2, 8}, 4096^2 order 8 with a varying medium
and with a 10-cell absorbing layer, 3D 256^3 and 512^3 order 4).

--impl reference runs the FP64 CPU oracle (the reference arm): each step is
one oracle CG iteration of the same workload (for the volume, one K + K*
pair at 40 steps scaled linearly to the full 800).
"""
import argparse
import csv
import hashlib
import io
import json
import os
import statistics
import subprocess
import sys
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "reconstruction iterations/sec (K+K* pairs)"
UNIT = "iterations/s"
WORKLOAD = "tree3d"
# per workload: description, timed kernel, committed ncu summary and the sources it was taken on
WORKLOADS = {
    "vessels": {
        "desc": ("2D 512x512, c in [1400,1600] m/s (Gaussian-filtered noise), order-8 staggered FDTD, 1500 steps, "
                 "512 sensors on a circle, p0 = 4 blobs + 6 Bezier vessels, 2% noise, db4 5 levels, "
                 "s in {1,2} x alpha in {1e-3,1e-2}, 100 CG iterations, FP32 fields + FP64 CG scalars"),
        "kernel": "wave2d_persist_kernel<R=7,varc>",
        "profile": "wave2d_persist_512_o8.txt",
        "sources": ("wave2d_persist.cu", "persist2d.cuh", "tile2d.cuh", "stencil.cuh"),
        "oracle_nt": None,
    },
    "tree3d": {
        "desc": ("3D 256^3, c = 1500 m/s, order-4 staggered FDTD, 800 steps, 4096 sensors on a Fibonacci sphere, "
                 "p0 = vessel tree + 5 blobs, 1% noise, 3D db4 4 levels, s = 1, alpha = 1e-2, 30 CG iterations, "
                 "FP32 fields + FP64 CG scalars"),
        "kernel": "step3d_tma_kernel<R=3>",
        "profile": "step3d_tma_256_o4.txt",
        "sources": ("wave3d_tma.cu", "stencil.cuh", "tma.cuh"),
        "oracle_nt": 40,  # oracle samples: one K + K* pair at 40 steps, scaled linearly to 800
    },
    "limited": {
        "desc": ("2D 512x512 limited view: c = 1500 m/s, 10-cell absorbing layer, 80 sensors in a row inside one "
                 "face, order-8 staggered FDTD, 2414 steps, data simulated on a 1024x1024 grid at half the time "
                 "step and sampled at every second step (no inverse crime), 2% noise, db4 5 levels, s = 1, "
                 "alpha = 1e-2 (relative), 15 GMRES iterations on the paper's image-space system"),
        "kernel": "wave2d_persist_kernel<R=7> with the absorbing layer",
        "profile": "wave2d_persist_512_o8_layer.txt",
        "sources": ("wave2d_persist.cu", "persist2d.cuh", "tile2d.cuh", "stencil.cuh"),
        "oracle_nt": 40,
    },
}
WORKLOAD_DESC = WORKLOADS[WORKLOAD]["desc"]
L2_FLUSH_BYTES = 256 << 20


def peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            d = json.load(f)
        return float(d["hbm_gbs"]), "measured"
    except Exception:
        return 6800.0, "fallback"


def kernel_traffic(workload):
    """DRAM bytes per launch of the workload's dominant kernel from the
    committed ncu summary, or None if absent or taken on a different source."""
    spec = WORKLOADS[workload]
    src = hashlib.sha256()
    for f in spec["sources"]:
        with open(os.path.join(ROOT, "paper_2507_02401_gb300", "csrc", f), "rb") as fh:
            src.update(fh.read())
    digest = src.hexdigest()[:16]
    path = os.path.join(ROOT, "profiles", spec["profile"])
    if not os.path.exists(path):
        return None, digest
    vals = {}
    for line in open(path):
        if ":" in line:
            k, v = line.split(":", 1)
            vals[k.strip()] = v.strip()
    if vals.get("source_sha256_16") != digest:
        return None, digest
    try:
        return float(vals["dram_bytes_per_launch"]), digest
    except (KeyError, ValueError):
        return None, digest


class ClockSampler:
    """nvidia-smi sampling of SM clock and throttle reasons during the timed region."""

    FIELDS = ["index", "clocks.sm", "clocks.max.sm", "power.draw", "clocks_event_reasons.active",
              "clocks_event_reasons.hw_slowdown", "clocks_event_reasons.hw_thermal_slowdown",
              "clocks_event_reasons.sw_thermal_slowdown", "clocks_event_reasons.sw_power_cap"]

    def __init__(self, gpu_index):
        self.proc = None
        self.gpu_index = gpu_index
        self.out = None

    def start(self):
        try:
            self.out = open(os.devnull, "w")
            self.proc = subprocess.Popen(
                ["nvidia-smi", "--query-gpu=" + ",".join(self.FIELDS), "--format=csv,noheader", "-lms", "200",
                 "-i", str(self.gpu_index)], stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except Exception:
            self.proc = None

    def stop(self):
        if self.proc is None:
            return None
        self.proc.terminate()
        try:
            text, _ = self.proc.communicate(timeout=5)
        except Exception:
            self.proc.kill()
            text = ""
        sm, mx, reasons = [], [], set()
        for row in csv.reader(io.StringIO(text)):
            if len(row) < len(self.FIELDS):
                continue
            row = [r.strip() for r in row]
            try:
                sm.append(float(row[1].split()[0]))
                mx.append(float(row[2].split()[0]))
            except ValueError:
                continue
            for name, v in zip(["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"],
                               row[5:9]):
                if v.lower() == "active":
                    reasons.add(name)
        if not sm:
            return None
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(mx), "reasons": sorted(reasons),
                "samples": len(sm)}


def dist_setup(use_cuda):
    import torch
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl" if use_cuda else "gloo")
    if use_cuda:
        torch.cuda.set_device(local)
    return rank, world, local


def barrier(world):
    if world > 1:
        import torch.distributed as dist
        dist.barrier()


def max_over_ranks(v, world, use_cuda):
    if world == 1:
        return v
    import torch
    import torch.distributed as dist
    t = torch.tensor([v], dtype=torch.float64, device="cuda" if use_cuda else "cpu")
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def job_throughput(units_per_rank, world, t_ms_max):
    """Whole-job rate: the units all ranks processed over the slowest rank's time."""
    return units_per_rank * world / (t_ms_max / 1e3)


def gpu_index(local):
    vis = os.environ.get("CUDA_VISIBLE_DEVICES")
    if vis:
        parts = [p for p in vis.split(",") if p.strip()]
        if local < len(parts) and parts[local].strip().isdigit():
            return int(parts[local])
    return local


def oracle_pairs_per_s(w, nt_sample):
    """One oracle K + K* pair of the workload at nt_sample steps, scaled
    linearly in nt to pairs per second at the full nt; (value, seconds)."""
    import oracle
    wave = oracle.Wave(w.shape, w.h, w.dt, nt_sample, w.order, w.c_array(), w.sensors)
    t0 = time.perf_counter()
    wave.adjoint(wave.forward(w.x_true))
    dt = time.perf_counter() - t0
    return (nt_sample - 1) / ((w.nt - 1) * dt), dt


def cpu_baseline(w, iters_sample, workload):
    """The FP64 oracle, as it stands, on the host cores: `iters_sample` CG
    iterations (one K, one K*, E_s, E_s* each) of the same workload, or for
    the volume one K + K* pair at a reduced step count scaled to the full one."""
    import oracle
    nt_s = WORKLOADS[workload]["oracle_nt"]
    if nt_s:
        value, dt = oracle_pairs_per_s(w, nt_s)
        return {"value": value, "unit": UNIT, "cores": oracle.max_threads(), "kind": "oracle",
                "sample": f"oracle FP64 K + K* of the full {'x'.join(map(str, w.shape))} grid at {nt_s} of "
                          f"{w.nt} steps ({dt:.1f} s), scaled linearly in steps; E_s/CG vector work not counted"}
    wave = oracle.Wave(w.shape, w.h, w.dt, w.nt, w.order, w.c_array(), w.sensors)
    wav = oracle.Wavelet(w.shape, w.family, w.levels)
    rng = np.random.default_rng(0)
    y = rng.standard_normal((w.ns, w.nt))
    t0 = time.perf_counter()
    oracle.cg(wave, wav, y, 1e-3, 1.0, iters_sample)
    dt = time.perf_counter() - t0
    # a solve of k iterations costs 1 + 2k wave solves; count iterations as (2k+1)/2 pairs
    pairs = (2 * iters_sample + 1) / 2.0
    return {"value": pairs / dt, "unit": UNIT, "cores": oracle.max_threads(), "kind": "oracle",
            "sample": f"oracle FP64 CG, {iters_sample} iterations (+ right-hand side) of the full "
                      f"{'x'.join(map(str, w.shape))} workload; {dt:.1f} s"}


def run_reference(args):
    """Reference arm: the FP64 CPU oracle; each step is one CG iteration of
    the workload (the volume: one K + K* pair at a reduced step count, scaled
    linearly to the full one)."""
    import synth
    import oracle
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return 0
    if args.workload == "batch64":
        return run_reference_batch(args, world)
    w = synth.workload(args.workload)
    nt_s = WORKLOADS[args.workload]["oracle_nt"]
    if nt_s:
        for _ in range(args.warmup):
            oracle_pairs_per_s(w, nt_s)
        t_full = 0.0
        for _ in range(args.steps):
            v, _ = oracle_pairs_per_s(w, nt_s)
            t_full += 1.0 / v
        dt = t_full
        step_desc = f"one oracle K + K* pair at {nt_s} of {w.nt} steps, scaled linearly to the full step count"
    else:
        wave = oracle.Wave(w.shape, w.h, w.dt, w.nt, w.order, w.c_array(), w.sensors)
        wav = oracle.Wavelet(w.shape, w.family, w.levels)
        H = oracle.normal_op(wave, wav, 1.0, 1e-3)
        rng = np.random.default_rng(0)
        p = rng.standard_normal(w.N)
        for _ in range(args.warmup):
            H(p)
        t0 = time.perf_counter()
        for _ in range(args.steps):
            q = H(p)
            a = float(p @ p) / float(p @ q)
            p = p - a * q  # the CG vector work of one iteration is negligible beside H
        dt = time.perf_counter() - t0
        step_desc = "one oracle CG iteration (K + K* + E_s + E_s*)"
    value = args.steps / dt
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * dt / args.steps,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": WORKLOADS[args.workload]["desc"], "step": step_desc},
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": oracle.max_threads(), "kind": "oracle",
                             "sample": f"{args.steps} timed steps ({step_desc}) after {args.warmup} warm-up"},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)
    return 0


def run_reference_batch(args, world):
    """Reference arm of the 64-instance workload: per size class one oracle
    K + K* pair at 40 steps, scaled linearly to every instance's nt; a step
    is one CG iteration of all 64 instances (wave work only)."""
    import synth
    import oracle
    ws = synth.batched_workloads()
    by_n = {}
    for w in ws:
        by_n.setdefault(w.shape[0], w)
    nt_s = 40

    def one_iteration():
        per_pt = {}
        for n, w in by_n.items():
            wave = oracle.Wave(w.shape, w.h, w.dt, nt_s, w.order, w.c_array(), w.sensors)
            t0 = time.perf_counter()
            wave.adjoint(wave.forward(w.x_true))
            per_pt[n] = (time.perf_counter() - t0) / (nt_s - 1)
        return sum(per_pt[w.shape[0]] * (w.nt - 1) for w in ws)

    for _ in range(args.warmup):
        one_iteration()
    dt = sum(one_iteration() for _ in range(args.steps))
    value = args.steps * len(ws) / dt
    step_desc = ("one oracle CG iteration of all 64 instances (K + K* per instance, timed per grid size at 40 "
                 "steps and scaled linearly to each instance's nt)")
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * dt / args.steps,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": "64 independent 2D reconstructions of uneven size (batched workload)",
                       "step": step_desc},
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": oracle.max_threads(), "kind": "oracle",
                             "sample": f"{args.steps} steps ({step_desc}) after {args.warmup} warm-up"},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)
    return 0


def lambda_max(plan, s, iters=20, seed=0):
    import torch
    g = torch.Generator(device="cuda").manual_seed(seed)
    v = torch.randn(plan.N, device="cuda", generator=g)
    v /= v.norm()
    lam = 0.0
    for _ in range(iters):
        hv = plan.EsT(plan.adjoint(plan.forward(plan.Es(v, s))), s)
        lam = float(hv.norm())
        v = hv / lam
    return lam


def run_ours(args):
    import torch

    import synth
    from paper_2507_02401_gb300 import Plan, _lib

    if not torch.cuda.is_available():
        print(json.dumps({"metric": METRIC, "error": "no CUDA device"}))
        return 1
    rank, world, local = dist_setup(True)
    spec = WORKLOADS[args.workload]
    w = synth.workload(args.workload, seed=(1001 if args.workload == "vessels" else 1004) + rank)
    if args.iters:
        w.iters = args.iters
    c = w.c if np.ndim(w.c) == 0 else w.c_array()
    plan = Plan(w.shape, w.h, w.dt, w.nt, w.order, c, w.sensors, w.family, w.levels)
    stream = torch.cuda.current_stream()
    x_true = torch.as_tensor(w.x_true, dtype=torch.float32, device="cuda")
    y_clean = plan.forward(x_true).cpu().numpy()
    y_np = synth.add_noise(y_clean, w.noise, np.random.default_rng(1234 + rank)).astype(np.float32)
    y = torch.as_tensor(y_np, device="cuda")
    combos = []
    for s in w.s:
        lam = lambda_max(plan, s, iters=args.power_iters)
        for a in w.alpha:
            combos.append((s, a * lam))
    u = torch.empty(plan.N, device="cuda")
    x = torch.empty(w.shape, device="cuda")
    flush = torch.empty(L2_FLUSH_BYTES // 4, device="cuda")
    flush.zero_()  # first use outside the timed region (the first launch of a kernel loads its module)
    # several (s, alpha) combinations: one step solves all of them with pat_solve_multi (two right-hand
    # sides per wave launch on the persistent engine); one combination: pat_solve
    multi = len(combos) > 1
    xs_multi = [torch.empty(w.shape, device="cuda") for _ in combos]
    iters_per_step = w.iters * (len(combos) if multi else 1)

    def solve(k, yy=y, xx=x, uu=u):
        if multi:
            _lib.pat_solve_multi(plan.handle, [yy] * len(combos), [a for _, a in combos], [s for s, _ in combos],
                                 w.iters, xs_multi, stream)
            return
        s, alpha = combos[k % len(combos)]
        _lib.pat_solve(plan.handle, yy, alpha, s, w.iters, None, uu, xx, None, stream)

    for k in range(args.warmup):
        solve(k)
    torch.cuda.synchronize()
    assert plan.check() == 0, _lib.pat_last_error()

    sampler = ClockSampler(gpu_index(local)) if rank == 0 else None
    _lib.pat_plan_profile(plan.handle, 1)
    barrier(world)
    torch.cuda.synchronize()
    if sampler:
        sampler.start()
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    ev0.record(stream)
    for k in range(args.steps):
        flush.zero_()  # L2 flush between steps (inside the timed region; ~0.01% of a step)
        solve(k)
    ev1.record(stream)
    torch.cuda.synchronize()
    barrier(world)
    clocks = sampler.stop() if sampler else None
    t_ms = max_over_ranks(ev0.elapsed_time(ev1), world, True)
    kernels, wave_calls, wave_ms, points = _lib.pat_plan_profile_read(plan.handle)
    _lib.pat_plan_profile(plan.handle, 0)
    status = plan.check()
    assert status == 0, f"device status {status}: {_lib.pat_last_error()}"

    # end to end through the C ABI with host buffers (copies inside the timed region)
    y_host = torch.empty((w.ns, w.nt), dtype=torch.float32, pin_memory=True)
    y_host.copy_(torch.as_tensor(y_np))
    x_host = torch.empty(w.shape, dtype=torch.float32, pin_memory=True)
    xs_host = [torch.empty(w.shape, dtype=torch.float32, pin_memory=True) for _ in combos]
    yh, xh = y_host.numpy(), x_host.numpy()
    y_dev = torch.empty((w.ns, w.nt), device="cuda")
    barrier(world)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for k in range(args.steps):
        if multi:  # pat_solve_multi takes device arrays: the copies are inside the timed region
            y_dev.copy_(y_host, non_blocking=True)
            solve(k, yy=y_dev)
            for xhm, xd in zip(xs_host, xs_multi):
                xhm.copy_(xd, non_blocking=True)
        else:
            s, alpha = combos[k % len(combos)]
            _lib.pat_solve(plan.handle, yh, alpha, s, w.iters, None, None, xh, None, stream)
    torch.cuda.synchronize()
    e2e_s = max_over_ranks(time.perf_counter() - t0, world, True)
    barrier(world)

    iters_total = world * args.steps * iters_per_step
    value = job_throughput(args.steps * iters_per_step, world, t_ms)
    bytes_per_pt = 16 if plan_varc(w) else 12
    # the persistent engine runs a whole K or K* per launch (two fields at once under pat_solve_multi),
    # the step engines one time step; achieved = the library's point-updates x algorithmic bytes over the
    # device time of its wave launches
    steps_per_launch = (w.nt - 1) if plan.path == 1 else 1
    launches = wave_calls * (w.nt - 1) // steps_per_launch
    launch_ms = wave_ms / max(launches, 1)
    achieved = bytes_per_pt * points / (wave_ms / 1e3) / 1e9 if wave_ms > 0 else 0.0
    peak, peak_kind = peaks()
    traffic, digest = kernel_traffic(args.workload)
    engine = {1: "persistent", 2: "step"}.get(plan.path, "?")
    gpts = world * args.steps * (2 * w.iters + 1) * (len(combos) if multi else 1) * (w.nt - 1) * w.N / (t_ms / 1e3) / 1e9
    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": t_ms / args.steps, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": {"workload": spec["desc"], "engine": engine, "iters_per_step": iters_per_step,
                   "solves_per_step": len(combos) if multi else 1,
                   "right_hand_sides_per_wave_launch": 2 if (multi and plan.path == 1) else 1,
                   "l2": "256 MiB buffer written before every step (inside the timed region)",
                   "parallelism": f"replicas x{world} (independent instances per rank)"},
        "gpoint_updates_per_s": gpts,
        "roofline": {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s",
                     "frac": achieved / peak, "traffic": traffic, "peak_kind": peak_kind,
                     "kernel": f"{spec['kernel']} ({engine} engine)",
                     "algorithmic_bytes_per_point_update": bytes_per_pt,
                     "launch_ms": launch_ms, "launches_timed": launches,
                     "launch": ("one K or K* application of two right-hand sides" if multi else
                                "one K or K* application") if steps_per_launch > 1 else
                               "one time step (averaged over whole K / K* applications, sampling and "
                               "injection launches included)",
                     "source_sha256_16": digest},
        "e2e": {"value": iters_total / e2e_s, "unit": UNIT, "h2d_bytes_per_step": int(y_np.nbytes),
                "d2h_bytes_per_step": int(w.N * 4 * (len(combos) if multi else 1))},
        "gpu_launches": int(kernels + args.steps),  # library kernels + one L2 flush per step
        "clocks": clocks,
    }
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        line["cpu_baseline"] = cpu_baseline(w, args.cpu_iters, args.workload)
    if rank == 0:
        print(json.dumps(line), flush=True)
    if world > 1:
        import torch.distributed as dist
        dist.destroy_process_group()
    plan.close()
    return 0


def run_sweep(args):
    """Per-step wave engines on HBM-sized grids: one JSON line per case with
    the time per step of K and K* (CUDA events, whole applications of 200
    steps, fields larger than L2) and the algorithmic GB/s against the HBM
    peak (12 B per point-update for a constant medium, 16 B for a varying one)."""
    import torch
    from paper_2507_02401_gb300 import Plan
    peak, peak_kind = peaks()
    cases = [((n, n), o, False, 0) for n in (2048, 4096, 8192, 16384) for o in (2, 8)]
    cases += [((4096, 4096), 8, True, 0), ((4096, 4096), 8, False, 10), ((256, 256, 256), 4, False, 0),
              ((512, 512, 512), 4, False, 0)]
    nt = 201
    if args.only:  # a grid ("4096x4096") or one case ("4096x4096-o8", "4096x4096-o8v" for the varying medium)
        def ids(cs):
            g = "x".join(map(str, cs[0]))
            return {g, f"{g}-o{cs[1]}" + ("v" if cs[2] else "") + ("s" if cs[3] else "")}
        cases = [cs for cs in cases if args.only in ids(cs)]
    for shape, order, varc, sponge in cases:
        h = 1e-4
        rng = np.random.default_rng(0)
        c = 1400.0 + 200.0 * rng.random(shape).astype(np.float32) if varc else 1500.0
        dt = 0.3 * h / 1600.0
        sens = np.stack([rng.uniform(0.1, 0.9, 64) * (n - 1) * h for n in shape[::-1]], axis=1)
        plan = Plan(shape, h, dt, nt, order, c, sens, 1, 0)
        if sponge:
            plan.set_sponge(sponge)  # absorbing layer, default damping rate
        x = torch.randn(shape, device="cuda")
        y = torch.empty((64, nt), device="cuda")
        xa = torch.empty(shape, device="cuda")
        res = {}
        for name, fn in (("K", lambda: plan.forward(x, out=y)), ("Kt", lambda: plan.adjoint(y, out=xa))):
            for _ in range(args.warmup):
                fn()
            ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            ev0.record()
            for _ in range(args.steps):
                fn()
            ev1.record()
            torch.cuda.synchronize()
            res[name] = ev0.elapsed_time(ev1) * 1e3 / args.steps / (nt - 1)
        assert plan.check() == 0
        N = int(np.prod(shape))
        bpp = 16 if varc else 12
        line = {"sweep": "x".join(map(str, shape)), "order": order, "medium": "varying" if varc else "constant",
                "absorbing_layer_cells": sponge,
                "engine": {1: "persistent", 2: "step"}.get(plan.path, "?"), "steps": nt - 1,
                "algorithmic_bytes_per_point_update": bpp, "peak_gbs": peak, "peak_kind": peak_kind}
        for name in ("K", "Kt"):
            us = res[name]
            gbs = N * bpp / us / 1e3
            line[name] = {"us_per_step": round(us, 2), "gpoint_updates_per_s": round(N / us / 1e3, 1),
                          "algorithmic_gbs": round(gbs, 1), "frac": round(gbs / peak, 3)}
        print(json.dumps(line), flush=True)
        plan.close()
        del x, y, xa
        torch.cuda.empty_cache()
    return 0


def run_limited(args):
    """Limited-view workload: one step = one 15-iteration GMRES reconstruction
    (the paper's solver) with the absorbing layer, from data simulated on a
    grid twice as fine; also reports the relative error of the GMRES image for
    s in {0, 0.5, 1, 1.5, 2} and the objective J per iterate at s = 1."""
    import torch

    import synth
    from paper_2507_02401_gb300 import Plan, _lib

    if not torch.cuda.is_available():
        print(json.dumps({"metric": METRIC, "error": "no CUDA device"}))
        return 1
    rank, world, local = dist_setup(True)
    spec = WORKLOADS["limited"]
    w = synth.workload("limited", seed=1005 + rank)
    ex = w.extra
    iters = args.iters or w.iters
    nf = w.shape[0] * ex["refine"]
    fine = Plan((nf, nf), ex["h_fine"], ex["dt_fine"], ex["nt_fine"], w.order, 1500.0, w.sensors, 1, 0)
    fine.set_sponge(ex["layer"] * ex["refine"])
    y_f = fine.forward(torch.as_tensor(ex["x_fine"], dtype=torch.float32, device="cuda")).cpu().numpy()
    fine.close()
    y_np = synth.add_noise(y_f[:, ::ex["refine"]].astype(np.float64), w.noise,
                           np.random.default_rng(1234 + rank)).astype(np.float32)
    plan = Plan(w.shape, w.h, w.dt, w.nt, w.order, 1500.0, w.sensors, w.family, w.levels)
    plan.set_sponge(ex["layer"])
    y = torch.as_tensor(y_np, device="cuda")
    s1 = 1.0
    alpha = w.alpha[0] * lambda_max(plan, s1, iters=args.power_iters)
    stream = torch.cuda.current_stream()
    x = torch.empty(w.shape, device="cuda")

    def solve():
        _lib.pat_solve_gmres(plan.handle, y, alpha, s1, iters, x, None, None, stream)

    for _ in range(args.warmup):
        solve()
    torch.cuda.synchronize()
    sampler = ClockSampler(gpu_index(local)) if rank == 0 else None
    barrier(world)
    torch.cuda.synchronize()
    if sampler:
        sampler.start()
    flush = torch.empty(L2_FLUSH_BYTES // 4, device="cuda")
    flush.zero_()  # first use outside the timed region (the first launch of a kernel loads its module)
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    ev0.record(stream)
    for _ in range(args.steps):
        flush.zero_()
        solve()
    ev1.record(stream)
    torch.cuda.synchronize()
    barrier(world)
    clocks = sampler.stop() if sampler else None
    t_ms = max_over_ranks(ev0.elapsed_time(ev1), world, True)
    # wave-kernel durations and launch counts from one more solve with the library's measurement hooks
    _lib.pat_plan_profile(plan.handle, 1)
    solve()
    torch.cuda.synchronize()
    kernels, wave_calls, wave_ms, points = _lib.pat_plan_profile_read(plan.handle)
    _lib.pat_plan_profile(plan.handle, 0)
    kernels *= args.steps  # per timed solve, times the timed solves
    # end to end through the C ABI with host arrays
    x_host = np.zeros(w.shape, dtype=np.float32)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for _ in range(args.steps):
        _lib.pat_solve_gmres(plan.handle, y_np, alpha, s1, iters, x_host, None, None, stream)
    e2e_s = max_over_ranks(time.perf_counter() - t0, world, True)
    # reconstruction quality (outside the timed region)
    errs = {}
    xt = w.x_true
    for s in w.s:
        a_s = w.alpha[0] * lambda_max(plan, s, iters=args.power_iters)
        xs, res, J = plan.solve_gmres(y, a_s, s, iters, want_log=(s == s1))
        errs[str(s)] = float(np.linalg.norm(xs.cpu().numpy() - xt) / np.linalg.norm(xt))
        if s == s1:
            J_curve, res_curve = [float(v) for v in J], [float(v) for v in res]
    # algorithmic bytes of the step kernel per time step (12 B per point-update, constant medium)
    steps_per_launch = (w.nt - 1) if plan.path == 1 else 1
    launches = wave_calls * (w.nt - 1) // steps_per_launch
    launch_ms = wave_ms / max(launches, 1)
    achieved = 12.0 * w.N * steps_per_launch / (launch_ms / 1e3) / 1e9 if wave_ms > 0 else 0.0
    peak, peak_kind = peaks()
    # GMRES vector kernels besides the library's counted wave and wavelet kernels, per solve
    extra = 4 + sum(1 + 3 * (j + 1) + 3 for j in range(iters)) + 1 + iters
    line = {
        "metric": METRIC, "value": world * args.steps * iters / (t_ms / 1e3), "unit": UNIT, "n_gpus": world,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": t_ms / args.steps, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": {"workload": spec["desc"], "engine": {1: "persistent", 2: "step"}.get(plan.path, "?"),
                   "solver": "GMRES", "iters_per_step": iters,
                   "l2": "256 MiB buffer written before every step (inside the timed region)",
                   "parallelism": f"replicas x{world} (independent instances per rank)"},
        "rel_error_by_s": errs, "J_per_iterate_s1": J_curve, "residual_per_iterate_s1": res_curve,
        "roofline": {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s", "frac": achieved / peak,
                     "traffic": kernel_traffic("limited")[0] if plan.path == 1 else None, "peak_kind": peak_kind,
                     "kernel": spec["kernel"],
                     "algorithmic_bytes_per_point_update": 12, "launch_ms": launch_ms, "launches_timed": launches,
                     "launch": "one K or K* application" if steps_per_launch > 1 else
                               "one time step (averaged over whole K / K* applications, injection included)",
                     "note": "512^2 fields are L2-resident"},
        "e2e": {"value": world * args.steps * iters / e2e_s, "unit": UNIT, "h2d_bytes_per_step": int(y_np.nbytes),
                "d2h_bytes_per_step": int(w.N * 4)},
        "gpu_launches": int(kernels + args.steps * (extra + 1)),
        "clocks": clocks,
    }
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        line["cpu_baseline"] = cpu_baseline(w, args.cpu_iters, "limited")
    if rank == 0:
        print(json.dumps(line), flush=True)
    if world > 1:
        import torch.distributed as dist
        dist.destroy_process_group()
    plan.close()
    return 0


def run_batch(args):
    """64 independent reconstructions of uneven size through the batched
    engine (one step = one 50-iteration batched solve of all instances),
    against the same 64 solves one after the other with pat_solve."""
    import torch

    import synth
    from paper_2507_02401_gb300 import Batch, Plan, _lib

    if not torch.cuda.is_available():
        print(json.dumps({"metric": METRIC, "error": "no CUDA device"}))
        return 1
    rank, world, local = dist_setup(True)
    ws = synth.batched_workloads(seed=1003 + rank)
    iters = args.iters or ws[0].iters
    plans = [Plan(w.shape, w.h, w.dt, w.nt, w.order, w.c, w.sensors, w.family, w.levels) for w in ws]
    batch = Batch(plans)
    stream = torch.cuda.current_stream()
    ys = batch.forward([w.x_true for w in ws])
    rng = np.random.default_rng(1234 + rank)
    y_np = [synth.add_noise(y.cpu().numpy().astype(np.float64), w.noise, rng).astype(np.float32)
            for y, w in zip(ys, ws)]
    ys = [torch.as_tensor(y, device="cuda") for y in y_np]
    ss = [w.s[0] for w in ws]
    g = torch.Generator(device="cuda").manual_seed(0)
    vs = [torch.randn(p.N, device="cuda", generator=g) for p in plans]
    vs = [v / v.norm() for v in vs]
    for _ in range(args.power_iters):  # lambda_max of E_s* K* K E_s per instance, through the batch
        hs = batch.adjoint(batch.forward([p.Es(v, s) for p, v, s in zip(plans, vs, ss)]))
        hv = [p.EsT(h, s) for p, h, s in zip(plans, hs, ss)]
        lams = [float(h.norm()) for h in hv]
        vs = [h / lam for h, lam in zip(hv, lams)]
    alphas = [w.alpha[0] * lam for w, lam in zip(ws, lams)]
    xs = [torch.empty(w.shape, device="cuda") for w in ws]
    flush = torch.empty(L2_FLUSH_BYTES // 4, device="cuda")
    flush.zero_()  # first use outside the timed region (the first launch of a kernel loads its module)

    def solve_batched():
        rc, per = _lib.pat_batch_solve(batch.handle, ys, alphas, ss, iters, xs, stream)
        assert rc == 0, (rc, per, _lib.load().pat_last_error())

    for _ in range(args.warmup):
        solve_batched()
    torch.cuda.synchronize()
    info = batch.info
    # batched K alone (algorithmic bytes of the step kernel)
    xs_in = [torch.as_tensor(w.x_true, dtype=torch.float32, device="cuda") for w in ws]
    yk = [torch.empty((p.ns, p.nt), device="cuda") for p in plans]
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    _lib.pat_batch_forward(batch.handle, xs_in, yk, stream)
    e1.record(stream)
    torch.cuda.synchronize()
    k_ms = e0.elapsed_time(e1)
    pts_k = sum(w.N * (w.nt - 1) for w in ws)
    sampler = ClockSampler(gpu_index(local)) if rank == 0 else None
    barrier(world)
    torch.cuda.synchronize()
    if sampler:
        sampler.start()
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    ev0.record(stream)
    for _ in range(args.steps):
        flush.zero_()
        solve_batched()
    ev1.record(stream)
    torch.cuda.synchronize()
    barrier(world)
    clocks = sampler.stop() if sampler else None
    t_ms = max_over_ranks(ev0.elapsed_time(ev1), world, True)
    x_batched = [x.cpu().numpy() for x in xs]

    # the plain single-instance path: the same 64 solves one after the other
    torch.cuda.synchronize()
    s0, s1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    x_seq = []
    s0.record(stream)
    for p, y, a, s in zip(plans, ys, alphas, ss):
        _, x1, _ = p.solve(y, a, s, iters, stream=stream)
        x_seq.append(x1)
    s1.record(stream)
    torch.cuda.synchronize()
    seq_ms = s0.elapsed_time(s1)
    diffs = [float(np.linalg.norm(xb - xq.cpu().numpy()) / max(np.linalg.norm(xq.cpu().numpy()), 1e-30))
             for xb, xq in zip(x_batched, x_seq)]

    # end to end: host data in, images out, through the batched solve
    y_host = [torch.as_tensor(y, dtype=torch.float32).pin_memory() for y in y_np]
    x_host = [torch.empty(w.shape, dtype=torch.float32).pin_memory() for w in ws]
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for _ in range(args.steps):
        for yd, yh in zip(ys, y_host):
            yd.copy_(yh, non_blocking=True)
        solve_batched()
        for xh, xd in zip(x_host, xs):
            xh.copy_(xd, non_blocking=True)
        torch.cuda.synchronize()
    e2e_s = max_over_ranks(time.perf_counter() - t0, world, True)

    n_inst = len(ws)
    iters_total = world * args.steps * n_inst * iters
    peak, peak_kind = peaks()
    achieved = 12.0 * pts_k / (k_ms / 1e3) / 1e9
    max_nt = max(w.nt for w in ws)
    line = {
        "metric": METRIC, "value": iters_total / (t_ms / 1e3), "unit": UNIT, "n_gpus": world,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": t_ms / args.steps, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": {"workload": f"{n_inst} independent 2D reconstructions, n in {{128,192,256,384,512}}, c = 1500, "
                               f"order 8, nt = ceil(sqrt(2) n / 0.3), 64-512 sensors on circles or arcs, "
                               f"alpha log-uniform in [1e-4, 1e-1] x lambda_max, s in {{1, 1.5, 2}}, db4 4 levels, "
                               f"{iters} CG iterations each; one step = one batched solve of all instances",
                   "engine": "batched", "tile_rows": info["tile_rows"], "ctas": info["ctas"],
                   "autotune_ms": info["tune_ms"], "graph_nodes_per_iteration": info["graph_nodes"],
                   "launch": info["launch"],
                   "launch_tune_ms": {"one per step": info["launch_tune_ms"][0],
                                      "one per application": info["launch_tune_ms"][1]},
                   "l2": "256 MiB buffer written before every step (inside the timed region)",
                   "parallelism": f"replicas x{world} (independent batches per rank)"},
        "solves_per_s": world * args.steps * n_inst / (t_ms / 1e3),
        "sequential": {"solves_per_s": n_inst / (seq_ms / 1e3), "ms": seq_ms,
                       "path": "pat_solve per instance (single-instance engines, FP64 CG scalars)"},
        "speedup_vs_sequential": (world * args.steps * n_inst / (t_ms / 1e3)) / (n_inst / (seq_ms / 1e3)),
        "max_rel_diff_vs_sequential": max(diffs),
        "roofline": {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s", "frac": achieved / peak,
                     "traffic": None, "peak_kind": peak_kind, "kernel": "batch_step_kernel<R=7> (batched K)",
                     "algorithmic_bytes_per_point_update": 12, "launch_ms": k_ms / max_nt,
                     "launch": "one time step of every running instance (mean over a whole batched K)",
                     "note": "the 64 instances' fields (~80 MB) are largely L2-resident"},
        "e2e": {"value": iters_total / e2e_s, "unit": UNIT,
                "h2d_bytes_per_step": int(sum(y.nbytes for y in y_np)),
                "d2h_bytes_per_step": int(sum(w.N * 4 for w in ws))},
        # graph nodes per CG iteration; right-hand side (batched K*, fills, E_s*, CG start) and final E_s; L2 flush
        "gpu_launches": int(args.steps * (iters * info["graph_nodes"] + max_nt + 12 * n_inst + 1)),
        "clocks": clocks,
    }
    if rank == 0 and args.accuracy:
        line["accuracy_vs_oracle"] = batch_accuracy(ws, plans, batch, iters, ys, alphas)
    if rank == 0:
        print(json.dumps(line), flush=True)
    if world > 1:
        import torch.distributed as dist
        dist.destroy_process_group()
    batch.close()
    return 0


def oracle_lambda_max(wave, wav, s, iters=15, seed=0):
    """Power iteration on E_s* K* K E_s with the FP64 oracle."""
    import oracle
    rng = np.random.default_rng(seed)
    v = rng.standard_normal(wave.N)
    v /= np.linalg.norm(v)
    H = oracle.normal_op(wave, wav, s, 0.0)
    lam = 0.0
    for _ in range(iters):
        hv = H(v)
        lam = float(np.linalg.norm(hv))
        v = hv / lam
    return lam


def batch_accuracy(ws, plans, batch, iters, ys_other, alphas_other, n_max=192, n_conv=128):
    """Accuracy of the batched and of the sequential (pat_solve) path against
    the FP64 oracle, on every instance of the batched workload with n <= n_max:
    data simulated by the oracle, alpha = alpha_rel * the oracle's lambda_max
    (the same absolute alpha on every side), the oracle's CG at the same
    iteration count and, for n <= n_conv, the oracle's converged minimiser
    (CG to ||b - H u|| <= 1e-10 ||b||).  Instances above n_max keep the
    benchmark's data and alpha (ys_other, alphas_other: they run in the batch
    but are not compared)."""
    import torch

    import oracle
    import synth
    from paper_2507_02401_gb300 import _lib
    idx = [i for i, w in enumerate(ws) if w.shape[0] <= n_max]
    ys, alphas = {}, {}
    ref = {}
    t0 = time.perf_counter()
    for i in idx:
        w = ws[i]
        wave = oracle.Wave(w.shape, w.h, w.dt, w.nt, w.order, w.c_array(), w.sensors)
        wav = oracle.Wavelet(w.shape, w.family, w.levels)
        y = synth.add_noise(wave.forward(w.x_true), w.noise, np.random.default_rng(3000 + i))
        a = w.alpha[0] * oracle_lambda_max(wave, wav, w.s[0])
        _, x_o, _ = oracle.cg(wave, wav, y, a, w.s[0], iters)
        conv = None
        if w.shape[0] <= n_conv:
            _, x_c, k, rr = oracle.cg_converged(wave, wav, y, a, w.s[0])
            conv = (x_c, k, rr)
        ys[i], alphas[i], ref[i] = y, a, (x_o, conv)
    t_oracle = time.perf_counter() - t0
    # GPU: one batched solve of all instances, then pat_solve per compared instance
    yb = [torch.as_tensor(ys[i], dtype=torch.float32, device="cuda") if i in ys else ys_other[i]
          for i in range(len(plans))]
    ab = [alphas.get(i, alphas_other[i]) for i in range(len(ws))]
    ss = [w.s[0] for w in ws]
    xs = [torch.empty(w.shape, device="cuda") for w in ws]
    rc, per = _lib.pat_batch_solve(batch.handle, yb, ab, ss, iters, xs, torch.cuda.current_stream())
    assert rc == 0, (rc, per)
    rows = []

    def rel(a, b):
        return float(np.linalg.norm(np.ravel(a) - np.ravel(b)) / np.linalg.norm(np.ravel(b)))

    for i in idx:
        w = ws[i]
        _, xq, _ = plans[i].solve(yb[i], ab[i], ss[i], iters)
        xb_np, xq_np = xs[i].cpu().numpy().astype(np.float64), xq.cpu().numpy().astype(np.float64)
        x_o, conv = ref[i]
        row = {"i": i, "n": w.shape[0], "s": w.s[0], "alpha_rel": w.alpha[0],
               "batched_vs_oracle": rel(xb_np, x_o), "sequential_vs_oracle": rel(xq_np, x_o)}
        if conv is not None:
            x_c, k, rr = conv
            row.update({"oracle_vs_converged": rel(x_o, x_c), "batched_vs_converged": rel(xb_np, x_c),
                        "sequential_vs_converged": rel(xq_np, x_c), "converged_iters": k,
                        "converged_rel_residual": rr})
        rows.append(row)
    bands = {}
    for name, lo, hi in (("alpha_rel<1e-3", 0.0, 1e-3), ("1e-3<=alpha_rel<1e-2", 1e-3, 1e-2),
                         ("alpha_rel>=1e-2", 1e-2, 1.0)):
        sel = [r for r in rows if lo <= r["alpha_rel"] < hi]
        if sel:
            bands[name] = {"instances": len(sel),
                           "max_batched_vs_oracle": max(r["batched_vs_oracle"] for r in sel),
                           "max_sequential_vs_oracle": max(r["sequential_vs_oracle"] for r in sel)}
    return {"compared": len(rows), "iters": iters, "oracle_seconds": t_oracle, "by_conditioning": bands,
            "instances": rows}


def run_prior_sweep(args):
    """E_s of the two prior forms on 2D grids: the db4 wavelet form (5 levels,
    fused level kernels) and the Fourier form (radix-2 FFT kernels), time per
    application (CUDA events, E_s and E_s* alternating) and GB/s against the
    algorithmic 8 B per pixel (read the input, write the output once)."""
    import torch
    from paper_2507_02401_gb300 import Plan
    peak, peak_kind = peaks()
    for n in (512, 2048, 4096):
        h = 1e-4
        plan = Plan((n, n), h, 0.3 * h / 1500.0, 2, 2, 1500.0, np.zeros((0, 2)), 4, 5)
        u = torch.randn(n * n, device="cuda")
        x = torch.empty((n, n), device="cuda")
        for kind in (0, 1):
            plan.set_prior(kind, 8.0)
            for _ in range(args.warmup):
                plan.Es(u, 1.0, out=x)
                plan.EsT(x, 1.0, out=u)
            ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            reps = max(args.steps, 10)
            ev0.record()
            for _ in range(reps):
                plan.Es(u, 1.0, out=x)
                plan.EsT(x, 1.0, out=u)
            ev1.record()
            torch.cuda.synchronize()
            us = ev0.elapsed_time(ev1) * 1e3 / (2 * reps)
            gbs = 8.0 * n * n / us / 1e3
            print(json.dumps({"prior": "wavelet db4 5 levels" if kind == 0 else "Fourier (FFT)", "grid": f"{n}x{n}",
                              "us_per_application": round(us, 2), "algorithmic_gbs": round(gbs, 1),
                              "frac": round(gbs / peak, 3), "peak_kind": peak_kind}), flush=True)
        plan.close()
    return 0


def dwt_bytes_per_cell(dim, levels):
    """Algorithmic bytes of one E_s or E_s* per grid cell: every level reads
    its input and writes its output once (8 B per cell of the level), the
    level sizes falling by 2^dim: 8 (1 - 2^(-dim m)) / (1 - 2^-dim)."""
    r = 2.0 ** -dim
    return 8.0 * (1.0 - r ** levels) / (1.0 - r)


def run_dwt_sweep(args):
    """The wavelet kernels (E_s = W^T S_s synthesis and E_s* = S_s W analysis,
    periodic db4) on HBM-sized grids: each application timed alone with CUDA
    events on the launching stream, a 256 MiB L2 flush before each, against
    the algorithmic bytes of dwt_bytes_per_cell (each application replayed
    from a captured CUDA graph, so that host-side call overhead stays out of
    the timed region)."""
    import torch
    from paper_2507_02401_gb300 import Plan
    peak, peak_kind = peaks()
    cases = [((2048, 2048), 5), ((4096, 4096), 5), ((8192, 8192), 5), ((256, 256, 256), 4), ((512, 512, 512), 4)]
    if args.only:
        cases = [c for c in cases if "x".join(map(str, c[0])) == args.only]
    stream = torch.cuda.current_stream()
    flush = torch.empty(L2_FLUSH_BYTES // 4, device="cuda")
    for shape, levels in cases:
        h = 1e-4
        sens = np.zeros((0, len(shape)))
        plan = Plan(shape, h, 0.3 * h / 1500.0, 2, 2, 1500.0, sens, 4, levels)
        N = int(np.prod(shape))
        g = torch.Generator(device="cuda").manual_seed(0)
        x = torch.randn(shape, device="cuda", generator=g)
        u = torch.empty(N, device="cuda")
        bpc = dwt_bytes_per_cell(len(shape), levels)
        line = {"dwt_sweep": "x".join(map(str, shape)), "wavelet": f"db4, {levels} levels, periodic",
                "algorithmic_bytes_per_cell": round(bpc, 3), "peak_gbs": peak, "peak_kind": peak_kind,
                "l2": "256 MiB buffer written before every timed application"}
        reps = max(args.steps, 10)
        for name, fn in (("EsT", lambda: plan.EsT(x, 1.0, out=u)), ("Es", lambda: plan.Es(u, 1.0, out=x))):
            for _ in range(args.warmup):
                fn()
            # the application's launches captured once as a CUDA graph, so that the timed region holds
            # device work only (the Python and ctypes marshalling of a call costs tens of microseconds)
            cs = torch.cuda.Stream()
            cs.wait_stream(stream)
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=cs):
                fn()
            torch.cuda.synchronize()
            ms = 0.0
            for _ in range(reps):
                flush.zero_()  # ~40 us of device work: the replay below is enqueued before it ends
                e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                e0.record(stream)
                graph.replay()
                e1.record(stream)
                torch.cuda.synchronize()
                ms += e0.elapsed_time(e1)
            us = ms * 1e3 / reps
            gbs = N * bpc / us / 1e3
            line[name] = {"us_per_application": round(us, 2), "algorithmic_gbs": round(gbs, 1),
                          "frac": round(gbs / peak, 3)}
        print(json.dumps(line), flush=True)
        plan.close()
        del x, u
        torch.cuda.empty_cache()
    return 0


def plan_varc(w):
    return np.ndim(w.c) != 0 and float(np.max(w.c)) != float(np.min(w.c))


def main():
    ap = argparse.ArgumentParser(description=__doc__.split("\n")[0])
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=8)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--workload", choices=sorted(WORKLOADS) + ["batch64"], default=WORKLOAD)
    ap.add_argument("--iters", type=int, default=0, help="override CG iterations per step")
    ap.add_argument("--cpu-iters", type=int, default=4, help="oracle CG iterations in the CPU baseline sample")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--accuracy", action="store_true",
                    help="with --workload batch64: per-instance errors against the FP64 oracle (n <= 192) and its "
                         "converged minimiser (n = 128), outside the timed region")
    ap.add_argument("--power-iters", type=int, default=20, help="power iterations for lambda_max")
    ap.add_argument("--only", default="", help="with --sweep: run only a grid (256x256x256) or a case (4096x4096-o8)")
    ap.add_argument("--prior-sweep", action="store_true",
                    help="time E_s of the wavelet and Fourier prior forms on 2D grids instead")
    ap.add_argument("--dwt-sweep", action="store_true",
                    help="time the wavelet kernels (E_s, E_s*) on 2D 2048^2..8192^2 and 3D 256^3, 512^3 instead")
    ap.add_argument("--sweep", action="store_true",
                    help="time the per-step wave engines on 2D 2048^2..16384^2 (orders 2, 8) and 3D grids instead")
    args = ap.parse_args()
    args.warmup = max(args.warmup, 3)  # timing rule: at least 3 untimed warm-up steps
    if args.impl == "reference":
        return run_reference(args)
    if args.sweep:
        return run_sweep(args)
    if args.prior_sweep:
        return run_prior_sweep(args)
    if args.dwt_sweep:
        return run_dwt_sweep(args)
    if args.workload == "batch64":
        return run_batch(args)
    if args.workload == "limited":
        return run_limited(args)
    return run_ours(args)


if __name__ == "__main__":
    sys.exit(main())
