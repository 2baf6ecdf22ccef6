"""Benchmark of the fused radiation-transfer step on GB300.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--workload box3d]
                    [--impl reference] [--no-e2e] [--no-cpu-baseline]

One step = one pass of the whole hot path (transport, velocity estimate,
absorption with the T^4 solve, scattering, quadrature and gas sources) over
the workload, which stays resident in HBM.  The default workload is the 3-D
periodic radiation-dominated box, 128^3 cells x 80 angles (S8), float32
intensities with the temperature solve finished in double.  Prints one JSON
line.  Under torchrun (N > 1) every rank runs its own independent copy of
the problem (replicas: the method needs no exchange between independent
problems) and rank 0 reports the whole-job rate over the slowest rank.

--impl reference times the FP64 CPU oracle on a bounded sample of the same
workload on the host cores (rank 0 only).
"""
import argparse
import hashlib
import json
import os
import statistics
import subprocess
import sys
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

PROFILE = os.path.join(ROOT, "profiles", "step_kernel_box3d.md")
# sources of the float step kernel (the kernel of opposite pairs, the quad kernel
# whose per-cell parts it uses, the packed-FP32 helpers and the tile geometry)
KERNEL_SRCS = [os.path.join(ROOT, "paper_1403_6126_gb300", "csrc", f)
               for f in ("rt_step_sym.cuh", "rt_step_quad.cuh", "rt_step_pair.cuh", "rt_step_kernel.cuh")]
NOMINAL_HBM_GBS = 8000.0


def algorithmic_bytes_per_cell(M, rs, velocity, live_T):
    """Bytes one fused step must move per cell: read and write I (M values of
    rs bytes); read rho, sigma_a, sigma_s, v (rs bytes each) and T (double);
    read E (for IV = 3 n.v J) and F, P_xx..P_zz (for the velocity estimate),
    double, when velocity terms are on; write T, E, F, P (10 moments), the
    gas energy source and the momentum source (3), all double.  At 80 angles
    and float intensities that is 848 bytes per cell."""
    b = 2 * M * rs                 # I^n in, I^{n+1} out
    b += 3 * rs + 3 * rs           # rho, sigma_a, sigma_s, v
    b += 8 + (8 if live_T else 0)  # T in (double), T out when it evolves
    if velocity:
        b += 7 * 8                 # E, F, P_dd of step n
    b += 10 * 8 + 8 + 3 * 8        # moments, dE_gas, dMom
    return b


def kernel_sha():
    """Hash of the float kernel's code: comments and blank lines are left
    out, so a changed comment keeps the recorded ncu figures valid."""
    h = hashlib.sha256()
    for path in KERNEL_SRCS:
        with open(path) as f:
            for line in f:
                code = line.split("//", 1)[0].rstrip()
                if code:
                    h.update(code.encode() + b"\n")
    return h.hexdigest()[:16]


def _profile_traffic():
    """Per-launch DRAM bytes from the committed ncu summary, or None when the
    kernel source changed since that capture."""
    try:
        text = open(PROFILE).read()
    except OSError:
        return None
    vals = {}
    for line in text.splitlines():
        if line.startswith("- ") and ":" in line:
            k, v = line[2:].split(":", 1)
            vals[k.strip()] = v.strip().strip("`")
    if vals.get("kernel_source_sha256_16") != kernel_sha():
        return None
    try:
        return float(vals["dram_bytes_per_launch"])
    except (KeyError, ValueError):
        return None


def _peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            p = json.load(f)
        return float(p["hbm_gbs"]), "measured"
    except Exception:
        return 6800.0, "fallback"


class ClockSampler:
    """nvidia-smi sampling of SM clocks and throttle reasons during the timed
    region."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index):
        self.gpu_index = gpu_index
        self.proc = None

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.gpu_index), "--query-gpu=" + self.FIELDS,
                                          "--format=csv,noheader,nounits", "-lms", "100"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except OSError:
            self.proc = None
        time.sleep(0.3)
        return self

    def __exit__(self, *exc):
        self.rows = []
        if self.proc is None:
            return
        time.sleep(0.2)
        self.proc.terminate()
        try:
            out, _ = self.proc.communicate(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
            out, _ = self.proc.communicate()
        for line in out.splitlines():
            parts = [p.strip() for p in line.split(",")]
            if len(parts) == 9:
                self.rows.append(parts)

    def summary(self):
        rows = getattr(self, "rows", [])
        if not rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["unsampled"]}
        sm = [float(r[1]) for r in rows if r[1].replace(".", "").isdigit()]
        mx = [float(r[2]) for r in rows if r[2].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for r in rows for i in range(4) if r[5 + i].lower() == "active"})
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": reasons, "samples": len(rows)}


def _dist():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return world, rank, local


def max_over_ranks(x, world, device="cuda"):
    """The slowest rank's figure: replicas report whole-job rates over the
    longest time any rank took (x unchanged when world == 1)."""
    if world <= 1:
        return x
    import torch
    import torch.distributed as dist
    t = torch.tensor([float(x)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def whole_job_rate(units_per_rank, world, seconds_max):
    """Units all replicas processed per second of the slowest one."""
    return units_per_rank * world / seconds_max


def _angles(name):
    import paper_1403_6126_gb300 as rt
    if name.startswith("s"):
        return rt.rt_angle_set(rt.RT_ANGLES_LEVEL_SYMMETRIC, int(name[1:]))
    return rt.rt_angle_set(rt.RT_ANGLES_GAUSS_LEGENDRE, int(name[2:]))


def _context(wl, n, w, stream=None, precision=None):
    import paper_1403_6126_gb300 as rt
    from paper_1403_6126_gb300 import workloads as wlmod
    prec = {"fp64": rt.RT_FP64, "fp32": rt.RT_FP32, "bf16": rt.RT_BF16}[precision or wl["precision"]]
    ctx = rt.Context(wl["shape"], n, w, wl["C"], wl["P"], dim=wl["dim"], lo=wl["lo"], hi=wl["hi"], bc=wl["bc"],
                     precision=prec, cfl=wl["cfl"], gamma=wl["gamma"], r_ideal=wl["R"], hold_T=wl["hold_T"],
                     estimate_v=wl["estimate_v"], stream=stream)
    for (axis, side), rule in wl["inflow"].items():
        ctx.set_inflow(axis, side, wlmod.inflow_values(rule, n))
    return ctx


def cpu_baseline(wl_name, steps, warmup, sample_n=None, threads=None, wl=None):
    """Times the FP64 oracle, as it stands, on the workload (or, with
    sample_n, the same recipe on a smaller box): `steps` timed steps after
    `warmup` untimed ones, OpenMP over `threads` host threads (default: all
    cores)."""
    import oracle
    from paper_1403_6126_gb300 import workloads as wlmod
    if wl is None:
        kw = {}
        if wl_name == "box3d" and sample_n:
            kw = dict(n=sample_n)
        wl = wlmod.by_name(wl_name, **kw)
    n, w = oracle.angles.by_name(wl["angles"])
    dx = tuple((wl["hi"][d] - wl["lo"][d]) / wl["shape"][2 - d] for d in range(3))
    inflow = {face: wlmod.inflow_values(rule, n) for face, rule in wl["inflow"].items()}
    p = oracle.Problem(wl["shape"], dx, n, w, C=wl["C"], P=wl["P"], dim=wl["dim"], bc=wl["bc"], inflow=inflow,
                       gamma=wl["gamma"], R=wl["R"], hold_T=wl["hold_T"], estimate_v=wl["estimate_v"])
    cores = os.cpu_count() or 1
    oracle.set_threads(threads or cores)
    I = wlmod.initial_intensity(wl, len(w))
    T = wl["T"].copy()
    dt = oracle.cfl_dt(p, wl["cfl"])
    for _ in range(warmup):
        out = oracle.step(p, dt, I, T, wl["rho"], wl["v"], wl["sa"], wl["ss"])
        I, T = out["I"], out["T"]
    t0 = time.perf_counter()
    for _ in range(steps):
        out = oracle.step(p, dt, I, T, wl["rho"], wl["v"], wl["sa"], wl["ss"])
        I, T = out["I"], out["T"]
    el = time.perf_counter() - t0
    units = p.N * p.M * steps
    used = oracle.max_threads()
    oracle.set_threads(cores)
    return dict(value=units / el, unit="cell-angle updates/s", cores=used, kind="oracle",
                sample="%s recipe at %s cells x %d angles, %d timed steps (+%d warm-up), FP64 C oracle, %d thread%s"
                       % (wl_name, "x".join(str(s) for s in wl["shape"][::-1] if s > 1), p.M, steps, warmup, used,
                          "s (OpenMP)" if used > 1 else ""),
                seconds=el, steps=steps, seconds_per_step=el / max(1, steps))


def cpu_baselines(args):
    """The oracle timed on the host cores: the headline figure on the timed
    workload itself (full size, two steps after one warm-up, every core),
    beside it one step of a 48^3 sample on one thread (the per-core rate),
    and the two small workloads (the 1-D slab in full, 2000 steps; the 2-D
    shadow problem over 10 steps), all on every core."""
    from paper_1403_6126_gb300 import workloads as wlmod
    kw = {"n": args.n} if args.workload == "box3d" and args.n else {}
    head = cpu_baseline(args.workload, 2, 1, wl=wlmod.by_name(args.workload, **kw))
    out = {k: head[k] for k in ("value", "unit", "cores", "kind", "sample")}
    one = cpu_baseline(args.workload, 1, 0, sample_n=48 if args.workload == "box3d" else None, threads=1)
    out["single_thread"] = {k: one[k] for k in ("value", "unit", "cores", "sample")}
    slab = wlmod.slab1d()
    s0 = cpu_baseline("slab1d", slab["steps"], 0, wl=slab)
    sh = cpu_baseline("shadow2d", 10, 0, wl=wlmod.shadow2d())
    out["small_configs"] = {
        "slab1d": {k: s0[k] for k in ("value", "unit", "cores", "sample", "seconds_per_step")},
        "shadow2d": {k: sh[k] for k in ("value", "unit", "cores", "sample", "seconds_per_step")}}
    return out


def arm_config(args, world):
    """The workload's description on the JSON line, the same for both arms:
    grid, angles, precision, whether T and the velocity terms are live, the
    CFL time step (cfl * min dx / Crat, sec. 4.1) and the L2 note."""
    from paper_1403_6126_gb300 import workloads as wlmod
    wl = wlmod.by_name(args.workload, **({"n": args.n} if args.workload == "box3d" and args.n else {}))
    name = wl["angles"]
    M = int(name[2:]) if name.startswith("gl") else int(name[1:]) * (int(name[1:]) + 2)
    N = int(np.prod(wl["shape"]))
    dims = [wl["shape"][2 - d] for d in range(wl["dim"])]
    dt = wl["cfl"] * min((wl["hi"][d] - wl["lo"][d]) / dims[d] for d in range(wl["dim"])) / wl["C"]
    velocity = bool(np.any(wl["v"] != 0)) or wl["estimate_v"]
    rs = 8 if wl["precision"] == "fp64" else 4
    return {"workload": "%s: %s cells x %d angles (%s), %s intensities, T live=%s, velocity=%s"
                        % (wl["name"], "x".join(str(s) for s in wl["shape"][::-1]), M, wl["angles"],
                           wl["precision"], not wl["hold_T"], velocity),
            "cells": N, "angles": M, "dt": dt,
            "l2": "inputs larger than L2: %.2f GB of intensity read per step" % (N * M * rs / 1e9),
            "parallelism": "replicas" if world > 1 else "single GPU"}


def run_reference(args):
    """The FP64 oracle on the host cores, on the GPU arm's own workload at
    full size.  At about 3 s per step of the 128^3 x 80 box on 16 cores, the
    run times at most --ref-steps steps (after one warm-up step) so that it
    ends within a few minutes; the line's steps and warmup say what was run."""
    world, rank, _ = _dist()
    if rank != 0:
        return 0
    from paper_1403_6126_gb300 import workloads as wlmod
    kw = {"n": args.n} if args.workload == "box3d" and args.n else {}
    steps, warmup = max(1, min(args.steps, args.ref_steps)), min(args.warmup, 1)
    res = cpu_baseline(args.workload, steps, warmup, wl=wlmod.by_name(args.workload, **kw))
    line = {
        "impl": "reference", "metric": "cell-angle updates/s", "value": res["value"], "unit": res["unit"],
        "n_gpus": world, "steps": steps, "warmup": warmup,
        "ms_per_step": 1e3 * res["seconds"] / steps, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": arm_config(args, world),
        "cpu_baseline": {k: res[k] for k in ("value", "unit", "cores", "kind", "sample")},
        "e2e": {"value": res["value"], "unit": res["unit"], "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line))
    return 0


def run_gpu(args):
    import torch

    world, rank, local = _dist()
    torch.cuda.set_device(local)
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl" if torch.cuda.is_available() else "gloo")
    import paper_1403_6126_gb300 as rt
    from paper_1403_6126_gb300 import build as rtbuild
    from paper_1403_6126_gb300 import workloads as wlmod

    rtbuild.build()
    kw = {}
    if args.workload == "box3d" and args.n:
        kw["n"] = args.n
    wl = wlmod.by_name(args.workload, **kw)
    n, w = _angles(wl["angles"])
    M = len(w)
    N = int(np.prod(wl["shape"]))
    stream = torch.cuda.Stream()
    ctx = _context(wl, n, w, stream=stream.cuda_stream)
    ctx.set_intensity(wlmod.initial_intensity(wl, M))
    ctx.set_material(wl["rho"], wl["T"], wl["v"], wl["sa"], wl["ss"])
    dt = ctx.cfl_dt()
    tuned = None
    if args.tile:
        ctx.set_tile(*[int(x) for x in args.tile.split("x")])
    elif not args.no_autotune:
        tuned = [dict(tile="%dx%dx%d" % t[:3], ms=t[3]) for t in ctx.autotune(3)]
    tile = ctx.tile()
    velocity = bool(np.any(wl["v"] != 0)) or wl["estimate_v"]
    rs = 8 if wl["precision"] == "fp64" else 4

    def barrier():
        if world > 1:
            import torch.distributed as dist
            dist.barrier()

    # warm-up
    for _ in range(args.warmup):
        ctx.step(dt)
    ctx.sync()
    torch.cuda.synchronize()

    starts = [torch.cuda.Event(enable_timing=True) for _ in range(args.steps)]
    ends = [torch.cuda.Event(enable_timing=True) for _ in range(args.steps)]
    t_all0 = torch.cuda.Event(enable_timing=True)
    t_all1 = torch.cuda.Event(enable_timing=True)
    sampler = ClockSampler(int(os.environ.get("CUDA_VISIBLE_DEVICES", str(local)).split(",")[0])
                           if os.environ.get("CUDA_VISIBLE_DEVICES", "").split(",")[0].isdigit() else local)
    with sampler:
        barrier()
        torch.cuda.synchronize()
        t_all0.record(stream)
        for k in range(args.steps):
            starts[k].record(stream)
            ctx.step(dt)
            ends[k].record(stream)
        t_all1.record(stream)
        torch.cuda.synchronize()
        barrier()
    ctx.sync()
    total_ms = t_all0.elapsed_time(t_all1)
    launch_ms = [s.elapsed_time(e) for s, e in zip(starts, ends)]
    total_ms = max_over_ranks(total_ms, world)
    ms_per_step = total_ms / args.steps
    units_per_step = N * M
    value = whole_job_rate(units_per_step * args.steps, world, total_ms / 1e3)

    bytes_per_launch = algorithmic_bytes_per_cell(M, rs, velocity, not wl["hold_T"]) * N
    avg_launch_s = statistics.mean(launch_ms) / 1e3
    peak, peak_kind = _peaks()
    achieved = bytes_per_launch / avg_launch_s / 1e9
    traffic = _profile_traffic()
    roofline = {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s", "frac": achieved / peak,
                "traffic": traffic, "peak_source": peak_kind + " (MEASURED_PEAKS.json hbm_gbs)" if peak_kind == "measured" else "fallback 6.8 TB/s",
                "frac_of_nominal_8tbs": achieved / NOMINAL_HBM_GBS,
                "algorithmic_bytes_per_launch": bytes_per_launch, "avg_launch_ms": avg_launch_s * 1e3,
                "kernel": ("step_kernel_%s<%d,%s,%d,%d,%d>"
                           % (("d" if rs == 8 else "sym" if wl["dim"] > 1 else "q", wl["dim"],
                               "true" if velocity else "false") + tile)),
                "tile": "%dx%dx%d" % tile, "autotune": tuned}

    # end to end through the C ABI with pinned host buffers: per step the gas
    # fields go host->device, the sources of the step come back
    e2e = None
    if not args.no_e2e:
        e2e = _e2e(ctx, wl, N, M, stream, args, world)
    clocks = sampler.summary()
    ctx.close()

    batched = serving = small = accuracy = bf16 = None
    if world == 1 and not args.no_small:
        small = bench_small(stream)
    if world == 1 and not args.no_accuracy:
        accuracy = bench_accuracy(stream)
    if world == 1 and not args.no_bf16:
        bf16 = bench_bf16(args, stream)
    if world == 1 and not args.no_batch:
        batched = bench_batched(args, stream)
    if world == 1 and not args.no_serve:
        serving = bench_serving(args)

    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        cpu = cpu_baselines(args)
    if rank == 0:
        config = arm_config(args, world)
        assert config["cells"] == N and config["angles"] == M and abs(config["dt"] - dt) <= 1e-15 * dt
        line = {
            "metric": "cell-angle updates/s", "value": value, "unit": "cell-angle updates/s", "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms_per_step, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f32" if rs == 4 else "f64", "data": "synthetic",
            "config": config,
            "roofline": roofline, "cpu_baseline": cpu, "e2e": e2e, "gpu_launches": args.steps, "clocks": clocks,
            "accuracy_vs_oracle": accuracy, "bf16_storage": bf16,
            "small_configs": small, "batched": batched, "serving": serving,
        }
        print(json.dumps(line))
    if world > 1:
        import torch.distributed as dist
        dist.destroy_process_group()
    return 0


def _e2e(ctx, wl, N, M, stream, args, world):
    import torch
    pin = lambda shape: torch.zeros(shape, dtype=torch.float64, pin_memory=True).numpy()
    rho, T, v, sa, ss = pin(N), pin(N), pin((3, N)), pin(N), pin(N)
    rho[:] = wl["rho"]; T[:] = wl["T"]; v[:] = wl["v"]; sa[:] = wl["sa"]; ss[:] = wl["ss"]
    dE, dM = pin(N), pin((3, N))
    import paper_1403_6126_gb300 as rt

    # the coupled loop of a gas code: its fields in, the sources of the step
    # out (the new T lands in the pinned T the next step sends back), as one
    # rt_step_coupled call (transfers overlapped with the step slab by slab)
    # and, for comparison, as rt_set_material + rt_step + rt_sources
    def coupled():
        rt.rt_step_coupled(ctx.ctx, 0.0, rho, T, v, sa, ss, dE, dM, T)

    def three_calls():
        rt.rt_set_material(ctx.ctx, rho, T, v, sa, ss)
        rt.rt_step(ctx.ctx, 0.0)
        rt.rt_sources(ctx.ctx, dE, dM, T)

    def timed(one):
        T[:] = wl["T"]
        for _ in range(max(1, args.warmup)):
            one()
        torch.cuda.synchronize()
        k = max(3, args.steps // 2)
        t0 = time.perf_counter()
        for _ in range(k):
            one()
        torch.cuda.synchronize()
        return k, max_over_ranks(time.perf_counter() - t0, world)

    k3, el3 = timed(three_calls)
    k, el = timed(coupled)
    h2d = 7 * N * 8
    d2h = (1 + 3 + 1) * N * 8
    return {"value": whole_job_rate(N * M * k, world, el), "unit": "cell-angle updates/s", "h2d_bytes_per_step": h2d,
            "d2h_bytes_per_step": d2h, "steps": k, "ms_per_step": 1e3 * el / k,
            "transfers": "rt_step_coupled: rho, T, v, sigma_a, sigma_s in, dE_gas, dMom, T_new out, pinned doubles, "
                         "every step, overlapped with the step slab by slab",
            "three_calls": {"value": whole_job_rate(N * M * k3, world, el3), "ms_per_step": 1e3 * el3 / k3,
                            "calls": "rt_set_material, rt_step, rt_sources"}}


def bench_batched(args, stream):
    """The batched workload (512 uneven 1-D and 2-D problems) in one
    persistent launch per step under a CUDA graph, against stepping the same
    contexts one launch each."""
    import torch
    import paper_1403_6126_gb300 as rt
    from paper_1403_6126_gb300 import workloads as wlmod
    wls = wlmod.batched(nprob=args.batch_n)
    ctxs, units, nbytes = [], 0, 0
    for wl in wls:
        n, w = _angles(wl["angles"])
        c = _context(wl, n, w, stream=stream.cuda_stream)
        c.set_intensity(wlmod.initial_intensity(wl, len(w)))
        c.set_material(wl["rho"], wl["T"], wl["v"], wl["sa"], wl["ss"])
        ctxs.append(c)
        N = int(np.prod(wl["shape"]))
        units += N * len(w)
        nbytes += algorithmic_bytes_per_cell(len(w), 4, False, True) * N
    b = rt.rt_batch_create(stream.cuda_stream)
    for c in ctxs:
        rt.rt_batch_add(b, c.ctx)
    tune_ms, chosen = rt.rt_batch_autotune(b, 3)
    K = args.batch_steps
    rt.rt_batch_step(b, 3)
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    rt.rt_batch_step(b, K)
    e1.record(stream)
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1) / K
    rt.rt_batch_destroy(b)
    for c in ctxs:          # the same problems, one launch per problem per step
        c.step(0.0)
    torch.cuda.synchronize()
    e0.record(stream)
    for _ in range(K):
        for c in ctxs:
            c.step(0.0)
    e1.record(stream)
    torch.cuda.synchronize()
    ms_one = e0.elapsed_time(e1) / K
    for c in ctxs:
        c.sync()
        c.close()
    peak, _ = _peaks()
    return {"workload": "%d problems (half 1-D 64..4096 cells x 8..48 angles, half 2-D 32..256^2 x 8/24/48 angles), "
                        "T live, float intensities" % len(wls),
            "value": units / (ms / 1e3), "unit": "cell-angle updates/s", "ms_per_step": ms, "steps": K,
            "cell_angles": units, "launches_per_step": 1,
            "autotune": {"ms_per_step": dict(zip(("512 threads", "256 threads", "128 threads"), tune_ms)),
                         "chosen": ("512 threads", "256 threads", "128 threads")[chosen]},
            "one_at_a_time": {"value": units / (ms_one / 1e3), "ms_per_step": ms_one, "launches_per_step": len(wls)},
            "hbm": {"achieved": nbytes / (ms / 1e3) / 1e9, "peak": peak, "unit": "GB/s",
                    "frac": nbytes / (ms / 1e3) / 1e9 / peak}}


def bench_small(stream):
    """The two small workloads: the 1-D slab (512 cells x 8 angles, FP64, 2000
    steps in one captured graph; launch/latency bound, so microseconds per
    step) and the 2-D shadow problem (256 x 128 cells x 80 angles, 4000
    steps, FP64 and FP32 intensities; its working set fits in L2, so the
    bandwidth is reported against the HBM peaks with that caveat)."""
    import torch
    from paper_1403_6126_gb300 import workloads as wlmod
    peak, _ = _peaks()
    out = {}
    runs = [("slab1d", wlmod.slab1d(), "fp64"), ("shadow2d_fp64", wlmod.shadow2d(), "fp64"),
            ("shadow2d_fp32", wlmod.shadow2d(), "fp32")]
    for key, wl, prec in runs:
        n, w = _angles(wl["angles"])
        M, N = len(w), int(np.prod(wl["shape"]))
        c = _context(wl, n, w, stream=stream.cuda_stream, precision=prec)
        c.set_intensity(wlmod.initial_intensity(wl, M))
        c.set_material(wl["rho"], wl["T"], wl["v"], wl["sa"], wl["ss"])
        dt = c.cfl_dt()
        tuned = [dict(tile="x".join(str(v) for v in t[:3]), ms=t[3]) for t in c.autotune(5)]
        c.run(dt, 10)           # warm-up, and the graph for 10 steps
        c.sync()
        steps = wl["steps"]
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        c.run(dt, steps)        # capture the graph for the timed length
        c.sync()
        e0.record(stream)
        c.run(dt, steps)
        e1.record(stream)
        c.sync()
        ms = e0.elapsed_time(e1) / steps
        rs = 8 if prec == "fp64" else 4
        bpc = algorithmic_bytes_per_cell(M, rs, False, not wl["hold_T"]) * N
        out[key] = {"workload": "%s: %s cells x %d angles, %s intensities, %d steps in one CUDA graph"
                                % (wl["name"], "x".join(str(x) for x in wl["shape"][::-1] if x > 1) or "1", M, prec, steps),
                    "us_per_step": ms * 1e3, "steps_per_s": 1e3 / ms, "cell_angle_updates_per_s": N * M / (ms / 1e3),
                    "algorithmic_gb_s": bpc / (ms / 1e3) / 1e9, "frac_of_measured_hbm": bpc / (ms / 1e3) / 1e9 / peak,
                    "working_set_mb": bpc / 1e6, "tile": "x".join(str(v) for v in c.tile()), "autotune": tuned,
                    "note": "working set fits in L2 (126 MB): a bandwidth fraction here is an L2 figure"}
        c.close()
    return out


def _stated_sample(name):
    """The oracle's stored values after a workload's full step count
    (tests/golden/stated_<name>.txt, written by make_stated_steps.py from the
    oracle alone): (dt, steps, scales, cells, E, F[3, k]), or None."""
    path = os.path.join(ROOT, "tests", "golden", "stated_%s.txt" % name)
    if not os.path.exists(path):
        return None
    scal, rows = {}, []
    with open(path) as f:
        for line in f:
            if line.startswith("#") or not line.strip():
                continue
            parts = line.split()
            if len(parts) == 2:
                scal[parts[0]] = float(parts[1])
            else:
                rows.append([float(x) for x in parts])
    a = np.array(rows)
    return scal["dt"], int(scal["steps"]), scal, a[:, 0].astype(np.int64), a[:, 1], a[:, 2:5].T


def _stated_workload(name):
    """The inputs the stored oracle values were computed from (float32-rounded
    fields; see tests/golden/make_stated_steps.py)."""
    from paper_1403_6126_gb300 import workloads as wlmod
    if name.startswith("serving_req"):
        base = wlmod.serving_request(int(name[len("serving_req"):]))
    else:
        base = wlmod.by_name(name, **({"n": 128} if name == "box3d" else {}))
    return wlmod.rounded_to_float32(base)


def _stated_errors(E, F, ref, dim):
    """E_r, |F_r| (active axes) at the stored cells and sum E_r, against the
    oracle's stored values."""
    _, _, scal, cells, Eo, Fo = ref
    Fo_abs = np.sqrt((Fo[:dim] ** 2).sum(axis=0))
    Fg = np.sqrt((F[:dim, cells] ** 2).sum(axis=0))
    return {"E_r": float(np.abs(E[cells] - Eo).max() / scal["E_max"]),
            "abs_F_r": float(np.abs(Fg - Fo_abs).max() / max(scal["F_max"], 1e-3 * scal["E_max"])),
            "sum_E_r": float(abs(E.sum() - scal["E_sum"]) / scal["E_sum"])}


def _stated_case(stream, name, precisions):
    """One workload after its full step count in each precision, against the
    oracle's stored sample; float against FP64 over the whole grid too."""
    from paper_1403_6126_gb300 import workloads as wlmod
    ref = _stated_sample(name)
    if ref is None:
        return None
    dt, steps = ref[0], ref[1]
    wl = _stated_workload(name)
    n, w = _angles(wl["angles"])
    I0 = wlmod.initial_intensity(wl, len(w)).astype(np.float32).astype(np.float64)
    dim = wl["dim"]
    out = {"workload": "%s %s x %d angles, %d steps; %d stored cells" % (
        name, "x".join(str(s) for s in wl["shape"][::-1] if s > 1), len(w), steps, len(ref[3]))}
    full = {}
    for prec in precisions:
        c = _context(wl, n, w, stream=stream.cuda_stream, precision=prec)
        c.set_intensity(I0)
        c.set_material(wl["rho"], wl["T"], wl["v"], wl["sa"], wl["ss"])
        c.run(dt, steps)
        c.sync()
        E, F, _ = c.moments()
        c.close()
        full[prec] = (E, np.sqrt((F[:dim] ** 2).sum(axis=0)))
        out[prec] = _stated_errors(E, F, ref, dim)
    if "fp64" in full and "fp32" in full:
        (E64, F64), (E32, F32) = full["fp64"], full["fp32"]
        out["fp32_vs_fp64_whole_grid"] = {
            "E_r": float(np.abs(E32 - E64).max() / np.abs(E64).max()),
            "abs_F_r": float(np.abs(F32 - F64).max() / max(F64.max(), 1e-3 * np.abs(E64).max())),
            "cells_E_over_1e-5": int((np.abs(E32 - E64) > 1e-5 * np.abs(E64).max()).sum())}
    return out


def bench_accuracy(stream):
    """The error of every GPU precision against the FP64 oracle after the full
    step count of each workload, at the oracle's stored sample of cells
    (tests/golden/stated_*.txt: written by tests/golden/make_stated_steps.py
    from the oracle alone; nothing here runs the oracle)."""
    return {"slab1d_512x8_2000_steps": _stated_case(stream, "slab1d", ("fp64", "fp32")),
            "shadow2d_256x128x80_4000_steps": _stated_case(stream, "shadow2d", ("fp64", "fp32", "bf16")),
            "box3d_128x80_500_steps": _stated_case(stream, "box3d", ("fp64", "fp32", "bf16"))}


def bench_bf16(args, stream):
    """The timed workload with bf16 intensity storage (RT_BF16)."""
    import torch
    from paper_1403_6126_gb300 import workloads as wlmod
    wl = wlmod.by_name(args.workload, **({"n": args.n} if args.n else {}))
    n, w = _angles(wl["angles"])
    M, N = len(w), int(np.prod(wl["shape"]))
    c = _context(wl, n, w, stream=stream.cuda_stream, precision="bf16")
    c.set_intensity(wlmod.initial_intensity(wl, M))
    c.set_material(wl["rho"], wl["T"], wl["v"], wl["sa"], wl["ss"])
    dt = c.cfl_dt()
    for _ in range(3):
        c.step(dt)
    c.sync()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    for _ in range(args.steps):
        c.step(dt)
    e1.record(stream)
    c.sync()
    ms = e0.elapsed_time(e1) / args.steps
    c.close()
    peak, _ = _peaks()
    velocity = bool(np.any(wl["v"] != 0)) or wl["estimate_v"]
    b = (algorithmic_bytes_per_cell(M, 4, velocity, not wl["hold_T"]) - 2 * M * 2) * N   # intensities at 2 bytes
    return {"workload": "%s: %s cells x %d angles, bf16 intensities (deviation from the cell mean)"
                        % (wl["name"], "x".join(str(x) for x in wl["shape"][::-1]), M),
            "ms_per_step": ms, "value": N * M / (ms / 1e3), "unit": "cell-angle updates/s",
            "algorithmic_gb_s": b / (ms / 1e3) / 1e9, "frac_of_measured_hbm": b / (ms / 1e3) / 1e9 / peak,
            "algorithmic_bytes_per_step": b}


def _submit_args(wl, angles=None):
    import ctypes
    import paper_1403_6126_gb300 as rt
    n, w = _angles(wl["angles"]) if angles is None else (np.ascontiguousarray(angles[0]), np.ascontiguousarray(angles[1]))
    g = rt.rt_grid()
    g.dim = wl["dim"]
    nz, ny, nx = wl["shape"]
    for d, nd in enumerate((nx, ny, nz)):
        g.n[d] = nd
        g.lo[d], g.hi[d] = wl["lo"][d], wl["hi"][d]
        g.bc[d][0], g.bc[d][1] = wl["bc"][d]
    a = rt.rt_angles()
    a.m = len(w)
    a.n = n.ctypes.data_as(ctypes.POINTER(ctypes.c_double))
    a.w = w.ctypes.data_as(ctypes.POINTER(ctypes.c_double))
    fields = [np.ascontiguousarray(wl[k], dtype=np.float64).reshape(-1) for k in ("rho", "T", "v", "sa", "ss")]
    return g, a, (n, w), fields


def _serving_accuracy(opts, budget_gb):
    """Request 8 of the serving stream (96^2 box2d, 24 angles, 200 steps,
    float32-rounded fields) served through the server (float) and solved
    alone by the FP64 path, each against the oracle's stored sample
    (tests/golden/stated_serving_req8.txt)."""
    import paper_1403_6126_gb300 as rt
    ref = _stated_sample("serving_req8")
    if ref is None:
        return None
    dt, steps = ref[0], ref[1]
    wl = _stated_workload("serving_req8")
    g, a, (nn, w), f = _submit_args(wl)
    N, dim = int(np.prod(wl["shape"])), wl["dim"]
    server = rt.rt_server_create(int(budget_gb * 2 ** 30), opts)
    try:
        t = rt.rt_submit(server, g, a, wl["C"], wl["P"], *f, steps)
        rt.rt_server_wait(server, t, 600.0)
        Es, Fs = np.zeros(N), np.zeros((3, N))
        rt.rt_poll(server, t, Es, Fs, None)
    finally:
        rt.rt_server_destroy(server)
    # the oracle (like the float server) started from the float32-rounded
    # equilibrium 1/(4 pi): the FP64 path gets the same start
    from paper_1403_6126_gb300 import workloads as wlmod
    c = _context(wl, nn, w, precision="fp64")
    c.set_intensity(wlmod.initial_intensity(wl, len(w)).astype(np.float32).astype(np.float64))
    c.set_material(*f)
    c.run(dt, steps)
    c.sync()
    E64, F64, _ = c.moments()
    c.close()
    return {"request": "serving request 8: %s x %d angles, %d steps; %d stored cells"
                       % ("x".join(str(s) for s in wl["shape"][::-1] if s > 1), len(w), steps, len(ref[3])),
            "served_fp32": _stated_errors(Es, Fs, ref, dim), "fp64_one_at_a_time": _stated_errors(E64, F64, ref, dim)}


def bench_serving(args):
    """The serving workload: a Poisson stream of 2-D / 3-D solves
    into the continuous-batching server under an HBM budget; solves/s and
    p50/p99 latency, against solving the same requests one at a time with
    the FP64 path."""
    import paper_1403_6126_gb300 as rt
    from paper_1403_6126_gb300 import workloads as wlmod
    wls = wlmod.serving(nreq=args.serve_n, steps=args.serve_steps)
    reqs = [_submit_args(wl) for wl in wls]
    o = rt.rt_options_default()
    o.estimate_v, o.hold_T = 1, 0

    failed = []

    def run(gaps, nreq):
        # a request whose T^4 Newton fails (the positivity limit of the
        # method on under-resolved velocity fields) is counted, not fatal
        server = rt.rt_server_create(int(args.serve_budget_gb * 2 ** 30), o)
        try:
            t0 = time.perf_counter()
            tickets = []
            for (g, a, _, f), wl, gap in zip(reqs[:nreq], wls[:nreq], gaps):
                while time.perf_counter() - t0 < gap:
                    time.sleep(0.0005)
                tickets.append(rt.rt_submit(server, g, a, wl["C"], wl["P"], *f, wl["steps"]))
            lat, nfail = [], 0
            for t in tickets:
                rt.rt_server_wait(server, t, 600.0)
                try:
                    lat.append(rt.rt_poll(server, t))
                except rt.RTError as e:
                    if e.status != rt.RT_E_NONFINITE:
                        raise
                    nfail += 1
            makespan = time.perf_counter() - t0
            steps = rt.rt_server_stats(server)["steps"]
        finally:
            rt.rt_server_destroy(server)
        failed.append(nfail)
        return makespan, np.array(lat), steps

    # capacity (all at once) and the 2x overload on the stream's first
    # --serve-cap-n requests (the same mix); the Poisson stream at 0.8x
    # capacity on all of them
    ncap = min(args.serve_cap_n, len(reqs))
    burst, _, _ = run(np.zeros(ncap), ncap)
    capacity = (ncap - failed[0]) / burst
    rng = np.random.default_rng(60)
    gaps = rng.exponential(1.0, len(reqs))
    arrivals = np.cumsum(gaps / (0.8 * capacity))
    arrivals -= arrivals[0]
    makespan, lat, steps = run(arrivals, len(reqs))
    over = np.cumsum(gaps[:ncap] / (2.0 * capacity))      # the first ncap at 2x capacity
    over -= over[0]
    over_makespan, over_lat, _ = run(over, ncap)
    # one at a time, FP64: a seeded sample stratified by dimension and angle
    # count (up to --serve-fp64-per-stratum requests from each of 2-D / 3-D
    # x 24 / 80 angles), each timed over at most --serve-fp64-steps steps
    # (one CUDA graph, after one untimed step) and scaled to its full step
    # count; the stream's total is each stratum's seconds per
    # cell-angle-step times the stratum's cell-angle-steps
    work = [int(np.prod(wl["shape"])) * len(r[2][1]) * wl["steps"] for r, wl in zip(reqs, wls)]
    strata = {}
    for i, (r, wl) in enumerate(zip(reqs, wls)):
        strata.setdefault((wl["dim"], len(r[2][1])), []).append(i)
    rng_s = np.random.default_rng(61)
    sample = {key: sorted(rng_s.choice(idx, size=min(args.serve_fp64_per_stratum, len(idx)), replace=False).tolist())
              for key, idx in sorted(strata.items())}
    t_fp64 = {}
    for key, idx in sample.items():
        for i in idx:
            (g, a, (n, w), f), wl = reqs[i], wls[i]
            c = _context(wl, n, w, precision="fp64")
            c.set_material(*f)
            S = min(wl["steps"], args.serve_fp64_steps)
            c.run(0.0, 1)
            c.sync()
            t0 = time.perf_counter()
            c.run(0.0, S)
            try:
                c.sync()
            except rt.RTError as e:
                if e.status != rt.RT_E_NONFINITE:
                    raise
            t_fp64[i] = (time.perf_counter() - t0) * wl["steps"] / S
            c.close()
    total = 0.0
    for key, idx in strata.items():
        rate = sum(t_fp64[i] for i in sample[key]) / sum(work[i] for i in sample[key])
        total += rate * sum(work[i] for i in idx)
    fp64_rate = len(reqs) / total
    mix = ", ".join("%d-D x %d angles: %d of %d" % (k[0], k[1], len(sample[k]), len(strata[k])) for k in sorted(strata))
    # both paths against the oracle's stored values for one request
    accuracy = _serving_accuracy(o, args.serve_budget_gb)
    return {"workload": "%d requests: 2-D 64..512^2 and 3-D 64..192^3 (sides in steps of 32), 24/80 angles, %d steps each, box gas fields; "
                        "Poisson arrivals at 0.8 x measured capacity" % (len(reqs), args.serve_steps),
            "value": (len(reqs) - failed[1]) / makespan, "unit": "solves/s", "p50_latency_s": float(np.percentile(lat, 50)),
            "p99_latency_s": float(np.percentile(lat, 99)), "capacity_solves_s": capacity,
            "capacity_requests": ncap,
            "batch_steps": steps, "budget_gb": args.serve_budget_gb,
            "failed_requests_per_run": failed,
            "overload_2x": {"value": (ncap - failed[2]) / over_makespan, "unit": "solves/s", "requests": ncap,
                            "p50_latency_s": float(np.percentile(over_lat, 50)),
                            "p99_latency_s": float(np.percentile(over_lat, 99))},
            "fp64_one_at_a_time": {"value": fp64_rate, "unit": "solves/s", "timed_requests": len(t_fp64),
                                   "note": "seeded sample stratified by dimension and angle count (%s), each "
                                           "request timed over %d steps and scaled to its step count; each "
                                           "stratum scaled to the stream by its cell-angle-steps"
                                           % (mix, args.serve_fp64_steps)},
            "accuracy_vs_oracle": accuracy}


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--workload", default="box3d")
    ap.add_argument("--n", type=int, default=0, help="box3d side (default 128)")
    ap.add_argument("--tile", default="", help="tile shape TXxTYxTZ (default: the library's choice)")
    ap.add_argument("--impl", default="gpu", choices=["gpu", "reference"])
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--ref-steps", type=int, default=5, help="most oracle steps the reference arm times")
    ap.add_argument("--no-batch", action="store_true")
    ap.add_argument("--no-small", action="store_true")
    ap.add_argument("--no-accuracy", action="store_true")
    ap.add_argument("--no-bf16", action="store_true")
    ap.add_argument("--no-autotune", action="store_true")
    ap.add_argument("--no-serve", action="store_true")
    ap.add_argument("--batch-n", type=int, default=512)
    ap.add_argument("--batch-steps", type=int, default=20)
    ap.add_argument("--serve-n", type=int, default=500)
    ap.add_argument("--serve-cap-n", type=int, default=64,
                    help="requests of the capacity and 2x-overload runs (the stream's first ones)")
    ap.add_argument("--serve-steps", type=int, default=200)
    ap.add_argument("--serve-fp64-per-stratum", type=int, default=4)
    ap.add_argument("--serve-fp64-steps", type=int, default=20)
    ap.add_argument("--serve-budget-gb", type=float, default=150.0)
    args = ap.parse_args()
    if args.warmup < 3 and args.impl == "gpu":
        args.warmup = 3
    if args.impl == "reference":
        return run_reference(args)
    return run_gpu(args)


if __name__ == "__main__":
    sys.exit(main())
