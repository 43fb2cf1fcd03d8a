#!/usr/bin/env python
"""Benchmark of the particle <-> fixed-mesh projection round trip on one GB300.

Workload: 1025 x 1025 periodic mesh (H = 1/1024), 2048 x 2048 jittered particles (h = H/2,
jitter 0.25 h), four FP32 channels (Taylor-Green u, v, p and a Zalesak slotted-disk
indicator).  One step = bin the particles (stable counting sort) -> quadratic P2M with the
shape functions built on the fly -> linear-FE M2P, all through the C ABI.

Prints one JSON line (rank 0).  `--impl reference` times the FP64 CPU oracle instead.
"""
from __future__ import annotations

import argparse
import json
import os
import subprocess
import tempfile
import sys
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "Mparticles/s for P2M+M2P round trip; %HBM peak; max rel err vs FP64 oracle"
UNIT = "Mparticles/s"
L2_BYTES = 129 * 1024 * 1024

# Mean edge-stencil size on the benchmark workload (oracle, 12,000 edges of 4,000 random nodes).
STENCIL_MEAN = 10.43
# FP32 arithmetic the method defines for one node of the quadratic P2M (the Delaunay search is
# integer and filtered-predicate work, not counted): barycentrics (30) + 3 edges x (244 + 77 k)
# (frame, Cholesky, two triangular solves; per stencil point the coordinates, monomials, moment
# update, coefficient and the apply of C = 4 values), + 24.
FLOP_PER_NODE_Q = 30 + 3 * (244 + 77 * STENCIL_MEAN) + 24
FP32_LANES_PER_SM = 128


def kernel_traffic(stage: str, solve: str):
    """DRAM bytes per launch of the dominant kernel, from the committed ncu summary
    (profiles/p2m_kernels_traffic.txt: lines 'key value'), or None when the kernel sources
    changed since those counters were taken."""
    import hashlib
    path = os.path.join(ROOT, "profiles", "p2m_kernels_traffic.txt")
    try:
        kv = dict(line.split()[:2] for line in open(path) if line.strip() and not line.startswith("#"))
    except Exception:
        return None
    h = hashlib.sha256()
    for f in sorted(os.listdir(os.path.join(ROOT, "paper_1610_05266_gb300", "csrc"))):
        h.update(open(os.path.join(ROOT, "paper_1610_05266_gb300", "csrc", f), "rb").read())
    if kv.get("sha256") != h.hexdigest():
        return None
    key = f"{stage}_{solve}"
    return int(kv[key]) if key in kv else None


def peaks():
    try:
        return json.load(open(os.path.join(ROOT, "MEASURED_PEAKS.json")))
    except Exception:
        return {}


def dist_setup():
    import torch
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1:
        import torch.distributed as dist
        os.environ.setdefault("MASTER_ADDR", "127.0.0.1")
        if torch.cuda.is_available():
            torch.cuda.set_device(local)
        dist.init_process_group("nccl" if torch.cuda.is_available() else "gloo")
    return world, rank, local


def free_port() -> int:
    import socket
    with socket.socket() as s:
        s.bind(("127.0.0.1", 0))
        return s.getsockname()[1]


def _replica(local: int, world: int, port: int, argv):
    """Entry of one replica process started by spawn_replicas."""
    os.environ.update({"RANK": str(local), "LOCAL_RANK": str(local), "WORLD_SIZE": str(world),
                       "MASTER_ADDR": "127.0.0.1", "MASTER_PORT": str(port)})
    sys.argv = [sys.argv[0]] + list(argv)
    main()


def spawn_replicas(n: int):
    """`--gpus N` without a launcher: start N processes, one per GPU (rank = local rank)."""
    import torch.multiprocessing as mp
    mp.start_processes(_replica, args=(n, free_port(), sys.argv[1:]), nprocs=n, join=True,
                       start_method="spawn")


def barrier(world):
    if world > 1:
        import torch.distributed as dist
        dist.barrier()


def max_over_ranks(x: float, world: int) -> float:
    """Largest value over the replicas (timing is the slowest rank's)."""
    if world == 1:
        return x
    import torch
    import torch.distributed as dist
    dev = "cuda" if dist.get_backend() == "nccl" else "cpu"
    t = torch.tensor([x], dtype=torch.float64, device=dev)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


class ClockSampler:
    """nvidia-smi clock/throttle samples during the timed region."""
    FIELDS = ("timestamp,index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.gpu = gpu_index
        self.proc = None
        self.path = os.path.join(tempfile.gettempdir(), f"pfem_clocks_{os.getpid()}.csv")

    def start(self):
        try:
            os.makedirs(os.path.dirname(self.path), exist_ok=True)
            self.f = open(self.path, "w")
            self.proc = subprocess.Popen(["nvidia-smi", f"--id={self.gpu}",
                                          f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
                                          "-lms", "50"], stdout=self.f, stderr=subprocess.DEVNULL)
            time.sleep(0.5)                  # let the sampler come up before the timed region
        except Exception:
            self.proc = None

    def mark(self, which: str):
        setattr(self, which, time.time())

    def stop(self):
        if self.proc is None:
            return None
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        self.f.close()
        import datetime
        rows = []
        for line in open(self.path):
            parts = [p.strip() for p in line.split(",")]
            if len(parts) >= 10:
                try:
                    ts = datetime.datetime.strptime(parts[0], "%Y/%m/%d %H:%M:%S.%f").timestamp()
                except ValueError:
                    continue
                rows.append((ts, parts[1:]))
        if not rows:
            return None
        t0, t1 = getattr(self, "t_start", 0.0), getattr(self, "t_end", 1e300)
        inside = [r for t, r in rows if t0 - 0.05 <= t <= t1 + 0.05]
        if not inside:   # timed region shorter than one sampling period: nearest samples
            inside = [min(rows, key=lambda x: abs(x[0] - 0.5 * (t0 + t1)))[1]]
        num = lambda v: float(v) if v.replace(".", "").isdigit() else None
        sm = [num(r[1]) for r in inside if num(r[1]) is not None]
        mx = [num(r[2]) for r in inside if num(r[2]) is not None]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[k] for r in inside for k in range(4) if r[5 + k] == "Active"})
        return {"sm_mhz": float(np.median(sm)) if sm else None,
                "sm_max_mhz": max(mx) if mx else None, "reasons": reasons,
                "samples": len(inside), "timed_s": t1 - t0}


def oracle_round_trip(pr, threads: int, node_range=None, particles=None):
    """One round trip of the FP64 oracle on the workload's FP32 positions: bins of all
    particles, quadratic P2M at the nodes of `node_range` (all nodes when None; OpenMP,
    `threads` threads) and linear-FE M2P of that mesh at the first `particles` particles (all
    when None; one thread).  Returns (seconds, mesh [n,n,C], vals [N',C], breakdown)."""
    import oracle as O
    n, N = pr.n, pr.N
    pos = np.ascontiguousarray(pr.pos.astype(np.float32).astype(np.float64))
    vals = np.ascontiguousarray(pr.vals)
    t0 = time.perf_counter()
    O.build_cells(n, pos)
    t_cells = time.perf_counter() - t0
    t0 = time.perf_counter()
    mesh = O.p2m(n, pos, vals, shape=1, nthreads=threads, node_range=node_range)
    t_p2m = time.perf_counter() - t0
    m = N if particles is None else min(particles, N)
    t0 = time.perf_counter()
    back = O.m2p(n, pos[:m], mesh)
    t_m2p = time.perf_counter() - t0
    nodes = n * n if node_range is None else node_range[1] - node_range[0]
    return t_cells + t_p2m + t_m2p, mesh, back, {
        "cells_s": t_cells, "p2m_nodes": nodes, "p2m_s": t_p2m, "m2p_particles": m,
        "m2p_s": t_m2p}


def run_reference(args, world, rank, workload=None):
    """The reference arm: the FP64 oracle on the host cores, rank 0 only.  Each step is one
    whole round trip of the workload while (steps + warm-up) whole steps fit in about four
    minutes; otherwise every step after the first warm-up step takes the same fraction of the
    mesh nodes and particles, and the line says so (its rate is measured on that sample, not
    extrapolated)."""
    if rank != 0:
        return
    from workloads import config_large
    pr = workload() if workload is not None else config_large()
    threads = os.cpu_count() or 1
    nn = pr.n * pr.n
    t_full, _, _, bd_full = oracle_round_trip(pr, threads)          # first warm-up step, whole
    budget_s = 240.0
    frac = min(1.0, budget_s / max(1e-9, t_full * (args.steps + max(args.warmup - 1, 0))))
    if frac >= 1.0:
        node_range, parts = None, None
        sample = (f"each step the whole workload: oracle bins of all {pr.N} particles, quadratic "
                  f"P2M at all {nn} nodes ({threads} OpenMP threads), M2P at all particles")
    else:
        k = max(1024, int(nn * frac))
        b = nn // 2 - k // 2
        node_range, parts = (b, b + k), max(1024, int(pr.N * frac))
        sample = (f"each timed step a sample: oracle bins of all {pr.N} particles, quadratic P2M "
                  f"at {k} of {nn} nodes, M2P at {parts} of {pr.N} particles; the rate is "
                  f"particles of the sample per second (whole step measured once: "
                  f"{t_full:.2f} s)")
    for _ in range(max(args.warmup - 1, 0)):
        oracle_round_trip(pr, threads, node_range, parts)
    times, last = [], None
    for _ in range(args.steps):
        t, _, _, last = oracle_round_trip(pr, threads, node_range, parts)
        times.append(t)
    t = float(np.mean(times))
    units = pr.N if frac >= 1.0 else pr.N * (node_range[1] - node_range[0]) / nn
    value = units / t / 1e6
    out = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world,
           "steps": args.steps, "warmup": args.warmup, "ms_per_step": t * 1e3,
           "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
           "data": "synthetic",
           "config": {"workload": pr.name, "mesh_nodes": f"{pr.n}x{pr.n}",
                      "particles": f"{pr.M}x{pr.M}", "channels": pr.C},
           "cpu_baseline": {"value": value, "unit": UNIT, "cores": threads, "kind": "oracle",
                            "sample": sample, "whole_step_s": t_full,
                            "step_is_whole_workload": frac >= 1.0, "breakdown": last},
           "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(out), flush=True)


def run_ours(args, world, rank, local):
    import torch
    import paper_1610_05266_gb300 as P
    from workloads import config_large

    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    P.load()
    pr = config_large()
    n, N, C = pr.n, pr.N, pr.C
    nn = n * n
    pos = torch.tensor(pr.pos, dtype=torch.float32, device=dev)
    vals = torch.tensor(pr.vals, dtype=torch.float32, device=dev)
    proj = P.Projector(n, N, C=C, pos_dtype=torch.float32, device=dev)
    mesh = torch.empty((n, n, C), dtype=torch.float32, device=dev)
    back = torch.empty((N, C), dtype=torch.float32, device=dev)
    flush = torch.empty(2 * L2_BYTES // 4, dtype=torch.float32, device=dev)
    solves = {"f32": P.PFEM_SOLVE_F32, "f32ref": P.PFEM_SOLVE_F32_REFINED,
              "f32ff": P.PFEM_SOLVE_F32_REFINED_FF, "f64": P.PFEM_SOLVE_F64}
    solve = solves[args.solve]
    sms = torch.cuda.get_device_properties(dev).multi_processor_count
    stream = torch.cuda.current_stream()

    ev = lambda: torch.cuda.Event(enable_timing=True)
    ctx = P.Context()
    proj.ctx = ctx
    def step(rec=None, stage=None):
        if stage is not None:
            ctx.set_stage_events(stage)
        if rec is not None:
            rec[0].record(stream)
        proj.build(pos)
        if rec is not None:
            rec[1].record(stream)
        proj.p2m(vals, shape=P.PFEM_SHAPE_QUADRATIC, solve=solve, out=mesh)
        if rec is not None:
            rec[2].record(stream)
        proj.m2p(pos, mesh, out=back)
        if rec is not None:
            rec[3].record(stream)

    for _ in range(max(args.warmup, 3) if not args.profile else args.warmup):
        step()
    torch.cuda.synchronize()
    proj.check("warm-up")

    clocks = ClockSampler(local)
    clocks.start()
    recs = [[ev() for _ in range(4)] for _ in range(args.steps)]
    stages = [[ev() for _ in range(5)] for _ in range(args.steps)]
    for st in stages:
        for e in st:
            e.record(stream)                 # create the handles before the timed region
    torch.cuda.synchronize()
    l0 = P.pfem_launch_count()
    barrier(world)
    torch.cuda.synchronize()
    clocks.mark("t_start")
    for k in range(args.steps):
        flush.zero_()                       # evict L2 between timed steps (outside the events)
        step(recs[k], stages[k])
    torch.cuda.synchronize()
    clocks.mark("t_end")
    barrier(world)
    launches = P.pfem_launch_count() - l0
    clk = clocks.stop()
    proj.check("timed steps")
    ctx.set_stage_events([])
    # the node location runs inside the solve kernel (k_p2m_tab): "geometry" is only the gap
    # between two events
    stage_ms = {name: float(np.mean([st[i].elapsed_time(st[i + 1]) for st in stages]))
                for i, name in enumerate(("star_table", "geometry", "solve", "fix_pass"))}
    step_ms = [r[0].elapsed_time(r[3]) for r in recs]
    cells_ms = [r[0].elapsed_time(r[1]) for r in recs]
    p2m_ms = [r[1].elapsed_time(r[2]) for r in recs]
    m2p_ms = [r[2].elapsed_time(r[3]) for r in recs]
    t_step = max_over_ranks(float(np.sum(step_ms)) / args.steps, world)
    value = world * N / (t_step * 1e-3) / 1e6

    pk = peaks()
    hbm_peak = pk.get("hbm_gbs", 6800.0)
    t_p2m = float(np.mean(p2m_ms)) * 1e-3
    t_m2p = float(np.mean(m2p_ms)) * 1e-3
    sm_mhz = (clk or {}).get("sm_mhz") or pk.get("sm_max_mhz", 2070.0)
    fp32_peak = sms * FP32_LANES_PER_SM * 2 * 2070.0e6 / 1e12   # TFLOP/s at the maximum SM clock
    p2m_flops = FLOP_PER_NODE_Q * nn
    # algorithmic bytes of the round trip: P2M reads pos + C vals per particle and writes C
    # per node; M2P reads pos per particle, C per node, writes C per particle (FP32)
    rt_bytes = N * (8 + 4 * C) + nn * 4 * C + N * 8 + nn * 4 * C + N * 4 * C
    m2p_bytes = N * 8 + nn * 4 * C + N * 4 * C
    # the dominant kernel of the step, timed by the stage events: integer and FP32 filter work of
    # the star table, or the location, FP32 solve and fixed-point residual of the node kernel
    dominant = max(stage_ms, key=stage_ms.get)
    roofline = {"bound": "alu", "kernel": {"star_table": "k_star_list + k_star_retry",
                                            "geometry": "none (gap between two events)",
                                            "solve": "k_p2m_tab (location, edge solves, apply)",
                                            "fix_pass": "k_p2m_fix_tab"}[dominant],
                "achieved": p2m_flops / t_p2m / 1e12, "peak": fp32_peak, "unit": "TFLOP/s",
                "frac": p2m_flops / t_p2m / 1e12 / fp32_peak,
                "algorithmic_flop_per_node": FLOP_PER_NODE_Q,
                "note": "FP32 arithmetic of the whole quadratic P2M call over the call's time",
                "peak_source": f"{sms} SMs (device query) x 128 FP32 lanes x 2 x 2070 MHz (derived)"}
    roofline["kernel_ms"] = stage_ms[dominant]
    roofline["traffic"] = kernel_traffic(dominant, args.solve)
    roofline["traffic_unit"] = "bytes per launch (ncu dram read+write), null when the sources changed since"
    out = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
           "warmup": args.warmup, "ms_per_step": t_step, "higher_is_better": True,
           "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
           "config": {"workload": pr.name, "mesh_nodes": f"{n}x{n}", "particles": f"{pr.M}x{pr.M}",
                      "channels": C, "jitter": pr.a, "shape": "quadratic", "solve": args.solve,
                      "bins": proj.nb, "l2": "flushed between timed steps (2x L2 write)",
                      "parallelism": "replicas only" if world > 1 else "single GPU"},
           "roofline": roofline,
           "hbm_view": {"round_trip_bytes": rt_bytes,
                        "round_trip_gbs": rt_bytes / (t_step * 1e-3) / 1e9,
                        "round_trip_frac": rt_bytes / (t_step * 1e-3) / 1e9 / hbm_peak,
                        "m2p_gbs": m2p_bytes / t_m2p / 1e9,
                        "m2p_frac": m2p_bytes / t_m2p / 1e9 / hbm_peak,
                        "peak_gbs": hbm_peak, "peak_source": "MEASURED_PEAKS.json hbm_gbs"},
           "breakdown_ms": {"build_cells": float(np.mean(cells_ms)), "p2m_quadratic": t_p2m * 1e3,
                            "m2p": t_m2p * 1e3, "p2m_stages": stage_ms},
           "gpu_launches": int(launches),
           "clocks": clk}
    if args.profile:
        if rank == 0:
            print(json.dumps(out), flush=True)
        return

    # --- end to end through the ABI with host buffers (copies inside the timed region): every
    # step copies positions and values from pinned host memory and the particle values back;
    # api.HostRoundTrip overlaps those copies with the compute of the neighbouring steps
    pos_h = torch.tensor(pr.pos, dtype=torch.float32).pin_memory()
    vals_h = torch.tensor(pr.vals, dtype=torch.float32).pin_memory()
    back_h = torch.empty((N, C), dtype=torch.float32).pin_memory()
    rt = P.HostRoundTrip(proj, C, dtype=torch.float32, solve=solve, stream=stream)
    for _ in range(3):
        rt.step(pos_h, vals_h, back_h)
    rt.wait()
    torch.cuda.synchronize()
    e0, e1 = ev(), ev()
    ke = max(3, args.steps // 2)
    barrier(world)
    e0.record(stream)
    rt.h2d.wait_event(e0)               # the first copy starts inside the timed region
    for _ in range(ke):
        rt.step(pos_h, vals_h, back_h)
    rt.join(stream)                     # ... and the last copy back ends inside it
    e1.record(stream)
    torch.cuda.synchronize()
    proj.check("end-to-end steps")
    t_e2e = max_over_ranks(e0.elapsed_time(e1) / ke, world)
    # the same steps with the copies in stream order (nothing overlapped), for comparison
    pos_d, vals_d = torch.empty_like(pos), torch.empty_like(vals)
    def serial_step():
        pos_d.copy_(pos_h, non_blocking=True)
        vals_d.copy_(vals_h, non_blocking=True)
        proj.build(pos_d)
        proj.p2m(vals_d, shape=P.PFEM_SHAPE_QUADRATIC, solve=solve, out=mesh)
        proj.m2p(pos_d, mesh, out=back)
        back_h.copy_(back, non_blocking=True)
    serial_step()
    torch.cuda.synchronize()
    e0.record(stream)
    for _ in range(ke):
        serial_step()
    e1.record(stream)
    torch.cuda.synchronize()
    t_serial = max_over_ranks(e0.elapsed_time(e1) / ke, world)
    out["e2e"] = {"value": world * N / (t_e2e * 1e-3) / 1e6, "unit": UNIT,
                  "h2d_bytes_per_step": int(pos_h.numel() * 4 + vals_h.numel() * 4),
                  "d2h_bytes_per_step": int(back_h.numel() * 4), "ms_per_step": t_e2e,
                  "api": "HostRoundTrip.step (public API): copies on their own streams, double-"
                         "buffered inputs, P2M waits for the values before its solve kernel",
                  "serial_copies_ms_per_step": t_serial,
                  "serial_copies_value": world * N / (t_serial * 1e-3) / 1e6}

    if rank != 0:
        return                  # replicas beyond rank 0 only take part in the timed regions

    # --- side measurements (outside the timed region)
    def timeit(fn, reps=5):
        fn()
        torch.cuda.synchronize()
        a, b = ev(), ev()
        a.record(stream)
        for _ in range(reps):
            fn()
        b.record(stream)
        torch.cuda.synchronize()
        return a.elapsed_time(b) / reps
    side = {}
    side["p2m_linear_ms"] = timeit(lambda: proj.p2m(vals, shape=P.PFEM_SHAPE_LINEAR, out=mesh))
    side["m2p_mesh_qcsf_ms"] = timeit(lambda: proj.m2p(pos, mesh, out=back, shape=P.PFEM_SHAPE_QUADRATIC))
    def projfemq():     # quadratic both ways: the paper's projFEMq interpolation pair
        proj.build(pos)
        proj.p2m(vals, shape=P.PFEM_SHAPE_QUADRATIC, solve=solve, out=mesh)
        proj.m2p(pos, mesh, out=back, shape=P.PFEM_SHAPE_QUADRATIC)
    side["projfemq_round_trip_ms"] = timeit(projfemq)
    side["projfemq_round_trip_mparticles_s"] = N / (side["projfemq_round_trip_ms"] * 1e-3) / 1e6
    for nm, sv in (("f64", P.PFEM_SOLVE_F64), ("f32ref", P.PFEM_SOLVE_F32_REFINED), ("f32", P.PFEM_SOLVE_F32)):
        side[f"p2m_quadratic_solve_{nm}_ms"] = timeit(
            lambda: proj.p2m(vals, shape=P.PFEM_SHAPE_QUADRATIC, solve=sv, out=mesh))
    def f32ff_round_trip():
        proj.build(pos)
        proj.p2m(vals, shape=P.PFEM_SHAPE_QUADRATIC, solve=P.PFEM_SOLVE_F32_REFINED_FF, out=mesh)
        proj.m2p(pos, mesh, out=back)
    side["f32ff_round_trip_ms"] = timeit(f32ff_round_trip)
    side["f32ff_round_trip_mparticles_s"] = N / (side["f32ff_round_trip_ms"] * 1e-3) / 1e6
    # the projection loop of the Zalesak procedure at this size: M2P of the field, midpoint move
    # in a mesh rotation field, re-binning, quadratic P2M; dt keeps every move within one bin
    gx = torch.arange(n, device=dev, dtype=torch.float32) / (n - 1)
    Y, X = torch.meshgrid(gx, gx, indexing="ij")
    inside = ((X - 0.5) ** 2 + (Y - 0.5) ** 2) < 0.45 ** 2
    vel = torch.stack([torch.where(inside, -2 * np.pi * (Y - 0.5), 0.0),
                       torch.where(inside, 2 * np.pi * (X - 0.5), 0.0)], -1).contiguous()
    lproj = P.Projector(n, N, C=C, pos_dtype=torch.float32, device=dev)
    lpos = pos.clone()
    lproj.build(lpos)
    lmesh = mesh.clone()
    state = {"pos": lpos, "mesh": lmesh}
    def loop_step(incremental):
        state["pos"], state["mesh"] = P.projection_loop(
            lproj, state["pos"], state["mesh"], vel, 2.5e-4, 1, solve=solve, incremental=incremental)
    side["loop_step_incremental_rebin_ms"] = timeit(lambda: loop_step(True), reps=5)
    side["loop_step_full_rebin_ms"] = timeit(lambda: loop_step(False), reps=5)
    side["loop_update_cells_ms"] = timeit(lambda: lproj.update(state["pos"]), reps=5)
    side["loop_build_cells_ms"] = timeit(lambda: lproj.build(state["pos"]), reps=5)
    side["loop_status"] = int(lproj.status()[0])
    del lproj, lpos, lmesh, state
    # plain FP64 single-instance form: FP64 positions and fields, FP64 solve
    pos64 = pos.double()                                     # the FP32 positions, exactly
    vals64 = torch.tensor(pr.vals, dtype=torch.float64, device=dev)
    proj64 = P.Projector(n, N, C=C, pos_dtype=torch.float64, device=dev)
    mesh64 = torch.empty((n, n, C), dtype=torch.float64, device=dev)
    back64 = torch.empty((N, C), dtype=torch.float64, device=dev)
    def step64():
        proj64.build(pos64)
        proj64.p2m(vals64, shape=P.PFEM_SHAPE_QUADRATIC, out=mesh64)
        proj64.m2p(pos64, mesh64, out=back64)
    t64 = timeit(step64, reps=3)
    side["fp64_round_trip_ms"] = t64
    side["fp64_round_trip_mparticles_s"] = N / (t64 * 1e-3) / 1e6
    proj64.check("fp64 round trip")
    # irregular input: uniform random particles (no lattice), same sizes, FP32 quadratic P2M
    from workloads import generators as WG
    pos_u = torch.tensor(WG.uniform01(WG.SEED_BASE + 62, 2 * N).reshape(N, 2), dtype=torch.float32,
                         device=dev)
    proj_u = P.Projector(n, N, C=C, pos_dtype=torch.float32, device=dev)
    proj_u.build(pos_u)
    side["uniform_random_p2m_linear_ms"] = timeit(
        lambda: proj_u.p2m(vals, shape=P.PFEM_SHAPE_LINEAR, out=mesh), reps=3)
    side["uniform_random_p2m_quadratic_ms"] = timeit(
        lambda: proj_u.p2m(vals, shape=P.PFEM_SHAPE_QUADRATIC, solve=solve, out=mesh), reps=3)
    side["uniform_random_status"] = int(proj_u.status()[0])
    del proj_u, pos_u
    out["side"] = side

    # --- differentiation workload: L = 1/2 sum_i (P2M_i - t_i)^2, backward to values and
    #     positions, recompute vs checkpoint of the shape-function weights
    if not args.no_grad:
        from workloads import config_grad
        gp_ = config_grad()
        gpos = torch.tensor(gp_.pos, dtype=torch.float32, device=dev)
        gvals = torch.tensor(gp_.vals, dtype=torch.float32, device=dev)
        gtarget = torch.tensor(gp_.target, dtype=torch.float32, device=dev)
        gproj = P.Projector(gp_.n, gp_.N, C=1, pos_dtype=torch.float32, device=dev)
        gproj.build(gpos)
        def fwd():
            return gproj.p2m(gvals, shape=P.PFEM_SHAPE_QUADRATIC)
        gmesh = fwd()
        gbar = (gmesh - gtarget).contiguous()
        t_fwd = timeit(fwd)
        t_bwd_rec = timeit(lambda: gproj.backward(gvals, gbar))
        wts = gproj.shape_weights(K=32, w_dtype=torch.float32)
        t_shape = timeit(lambda: gproj.shape_weights(K=32, w_dtype=torch.float32))
        t_fwd_ck = timeit(lambda: gproj.p2m(gvals, weights=wts))
        t_bwd_ck = timeit(lambda: gproj.backward(gvals, gbar, weights=wts))
        t_bwd_ck_vals = timeit(lambda: gproj.backward(gvals, gbar, weights=wts, want_pos=False))
        code, _ = gproj.backward_status()
        out["gradient"] = {"workload": gp_.name, "dtype": "f32", "status": code,
                           "forward_fused_ms": t_fwd,
                           "backward_recompute_ms": t_bwd_rec,
                           "checkpoint_weights_ms": t_shape,
                           "forward_from_checkpoint_ms": t_fwd_ck,
                           "backward_checkpoint_ms": t_bwd_ck,
                           "backward_checkpoint_values_only_ms": t_bwd_ck_vals,
                           "step_recompute_ms": t_fwd + t_bwd_rec,
                           "step_checkpoint_ms": t_shape + t_fwd_ck + t_bwd_ck}
        del gproj, wts
        torch.cuda.empty_cache()

    # --- batched uneven problems (256, persistent launches, tuned, CUDA graph) vs the plain
    #     FP64 single-instance form, problem by problem
    if not args.no_batched:
        from paper_1610_05266_gb300 import tuner
        from workloads import config_batched
        probs = config_batched()
        bpos = torch.tensor(np.concatenate([p.pos for p in probs]), dtype=torch.float32, device=dev)
        bvals = torch.tensor(np.concatenate([p.vals for p in probs]), dtype=torch.float32, device=dev)
        batch = P.Batch([(p.n, p.N) for p in probs], C=3, dtype=torch.float32, device=dev)
        t0 = time.time()
        cfg = tuner.tune_batch(batch, bpos, bvals, P.PFEM_SHAPE_QUADRATIC, solve)
        tune_s = time.time() - t0
        batch.capture(bpos, bvals, solve=solve)
        tb = timeit(batch.replay, reps=3)
        code, _ = batch.status()
        Nb = batch.N_total
        rng_b = np.random.default_rng(11)
        checked = sorted(int(p) for p in rng_b.choice(len(probs), 4, replace=False))
        single_ms, single_mesh = 0.0, {}
        for ip, pb in enumerate(probs):
            pp = torch.tensor(pb.pos, dtype=torch.float64, device=dev)
            vv = torch.tensor(pb.vals, dtype=torch.float64, device=dev)
            pj = P.Projector(pb.n, pb.N, C=3, pos_dtype=torch.float64, device=dev)
            torch.cuda.synchronize()
            b0, b1 = ev(), ev()
            b0.record(stream)
            pj.build(pp)
            mm = pj.p2m(vv)
            pj.m2p(pp, mm)
            b1.record(stream)
            torch.cuda.synchronize()
            single_ms += b0.elapsed_time(b1)
            if ip in checked:
                single_mesh[ip] = mm.cpu().numpy()
        acc_b = None
        if rank == 0 and not args.no_oracle:
            import oracle as O
            eb, es = 0.0, 0.0
            for ip in checked:
                pb = probs[ip]
                p32 = pb.pos.astype(np.float32).astype(np.float64)
                ref32 = O.p2m(pb.n, p32, pb.vals, shape=1, nthreads=os.cpu_count() or 1)
                ref64 = O.p2m(pb.n, pb.pos, pb.vals, shape=1, nthreads=os.cpu_count() or 1)
                mb = batch.mesh_view(ip).cpu().numpy().astype(np.float64)
                eb = max(eb, float((np.abs(mb - ref32).reshape(-1, 3).max(0) /
                                    np.abs(ref32).reshape(-1, 3).max(0)).max()))
                es = max(es, float((np.abs(single_mesh[ip] - ref64).reshape(-1, 3).max(0) /
                                    np.abs(ref64).reshape(-1, 3).max(0)).max()))
            acc_b = {"batched_fp32_max_rel_err": eb, "fp64_single_instance_max_rel_err": es,
                     "compared": f"all nodes of problems {checked} against the FP64 oracle (the "
                                 f"batch on its FP32 positions, the FP64 form on the FP64 ones)"}
        out["batched"] = {"workload": "256 problems, n in 65..513, h/H in {1/4,1/2,1}, a=0.3, TG k in 1..8, C=3",
                          "particles": Nb, "nodes": batch.nodes_total,
                          "graph_replay_ms": tb, "mparticles_s": Nb / (tb * 1e-3) / 1e6,
                          "dtype": "f32", "solve": args.solve, "status": code,
                          "tuned": {k: v for k, v in cfg.items() if not k.startswith("_")},
                          "tune_s": tune_s,
                          "fp64_single_instance_ms": single_ms,
                          "fp64_single_instance_mparticles_s": Nb / (single_ms * 1e-3) / 1e6,
                          "speedup_vs_fp64_single": single_ms / tb,
                          "accuracy": acc_b}
        del batch, bpos, bvals
        torch.cuda.empty_cache()

    # --- precision study: 4097^2 mesh, 8192^2 particles (67M), Rayleigh-Taylor density
    if not args.no_precision:
        from workloads import config_precision
        pp = config_precision()
        ppos32 = torch.tensor(pp.pos, dtype=torch.float32, device=dev)
        pproj = P.Projector(pp.n, pp.N, C=1, pos_dtype=torch.float32, device=dev)
        pproj.build(ppos32)
        variants = {}
        # node rows 2040..2055 cross the interface y = 0.5 + 0.05 cos(2 pi x), where the
        # density varies fastest; the oracle computes every node of those rows
        J0, J1 = 2040, 2056
        refs = None
        if rank == 0 and not args.no_oracle:
            import oracle as O
            ref_rows = O.p2m(pp.n, pp.pos.astype(np.float32).astype(np.float64), pp.vals, shape=1,
                             nthreads=os.cpu_count() or 1, node_range=(J0 * pp.n, J1 * pp.n))
            refs = ref_rows[J0:J1, :, 0]
        for vt, vname in ((torch.float32, "f32"), (torch.bfloat16, "bf16")):
            vv = torch.tensor(pp.vals, dtype=torch.float32, device=dev).to(vt)
            for sv, sname in ((P.PFEM_SOLVE_F64, "solve_f64"), (P.PFEM_SOLVE_F32, "solve_f32"),
                              (P.PFEM_SOLVE_F32_REFINED, "solve_f32_refined"),
                              (P.PFEM_SOLVE_F32_REFINED_FF, "solve_f32_refined_ff")):
                mesh_p = pproj.p2m(vv, shape=P.PFEM_SHAPE_QUADRATIC, solve=sv)
                t_v = timeit(lambda: pproj.p2m(vv, shape=P.PFEM_SHAPE_QUADRATIC, solve=sv, out=mesh_p), reps=2)
                ent = {"p2m_ms": t_v}
                if refs is not None:
                    got = mesh_p[J0:J1, :, 0].float().cpu().numpy().astype(np.float64)
                    ent["max_rel_err_vs_fp64_oracle"] = float(np.abs(got - refs).max() / np.abs(refs).max())
                variants[f"{vname}_{sname}"] = ent
        code, _ = pproj.status()
        out["precision_study"] = {"workload": "4097x4097 mesh, 8192x8192 particles, RT density (C=1)",
                                  "variants": variants, "status": code,
                                  "error_sample": (f"every node of rows {J0}..{J1 - 1} ({(J1 - J0) * pp.n} "
                                                   f"nodes across the interface), error / max|rho|")}
        del pproj, ppos32
        torch.cuda.empty_cache()

    # --- the FP64 oracle over the whole workload (every node, every particle): the CPU baseline
    #     and the reference of the accuracy figures
    if rank == 0 and not args.no_oracle:
        threads = os.cpu_count() or 1
        t_or, ref_mesh, ref_back, bd = oracle_round_trip(pr, threads)
        if not args.no_cpu_baseline:
            out["cpu_baseline"] = {"value": N / t_or / 1e6, "unit": UNIT, "cores": threads,
                                   "kind": "oracle",
                                   "sample": ("the whole workload, not sampled: oracle bins of all "
                                              "particles (1 thread), quadratic P2M at all nodes (all "
                                              "cores, OpenMP), M2P at all particles (1 thread)"),
                                   "wall_seconds": t_or, "breakdown": bd}
        import oracle as O
        pos32 = np.ascontiguousarray(pr.pos.astype(np.float32).astype(np.float64))
        vmax = np.abs(ref_mesh).reshape(-1, C).max(0)
        bmax = np.abs(ref_back).max(0)

        def mesh_err(m):
            d = np.abs(m.cpu().numpy().astype(np.float64) - ref_mesh).reshape(-1, C).max(0)
            return float((d / vmax).max())
        variants = {}
        for nm in ("f32ref", "f32ff", "f32", "f64"):
            mm = torch.empty_like(mesh)
            proj.p2m(vals, shape=P.PFEM_SHAPE_QUADRATIC, solve=solves[nm], out=mm)
            variants[f"p2m_fp32_values_solve_{nm}"] = mesh_err(mm)
        proj.check("accuracy variants")
        variants["p2m_fp64_single_instance"] = mesh_err(mesh64)
        step()
        torch.cuda.synchronize()
        m_gpu = mesh.cpu().numpy().astype(np.float64)
        b_gpu = back.cpu().numpy().astype(np.float64)
        b_of_gpu_mesh = O.m2p(n, pos32, m_gpu)
        out["max_rel_err"] = {
            "solve": args.solve,
            "p2m_vs_fp64_oracle": mesh_err(mesh),
            "m2p_vs_fp64_oracle_same_mesh": float((np.abs(b_gpu - b_of_gpu_mesh).max(0) / bmax).max()),
            "round_trip_vs_fp64_oracle": float((np.abs(b_gpu - ref_back).max(0) / bmax).max()),
            "variants": variants,
            "compared": f"all {nn} nodes and all {N} particles; per channel max|gpu - oracle| / "
                        f"max|oracle|, maximum over the {C} channels",
        }

    if rank == 0:
        print(json.dumps(out), flush=True)


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=200)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--solve", choices=["f32", "f32ref", "f32ff", "f64"], default="f32ref",
                    help="moment solve of the headline P2M: f32ref = FP32 Cholesky + one "
                         "refinement step, residual in 64-bit fixed point (default); f32ff = the same "
                         "by its other name; f64 = FP64 assembly and solve; f32 = plain FP32 "
                         "Cholesky (a side variant outside the stated accuracy target)")
    ap.add_argument("--profile", action="store_true", help="timed loop only (for ncu)")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-oracle", action="store_true")
    ap.add_argument("--no-batched", action="store_true")
    ap.add_argument("--no-grad", action="store_true")
    ap.add_argument("--no-precision", action="store_true")
    args = ap.parse_args()
    if args.gpus > 1 and "WORLD_SIZE" not in os.environ and args.impl == "ours":
        spawn_replicas(args.gpus)
        return
    world, rank, local = dist_setup()
    if args.impl == "reference":
        run_reference(args, world, rank)
    else:
        run_ours(args, world, rank, local)
    if world > 1:
        import torch.distributed as dist
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
