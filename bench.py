"""Benchmark of the IGKS hot path on GB300: cell-updates/s of full implicit iterations
(ghosts, spectral radius, gradients, gas-kinetic flux with SA terms, residual, norms,
both LU-SGS sweeps and the update).

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl igks|reference]
      default: the 64-airfoil batch (64 seeded NACA 4-digit sections, SA, O-meshes of
      8k-80k cells, 2.26M cells in one context, FP32 sweeps with FP64 flux, residual and
      update, autotuned launch configuration), with the turbulent flat plate (FP64 and
      FP32 sweeps) and a bounded serving leg (converged solves/hour, p50/p99) beside it
  python bench.py --workload turbulent_plate|laminar_plate|naca0012 [--precision fp64|mixed]
  python bench.py --workload serving      request stream served vs the plain FP64 path
  python bench.py --workload cavity       implicit vs explicit, Table 1 vortex centres

One step = one iteration of the whole hot path over every solve of the workload.
`value` is device time (CUDA events on the library's stream around each step, L2 flushed
between steps by writing a 256 MiB buffer outside the timed intervals). `e2e` is the same
metric through the public API with host buffers: each step copies every solve's state in
from pinned host memory, iterates once (reading the per-solve status back) and copies the
states out. Under torchrun each rank runs an independent replica (the method does not
shard: replicas only) and rank 0 prints one JSON line with the max time over ranks.
--impl reference times the CPU oracle (single thread) on a bounded sample of the same
workload.
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402

from igks_inputs import fields as F  # noqa: E402
from igks_inputs import meshgen as G  # noqa: E402

WORKLOADS = {
    "turbulent_plate": (G.turbulent_plate, F.turbulent_plate_flow,
                        "turbulent flat plate, SA, Ma 0.2, Re 5e6, 128x64 quads + 12288 triangles"),
    "laminar_plate": (G.laminar_plate, F.laminar_plate_flow,
                      "laminar flat plate, Ma 0.15, Re 1e5, 64x32 quads"),
    "naca0012": (G.naca0012, F.naca_flow, "NACA 0012, SA, Ma 0.15, Re 6e6, AoA 10, hybrid O-mesh"),
}
METRIC = "cell-updates/s"
SM_COUNT, SM_MAX_MHZ = 152, 2070.0
# FP64 units of GB300: 2 FP64 FMA per SM per clock (1.25 TFLOP/s nominal at 2.07 GHz); the
# ALU peak of the flux kernel is this count at the SM clock sampled during the run
FP64_FLOP_PER_SM_CLK = 4.0
# Algorithmic FP64 work of the gas-kinetic flux per face: 2 kflop, the upper end of the
# method's own count (two erfc/exp pairs, ten 4x4 moment solves, the moment tables to
# order 6-7 and the flux assembly); what the kernel executes on top (the instructions
# inside the library's erfc/exp/divide) does not count as work done; FP64 and double-float
# solves execute about half of it (igks_gks.cuh), so their rate can pass the peak
FLUX_ALG_FLOPS_PER_FACE = 2000.0
# ncu figures per face / per cell of one launch, by workload, with the capture they come
# from (executed FP64 flops = 2 x DFMA + DADD + DMUL thread instructions; DRAM = read +
# write bytes); by bytes of the sweep type where precisions differ. None: not captured for
# that workload.
NCU = {
    "naca_batch": {"source": "ncu, k_flux_moment on the first 8 airfoils of the batch (573454 faces), per face",
                   "flux_exec_flops_per_face": {4: 2125.4}, "flux_dram_bytes_per_face": {4: 198.3}},
    "turbulent_plate": {"source": "ncu, the flux and the one-block-per-solve sweeps on the turbulent flat plate "
                                  "(35056 faces, 20480 cells)",
                        "flux_exec_flops_per_face": {4: 2121.2, 8: 1058.5},
                        "flux_dram_bytes_per_face": {4: 168.1, 8: 176.5},
                        "sweep_dram_bytes_per_cell": {("k_sweep_fwd", 8): 301.5, ("k_sweep_bwd", 8): 300.4,
                                                      ("k_sweep_fwd", 4): 168.2, ("k_sweep_bwd", 4): 163.9}},
}


def alg_bytes(kernel, t, nc, nf):
    """Algorithmic (compulsory) bytes of one launch: every array the kernel needs streamed
    once, neighbour re-reads from cache. t = bytes of the sweep type."""
    cell_flux_inputs = 17 * 8          # W 5, (limited) gradient 8, centroid 2, mu 2
    per = {
        "k_ghost": nc * (5 * 8 + 2 * 8) + nf * (3 * 4 + 3 * 8 + 8),   # states, viscosities, face ids/geometry, lambda_f
        "k_gradient": nc * (5 * 8 + 2 * 8 + 8 + 8 * 8 + 4 * 8 + 8 + 8) + nf * (2 * 4 + 8 + 8),
        "k_flux": nf * (4 * 4 + 8 * 8 + 10 * 8) + nc * cell_flux_inputs,
        "k_residual": nc * (8 + 8 * 8 + 5 * 8 + 3 * 8) + nf * (6 * 8 + 4 * 8),
        # record in (32 B static, 13 values, three stencil entries of 4), increments out
        "k_sweep_fwd": nc * (32 + 25 * t + 5 * t),
        "k_sweep_bwd": nc * (32 + 25 * t + 5 * t),
        # W, M, Lambda, velocity, SA diagonal in; record heads (2 x 13 T) and about four
        # stencil entries of 4 T out; face geometry and spectral radius
        "k_sweep_prep": nc * (2 * 5 * 8 + 8 + 2 * 8 + 8 + 26 * t + 16 * t) + nf * (6 * 8),
    }
    return per.get(kernel)


def _max_over_ranks(dist, x, device):
    """The largest x over all ranks (x itself without a process group): every timed
    quantity is reported as the slowest rank's."""
    if not dist:
        return x
    import torch
    t = torch.tensor([float(x)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def _dist(backend="nccl"):
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    if ws > 1:
        import torch.distributed as dist
        dist.init_process_group(backend)
        return dist, dist.get_rank(), ws
    return None, 0, 1


def _peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        with open(p) as f:
            return json.load(f), "measured"
    return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0}, "fallback"


class ClockSampler:
    """nvidia-smi clocks and throttle reasons sampled during the timed region."""

    def __init__(self, index):
        self.index = index
        self.rows = []
        self.proc = None

    def __enter__(self):
        q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--id={self.index}", f"--query-gpu={q}",
                                          "--format=csv,noheader,nounits", "-lms", "100"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
        except OSError:
            self.proc = None
        return self

    def _read(self):
        for line in self.proc.stdout:
            self.rows.append([c.strip() for c in line.split(",")])

    def __exit__(self, *a):
        if self.proc:
            time.sleep(0.25)
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()

    def summary(self):
        if not self.rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["unavailable"]}
        sm = [float(r[1]) for r in self.rows if len(r) > 2 and r[1].replace(".", "").isdigit()]
        mx = [float(r[2]) for r in self.rows if len(r) > 2 and r[2].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[k] for r in self.rows if len(r) >= 9 for k in range(4) if r[5 + k] == "Active"})
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": reasons, "samples": len(self.rows)}


def cpu_baseline(mesh, flow, budget_s=15.0):
    """The oracle as it stands, single-threaded, on the same workload (bounded sample)."""
    import oracle as O
    ora = O.Oracle(mesh, flow)
    ora.iterate(1)
    t0 = time.perf_counter()
    n = 0
    while True:
        ora.iterate(1)
        n += 1
        if time.perf_counter() - t0 >= budget_s or n >= 200:
            break
    dt = time.perf_counter() - t0
    return {"value": mesh.n_cells * n / dt, "unit": METRIC, "cores": 1, "kind": "oracle",
            "sample": f"{n} iterations (after the first) of the {mesh.n_cells}-cell workload from the free "
                      f"stream, {dt:.1f} s, single-threaded C oracle (-O2 -ffp-contract=off)"}


def run_reference(args, mesh, flow, desc, budget_s=150.0):
    """The reference arm: the CPU oracle, single-threaded, on the same workload. One step
    is one full oracle iteration; warm-up and timed steps are capped so the whole run stays
    within about budget_s seconds (the sample actually timed is stated)."""
    if int(os.environ.get("RANK", "0")) != 0:
        return                      # under torchrun only rank 0 runs the reference arm
    import oracle as O
    ora = O.Oracle(mesh, flow)
    t0 = time.perf_counter()
    ora.iterate(1)
    t_one = time.perf_counter() - t0
    n_warm = min(args.warmup, max(1, int(0.2 * budget_s / t_one)))
    n_time = min(args.steps, max(3, int(0.8 * budget_s / t_one)))
    if n_warm > 1:
        ora.iterate(n_warm - 1)
    t0 = time.perf_counter()
    ora.iterate(n_time)
    dt = time.perf_counter() - t0
    v = mesh.n_cells * n_time / dt
    sample = (f"{n_time} timed iterations (of --steps {args.steps}) after {n_warm} warm-up of the "
              f"{mesh.n_cells}-cell workload, single-threaded C oracle")
    line = {"metric": METRIC, "value": v, "unit": METRIC, "impl": "reference", "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * dt / n_time,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic", "config": {"workload": desc, "cells": mesh.n_cells, "faces": mesh.n_faces},
            "cpu_baseline": {"value": v, "unit": METRIC, "cores": 1, "kind": "oracle", "sample": sample},
            "e2e": {"value": v, "unit": METRIC, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


def run_reference_batch(args, budget_s=150.0):
    """The reference arm on the batch workload: the CPU oracle, single-threaded. One step
    is one oracle iteration of one airfoil of the batch (airfoil k mod 64 at step k, from
    the free stream); value = cells iterated / time. The steps are capped so that the run
    stays within about budget_s seconds; the sample actually timed is stated."""
    if int(os.environ.get("RANK", "0")) != 0:
        return
    import oracle as O
    cases = batch_cases(args.batch)
    oras = {}

    def step(k):
        m, fl = cases[k % len(cases)]
        if k % len(cases) not in oras:
            oras[k % len(cases)] = O.Oracle(m, fl)
        oras[k % len(cases)].iterate(1)
        return m.n_cells

    t_start = time.perf_counter()
    for k in range(args.warmup):
        step(k)
        if time.perf_counter() - t_start > 0.2 * budget_s:
            break
    t0 = time.perf_counter()
    cells, n = 0, 0
    for k in range(args.steps):
        cells += step(args.warmup + k)
        n += 1
        if time.perf_counter() - t0 > 0.8 * budget_s:
            break
    dt = time.perf_counter() - t0
    v = cells / dt
    sample = (f"{n} timed steps (of --steps {args.steps}), each one oracle iteration of one airfoil of the "
              f"64-airfoil batch in turn ({cells} cell-updates), after {args.warmup} warm-up steps, "
              f"single-threaded C oracle")
    desc = (f"{len(cases)} seeded NACA 4-digit airfoils (m 0-0.06, p 0.2-0.6, t 0.08-0.18), Ma 0.1-0.75, "
            f"AoA -4..8 deg, Re_c 1e6-1e7, SA, hybrid O-meshes of 8k-80k cells in one context")
    line = {"metric": METRIC, "value": v, "unit": METRIC, "impl": "reference", "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * dt / max(n, 1),
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic", "config": {"workload": desc, "solves": len(cases),
                                            "cells": sum(m.n_cells for m, _ in cases),
                                            "faces": sum(m.n_faces for m, _ in cases), "precision": "fp64"},
            "cpu_baseline": {"value": v, "unit": METRIC, "cores": 1, "kind": "oracle", "sample": sample},
            "e2e": {"value": v, "unit": METRIC, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


def _given_launch(ctx, spec):
    """Apply a launch configuration given as flux_block,sweep_threads,groups[,sweep_cluster]."""
    v = [int(x) for x in spec.split(",")]
    fb, stt, gr, cl = (v + [1])[:4]
    tuning = dict(sweep_threads=stt, flux_block=fb, sweep_mode=1, sweep_cluster=cl, groups=gr, ms_per_iter=0.0)
    ctx.set_launch(tuning)
    return tuning


def measure(args, mesh, flow, precision, dev, dist, ws, with_e2e):
    """Time args.steps iterations of one solve at one sweep precision."""
    import torch
    from paper_1709_00803_gb300 import igks

    stream = torch.cuda.Stream()
    prec = {"mixed": igks.PREC_MIXED, "df64": igks.PREC_DF64}.get(precision, igks.PREC_FP64)
    ctx = igks.Context(precision=prec, device=dev, stream=stream.cuda_stream, timing=1,
                       sweep_cluster=getattr(args, "sweep_cluster", 0))
    sid = ctx.mesh_upload(mesh)
    ctx.set_flow(sid, flow)
    ctx.init_freestream(sid)
    info = ctx.mesh_info(sid)
    # launch configuration for this solve (autotune restores the state it started from)
    tuning = _given_launch(ctx, args.launch) if args.launch else ctx.autotune(5)
    ctx.enqueue(args.warmup)
    stream.synchronize()
    flush = torch.empty(64 * 1024 * 1024, dtype=torch.float32, device=f"cuda:{dev}")
    starts = [torch.cuda.Event(enable_timing=True) for _ in range(args.steps)]
    ends = [torch.cuda.Event(enable_timing=True) for _ in range(args.steps)]
    ktimes = {}
    if dist:
        dist.barrier()
    torch.cuda.synchronize()
    with ClockSampler(dev) as clk:
        for k in range(args.steps):
            with torch.cuda.stream(stream):
                flush.fill_(float(k))        # evict the solve's working set from L2
            starts[k].record(stream)
            ctx.enqueue(1)
            ends[k].record(stream)
            stream.synchronize()
            for name, t in ctx.kernel_times().items():
                ktimes.setdefault(name, []).append(t)
    torch.cuda.synchronize()
    if dist:
        dist.barrier()
    total_ms = float(sum(s.elapsed_time(e) for s, e in zip(starts, ends)))
    total_ms = _max_over_ranks(dist, total_ms, f"cuda:{dev}")
    _, st = ctx.iterate(0)
    if st[sid]["state"] != 0 or st[sid]["iters"] != args.warmup + args.steps:
        raise RuntimeError(f"the solve stopped during the timed steps: {st[sid]}")
    res = {"value": ws * mesh.n_cells * args.steps / (total_ms / 1e3), "ms_per_step": total_ms / args.steps,
           "kernel_ms": {k: round(statistics.mean(v), 5) for k, v in ktimes.items()},
           "launches_per_step": ctx.launches_per_iteration(), "clocks": clk.summary(), "info": info,
           "levels": (info["levels_fwd"], info["levels_bwd"]), "autotune": tuning,
           "solver_state": {"iters": st[sid]["iters"], "res_l2_rel": st[sid]["res_l2_rel"], "cfl": st[sid]["cfl"]}}
    if with_e2e:
        W_host = torch.empty((5, mesh.n_cells), dtype=torch.float64).pin_memory().numpy()
        ctx.get_fields(sid, out=W_host)
        n_e2e = max(5, min(args.steps, 50))
        if dist:
            dist.barrier()
        t0 = time.perf_counter()
        for _ in range(n_e2e):
            ctx.set_fields(sid, W_host)          # H2D: the step's input state
            ctx.iterate(1)                       # one iteration, per-solve status read back
            ctx.get_fields(sid, out=W_host)      # D2H: the step's result
        e2e_s = time.perf_counter() - t0
        e2e_s = _max_over_ranks(dist, e2e_s, f"cuda:{dev}")
        res["e2e"] = {"value": ws * mesh.n_cells * n_e2e / e2e_s, "unit": METRIC,
                      "h2d_bytes_per_step": int(W_host.nbytes), "d2h_bytes_per_step": int(W_host.nbytes) + 48}
    ctx.destroy()
    return res


def measure_batch(args, cases, precision, dev, dist, ws, with_e2e=False):
    """Time args.steps iterations of many solves in one context (one launch per kernel
    covers every solve); only cells of solves still running count as updated."""
    import torch
    from paper_1709_00803_gb300 import igks

    stream = torch.cuda.Stream()
    prec = igks.PREC_MIXED if precision == "mixed" else igks.PREC_FP64
    ctx = igks.Context(precision=prec, device=dev, stream=stream.cuda_stream, timing=1,
                       sweep_cluster=getattr(args, "sweep_cluster", 0))
    for mesh, flow in cases:
        sid = ctx.mesh_upload(mesh)
        ctx.set_flow(sid, flow)
    for k in range(len(cases)):
        ctx.init_freestream(k)
    ncells = np.array([m.n_cells for m, _ in cases])
    ctx.enqueue(args.warmup)
    stream.synchronize()
    if args.launch:                   # a given launch configuration instead of tuning
        tuning = _given_launch(ctx, args.launch)
    else:
        tuning = ctx.autotune(5)      # launch configuration for this batch (state restored)
    s0, s1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    _, st = ctx.iterate(0)
    it0 = np.array([q["iters"] for q in st])
    live0 = int(ncells[np.array([q["state"] == 0 for q in st])].sum())
    if dist:
        dist.barrier()
    torch.cuda.synchronize()
    # the K steps as one window: the groups of solves run on streams of their own and drift
    # against each other, so that one group's sweeps overlap another's flux; the state and
    # mesh data of a step (2+ GB) are far larger than the 129 MB L2, so nothing is flushed
    with ClockSampler(dev) as clk:
        s0.record(stream)
        ctx.enqueue(args.steps)
        s1.record(stream)
        stream.synchronize()
    total_ms = _max_over_ranks(dist, float(s0.elapsed_time(s1)), f"cuda:{dev}")
    _, st = ctx.iterate(0)
    updates = int((ncells * (np.array([q["iters"] for q in st]) - it0)).sum())
    states = [q["state"] for q in st]
    # the per-kernel split, one group (the kernels one after another), a few more iterations
    ctx.set_launch(dict(tuning, groups=1))
    ktimes = {}
    for _ in range(3):
        ctx.enqueue(1)
        stream.synchronize()
        for name, t in ctx.kernel_times().items():
            ktimes.setdefault(name, []).append(t)
    ctx.set_launch(tuning)
    res = {"value": ws * updates / (total_ms / 1e3), "ms_per_step": total_ms / args.steps,
           "kernel_ms": {k: round(statistics.mean(v), 5) for k, v in ktimes.items()},
           "kernel_ms_note": "one group, the kernels in sequence, 3 iterations after the timed window",
           "launches_per_step": ctx.launches_per_iteration(), "clocks": clk.summary(),
           "solves": len(cases), "running": states.count(0), "converged": states.count(1),
           "diverged": sum(1 for x in states if x < 0), "live_cells_first_last": [live0, int(ncells[np.array([x == 0 for x in states])].sum())],
           "autotune": tuning}
    if with_e2e:
        # every solve's state in from pinned host memory (igks_set_fields_all: one copy per
        # solve, checked on the device), one iteration through the public API (igks_iterate
        # reads the per-solve status back), every state out again (igks_get_fields_all)
        host = torch.empty((5, int(ncells.sum())), dtype=torch.float64).pin_memory().numpy()
        ctx.get_fields_all(out=host)
        n_e2e = max(3, min(args.steps, 10))
        if dist:
            dist.barrier()
        t0 = time.perf_counter()
        for _ in range(n_e2e):
            ctx.set_fields_all(host)
            _, st = ctx.iterate(1)
            ctx.get_fields_all(out=host)
        e2e_s = _max_over_ranks(dist, time.perf_counter() - t0, f"cuda:{dev}")
        nbytes = int(host.nbytes)
        res["e2e"] = {"value": ws * int(ncells.sum()) * n_e2e / e2e_s, "unit": METRIC,
                      "h2d_bytes_per_step": nbytes, "d2h_bytes_per_step": nbytes + 48 * len(cases),
                      "steps": n_e2e}
    ctx.destroy()
    return res


def fp64_peak(clocks):
    """Derived FP64 peak in TFLOP/s: the FP64 units of the 152 SMs at the median SM clock
    sampled during the timed region (the maximum clock if no sample was taken)."""
    mhz = (clocks or {}).get("sm_mhz") or SM_MAX_MHZ
    return SM_COUNT * FP64_FLOP_PER_SM_CLK * mhz * 1e6 / 1e12, mhz


def rooflines(res, mesh, precision, workload, probe_tflops=None):
    """The dominant kernel against the roofline that bounds it. The flux kernel is bound by
    the FP64 pipe: achieved = algorithmic flops (FLUX_ALG_FLOPS_PER_FACE x faces) over its
    CUDA-event time, against the derived FP64 peak at the sampled clock. The other kernels
    against HBM: algorithmic bytes over time, against the measured copy bandwidth."""
    peaks, src = _peaks()
    hbm = float(peaks.get("hbm_gbs", 6800.0))
    t = 4 if precision == "mixed" else 8
    km = res["kernel_ms"]
    ncu = NCU.get(workload, {})
    dom = max(km, key=km.get)
    b = alg_bytes(dom, t, mesh.n_cells, mesh.n_faces)
    ach = b / (km[dom] / 1e3) / 1e9
    per_cell = ncu.get("sweep_dram_bytes_per_cell", {}).get((dom, t))
    dominant = {"bound": "hbm", "kernel": dom, "achieved": ach, "peak": hbm, "unit": "GB/s", "frac": ach / hbm,
                "traffic": per_cell * mesh.n_cells if per_cell else None,
                "peak_source": f"hbm_gbs of MEASURED_PEAKS.json ({src}, burst copy)",
                "alg_bytes_per_launch": b}
    peak, mhz = fp64_peak(res.get("clocks"))
    flux_t = km["k_flux"]
    ach_f = FLUX_ALG_FLOPS_PER_FACE * mesh.n_faces / (flux_t / 1e3) / 1e12
    exe = ncu.get("flux_exec_flops_per_face", {}).get(t)
    dram = ncu.get("flux_dram_bytes_per_face", {}).get(t)
    flux = {"bound": "alu", "kernel": "k_flux", "achieved": ach_f, "peak": peak, "unit": "TFLOP/s",
            "frac": ach_f / peak, "traffic": dram * mesh.n_faces if dram else None,
            "peak_source": f"derived: {SM_COUNT} SMs x 2 FP64 FMA/clk x 2 flop x {mhz:.0f} MHz (median SM clock "
                           f"sampled during the timed region)",
            "alg_flops_per_face": FLUX_ALG_FLOPS_PER_FACE, "faces_per_launch": mesh.n_faces,
            "ms_per_launch": flux_t}
    if probe_tflops:
        flux.update(peak_measured_probe=probe_tflops, frac_of_probe=ach_f / probe_tflops)
    if exe:
        flux.update(executed_flops_per_face=exe, executed_tflops=exe * mesh.n_faces / (flux_t / 1e3) / 1e12,
                    executed_source=ncu["source"])
    if dominant["kernel"] == "k_flux":
        dominant = dict(flux, alg_bytes_per_launch=b, hbm_achieved_gbs=ach, hbm_frac=ach / hbm)
    return dominant, flux


def per_kernel(res, mesh, precision):
    """Every kernel of the iteration against the roofline that bounds it: algorithmic bytes
    (HBM) or FP64 flops (the flux) per launch over its event-timed duration; the sweeps
    also per dependency level (their bound is the depth of the sweep order)."""
    peaks, _ = _peaks()
    hbm = float(peaks.get("hbm_gbs", 6800.0))
    peak, _ = fp64_peak(res.get("clocks"))
    t = 4 if precision == "mixed" else 8
    out = {}
    for k, ms in res["kernel_ms"].items():
        row = {"ms": ms}
        b = alg_bytes(k, t, mesh.n_cells, mesh.n_faces)
        if b:
            row.update(alg_bytes=b, gbs=b / (ms / 1e3) / 1e9, hbm_frac=b / (ms / 1e3) / 1e9 / hbm)
        if k == "k_flux":
            tf = FLUX_ALG_FLOPS_PER_FACE * mesh.n_faces / (ms / 1e3) / 1e12
            row.update(fp64_tflops=tf, fp64_frac=tf / peak)
        lv = res.get("levels")
        if lv and k in ("k_sweep_fwd", "k_sweep_bwd"):
            n = lv[0] if k == "k_sweep_fwd" else lv[1]
            row.update(levels=n, us_per_level=1e3 * ms / n)
        out[k] = row
    return out


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=200)
    ap.add_argument("--warmup", type=int, default=20)
    ap.add_argument("--impl", default="igks", choices=["igks", "reference"])
    ap.add_argument("--precision", default=None, choices=["fp64", "df64", "mixed"],
                    help="headline sweep precision (default: mixed for the batch, fp64 for one solve)")
    ap.add_argument("--workload", default="naca_batch", choices=list(WORKLOADS) + ["naca_batch", "serving", "cavity"])
    ap.add_argument("--explicit-cap", type=int, default=2000000, help="cavity: explicit iterations at most")
    ap.add_argument("--sweep-cluster", type=int, default=0,
                    help="blocks (thread-block cluster) per solve in the sweeps; 0: the library's choice")
    ap.add_argument("--requests", type=int, default=12, help="requests of the serving workload")
    ap.add_argument("--cells-lo", type=int, default=2000)
    ap.add_argument("--cells-hi", type=int, default=12000)
    ap.add_argument("--slots", type=int, default=64, help="serving: live solves at most")
    ap.add_argument("--iters-per-step", type=int, default=100)
    ap.add_argument("--max-iters", type=int, default=20000)
    ap.add_argument("--eq40", type=float, default=3e-8,
                    help="serving: also stop at the paper's Eq. 40 ratio (0: residual 1e-10 only)")
    ap.add_argument("--batch", type=int, default=64, help="solves of the naca_batch workload")
    ap.add_argument("--ordering", default="as_given", choices=["as_given", "multicolor"],
                    help="cell numbering = LU-SGS sweep order (the oracle baseline runs the same)")
    ap.add_argument("--cpu-budget", type=float, default=15.0)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-other", action="store_true", help="skip the other precision / the flat plate")
    ap.add_argument("--no-serving", action="store_true", help="batch: skip the bounded serving leg")
    ap.add_argument("--launch", default="", help="flux_block,sweep_threads,groups[,sweep_cluster] instead of autotune")
    ap.add_argument("--open-loop", type=int, default=1, help="serving: 1 Poisson arrivals after the capacity "
                    "run, 0 latencies of the capacity run")
    ap.add_argument("--plain-sample", type=int, default=0, help="serving: estimate the plain path from this many "
                    "iterations of each request (0: run each to its stop)")
    args = ap.parse_args()
    args.warmup = max(args.warmup, 3)
    if args.workload == "naca_batch":
        if args.impl == "reference":
            return run_reference_batch(args)
        return main_batch(args)
    if args.precision is None:
        args.precision = "fp64"
    if args.workload == "serving":
        return main_serving(args)
    if args.workload == "cavity":
        return main_cavity(args)
    mk, fl_fn, desc = WORKLOADS[args.workload]
    mesh, flow = mk(), fl_fn()
    if args.ordering == "multicolor":
        from paper_1709_00803_gb300 import igks as _ig
        perm, ncol = _ig.order_cells(mesh, _ig.ORDER_MULTICOLOR)
        mesh = mesh.renumbered(perm)
        desc += f", multicolour cell order ({ncol} colours)"
    if args.impl == "reference":
        return run_reference(args, mesh, flow, desc)

    import torch
    dist, rank, ws = _dist()
    dev = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(dev)
    head = measure(args, mesh, flow, args.precision, dev, dist, ws, with_e2e=True)
    other_p = "mixed" if args.precision == "fp64" else "fp64"
    other = None if args.no_other else measure(args, mesh, flow, other_p, dev, dist, ws, with_e2e=False)
    dominant, flux_roof = rooflines(head, mesh, args.precision, args.workload)
    out = {"metric": METRIC, "value": head["value"], "unit": METRIC, "n_gpus": ws, "steps": args.steps,
           "warmup": args.warmup, "ms_per_step": head["ms_per_step"], "higher_is_better": True,
           "scaling": "weak", "vs_baseline": None,
           "dtype": {"fp64": "f64", "df64": "f64 flux/residual/update + double-float (2 x f32) sweeps"}.get(
               args.precision, "f64 flux/residual/update + f32 sweeps"),
           "data": "synthetic",
           "config": {"workload": desc, "cells": mesh.n_cells, "faces": mesh.n_faces,
                      "sweep_levels": [head["info"]["levels_fwd"], head["info"]["levels_bwd"]],
                      "precision": args.precision, "ordering": args.ordering,
                      "parallelism": "replicas" if ws > 1 else "single solve",
                      "l2": "flushed between steps (256 MiB write outside the timed intervals)"},
           "e2e": head["e2e"], "gpu_launches": head["launches_per_step"] * args.steps,
           "kernel_ms": head["kernel_ms"], "roofline": dominant, "roofline_flux": flux_roof,
           "per_kernel": per_kernel(head, mesh, args.precision),
           "clocks": head["clocks"], "solver_state": head["solver_state"], "autotune": head["autotune"]}
    if other:
        out["other"] = {"precision": other_p, "value": other["value"], "ms_per_step": other["ms_per_step"],
                        "kernel_ms": other["kernel_ms"], "clocks": other["clocks"]}
    if rank == 0 and ws == 1 and not args.no_cpu_baseline:
        out["cpu_baseline"] = cpu_baseline(mesh, flow, args.cpu_budget)
        out["cpu_baseline"]["cores_available"] = os.cpu_count()
    if rank == 0:
        print(json.dumps(out), flush=True)
    if dist:
        dist.barrier()
        dist.destroy_process_group()


def batch_cases(n):
    cases = []
    for sp in G.naca_batch_specs(n):
        mesh = G.naca_scaled(sp["m"], sp["p"], sp["t"], sp["cells"], sp["mesh_seed"])
        cases.append((mesh, F.naca_flow(mach=sp["mach"], reynolds=sp["reynolds"], aoa_deg=sp["aoa"])))
    return cases


class _Totals:
    def __init__(self, cases):
        self.n_cells = sum(m.n_cells for m, _ in cases)
        self.n_faces = sum(m.n_faces for m, _ in cases)


def serving_leg(args, dev, n_small=11, budget_s=120.0):
    """A bounded serving run beside the headline: the 64 x 32 laminar flat plate (whose
    oracle solution to density residual 1e-10 is stored) plus n_small seeded requests of
    the serving stream (2k-12k cells, SA, stop at residual 1e-10 or Eq. 40 <= 3e-8), all
    submitted at once to one server (FP32 sweeps, continuous batching). Reports converged
    solves/hour over the makespan, p50/p99 time to converged, and the plate's error
    against the oracle's field."""
    from paper_1709_00803_gb300 import igks
    cases = [(G.laminar_plate(), F.laminar_plate_flow(), None)] + serving_cases(n_small, 2000, 12000, 3e-8)
    srv = igks.Server(precision=igks.PREC_MIXED, max_slots=64, max_cohort=64, iters_per_step=args.iters_per_step,
                      max_iters=args.max_iters, keep_fields=1)
    t0 = srv.now()
    ids = [srv.submit(m, fl, tag=k) for k, (m, fl, _) in enumerate(cases)]
    results, wall0 = {}, time.perf_counter()
    while len(results) < len(cases) and time.perf_counter() - wall0 < budget_s:
        srv.step()
        for r in srv.poll():
            results[r["id"]] = r
    timed_out = len(results) < len(cases)
    lat = sorted(r["t_finish"] - r["t_submit"] for r in results.values() if r["state"] == igks.CONVERGED)
    makespan = (max(r["t_finish"] for r in results.values()) - t0) if results else None
    plate = results.get(ids[0])
    err = None
    gold = os.path.join(ROOT, "tests", "golden", "converged_laminar_plate.npz")
    if plate and plate["state"] == igks.CONVERGED and os.path.exists(gold):
        W = srv.take_fields(ids[0])
        ref = np.load(gold)["W"]
        err = float(np.max(np.linalg.norm(W[:4] - ref[:4], axis=1) / np.linalg.norm(ref[:4], axis=1)))
    srv.destroy()
    conv = len(lat)
    return {"requests": len(cases), "finished": len(results), "converged": conv,
            "solves_per_hour": conv / makespan * 3600.0 if makespan else None, "makespan_s": makespan,
            "p50_s": _pct(lat, 50), "p99_s": _pct(lat, 99), "budget_s": budget_s, "hit_budget": timed_out,
            "laminar_plate_rel_l2_vs_oracle": err,
            "laminar_plate_iters": plate["iters"] if plate else None,
            "stream": f"laminar flat plate 64x32 (residual 1e-10) + {n_small} seeded requests (flat plate or NACA "
                      f"4-digit, SA, 2k-12k cells, residual 1e-10 or Eq. 40 <= 3e-8), all submitted at once, "
                      f"FP32 sweeps, cap {args.max_iters} iterations"}


def cpu_baseline_batch(cases, budget_s=15.0):
    """The oracle as it stands, single-threaded, on a bounded sample of the batch: whole
    iterations of its airfoils in order until budget_s has passed."""
    import oracle as O
    cells, used, dt = 0, 0, 0.0
    for m, fl in cases:
        ora = O.Oracle(m, fl)
        t1 = time.perf_counter()
        ora.iterate(1)
        dt += time.perf_counter() - t1
        cells += m.n_cells
        used += 1
        if dt >= budget_s:
            break
    return {"value": cells / dt, "unit": METRIC, "cores": 1, "kind": "oracle",
            "sample": f"one oracle iteration (from the free stream; set-up not timed) of each of the first {used} "
                      f"airfoils of the batch ({cells} cell-updates), {dt:.1f} s, single-threaded C oracle "
                      f"(-O2 -ffp-contract=off)"}


def main_batch(args):
    """The headline: many uneven airfoil solves in one context (FP32 sweeps by default),
    with the turbulent flat plate and a bounded serving run beside it."""
    import torch
    from paper_1709_00803_gb300 import igks
    dist, rank, ws = _dist()
    dev = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(dev)
    cases = batch_cases(args.batch)
    tot = _Totals(cases)
    precision = args.precision or "mixed"
    probe = igks.fp64_probe(dev)
    head = measure_batch(args, cases, precision, dev, dist, ws, with_e2e=True)
    dominant, flux_roof = rooflines(head, tot, precision, "naca_batch", probe)
    desc = (f"{len(cases)} seeded NACA 4-digit airfoils (m 0-0.06, p 0.2-0.6, t 0.08-0.18), Ma 0.1-0.75, "
            f"AoA -4..8 deg, Re_c 1e6-1e7, SA, hybrid O-meshes of 8k-80k cells in one context")
    out = {"metric": METRIC, "value": head["value"], "unit": METRIC, "n_gpus": ws, "steps": args.steps,
           "warmup": args.warmup, "ms_per_step": head["ms_per_step"], "higher_is_better": True,
           "scaling": "weak", "vs_baseline": None,
           "dtype": {"fp64": "f64", "df64": "f64 flux/residual/update + double-float (2 x f32) sweeps"}.get(
               precision, "f64 flux/residual/update + f32 sweeps"),
           "data": "synthetic",
           "config": {"workload": desc, "solves": len(cases), "cells": tot.n_cells, "faces": tot.n_faces,
                      "precision": precision, "parallelism": "replicas" if ws > 1 else "one context, all solves",
                      "l2": "not flushed: the state and mesh data of a step (%.1f GB) exceed the 129 MB L2"
                            % (sum(igks.footprint_bytes(m) for m, _ in cases) / 1e9),
                      "timing": "one window of --steps iterations between CUDA events on the library stream"},
           "e2e": head["e2e"], "gpu_launches": head["launches_per_step"] * args.steps,
           "kernel_ms": head["kernel_ms"], "roofline": dominant, "roofline_flux": flux_roof,
           "clocks": head["clocks"], "per_kernel": per_kernel(head, tot, precision),
           "batch": {k: head[k] for k in ("solves", "running", "converged", "diverged", "live_cells_first_last",
                                          "autotune")}}
    if not args.no_other:
        # the turbulent flat plate, one solve, both sweep precisions
        mesh, flow = G.turbulent_plate(), F.turbulent_plate_flow()
        plate = {}
        for prec in ("fp64", "df64", "mixed"):
            r = measure(args, mesh, flow, prec, dev, dist, ws, with_e2e=False)
            plate[prec] = {"value": r["value"], "ms_per_step": r["ms_per_step"], "kernel_ms": r["kernel_ms"],
                           "sweep_levels": list(r["levels"]), "clocks": r["clocks"], "autotune": r["autotune"]}
        out["turbulent_plate"] = dict(plate, workload=WORKLOADS["turbulent_plate"][2], cells=mesh.n_cells,
                                      faces=mesh.n_faces)
    if not args.no_serving and ws == 1:
        out["serving"] = serving_leg(args, dev)
    if rank == 0 and ws == 1 and not args.no_cpu_baseline:
        out["cpu_baseline"] = cpu_baseline_batch(cases, args.cpu_budget)
        out["cpu_baseline"]["cores_available"] = os.cpu_count()
    if rank == 0:
        print(json.dumps(out), flush=True)
    if dist:
        dist.barrier()
        dist.destroy_process_group()


def serving_cases(n, cells_lo, cells_hi, eq40_target):
    """The serving request stream: seeded flat plates and NACA sections (SA), flow and size
    drawn per request; each flow stops at res_target (1e-10) or, when eq40_target > 0, at
    the paper's Eq. 40 criterion, whichever comes first."""
    cases = []
    for sp in G.serving_specs(n, 5, cells_lo, cells_hi):
        if sp["kind"] == "plate":
            mesh = G.plate_scaled(sp["cells"], sp["mesh_seed"])
            fl = F.turbulent_plate_flow()
            fl.mach, fl.reynolds = sp["mach"], sp["reynolds"]
        else:
            mesh = G.naca_scaled(sp["m"], sp["p"], sp["t"], sp["cells"], sp["mesh_seed"])
            fl = F.naca_flow(mach=sp["mach"], reynolds=sp["reynolds"], aoa_deg=sp["aoa"])
        fl.eq40_target = eq40_target
        cases.append((mesh, fl, sp))
    return cases


def _pct(xs, q):
    return float(np.percentile(np.asarray(xs, dtype=np.float64), q)) if len(xs) else None


def _serve(igks, cases, args, arrivals=None):
    """Run the request stream through one server (mixed precision). arrivals=None submits
    everything at once (capacity); otherwise request k is submitted once the server clock
    passes arrivals[k]. Returns the results and the makespan."""
    srv = igks.Server(precision=igks.PREC_MIXED, max_slots=args.slots, max_cohort=args.slots,
                      iters_per_step=args.iters_per_step, max_iters=args.max_iters, keep_fields=0)
    n = len(cases)
    start = srv.now()
    nxt, results = 0, []
    if arrivals is None:
        for k, (m, fl, _) in enumerate(cases):
            srv.submit(m, fl, tag=k)
        nxt = n
    while len(results) < n:
        now = srv.now() - start
        while nxt < n and arrivals[nxt] <= now:
            srv.submit(cases[nxt][0], cases[nxt][1], tag=nxt)
            nxt += 1
        st = srv.status()
        if st["live"] + st["queued"] == 0:
            time.sleep(max(0.0, min(0.05, arrivals[nxt] - now)))
            continue
        srv.step()
        results += srv.poll()
    srv.destroy()
    for r in results:
        r["t_arrival"] = (arrivals[r["tag"]] if arrivals is not None else 0.0) + start
    return results, max(r["t_finish"] for r in results) - start


def _plain(igks, cases, args, served=None):
    """The plain path: each request alone, FP64 sweeps, one after the other. With
    --plain-sample N each request runs only N iterations alone, and its service time is
    estimated as the iterations its served solve took times the measured time per plain
    iteration (plus the set-up measured); its outcome is taken from the served solve."""
    out = []
    for k, (m, fl, _) in enumerate(cases):
        t = time.perf_counter()
        ctx = igks.Context(precision=igks.PREC_FP64, check_every=100)
        sid = ctx.mesh_upload(m); ctx.set_flow(sid, fl); ctx.init_freestream(sid)
        if args.plain_sample > 0 and served is not None:
            ctx.iterate(1)
            t1 = time.perf_counter()
            ctx.iterate(args.plain_sample)
            per = (time.perf_counter() - t1) / args.plain_sample
            setup = t1 - t
            r = served[k]
            out.append(dict(service=setup + per * r["iters"], state=r["state"], iters=r["iters"], estimated=True,
                            ms_per_iteration=1e3 * per))
        else:
            rc, st = ctx.iterate(args.max_iters)
            out.append(dict(service=time.perf_counter() - t, state=st[sid]["state"], iters=st[sid]["iters"]))
        ctx.destroy()
    return out


def main_serving(args):
    """Continuous batching of a Poisson stream of steady solves against the plain
    one-solve-at-a-time FP64 path on the same GPU."""
    import torch
    from paper_1709_00803_gb300 import igks
    dist, rank, ws = _dist()
    dev = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(dev)
    all_cases = serving_cases(args.requests, args.cells_lo, args.cells_hi, args.eq40)
    cases = all_cases[rank::ws]          # replicas: each rank serves its share of the stream
    conv = lambda st: st == igks.CONVERGED
    # capacity: everything submitted at once
    with ClockSampler(dev) as clk:
        res_cap, T_cap = _serve(igks, cases, args)
    n_conv = sum(conv(r["state"]) for r in res_cap)
    cap_per_s = len(res_cap) / T_cap
    # progress on stderr: the capacity run alone, in case a later phase is cut short
    print(json.dumps({"phase": "capacity", "requests": len(res_cap), "converged": n_conv, "makespan_s": T_cap,
                      "solves_per_hour": n_conv / T_cap * 3600.0,
                      "iterations": [r["iters"] for r in res_cap], "states": [r["state"] for r in res_cap],
                      "cells": [m.n_cells for m, _, _ in cases]}), file=sys.stderr, flush=True)
    # open loop: Poisson arrivals at 0.8 x the measured capacity
    gaps = np.array([sp["gap"] for _, _, sp in cases])
    arrivals = np.cumsum(gaps) / (0.8 * cap_per_s) if args.open_loop else np.zeros(len(cases))
    if args.open_loop:
        res_open, T_open = _serve(igks, cases, args, arrivals)
    else:                              # latencies of the all-at-once run (a heavier load)
        res_open, T_open = res_cap, T_cap
        for r in res_open:
            r["t_arrival"] = r["t_submit"]
    lat = [r["t_finish"] - r["t_arrival"] for r in res_open if conv(r["state"])]
    # plain FP64, one at a time; its latency under the same arrivals follows from its
    # service times (one FIFO server)
    by_tag = {r["tag"]: r for r in res_cap}
    plain = _plain(igks, cases, args, served=[by_tag[k] for k in range(len(cases))])
    fin, lat_plain = 0.0, []
    for a, p in zip(arrivals, plain):
        fin = max(fin, a) + p["service"]
        if conv(p["state"]):
            lat_plain.append(fin - a)
    T_plain = sum(p["service"] for p in plain)
    n_plain = sum(conv(p["state"]) for p in plain)
    loc = dict(n=len(cases), conv=n_conv, T_cap=T_cap, lat=lat, conv_plain=n_plain, T_plain=T_plain,
               lat_plain=lat_plain, cells=sum(m.n_cells for m, _, _ in cases),
               iters=[r["iters"] for r in res_cap], states=[r["state"] for r in res_cap],
               clocks=clk.summary())
    parts = [loc]
    if dist:
        parts = [None] * ws
        dist.all_gather_object(parts, loc)
    T = max(p["T_cap"] for p in parts)
    served = sum(p["conv"] for p in parts) / T * 3600.0
    plain_rate = sum(p["conv_plain"] for p in parts) / max(p["T_plain"] for p in parts) * 3600.0
    lat_all = sum((p["lat"] for p in parts), [])
    latp_all = sum((p["lat_plain"] for p in parts), [])
    stop = "density residual 1e-10" + (f" or Eq. 40 ratio <= {args.eq40:g}" if args.eq40 > 0 else "")
    out = {"metric": "converged solves/hour", "value": served, "unit": "solves/hour", "n_gpus": ws,
           "steps": None, "warmup": 0, "ms_per_step": None, "higher_is_better": True, "scaling": "weak",
           "vs_baseline": None, "dtype": "f64 flux/residual/update + f32 sweeps", "data": "synthetic",
           "config": {"workload": f"{args.requests} seeded requests (flat plate or NACA 4-digit, SA; cells "
                                  f"log-uniform {args.cells_lo}-{args.cells_hi}; Ma 0.1-0.75, AoA -4..8, "
                                  f"Re 1e6-1e7), stop at {stop}, cap {args.max_iters} iterations",
                      "slots": args.slots, "iters_per_step": args.iters_per_step,
                      "latency": "Poisson arrivals at 0.8 x the measured capacity" if args.open_loop else
                                 "all requests submitted at once (the capacity run)",
                      "plain": (f"estimated: {args.plain_sample} plain FP64 iterations of each request alone "
                                f"timed, times the iterations of its served solve") if args.plain_sample > 0 else
                               "each request run alone to its stop"},
           "served": {"solves_per_hour": served, "converged": sum(p["conv"] for p in parts),
                      "requests": sum(p["n"] for p in parts), "makespan_s": T,
                      "p50_s": _pct(lat_all, 50), "p99_s": _pct(lat_all, 99),
                      "arrival_rate_per_s": 0.8 * sum(p["n"] for p in parts) / T},
           "plain_fp64_one_at_a_time": {"solves_per_hour": plain_rate,
                                        "converged": sum(p["conv_plain"] for p in parts),
                                        "busy_s": max(p["T_plain"] for p in parts),
                                        "p50_s": _pct(latp_all, 50), "p99_s": _pct(latp_all, 99)},
           "served_over_plain": served / plain_rate if plain_rate > 0 else None,
           "iterations": sum((p["iters"] for p in parts), []), "states": sum((p["states"] for p in parts), []),
           "clocks": parts[0]["clocks"]}
    if rank == 0:
        print(json.dumps(out), flush=True)
    if dist:
        dist.barrier()
        dist.destroy_process_group()

def main_cavity(args):
    """The paper's cavity (Re 1000, 100 x 100): implicit and explicit scheme from rest on the
    same kernels, each run until the primary vortex's stream function is within 0.1% of its
    settled value (the implicit solution after 40000 iterations), with the iterations and
    device time of each (the comparison of Table 2), and the settled vortex centres against
    Table 1. With the paper's adiabatic walls the lid's work keeps heating the fluid, so the
    conserved state drifts slowly and neither the Eq. 40 ratio nor the density residual is
    a fair stopping rule for the comparison; the velocity field does settle."""
    import torch
    from paper_1709_00803_gb300 import igks
    from paper_1709_00803_gb300 import postproc as P
    dist, rank, ws = _dist()
    dev = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(dev)
    n = 100
    m = G.cavity(n)

    def start(scheme):
        fl = F.cavity_flow(scheme=scheme)
        ctx = igks.Context(precision=1 if scheme == 0 else 0, check_every=10 ** 6)
        sid = ctx.mesh_upload(m); ctx.set_flow(sid, fl); ctx.init_freestream(sid)
        ctx.set_fields(sid, F.rest_state(m, fl))
        return ctx, sid

    with ClockSampler(dev) as clk:
        ctx, sid = start(0)
        ctx.iterate(40000)
        ref = P.cavity_vortices(ctx.get_fields(sid), n)
        _, st = ctx.iterate(0)
        settled = dict(eq40=st[sid]["eq40_ratio"], res_l2_rel=st[sid]["res_l2_rel"])
        ctx.destroy()
        psi_ref = ref["primary"]["psi"]
        runs = {}
        for name, scheme, every, cap in (("implicit", 0, 100, 40000), ("explicit", 1, 5000, args.explicit_cap)):
            ctx, sid = start(scheme)
            done, t_dev, hit = 0, 0.0, False
            while done < cap:
                torch.cuda.synchronize()
                t0 = time.perf_counter()
                ctx.iterate(every)
                t_dev += time.perf_counter() - t0
                done += every
                psi = P.cavity_vortices(ctx.get_fields(sid), n)["primary"]["psi"]
                if abs(psi - psi_ref) <= 1e-3 * abs(psi_ref):
                    hit = True
                    break
            runs[name] = dict(iterations=done, seconds=t_dev, reached=hit, psi=psi,
                              ms_per_iteration=1e3 * t_dev / done)
            ctx.destroy()
    ok = runs["explicit"]["reached"] and runs["implicit"]["reached"]
    out = {"metric": "cavity: explicit / implicit time to the settled primary vortex (0.1%)", "unit": "ratio",
           "value": runs["explicit"]["seconds"] / runs["implicit"]["seconds"] if ok else None,
           "n_gpus": 1, "higher_is_better": True, "data": "synthetic",
           "config": {"workload": "lid-driven cavity, Re 1000, Ma 0.1 sqrt(3), 100 x 100 uniform quads, from rest",
                      "stop": "primary-vortex stream function within 0.1% of the implicit solution after 40000 "
                              "iterations (checked every 100 implicit / 5000 explicit iterations)"},
           "implicit": runs["implicit"], "explicit": runs["explicit"],
           "iteration_ratio": runs["explicit"]["iterations"] / runs["implicit"]["iterations"] if ok else None,
           "paper_table2": {"explicit_iterations": 608000, "implicit_iterations": 4430, "speedup": 64.1},
           "settled": dict(settled, vortices=ref), "paper_table1_igks": {
               "primary": {"omega": 2.0861, "psi": -0.1178, "x": 0.5335, "y": 0.5681},
               "left": {"psi": 2.2461e-4, "x": 0.0820, "y": 0.0716}, "right": {"psi": 1.7123e-3, "x": 0.8720, "y": 0.1132}},
           "clocks": clk.summary()}
    if rank == 0:
        print(json.dumps(out), flush=True)

if __name__ == "__main__":
    main()
