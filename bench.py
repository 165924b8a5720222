#!/usr/bin/env python
"""Benchmark of the five-equation RHS hot path (WENO5-JS + HLLC + SSP-RK3).

Metric: grind time, ns per (cell x equation x RHS evaluation), lower is better,
and the fraction of the HBM roofline it reaches, for the FP64 form (reference
operation order, bit-identical to the oracle; the headline value), the
FP64-fast selection (the same kernels), the mixed-precision form (512^3) and
the MLP-gated form (256^3, trained weights from paper_2409_10729_gb300/gate_weights.npy),
plus the third-order reconstruction option (WENO3-JS) and a tanh-refined
(non-uniform) grid in the FP64 (256^3) and mixed (512^3) forms, and a
three-fluid droplet case (256^3, 9 equations) in both.

Workload (per GPU): the 3-D shock / droplet array, 256^3 cells, 7 equations,
FP64, SSP-RK3 at CFL 0.4 (the timed "step" is one RK3 step = 3 RHS
evaluations).  The mixed form runs the same setup at 512^3.  Inputs are
seeded synthetic states generated by paper_2409_10729_gb300.inputs.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]

Under torchrun each rank runs its own replica (weak scaling, no collective in
the data path); rank 0 prints one JSON line.  `--impl reference` times the
serial CPU oracle on the host cores (rank 0 only).
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

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "grind time ns/(cell·eq·RHS) & % HBM roofline: FP64 vs mixed vs MLP-gated"
UNIT = "ns/(cell*eq*RHS)"
CFL = 0.4

# Algorithmic work per cell and direction of one sweep, counted from the
# oracle's formulas (every +, -, *, /, sqrt and Davis min/max counts 1), for
# nf fluids in ndim dimensions (neq = 2 nf + ndim):
#   cons->prim   6 nf + 3 ndim + 1        (two fluids, 3-D: 22)
#   WENO5-JS     107 per field (beta 33, two faces x 37); WENO3-JS 38
#   HLLC         19 nf + 12 ndim + 48 per face, star region (122)
#   divergence   2 neq + 4 (nf - 1) with the volume-fraction terms (18)
# The last sweep adds the accumulation (neq), the stage update (4 per field,
# mean over the three stages) and a third of the wave speed (cons->prim + 23,
# once per step).
WENO_FLOPS = {5: 107, 3: 38}


def flops_cell_dir(nf=2, ndim=3, order=5):
    neq = 2 * nf + ndim
    return (6 * nf + 3 * ndim + 1) + WENO_FLOPS[order] * neq + (19 * nf + 12 * ndim + 48) + \
        (2 * neq + 4 * (nf - 1))


def flops_last_sweep_extra(nf=2, ndim=3):
    neq = 2 * nf + ndim
    return neq + 4 * neq + ((6 * nf + 3 * ndim + 1) + 23) / 3.0


FLOPS_CELL_DIR_3D = flops_cell_dir()                   # 911
FLOPS_CELL_DIR_3D_WENO3 = flops_cell_dir(order=3)      # 428
# Algorithmic bytes per cell, equation and RHS: stage 1 reads q^n and writes
# q^(1); stages 2-3 read q^(k) and q^n and write q^(k+1): 8/3 state arrays.
ALG_BYTES = {"fp64": 8.0 / 3.0 * 8.0, "fp64_fast": 8.0 / 3.0 * 8.0, "mixed": (12.0 + 16.0 + 20.0) / 3.0,
             "gated": (12.0 + 16.0 + 20.0) / 3.0}


def max_over_ranks(value: float, world: int) -> float:
    """The largest of the ranks' values (the slowest rank's time); the
    process group's own device (CUDA under NCCL, CPU under gloo)."""
    if world == 1:
        return float(value)
    import torch
    import torch.distributed as dist
    dev = "cuda" if dist.get_backend() == "nccl" else "cpu"
    t = torch.tensor([float(value)], dtype=torch.float64, device=dev)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def aggregate_grind(seconds: float, steps: int, ncell: int, neq: int, world: int) -> float:
    """Whole-job grind time in ns per (cell x equation x RHS evaluation): the
    slowest rank's time over the cells of all ranks (each rank runs its own
    replica: weak scaling), 3 RHS evaluations per SSP-RK3 step."""
    return seconds * 1e9 / (steps * 3 * ncell * neq * world)


def dist_env():
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return rank, world, local


def measured_peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(path) as f:
            d = json.load(f)
        return float(d["hbm_gbs"]), "measured"
    except Exception:
        return 6800.0, "fallback"


class ClockSampler:
    """nvidia-smi clock/throttle samples while the timed region runs."""

    FIELDS = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.hw_slowdown,"
              "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
              "clocks_event_reasons.sw_power_cap")

    def __init__(self, device_index: int):
        self.proc = None
        self.out_path = os.path.join("/tmp", f"mfc5_clocks_{os.getpid()}.csv")
        try:
            self.fh = open(self.out_path, "w")
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(device_index), f"--query-gpu={self.FIELDS}",
                 "--format=csv,noheader,nounits", "-lms", "200"], stdout=self.fh, stderr=subprocess.DEVNULL)
        except Exception:
            self.proc = None

    def stop(self):
        if self.proc is None:
            return None
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        self.fh.close()
        with open(self.out_path) as f:
            out = parse_clock_samples(f)
        os.unlink(self.out_path)
        return out


def parse_clock_samples(lines):
    """Median SM clock, the largest max clock and the active throttle reasons
    of nvidia-smi samples (csv, noheader, nounits, fields as ClockSampler
    queries them); None without a usable sample."""
    sm, smax, reasons = [], [], set()
    names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
    for line in lines:
        parts = [x.strip() for x in line.split(",")]
        if len(parts) < 7:
            continue
        try:
            sm.append(float(parts[0]))
            smax.append(float(parts[1]))
        except ValueError:
            continue
        for nm, v in zip(names, parts[3:7]):
            if v.lower().startswith("active"):
                reasons.add(nm)
    if not sm:
        return None
    return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(smax), "reasons": sorted(reasons),
            "samples": len(sm)}


def read_traffic(kernel: str):
    """DRAM bytes per launch of `kernel` from the committed ncu summary, if it
    was taken on the current kernel source (else None)."""
    import hashlib
    path = os.path.join(ROOT, "profiles", "traffic.txt")
    src = b""
    for f in ("sweep.cuh", "tile.cuh", "physics.cuh", "physics_exact.cuh", "mfc_internal.cuh"):
        with open(os.path.join(ROOT, "paper_2409_10729_gb300", "csrc", f), "rb") as fh:
            src += fh.read()
    sha = hashlib.sha256(src).hexdigest()[:16]
    try:
        with open(path) as fh:
            for line in fh:
                parts = line.split()
                if len(parts) >= 3 and parts[0] == kernel and parts[2] == sha:
                    return float(parts[1])
    except OSError:
        pass
    return None


def pipe_busy(form, name):
    """Busy fraction of the FP64 (FP64 forms) or FP32 FMA (FP32 forms) pipe of
    the dominant kernel, from the committed ncu summary of the same kernel
    source (None if the kernels changed since)."""
    pipe = "fp64" if form.startswith("fp64") else "fma"
    v = read_traffic(f"{form}:{name}:pipe_{pipe}")
    return None if v is None else {"pipe": pipe, "frac": v, "source": "ncu sm__inst_executed_pipe_" + pipe +
                                   " at 160^3, profiles/traffic.txt"}


def stretched(p):
    """The same case on a grid refined with a hyperbolic tangent about the
    domain centre in every direction (Sec. III-A): cells there half as wide."""
    from paper_2409_10729_gb300 import inputs as I
    return dict(p, edges=[I.tanh_edges(p["n"][d], p["lo"][d], p["hi"][d], 0.5 * (p["lo"][d] + p["hi"][d]),
                                       strength=8.0, refine=0.5) if d < p["ndim"] else None for d in range(3)])


def gate_weights():
    import numpy as np
    return np.load(os.path.join(ROOT, "paper_2409_10729_gb300", "gate_weights.npy"))


def split_steps(steps: int, regions: int = 5):
    """K timed steps as up to `regions` consecutive regions of nearly equal
    length (every region at least one step)."""
    r = max(1, min(regions, steps))
    base, extra = divmod(steps, r)
    return [base + (1 if i < extra else 0) for i in range(r)]


def time_form(form, p, w, steps, warmup, device_index, rank, world, kernel_steps=3):
    """Run `warmup` + `steps` RK3 steps of one form, replaying the captured
    step graph exactly as the product does, timed with CUDA events on the
    context's stream as consecutive regions (median per-step time over the
    regions next to the total); then a separate, shorter pass with per-kernel
    events (direct launches) for the kernel split.  Returns a result dict."""
    import torch
    from paper_2409_10729_gb300 import mfc
    s = mfc.Solver(p, form)
    if form == "gated":
        s.set_mlp_weights(gate_weights())
    s.set_state_prim(w)
    s.step_rk3(CFL, warmup)
    torch.cuda.synchronize()
    if world > 1:
        torch.distributed.barrier()
    sampler = ClockSampler(device_index)
    stream = torch.cuda.current_stream()
    parts = split_steps(steps)
    evs = [torch.cuda.Event(enable_timing=True) for _ in range(len(parts) + 1)]
    t_adv = 0.0
    evs[0].record(stream)
    for i, k in enumerate(parts):
        t_adv += s.step_rk3(CFL, k)
        evs[i + 1].record(stream)
    torch.cuda.synchronize()
    clocks = sampler.stop()
    region_ms = [evs[i].elapsed_time(evs[i + 1]) for i in range(len(parts))]
    ms = max_over_ranks(evs[0].elapsed_time(evs[-1]), world)
    per_step = sorted(r / k for r, k in zip(region_ms, parts))
    median_step_ms = max_over_ranks(statistics.median(per_step), world)
    if world > 1:
        torch.distributed.barrier()
    gate = (*s.gate_stats(), s.gate_flat()) if form == "gated" else None
    launches = s.launches_per_step() * steps
    # per-kernel split: direct launches bracketed by per-kernel events
    ks = max(1, min(kernel_steps, steps))
    s.set_timing(True)
    s.step_rk3(CFL, ks)
    kt = s.kernel_times()
    launches += s.launches_per_step() * ks
    s.set_timing(False)
    ncell = p["n"][0] * p["n"][1] * p["n"][2]
    neq = 2 * len(p["gamma"]) + p["ndim"]
    grind = aggregate_grind(ms * 1e-3, steps, ncell, neq, world)
    grind_median = aggregate_grind(median_step_ms * 1e-3, 1, ncell, neq, world)
    s.close()
    del s
    torch.cuda.empty_cache()
    return {"ms": ms, "grind": grind, "grind_median": grind_median, "median_step_ms": median_step_ms,
            "region_steps": parts, "region_ms": region_ms, "kernels": kt, "kernel_steps": ks,
            "launches": launches, "clocks": clocks, "t_advanced": t_adv, "ncell": ncell, "neq": neq,
            "steps": steps, "gate": gate}


def roofline_for(form, res, peak_alu, alu_src, hbm_peak, hbm_src):
    """Roofline object for the dominant kernel of one form.

    FP64 forms: algorithmic +, -, *, /, sqrt per second beside the FMA-chain
    probe's rate.  About half of those operations (quotients, square roots,
    WENO's products) are formed on the integer pipes, so their ratio to the
    FP64 pipe's rate bounds nothing: pipe_roofline states what does.  FP32
    forms: TFLOP/s against the FP32 probe at 2 flops per FMA."""
    kt = res["kernels"]
    base = form.replace("_weno3", "").replace("_stretched", "").replace("_3fluid", "")
    name = max((k for k in kt if kt[k][1] > 0), key=lambda k: kt[k][0])
    total_ms, count = kt[name]
    avg_s = total_ms / count * 1e-3
    ncell = res["ncell"]
    nf, neq = (res["neq"] - 3) // 2, res["neq"]
    flops = flops_cell_dir(nf, 3, 3 if form.endswith("_weno3") else 5)
    if name == "sweep_y":
        flops += neq
    if name == "sweep_z":   # with the stage update, unless that is a kernel of its own
        flops += neq if kt.get("stage_update", (0, 0))[1] else flops_last_sweep_extra(nf, 3)
    achieved = flops * ncell / avg_s / 1e12
    share = total_ms / sum(v[0] for v in kt.values())
    if base == "fp64":   # the reference-order form (no FMA contraction)
        peak, unit = peak_alu / 2.0, "Top/s"
        src = (f"{alu_src}: {peak_alu:.3f} TFLOP/s = {peak_alu / 2:.3f} T FP64 FMA instructions/s; one algorithmic "
               "operation (+, -, *, /, sqrt, min/max) per FP64 instruction slot; those formed on the integer "
               "pipes take none, so the fraction can pass 1")
    else:
        peak, unit = peak_alu, "TFLOP/s"
        src = f"{alu_src} ({'FP64' if base == 'fp64_fast' else 'FP32'}, 2 flops per FMA)"
    return {"bound": "alu", "kernel": name, "achieved": round(achieved, 4), "peak": round(peak, 4),
            "unit": unit, "frac": round(achieved / peak, 4), "peak_source": src,
            "traffic": read_traffic(f"{form}:{name}") if form == base else None, "share_of_step": round(share, 3),
            "avg_launch_ms": round(total_ms / count, 4),
            "algorithmic_flops_per_cell": flops,
            "pipe_busy_ncu": pipe_busy(form, name) if form == base else None,
            "hbm": {"achieved_gbs": round(ALG_BYTES[base] / res["grind"], 1), "peak": hbm_peak,
                    "frac": round(ALG_BYTES[base] / res["grind"] / hbm_peak, 4), "peak_source": hbm_src}}


def pipe_roofline(form, roof, fp64_peak):
    """The roofline as printed.  FP64 forms, which both run the same kernels, are
    bound by the FP64 pipe, whose rate is the FMA-chain probe's FMA instructions
    per second (its TFLOP/s over 2): frac is the pipe's busy fraction that ncu
    counted on the same kernel source (None where it has no figure), achieved the
    instruction rate that this means, and the algorithmic operations per second,
    integer pipes included, are a figure by themselves."""
    if not form.startswith("fp64"):
        return roof
    busy = pipe_busy("fp64", roof["kernel"]) if form in ("fp64", "fp64_fast") else None
    frac = busy["frac"] if busy else None
    peak = fp64_peak / 2.0
    return dict(roof, unit="T FP64 instructions/s", peak=round(peak, 4), frac=frac,
                achieved=None if frac is None else round(frac * peak, 4), pipe_busy_ncu=busy,
                algorithmic_tops=roof["achieved"],
                peak_source=f"measured FMA-chain probe: {fp64_peak:.3f} TFLOP/s at 2 flops per FMA instruction")


def host_info():
    """Core count and CPU model of this host (nproc, lscpu)."""
    info = {"nproc": os.cpu_count() or 1, "model": None}
    try:
        out = subprocess.run(["lscpu"], capture_output=True, text=True, timeout=10).stdout
        for line in out.splitlines():
            k, _, v = line.partition(":")
            if k.strip() in ("Model name", "Model"):
                if info["model"] is None or k.strip() == "Model name":
                    info["model"] = v.strip()
    except Exception:
        pass
    if info["model"] is None:
        try:
            with open("/proc/cpuinfo") as fh:
                for line in fh:
                    if line.lower().startswith(("model name", "cpu part")):
                        info["model"] = line.partition(":")[2].strip()
                        break
        except OSError:
            pass
    try:
        info["nproc"] = len(os.sched_getaffinity(0))
    except Exception:
        pass
    return info


def baseline_entry(grind: float, sample: str):
    """cpu_baseline object: the serial oracle's grind on one core, the host,
    and the ideal-scaling figure (single-core grind / nproc)."""
    h = host_info()
    return {"value": round(grind, 4), "unit": UNIT, "cores": 1, "kind": "oracle", "sample": sample,
            "host": {"nproc": h["nproc"], "cpu_model": h["model"]},
            "ideal_scaling_all_cores": {"value": round(grind / h["nproc"], 4), "unit": UNIT,
                                        "cores": h["nproc"],
                                        "note": "single-core grind / nproc (ideal scaling), not measured"}}


def headline_config(ncell=256 ** 3, neq=7, n_gpus=1):
    """The workload the headline value is quoted on (both arms print it)."""
    return {"workload": "3-D shock-droplet array, 256^3 cells, 7 equations, FP64, SSP-RK3 at CFL 0.4 "
                        "(step = one RK3 step = 3 RHS evaluations)",
            "cells": ncell, "neq": neq, "precision": "fp64", "parallelism": f"replicas x{n_gpus}",
            "l2": "no flush: each state array is 0.94 GB (7 fields x 256^3 x 8 B) > 129 MB L2"}


def cpu_baseline(target_s=15.0):
    """The oracle, as it stands, on a z-slab of the 256^3 shock-droplet state:
    one RHS evaluation per sample, sized to about target_s seconds."""
    import numpy as np
    import oracle as O
    from paper_2409_10729_gb300 import inputs as I
    p, w = I.shock_droplets(256)
    z0 = 96
    q_all = None

    def sample(k):
        ps = dict(p)
        ps["n"] = [256, 256, k]
        ps["lo"] = [0.0, 0.0, z0 / 256.0]
        ps["hi"] = [1.0, 1.0, (z0 + k) / 256.0]
        ws = np.ascontiguousarray(w[:, z0:z0 + k])
        q = O.prim_to_cons(ps, ws)
        t0 = time.perf_counter()
        O.rhs(ps, q)
        return time.perf_counter() - t0, ps

    t1, _ = sample(2)
    k = max(2, min(160, int(target_s / max(t1 / 2, 1e-6))))
    t, ps = sample(k)
    ncell = 256 * 256 * k
    grind = t * 1e9 / (ncell * 7)
    return baseline_entry(grind, f"one oracle RHS on a 256x256x{k} z-slab (z from {z0}) of the 256^3 "
                                 f"shock-droplet initial state, {t:.1f} s"), t, k


def run_reference(args):
    rank, world, local = dist_env()
    if rank != 0:
        return
    import oracle as O
    O.build()
    # size each step so the whole run stays within ~3 minutes
    per_step = max(2.0, min(20.0, 150.0 / max(1, args.steps + args.warmup)))
    base, t, k = cpu_baseline(per_step)
    import numpy as np
    from paper_2409_10729_gb300 import inputs as I
    p, w = I.shock_droplets(256)
    z0 = 96
    ps = dict(p)
    ps["n"] = [256, 256, k]
    ps["lo"] = [0.0, 0.0, z0 / 256.0]
    ps["hi"] = [1.0, 1.0, (z0 + k) / 256.0]
    q = O.prim_to_cons(ps, np.ascontiguousarray(w[:, z0:z0 + k]))
    for _ in range(args.warmup):
        O.rhs(ps, q)
    t0 = time.perf_counter()
    for _ in range(args.steps):
        O.rhs(ps, q)
    el = time.perf_counter() - t0
    grind = el * 1e9 / (args.steps * 256 * 256 * k * 7)
    line = {"metric": METRIC, "value": round(grind, 4), "unit": UNIT, "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": round(el * 1e3 / args.steps, 2),
            "higher_is_better": False, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic", "impl": "reference",
            "config": headline_config(n_gpus=args.gpus),
            "cpu_baseline": baseline_entry(grind, f"each step: one oracle RHS on a 256x256x{k} z-slab (z from "
                                                  f"{z0}) of the 256^3 shock-droplet initial state "
                                                  f"({256 * 256 * k} cells), serial, one core"),
            "e2e": {"value": round(grind, 4), "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


def run_ours(args):
    import numpy as np
    import torch
    rank, world, local = dist_env()
    torch.cuda.set_device(local)
    if world > 1:
        torch.distributed.init_process_group("nccl", device_id=torch.device("cuda", local))
    from paper_2409_10729_gb300 import build as B
    if rank == 0:
        B.build()
    if world > 1:
        torch.distributed.barrier()
    from paper_2409_10729_gb300 import inputs as I
    from paper_2409_10729_gb300 import mfc

    hbm_peak, hbm_src = measured_peaks()
    fp64_peak = mfc.alu_peak(True)
    fp32_peak = mfc.alu_peak(False)

    p, w = I.shock_droplets(256)
    res = time_form("fp64", p, w, args.steps, args.warmup, local, rank, world)
    forms = {"fp64": res}
    forms["fp64_fast"] = time_form("fp64_fast", p, w, args.steps, args.warmup, local, rank, world)
    # the third-order reconstruction option (weno_order = 3), same workload
    forms["fp64_weno3"] = time_form("fp64", dict(p, weno_order=3), w, max(2, args.steps // 2), args.warmup,
                                    local, rank, world)
    # a tanh-refined grid in every direction (cells at the centre half as wide)
    forms["fp64_stretched"] = time_form("fp64", stretched(p), w, max(2, args.steps // 2), args.warmup,
                                        local, rank, world)
    # three fluids: water and oil droplets in air (9 equations)
    p3, w3 = I.shock_droplets_3fluid(256)
    forms["fp64_3fluid"] = time_form("fp64", p3, w3, max(2, args.steps // 2), args.warmup, local, rank, world)
    if not args.no_mixed:
        forms["gated"] = time_form("gated", p, w, args.steps, args.warmup, local, rank, world)
        pm, wm = I.shock_droplets(512)
        forms["mixed"] = time_form("mixed", pm, wm, max(2, args.steps // 2), args.warmup, local, rank, world)
        forms["mixed_weno3"] = time_form("mixed", dict(pm, weno_order=3), wm, max(2, args.steps // 2),
                                         args.warmup, local, rank, world)
        forms["mixed_stretched"] = time_form("mixed", stretched(pm), wm, max(2, args.steps // 2), args.warmup,
                                             local, rank, world)
        forms["mixed_3fluid"] = time_form("mixed", p3, w3, max(2, args.steps // 2), args.warmup, local, rank, world)
        del wm

    # end to end through the C ABI with pinned host buffers: per step, copy
    # q^n in, one RK3 step, copy q^{n+1} out
    s = mfc.Solver(p, "fp64")
    s.set_state_prim(w)
    q_host = torch.empty(s.shape, dtype=torch.float64).pin_memory().numpy()
    q_out = torch.empty(s.shape, dtype=torch.float64).pin_memory().numpy()
    s.get_state(q_host)
    e2e_steps = max(2, min(args.steps, 5))
    s.set_state(q_host)
    s.step_rk3(CFL, 1)
    s.get_state(q_out)
    torch.cuda.synchronize()
    if world > 1:
        torch.distributed.barrier()
    t0 = time.perf_counter()
    for _ in range(e2e_steps):
        s.set_state(q_host)
        s.step_rk3(CFL, 1)
        s.get_state(q_out)
    torch.cuda.synchronize()
    e2e_s = max_over_ranks(time.perf_counter() - t0, world)
    ncell, neq = res["ncell"], res["neq"]
    e2e_grind = aggregate_grind(e2e_s, e2e_steps, ncell, neq, world)
    s.close()

    if rank != 0:
        if world > 1:
            torch.distributed.barrier()
            torch.distributed.destroy_process_group()
        return
    base = None
    if world == 1 and not args.no_cpu_baseline:
        base, _, _ = cpu_baseline()

    roof = pipe_roofline("fp64", roofline_for("fp64", res, fp64_peak, "measured (FP64 FMA-chain probe)", hbm_peak,
                                              hbm_src), fp64_peak)
    out_forms = {}
    for name, r in forms.items():
        peak = fp32_peak if name.startswith(("mixed", "gated")) else fp64_peak
        rf = pipe_roofline(name, roofline_for(name, r, peak, "measured FMA-chain probe", hbm_peak, hbm_src), fp64_peak)
        out_forms[name] = {"grind": round(r["grind"], 5), "grind_median": round(r["grind_median"], 5), "unit": UNIT,
            "ms_per_step": round(r["ms"] / r["steps"], 3),
            "cells": r["ncell"],
            "hbm_frac": rf["hbm"]["frac"], "hbm_gbs_algorithmic": rf["hbm"]["achieved_gbs"],
            "alu_frac": rf["frac"], "algorithmic_tops": rf.get("algorithmic_tops", rf["achieved"]),
            "dominant_kernel": rf["kernel"],
            "kernel_ms": {k: round(v[0] / max(1, v[1]), 4) for k, v in r["kernels"].items() if v[1]},
            "clocks": r["clocks"]}
        if r["gate"]:
            g, f, c, fl = r["gate"]
            out_forms[name]["fraction_gated_linear"] = round(g / max(c, 1), 4)
            out_forms[name]["fraction_fallback"] = round(f / max(c, 1), 4)
            out_forms[name]["fraction_flat_warp_steps"] = round(fl / max(c, 1), 4)
    line = {
        "metric": METRIC, "value": round(res["grind"], 5), "unit": UNIT, "n_gpus": world,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": round(res["ms"] / args.steps, 3),
        "higher_is_better": False, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
        "data": "synthetic",
        "config": headline_config(ncell, neq, world),
        "timing": {"how": "CUDA events on the context stream around replays of the captured step graph "
                          f"(the product path), the {args.steps} steps as {len(res['region_steps'])} consecutive "
                          "regions; value from their total, median_ms_per_step = median over the regions; "
                          "per-kernel split from a separate pass of direct launches with per-kernel events",
                   "region_steps": res["region_steps"], "region_ms": [round(x, 3) for x in res["region_ms"]],
                   "median_ms_per_step": round(res["median_step_ms"], 3),
                   "median_grind": round(res["grind_median"], 5),
                   "kernel_pass_steps": res["kernel_steps"]},
        "roofline": roof,
        "forms": out_forms,
        "e2e": {"value": round(e2e_grind, 5), "unit": UNIT, "h2d_bytes_per_step": ncell * neq * 8,
                "d2h_bytes_per_step": ncell * neq * 8, "steps": e2e_steps,
                "copies": "mfc_set_state / mfc_get_state from page-locked host buffers, copied by the SMs "
                          "through the buffers' device mapping"},
        "gpu_launches": sum(r["launches"] for r in forms.values()),
        "clocks": res["clocks"],
        "cpu_baseline": base,
        "alu_peaks_tflops": {"fp64": round(fp64_peak, 3), "fp32": round(fp32_peak, 2)},
    }
    print(json.dumps(line), flush=True)
    if world > 1:
        torch.distributed.barrier()
        torch.distributed.destroy_process_group()


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--no-mixed", action="store_true", help="skip the mixed-precision form")
    ap.add_argument("--no-cpu-baseline", action="store_true", help="skip the oracle timing")
    args = ap.parse_args()
    if args.warmup < 3:
        args.warmup = 3
    if args.impl == "reference":
        run_reference(args)
    else:
        run_ours(args)


if __name__ == "__main__":
    main()
