"""Throughput benchmark of the fused phonon-LBM stream-collide step.

Workload: 8192 x 8192 fully periodic D2Q8 lattice, sine temperature mode of
wavelength 512 cells plus seeded U[-1e-6, 1e-6) noise, Kn_N = 0.01,
Kn_R = 0.1 measured on the 512-cell wavelength, populations stored as FP32
deviations (``--precision`` selects fp16/bf16/fp64 storage).  One bench
step = one time step of Eq. 13 over the whole lattice (pull-stream, seam and
wall rules, collision); the FP64 residual / energy reduction runs every 100
steps inside the timed region (on the last step of a shorter run), fused
into that step's launch.  The population buffers (2 x 2.1 GB) exceed
the 129 MB L2, so no flush is needed between steps.

Metric: GLUPS (10^9 lattice-site updates per second, whole job).  Also
reported: the roofline of the dominant stream-collide kernel (algorithmic
bytes: one state buffer read and one written per launch, which is one site
update for the single-step kernels and several for the multi-step kernel,
over its mean launch time from the library's CUDA events on the lattice's
stream), an end-to-end figure through the public API with host buffers, the
FP64 oracle on the host cores as a CPU baseline, and (``steady_state``) the
metric's second half: time to steady state (r < 1e-8) of 64 held-out
channels from the cold, the analytic (Eq. 68) and the learned start, with
each end state's error against an FP64 reference (``--no-steady`` skips it;
``--workload warmstart`` runs the full 512-channel study).

Multi-GPU: ``--gpus N`` (under torchrun) runs N independent replicas, one
lattice per rank, with no data-path collective (weak scaling); the job time
is the maximum over ranks.

``--impl reference`` times the FP64 CPU oracle instead (host cores, bounded
sample of the same workload), rank 0 only.
"""
from __future__ import annotations

import argparse
import hashlib
import json
import math
import os
import re
import statistics
import subprocess
import sys
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

from paper_2010_01847_gb300 import inputs  # noqa: E402

RESIDUAL_EVERY = 100
FALLBACK_HBM_GBS = 6800.0
METRIC = "GLUPS & % HBM roofline; time-to-steady-state, warm-started vs plain LBM"
STORAGE_BYTES = {"fp32": 4, "fp16": 2, "bf16": 2, "fp64": 8}
DTYPE = {"fp32": "f32", "fp16": "f32", "bf16": "f32", "fp64": "f64"}


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=2000)
    ap.add_argument("--warmup", type=int, default=20)
    ap.add_argument("--impl", default="native", choices=["native", "reference"])
    ap.add_argument("--precision", default="fp32", choices=list(STORAGE_BYTES))
    ap.add_argument("--kernel", default="auto")
    ap.add_argument("--wave-steps", type=int, default=0,
                    help="multi-step kernel: steps per launch (0 = autotuned or default)")
    ap.add_argument("--wave-rows", type=int, default=0,
                    help="multi-step kernel: rows per segment (0 = autotuned or default)")
    ap.add_argument("--rounding", default="nearest", choices=["nearest", "stochastic"],
                    help="rounding of 16-bit storage")
    ap.add_argument("--nx", type=int, default=inputs.THROUGHPUT_8192.nx)
    ap.add_argument("--ny", type=int, default=inputs.THROUGHPUT_8192.ny)
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-cpu", action="store_true")
    ap.add_argument("--cpu-seconds", type=float, default=15.0)
    ap.add_argument("--workload", default="heat_mode",
                    choices=["heat_mode", "batch", "warmstart", "train", "d3q14", "small"],
                    help="heat_mode: 8192^2 throughput (default); batch: 512 channels "
                         "solved to steady state; warmstart: learned warm start vs cold "
                         "start on 512 held-out channels; train: the warm-start network's "
                         "training speed alone; d3q14: 3-D D3Q14 throughput "
                         "on a periodic nz x ny x nx lattice (--n3 cells per side); small: "
                         "the 128x32 Poiseuille channel (FP64, FP32) and the 4096x4 "
                         "second-sound pulse (FP32), time per step and error vs the oracle")
    ap.add_argument("--n3", type=int, default=512)
    ap.add_argument("--train-instances", type=int, default=4096)
    ap.add_argument("--train-steps", type=int, default=4000)
    ap.add_argument("--instances", type=int, default=512)
    ap.add_argument("--tol", type=float, default=1e-8)
    ap.add_argument("--check-every", type=int, default=500,
                    help="steps per residual window (FP32 rounding puts a floor of about "
                         "1e-6/K under the residual of high-tau channels)")
    ap.add_argument("--max-steps", type=int, default=400000)
    ap.add_argument("--reference-instances", type=int, default=64,
                    help="held-out channels whose end states are compared with an FP64 "
                         "reference (warmstart workload)")
    ap.add_argument("--no-steady", action="store_true",
                    help="default workload: skip the time-to-steady-state leg")
    ap.add_argument("--sequential-sample", type=int, default=0,
                    help="batch workload: channels of the one-at-a-time baseline "
                         "(0 = all of them)")
    return ap.parse_args()


def dist_env():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return world, rank, local


def max_over_ranks(value, dist=None, device=None):
    """The job's time: the maximum of a per-rank value over all ranks (the
    slowest replica sets it); the value itself without a process group."""
    if dist is None:
        return value
    import torch
    t = torch.tensor([float(value)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return t.item()


def job_value(world, sites, steps, seconds):
    """Whole-job GLUPS: site updates of all ranks over the job's time."""
    return world * sites * steps / seconds / 1e9


def workload(args):
    w = inputs.THROUGHPUT_8192
    return dict(nx=args.nx, ny=args.ny, kn_N=w.kn_N, kn_R=w.kn_R, length=w.length)


def cpu_info():
    model = ""
    try:
        out = subprocess.run(["lscpu"], capture_output=True, text=True, timeout=10).stdout
        m = re.search(r"Model name:\s*(.+)", out)
        model = m.group(1).strip() if m else ""
    except Exception:
        pass
    return os.cpu_count() or 1, model


def oracle_sample(w, seconds: float):
    """Time the FP64 oracle on a bounded sample of the workload: a periodic
    2048 x 2048 window of the same fields, as many steps as fit ~`seconds`."""
    import oracle
    cores, model = cpu_info()
    oracle.set_threads(cores)
    side = min(2048, w["nx"], w["ny"])
    tau_N = oracle.tau_from_kn(w["kn_N"], w["length"])
    tau_R = oracle.tau_from_kn(w["kn_R"], w["length"])
    e = inputs.sine_mode(side, side, 512.0, 1e-3, noise=1e-6)
    lat = oracle.run(side, side, tau_N, tau_R, e)
    t0 = time.perf_counter()
    lat.step(1)
    one = time.perf_counter() - t0
    steps = max(1, int(seconds / max(one, 1e-6)))
    t0 = time.perf_counter()
    lat.step(steps)
    dt = time.perf_counter() - t0
    glups = side * side * steps / dt / 1e9
    return {"value": glups, "unit": "GLUPS", "cores": oracle.get_threads(), "kind": "oracle",
            "sample": f"{side}x{side} periodic window of the workload, {steps} steps, "
                      f"{dt:.1f} s, FP64, host '{model}'"}


def oracle_rate(instances, seconds: float):
    """FP64 oracle (all host cores) on a bounded sample of batched channels:
    each instance from a cold start for as many steps as fit its share of
    `seconds`; returns (GLUPS, cores, description)."""
    import oracle
    cores, model = cpu_info()
    oracle.set_threads(cores)
    updates, spent = 0.0, 0.0
    for i in instances:
        lat = oracle.run(i["nx"], i["ny"], i["tau_N"], i["tau_R"], np.ones((i["ny"], i["nx"])),
                         bc_x=i["bc_x"], bc_y=i["bc_y"], delta_e=i["delta_e"])
        t0 = time.perf_counter()
        lat.step(1)
        one = time.perf_counter() - t0
        n = max(1, int(seconds / len(instances) / max(one, 1e-6)))
        t0 = time.perf_counter()
        lat.step(n)
        spent += time.perf_counter() - t0
        updates += n * i["nx"] * i["ny"]
    widths = ", ".join(str(i["ny"]) for i in instances)
    return updates / spent / 1e9, oracle.get_threads(), \
        f"{len(instances)} channels (W = {widths}), {updates:.3g} site updates in {spent:.1f} s, " \
        f"FP64, host '{model}'"


class ClockSampler:
    """nvidia-smi clock/throttle samples while the timed region runs."""
    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.proc = None

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--id={self.index}", f"--query-gpu={self.Q}",
                 "--format=csv,noheader,nounits", "-lms", "100"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except Exception:
            self.proc = None
        return self

    def __exit__(self, *exc):
        self.lines = []
        if self.proc is not None:
            self.proc.terminate()
            try:
                out, _ = self.proc.communicate(timeout=5)
            except Exception:
                self.proc.kill()
                out, _ = self.proc.communicate()
            self.lines = [l for l in out.splitlines() if l.strip()]

    def summary(self):
        sm, mx, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for l in getattr(self, "lines", []):
            f = [x.strip() for x in l.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                mx.append(float(f[2]))
            except ValueError:
                continue
            for n, v in zip(names, f[5:9]):
                if v.lower() == "active":
                    reasons.add(n)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": [], "samples": 0}
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(mx),
                "reasons": sorted(reasons), "samples": len(sm)}


def measured_peak():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(path) as fh:
            d = json.load(fh)
        for key in ("hbm_gbs", "hbm_GBs", "hbm"):
            if key in d:
                v = d[key]
                v = v.get("value", v) if isinstance(v, dict) else v
                return float(v), "measured"
    except Exception:
        pass
    return FALLBACK_HBM_GBS, "fallback"


# FP32 operations of the collision per node and step in the kernels that
# compute in FP32 (FP32 and 16-bit storage): 15 for the moments, 9 for the
# flux terms, 3 per population
FP32_OPS_PER_UPDATE = {"fp32": 48, "fp16": 48, "bf16": 48}
NOMINAL_SM_MHZ = 2070.0

# sources that define each stream-collide kernel
KERNEL_SOURCES = {
    "step_vector": ["lbm_device.cuh", "vector_pull.cuh", "stream_collide.cu"],
    "step_pipe16": ["lbm_device.cuh", "refs16.cuh", "pairs16.cuh", "vector_pull.cuh",
                    "pipe16.cu"],
    "step_staged": ["lbm_device.cuh", "mbarrier.cuh", "staged.cu"],
    "step_scalar": ["lbm_device.cuh", "refs16.cuh", "stream_collide.cu"],
    "step_wave": ["lbm_device.cuh", "wave.cuh", "wave.cu"],
    "step_wave16": ["lbm_device.cuh", "refs16.cuh", "wave.cuh", "wave16.cu"],
}


def kernel_source_hash(kernel_name):
    h = hashlib.sha256()
    csrc = os.path.join(ROOT, "paper_2010_01847_gb300", "csrc")
    for f in KERNEL_SOURCES[kernel_name]:
        with open(os.path.join(csrc, f), "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()[:16]


def ncu_traffic(kernel_name, precision, nx, ny, shape=None):
    """DRAM bytes per launch from the committed ncu summary, if it was taken
    on the current sources of that kernel (else None), scaled by sites.  A
    multi-step kernel's line names its shape (`step_wave:5x128`: steps per
    launch x segment rows, which set the overlap rows it reads)."""
    path = os.path.join(ROOT, "profiles", "dram_traffic.txt")
    if not os.path.exists(path) or kernel_name not in KERNEL_SOURCES:
        return None
    src = kernel_source_hash(kernel_name)
    key = kernel_name if shape is None else f"{kernel_name}:{shape['steps']}x{shape['rows']}"
    for line in open(path):
        f = line.split()
        if len(f) < 7 or f[0].startswith("#"):
            continue
        kname, prec, snx, sny, nbytes, shash = f[0], f[1], int(f[2]), int(f[3]), float(f[4]), f[5]
        if kname == key and prec == precision and shash == src:
            return nbytes * (nx * ny) / (snx * sny)   # traffic grows with the sites
    return None


def run_reference(args):
    """The FP64 oracle on the host cores, each bench step one timed oracle
    step on a periodic window of the workload sized so the whole run stays
    within about 90 s.  Rank 0 only."""
    world, rank, _ = dist_env()
    if rank != 0:
        return
    import oracle
    w = workload(args)
    cores, model = cpu_info()
    oracle.set_threads(cores)
    tau_N = oracle.tau_from_kn(w["kn_N"], w["length"])
    tau_R = oracle.tau_from_kn(w["kn_R"], w["length"])
    cal = oracle.run(512, 512, tau_N, tau_R, inputs.sine_mode(512, 512, 512.0, 1e-3, noise=1e-6))
    t0 = time.perf_counter()
    cal.step(2)
    rate = 2 * 512 * 512 / (time.perf_counter() - t0)
    budget = min(args.cpu_seconds, 90.0 / max(args.steps + args.warmup, 1))
    side = int(min(2048, max(64, math.sqrt(rate * budget))) // 64 * 64)
    side = min(side, w["nx"], w["ny"])
    lat = oracle.run(side, side, tau_N, tau_R, inputs.sine_mode(side, side, 512.0, 1e-3,
                                                                noise=1e-6))
    lat.step(max(args.warmup, 0))
    total = 0.0
    for _ in range(args.steps):
        t0 = time.perf_counter()
        lat.step(1)
        total += time.perf_counter() - t0
    value = side * side * args.steps / total / 1e9
    sample = {"value": value, "unit": "GLUPS", "cores": oracle.get_threads(), "kind": "oracle",
              "sample": f"{side}x{side} periodic window of the workload, {args.steps} timed "
                        f"steps ({total:.1f} s), FP64, host '{model}'"}
    # the line describes what was timed: the window, its own time per step;
    # the time a full-size step would take at the same rate is a field apart
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": "GLUPS",
        "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": total / args.steps * 1e3,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
        "data": "synthetic",
        "config": {"workload": f"heat_mode_window_{side}x{side}",
                   "window_of": f"heat_mode_{w['nx']}x{w['ny']}", "kn_N": w["kn_N"],
                   "kn_R": w["kn_R"], "length_cells": w["length"], "storage": "fp64 (oracle)",
                   "lattice": "D2Q8"},
        "ms_per_step_extrapolated_full_size": w["nx"] * w["ny"] / (value * 1e9) * 1e3,
        "cpu_baseline": sample,
        "e2e": {"value": value, "unit": "GLUPS", "h2d_bytes_per_step": 0,
                "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)


def run_native(args):
    import torch
    import paper_2010_01847_gb300 as plbm

    world, rank, local = dist_env()
    if world > 1:
        import torch.distributed as dist
        torch.cuda.set_device(local)
        dist.init_process_group("nccl")
    else:
        dist = None
        torch.cuda.set_device(0)
    dev = torch.device("cuda", torch.cuda.current_device())
    w = workload(args)
    nx, ny = w["nx"], w["ny"]
    tau_N = plbm.tau_from_kn(w["kn_N"], w["length"])
    tau_R = plbm.tau_from_kn(w["kn_R"], w["length"])
    e = inputs.sine_mode(nx, ny, 512.0, 1e-3, noise=1e-6)
    e_dev = torch.from_numpy(e).to(dev)
    z_dev = torch.zeros_like(e_dev)

    lat = plbm.Lattice(nx, ny, tau_N, tau_R, precision=args.precision, kernel=args.kernel,
                       rounding=args.rounding if STORAGE_BYTES[args.precision] == 2 else "nearest")
    lat.init(e_dev, z_dev, z_dev)
    tuned = None
    if args.kernel == "auto":
        # set-up, untimed: pick the fastest kernel / shape on this GPU
        tuned = lat.autotune(20)
    if args.wave_steps or args.wave_rows:
        wc = lat.wave_config
        lat.set_wave_config(args.wave_steps or wc["steps"], args.wave_rows or wc["rows"])
    stream = torch.cuda.current_stream(dev)

    # residual window: every RESIDUAL_EVERY-th step, or once per run when
    # the run is shorter, so a short timed region still carries the
    # residual's cost (at a higher weight than a long one)
    window = max(1, min(RESIDUAL_EVERY, args.steps))

    def chunked(nsteps):
        """Advance nsteps in windows: each whole window is one
        lbm_step_residual call, whose last step also reduces the residual
        inside its stream-collide launch; a shorter tail is plain steps."""
        done = 0
        while done < nsteps:
            k = min(window, nsteps - done)
            if k == window:
                lat.step_residual(k)
            else:
                lat.step(k)
            done += k

    chunked(max(args.warmup, 3))
    torch.cuda.synchronize()
    if dist:
        dist.barrier()
    torch.cuda.synchronize()
    sampler = ClockSampler(dev.index)
    launches0 = lat.kernel_launches
    # the library brackets every stream-collide launch with CUDA events on
    # the lattice's stream (no graphs meanwhile: at these sizes a launch is
    # far longer than its launch latency)
    lat.set_launch_timing(True)
    with sampler:
        t0 = torch.cuda.Event(enable_timing=True)
        t1 = torch.cuda.Event(enable_timing=True)
        t0.record(stream)
        chunked(args.steps)
        t1.record(stream)
        torch.cuda.synchronize()
    if dist:
        dist.barrier()
    torch.cuda.synchronize()
    elapsed = t0.elapsed_time(t1) / 1e3
    launches = lat.kernel_launches - launches0        # counted by the library
    timed = {which: lat.launch_time(which)
             for which in (plbm.TIMED_WAVE, plbm.TIMED_SINGLE, plbm.TIMED_RESIDUAL)}
    lat.set_launch_timing(False)
    elapsed = max_over_ranks(elapsed, dist, dev)
    sites = nx * ny
    value = job_value(world, sites, args.steps, elapsed)

    # roofline of the dominant stream-collide kernel (the kind of launch
    # with the most time): one state buffer read and one written per launch
    # (16-bit storage includes the tiles' references), i.e. per site update
    # for single steps and per `steps / launches` updates for the
    # multi-step kernel
    bps = lat.bytes_per_site_update
    dom = max(timed, key=lambda w: timed[w][0])
    kern_ms, kern_launches, kern_steps = timed[dom]
    avg_launch = kern_ms / 1e3 / kern_launches
    achieved = bps * sites / avg_launch / 1e9
    peak, peak_kind = measured_peak()
    shape = None
    if dom == plbm.TIMED_WAVE:
        kname = "step_wave16" if STORAGE_BYTES[args.precision] == 2 else "step_wave"
        shape = lat.wave_config
    elif dom == plbm.TIMED_RESIDUAL:
        kname = "step_vector_residual"
    else:
        kname = "step_" + ("vector" if lat.kernel == "wave" else lat.kernel)
        if kname == "step_vector" and STORAGE_BYTES[args.precision] == 2:
            kname = "step_pipe16"           # plain 16-bit steps: the pipelined node-pair kernel
    roof = {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s",
            "frac": achieved / peak, "traffic": ncu_traffic(kname, args.precision, nx, ny, shape),
            "peak_source": f"{peak_kind} ({'MEASURED_PEAKS.json hbm_gbs' if peak_kind == 'measured' else 'profiling-recipe fallback 6.8 TB/s'})",
            "kernel": kname, "bytes_per_launch_site": bps,
            "steps_per_launch": kern_steps / kern_launches,
            "bytes_per_site_update": bps * kern_launches / kern_steps,
            "avg_launch_us": avg_launch * 1e6,
            "launch_mix": {n: {"ms": v[0], "launches": v[1], "steps": v[2]}
                           for n, v in (("multi_step", timed[plbm.TIMED_WAVE]),
                                        ("single", timed[plbm.TIMED_SINGLE]),
                                        ("residual", timed[plbm.TIMED_RESIDUAL]))}}

    # end to end through the public API with pinned host buffers
    e2e = None
    if not args.no_e2e:
        # the workload's input is the energy field (q = 0 at the start: lbm_init
        # takes no flux arrays); its result the three fields (e, qx, qy)
        host = torch.from_numpy(e).pin_memory()
        out = [torch.empty((ny, nx), dtype=torch.float64).pin_memory() for _ in range(3)]
        hp = host.numpy()
        op = [o.numpy() for o in out]
        # pinning ~2 GB above leaves the GPU idle for a second or more: warm
        # it up again, untimed, for the warm-up steps and at least 0.3 s of
        # stepping (20 steps of the 8192^2 lattice take 4 ms, too short for
        # the clocks to come back: the first e2e runs lost ~50 ms that way)
        chunked(max(args.warmup, 3))
        torch.cuda.synchronize()
        t_warm = time.perf_counter()
        while time.perf_counter() - t_warm < 0.3:
            chunked(window)
            torch.cuda.synchronize()
        # three end-to-end runs, the median reported; each with its parts
        # (the synchronize after the steps costs nothing: lbm_moments waits
        # for them anyway)
        runs = []
        for _ in range(3):
            if dist:
                dist.barrier()
            t_start = time.perf_counter()
            lat.init(hp)
            t_init = time.perf_counter()
            chunked(args.steps)
            torch.cuda.synchronize()
            t_steps = time.perf_counter()
            lat.moments(out=op)                 # device -> pinned host
            t_end = time.perf_counter()
            total = max_over_ranks(t_end - t_start, dist, dev)
            runs.append((total, {"init_ms": (t_init - t_start) * 1e3,
                                 "steps_ms": (t_steps - t_init) * 1e3,
                                 "moments_ms": (t_end - t_steps) * 1e3}))
        runs.sort(key=lambda r: r[0])
        t_e2e, parts = runs[1]
        e2e = {"value": job_value(world, sites, args.steps, t_e2e), "unit": "GLUPS",
               "h2d_bytes_per_step": 8 * sites / args.steps,
               "d2h_bytes_per_step": 3 * 8 * sites / args.steps,
               "what": "lbm_init from pinned host (e; q = 0) + steps + lbm_moments "
                       "(e, qx, qy) into pinned host; median of 3 runs",
               "runs": [job_value(world, sites, args.steps, r[0]) for r in runs],
               "median_run_ms": parts}

    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu:
        cpu = oracle_sample(w, args.cpu_seconds)

    # time to steady state, learned vs analytic vs cold start (the metric's
    # second half), on a bounded held-out set: one GPU, rank 0 alone
    kernel_name = lat.kernel
    staged_shape = lat.staged_config if kernel_name == "staged" else None
    wave_shape = lat.wave_config if kernel_name == "wave" else None
    steady = None
    if rank == 0 and world == 1 and not args.no_steady:
        lat.close()
        torch.cuda.synchronize()
        steady = steady_state_study(n_train=1024, train_steps=2000, n_test=64, n_ref=64,
                                    tol=1e-8, check_every=500, max_steps=400000)

    if rank == 0:
        clocks = sampler.summary()
        if FP32_OPS_PER_UPDATE.get(args.precision):
            # the same launches against the FP32 pipe: the collision's
            # operations per useful site update (an FMA counts one) over the
            # launch time, against 128 FP32 lanes per SM at the sampled
            # maximum SM clock; halo columns and overlap rows that the
            # multi-step kernel computes twice are not counted
            ops = FP32_OPS_PER_UPDATE[args.precision]
            mhz = clocks.get("sm_max_mhz") or NOMINAL_SM_MHZ
            sms = torch.cuda.get_device_properties(dev).multi_processor_count
            peak_ops = sms * 128 * mhz * 1e6 / 1e12
            got = ops * sites * roof["steps_per_launch"] / (roof["avg_launch_us"] * 1e-6) / 1e12
            roof["fp32_pipe"] = {"bound": "alu", "ops_per_site_update": ops, "achieved": got,
                                 "peak": peak_ops, "unit": "TOP/s", "frac": got / peak_ops,
                                 "peak_source": f"{sms} SMs x 128 FP32 lanes x {mhz:g} MHz"}
        line = {
            "metric": METRIC, "value": value, "unit": "GLUPS", "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": elapsed / args.steps * 1e3, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": DTYPE[args.precision],
            "data": "synthetic",
            "config": {"workload": f"heat_mode_{nx}x{ny}", "lattice": "D2Q8 (paper's D2Q9 "
                       "label: rest population identically zero, not stored)",
                       "kn_N": w["kn_N"], "kn_R": w["kn_R"], "length_cells": w["length"],
                       "storage": (f"{args.precision} deviation" +
                                   (f", tile references, {args.rounding} rounding"
                                    if STORAGE_BYTES[args.precision] == 2 else "")),
                       "kernel": kernel_name,
                       "staged_shape": staged_shape,
                       "wave_shape": wave_shape,
                       "autotuned": tuned is not None,
                       "residual_every": window,
                       "l2": "inputs larger than L2 (2 x population buffers >> 129 MB); "
                             "no flush", "parallelism": f"replicas x{world}"},
            "roofline": roof, "clocks": clocks, "gpu_launches": launches,
            "e2e": e2e, "cpu_baseline": cpu, "steady_state": steady,
        }
        print(json.dumps(line), flush=True)
    lat.close()
    if dist:
        dist.destroy_process_group()


def run_d3q14(args):
    """Throughput of the D3Q14 stream-collide step (lbm_nd_*): periodic n^3
    lattice, x-directed sine mode of wavelength 512 cells (+ U[-1e-6, 1e-6)
    noise), Kn as the 2-D heat-mode workload, FP32 or FP64 storage."""
    import torch
    import paper_2010_01847_gb300 as plbm
    torch.cuda.set_device(0)
    dev = torch.device("cuda", 0)
    n = args.n3
    w = inputs.THROUGHPUT_8192
    speed = plbm.LatticeND.lattice_speed(plbm.D3Q14)
    tau_N, tau_R = w.kn_N * w.length * speed, w.kn_R * w.length * speed
    x = np.arange(n, dtype=np.float64)
    e = np.empty((n, n, n))
    e[...] = 1.0 + 1e-3 * np.sin(2 * np.pi * x / 512.0)
    e += inputs.uniform_noise(e.shape, 1e-6)
    prec = args.precision if args.precision in ("fp32", "fp64") else "fp32"
    lat = plbm.LatticeND(plbm.D3Q14, (n, n, n), tau_N, tau_R, precision=prec)
    lat.init(e)
    e0 = lat.energy()
    stream = torch.cuda.current_stream(dev)
    lat.step(max(args.warmup, 3))
    torch.cuda.synchronize()
    sampler = ClockSampler(dev.index)
    with sampler:
        t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        launches = lat.kernel_launches
        t0.record(stream)
        lat.step(args.steps)
        t1.record(stream)
        torch.cuda.synchronize()
        launches = lat.kernel_launches - launches
    elapsed = t0.elapsed_time(t1) / 1e3
    sites = n ** 3
    # one read and one write of the state per launch, of one or two steps
    pairs = args.steps - launches
    bps = 2 * 14 * STORAGE_BYTES[prec] * launches / args.steps
    achieved = bps * sites * args.steps / elapsed / 1e9
    peak, peak_kind = measured_peak()
    drift = abs(lat.energy() - e0) / abs(e0)
    line = {
        "metric": "GLUPS & % HBM roofline (D3Q14)", "value": sites * args.steps / elapsed / 1e9,
        "unit": "GLUPS", "n_gpus": 1, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": elapsed / args.steps * 1e3, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": DTYPE[prec], "data": "synthetic",
        "config": {"workload": f"d3q14_heat_mode_{n}^3", "lattice": "D3Q14",
                   "kn_N": w.kn_N, "kn_R": w.kn_R, "length_cells": w.length,
                   "storage": f"{prec} deviation",
                   "l2": "inputs larger than L2; no flush"},
        "roofline": {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s",
                     "frac": achieved / peak, "traffic": None,
                     "peak_source": peak_kind,
                     "kernel": "step2_d3q14" if pairs else "step_nd",
                     "bytes_per_site_update": bps},
        "clocks": sampler.summary(), "gpu_launches": launches, "e2e": None,
        "cpu_baseline": None, "energy_drift": drift,
    }
    print(json.dumps(line), flush=True)
    lat.close()


def run_small(args):
    """The two small named workloads: the 128x32 phonon Poiseuille channel
    (10 000 steps, FP64 and FP32 storage) and the 4096x4 second-sound pulse
    (5 000 steps, Kn_R = 0.1, 1, 10, FP32).  Both are far too small to fill
    the GPU: FP32 runs the channel cluster-resident (the whole lattice in one
    cluster's shared memory, all steps in one launch) and the pulse on register
    tiles (several steps per launch; `kernel` then names that of the single
    steps), FP64 as graph-captured launches, one per step.  The CPU-baseline leg (skipped
    with --no-cpu) runs the FP64 oracle on the same inputs, on all host
    cores: its time per step, and the GPU result's error against it (err_e,
    err_q as in the parity tests)."""
    import torch
    import paper_2010_01847_gb300 as plbm
    torch.cuda.set_device(0)
    stream = torch.cuda.current_stream()
    runs = []

    def cpu_leg(w, fields, tau_N, tau_R, steps, g):
        import oracle
        cores, model = cpu_info()
        oracle.set_threads(cores)
        t_o = time.perf_counter()
        o = oracle.run(w.nx, w.ny, tau_N, tau_R, *fields, steps=steps, bc_x=w.bc_x,
                       bc_y=w.bc_y, delta_e=w.delta_e).moments()
        t_o = time.perf_counter() - t_o
        de = np.abs(o[0] - o[0].mean()).max()
        qmax = max(np.abs(o[1]).max(), np.abs(o[2]).max())
        return {"kind": "oracle", "us_per_step": t_o / steps * 1e6,
                "value": w.nx * w.ny * steps / t_o / 1e9, "unit": "GLUPS",
                "cores": oracle.get_threads(), "sample": f"full run, FP64, host '{model}'",
                "gpu_err_e": float(np.abs(g[0] - o[0]).max() / de),
                "gpu_err_q": float(max(np.abs(g[1] - o[1]).max(),
                                       np.abs(g[2] - o[2]).max()) / qmax)}

    def one(w, precision):
        tau_N = plbm.tau_from_kn(w.kn_N, w.length)
        tau_R = plbm.tau_from_kn(w.kn_R, w.length)
        fields = inputs.initial_fields(w)
        lat = plbm.Lattice(w.nx, w.ny, tau_N, tau_R, w.bc_x, w.bc_y, w.delta_e,
                           precision=precision)
        lat.init(*fields)
        warm = 64                                      # warm-up; captures the step graphs
        lat.step(warm)
        torch.cuda.synchronize()
        t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        launches0 = lat.kernel_launches
        t0.record(stream)
        lat.step(w.steps)
        t1.record(stream)
        torch.cuda.synchronize()
        launches = lat.kernel_launches - launches0
        us = t0.elapsed_time(t1) * 1e3 / w.steps
        g = lat.moments()
        lat_kernel = lat.kernel
        lat.close()
        runs.append({"workload": w.name, "storage": precision, "steps": w.steps,
                     "us_per_step": us, "glups": w.nx * w.ny / us / 1e3, "kernel": lat_kernel,
                     "gpu_launches": launches,
                     "cpu_baseline": None if args.no_cpu else
                     cpu_leg(w, fields, tau_N, tau_R, warm + w.steps, g)})

    one(inputs.POISEUILLE_128x32, "fp64")
    one(inputs.POISEUILLE_128x32, "fp32")
    for kn_R in (0.1, 1.0, 10.0):
        one(inputs.second_sound_4096x4(kn_R), "fp32")
    line = {"metric": "time per step, small named workloads",
            "value": runs[1]["us_per_step"], "unit": "us/step", "n_gpus": 1,
            "higher_is_better": False, "dtype": "f32", "data": "synthetic",
            "config": {"workload": "poiseuille_128x32 (value: FP32) + second_sound_4096x4",
                       "kernels": "FP32: cluster-resident, all steps in one launch (128x32); "
                                  "register tiles, several steps per launch (4096x4); FP64: "
                                  "graph-captured launches"},
            "runs": runs, "gpu_launches": sum(r["gpu_launches"] for r in runs)}
    print(json.dumps(line), flush=True)


def batch_instances(n, seed=inputs.SEED):
    """The batched-channel workload: seeded candidates (width W in [16, 512],
    length 4W, Kn_N log-U[1e-3, 1e-1], Kn_R log-U[0.1, 10], walls, periodic
    temperature gradient with delta_e = 1e-3) whose tau is at least 0.6, the
    scheme's linear-stability bound with margin; returns (kept, rejected)."""
    import paper_2010_01847_gb300 as plbm
    kept, rejected = [], 0
    for c in inputs.batch_channels(8 * n, seed=seed):
        tau_N = plbm.tau_from_kn(c["kn_N"], c["d"])
        tau_R = plbm.tau_from_kn(c["kn_R"], c["d"])
        tau = 1.0 / (1.0 / tau_N + 1.0 / tau_R) + 0.5
        if tau < 0.6:
            rejected += 1
            continue
        kept.append(dict(nx=c["nx"], ny=c["ny"], tau_N=tau_N, tau_R=tau_R,
                         bc_x=inputs.PERIODIC_GRADIENT, bc_y=inputs.WALLS, delta_e=1e-3,
                         W=c["W"], kn_N=c["kn_N"], kn_R=c["kn_R"]))
        if len(kept) == n:
            break
    return kept, rejected


def run_batch(args):
    """Time to steady state (r < tol on two consecutive checks every
    --check-every steps) of the batched channels from a cold start (e = 1,
    q = 0), with the plain single-lattice solver run on every channel, one
    after the other, as the baseline."""
    import torch
    import paper_2010_01847_gb300 as plbm
    torch.cuda.set_device(0)
    inst, rejected = batch_instances(args.instances)
    sites = np.array([i["nx"] * i["ny"] for i in inst], dtype=np.float64)
    b = plbm.Batch(inst)
    b.init()
    tune_us = b.autotune(10)
    b.init()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    steps, r = b.solve(args.tol, args.check_every, args.max_steps)
    t_batch = time.perf_counter() - t0
    updates = float((steps * sites).sum())
    # the plain single-lattice solver, one channel at a time (the fastest
    # kernel each: cluster-resident up to 16384 nodes, else the one the
    # autotuner picks -- multi-step or vector launches -- with the residual
    # fused every check window): all channels, or a seeded sample with
    # --sequential-sample n > 0
    if args.sequential_sample > 0:
        rng = np.random.default_rng(5)
        sample = sorted(rng.choice(len(inst), size=min(args.sequential_sample, len(inst)),
                                   replace=False).tolist())
    else:
        sample = list(range(len(inst)))
    t_seq = 0.0
    seq_updates = 0.0
    for k in sample:
        i = inst[k]
        lat = plbm.Lattice(i["nx"], i["ny"], i["tau_N"], i["tau_R"], i["bc_x"], i["bc_y"],
                           i["delta_e"])
        lat.init(np.ones((i["ny"], i["nx"])))
        if i["nx"] * i["ny"] > 16384:
            lat.autotune(20)          # untimed set-up: the fastest kernel for this channel
        torch.cuda.synchronize()
        t1 = time.perf_counter()
        lat.residual()
        good, n = 0, 0
        while n < args.max_steps:
            rr, _ = lat.step_residual(args.check_every)
            n += args.check_every
            good = good + 1 if rr < args.tol else 0
            if good >= 2:
                break
        t_seq += time.perf_counter() - t1
        seq_updates += n * i["nx"] * i["ny"]
        lat.close()
    cpu = None
    if not args.no_cpu:
        g_cpu, cores, desc = oracle_rate([inst[k] for k in sample[::max(1, len(sample) // 4)][:4]],
                                         args.cpu_seconds)
        cpu = {"value": g_cpu, "unit": "GLUPS", "cores": cores, "kind": "oracle",
               "sample": desc, "estimated_seconds_all": updates / (g_cpu * 1e9)}
    line = {
        "metric": "time to steady state (r < 1e-8), batched channels, cold start",
        "value": t_batch, "unit": "s", "n_gpus": 1, "higher_is_better": False,
        "dtype": "f32", "data": "synthetic",
        "config": {"workload": f"batched_channels_{len(inst)}", "instances": len(inst),
                   "rejected_unstable_candidates": rejected,
                   "total_sites": int(sites.sum()), "tol": args.tol,
                   "check_every": args.check_every,
                   "schedule": b.schedule, "wave": b.wave, "autotune_us_per_step": tune_us},
        "steps": {"min": int(steps.min()), "median": float(np.median(steps)),
                  "max": int(steps.max()), "all_converged": bool(np.all(r < args.tol))},
        "site_updates": updates, "glups": updates / t_batch / 1e9,
        "plain_sequential": {
            "instances": len(sample), "measured_all": len(sample) == len(inst),
            "seconds": t_seq, "site_updates": seq_updates,
            "glups": seq_updates / t_seq / 1e9,
            "seconds_all": t_seq if len(sample) == len(inst)
            else t_seq * updates / max(seq_updates, 1.0)},
        "batched_over_sequential": (t_seq if len(sample) == len(inst)
                                    else t_seq * updates / max(seq_updates, 1.0)) / t_batch,
        "cpu_baseline": cpu,
    }
    print(json.dumps(line), flush=True)


def steady_state_study(n_train, train_steps, n_test, n_ref, tol, check_every, max_steps,
                       w_range=(16, 512)):
    """Time to steady state (r < tol) of held-out walled channels with the
    periodic gradient from three starts, and their accuracy.

    Training: n_train channels' steady states from the batched solver (on
    channels shortened to 8 columns, whose steady rows are the full ones';
    solved from the analytic start),
    the network trained on the GPU (train_steps Adam steps, minibatches of
    512).  Held-out: n_test channels of length 4W from a seed training never
    saw, solved from the cold start (e = e_ref, q = 0), the analytic start
    (Eq. 68 flux, affine e) and the learned start.  Reference: the first
    n_ref held-out channels solved with FP64 storage to r < 1e-12 (shortened
    copies); each start's end state is compared with it row by row."""
    import torch
    from paper_2010_01847_gb300 import warmstart
    t0 = time.perf_counter()
    train = warmstart.channels(n_train, seed=inputs.SEED + 1, nx=warmstart.TRAIN_NX,
                               w_range=w_range)
    # the training steady states, solved from the analytic start (Eq. 68)
    prof, tsteps, tr, t_gen = warmstart.steady_profiles(train, tol, check_every, max_steps,
                                                        schedule="tune", start="analytic")
    ws = warmstart.WarmStart(seed=0, max_batch=max(512, n_train))
    torch.cuda.synchronize()
    t1 = time.perf_counter()
    hist = ws.train(train, prof, steps=train_steps, batch=512, lr=1e-3)
    torch.cuda.synchronize()
    t_train = time.perf_counter() - t1
    test = warmstart.channels(n_test, seed=inputs.SEED + 2, w_range=w_range)
    t2 = time.perf_counter()
    pred = ws.predict(test)
    torch.cuda.synchronize()
    t_pred = time.perf_counter() - t2
    t3 = time.perf_counter()
    ana = warmstart.analytic_profiles(test)
    torch.cuda.synchronize()
    t_ana = time.perf_counter() - t3
    runs = {}
    schedule = "tune"           # autotuned on the cold batch, then kept for all three
    for name, start in (("cold", None), ("analytic", ana), ("learned", pred)):
        steps, r, secs, b = warmstart.solve(test, start, tol, check_every, max_steps,
                                            schedule=schedule)
        schedule = warmstart.schedule_of(b)
        runs[name] = {"seconds": secs, "steps": steps, "r": r, "batch": b}
    ref_set = test[:n_ref]
    t4 = time.perf_counter()
    ref, rsteps, rr = warmstart.reference_profiles(ref_set)
    t_ref = time.perf_counter() - t4
    sites = np.array([i["nx"] * i["ny"] for i in test], dtype=np.float64)
    out = {"tol": tol, "check_every": check_every,
           "train_instances": len(train), "train_steps": train_steps,
           "held_out": len(test), "widths": list(w_range), "schedule": schedule}
    for name, run in runs.items():
        b = run["batch"]
        ee, eq = warmstart.profile_errors(b.profiles()[:n_ref], ref, ref_set)
        out[name] = {"seconds": run["seconds"],
                     "steps_median": float(np.median(run["steps"])),
                     "steps_max": int(run["steps"].max()),
                     "site_updates": float((run["steps"] * sites).sum()),
                     "converged": bool(np.all(run["r"] < tol)),
                     "err_vs_reference": {"e_max": float(ee.max()), "q_max": float(eq.max()),
                                          "e_median": float(np.median(ee)),
                                          "q_median": float(np.median(eq))}}
        b.close()
    out["speedup_learned_vs_cold"] = out["cold"]["seconds"] / out["learned"]["seconds"]
    out["speedup_learned_vs_analytic"] = out["analytic"]["seconds"] / out["learned"]["seconds"]
    out["speedup_analytic_vs_cold"] = out["cold"]["seconds"] / out["analytic"]["seconds"]
    out["training"] = {"data_generation_seconds": t_gen,
                       "data_steps_median": float(np.median(tsteps)),
                       "train_seconds": t_train, "loss_first": float(hist[0]),
                       "loss_last": float(hist[-1]), "predict_seconds": t_pred}
    out["analytic_profile_seconds"] = t_ana
    # the whole learned pipeline (generate data, train, predict, solve)
    out["learned_pipeline_seconds"] = t_gen + t_train + t_pred + out["learned"]["seconds"]
    out["speedup_learned_pipeline_vs_cold"] = out["cold"]["seconds"] / \
        out["learned_pipeline_seconds"]
    out["reference"] = {"channels": len(ref_set), "storage": "fp64", "tol": 1e-12,
                        "seconds": t_ref, "converged": bool(np.all(rr < 1e-12)),
                        "how": "held-out channels shortened to 8 columns with the same "
                               "gradient (their steady rows are the full channels'), "
                               "solved to r < 1e-12"}
    out["study_seconds"] = time.perf_counter() - t0
    return out


def run_train(args):
    """Training speed of the warm-start network alone: --train-steps Adam
    steps (the device training loop, lbm_mlp_train) on minibatches of 512
    from --train-instances synthetic samples (inputs uniform in [-1, 1],
    targets N(0, 0.1^2); the time does not depend on the values)."""
    import torch
    import paper_2010_01847_gb300 as plbm
    from paper_2010_01847_gb300 import warmstart
    torch.cuda.set_device(0)
    n = args.train_instances
    rng = np.random.default_rng(inputs.SEED)
    x = torch.from_numpy(rng.uniform(-1, 1, (n, warmstart.WIDTHS[0])).astype(np.float32)).cuda()
    t = torch.from_numpy(rng.normal(0, 0.1, (n, warmstart.WIDTHS[-1])).astype(np.float32)).cuda()
    net = plbm.Mlp(list(warmstart.WIDTHS), max_batch=max(512, n))
    net.init_params(0)
    net.train(x, t, 10, 512, 1e-3, 1e-5)          # capture, first launches (untimed)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    hist = net.train(x, t, args.train_steps, 512, 1e-3, 1e-5)
    torch.cuda.synchronize()
    dt = time.perf_counter() - t0
    line = {"metric": "warm-start network training time", "value": dt, "unit": "s",
            "n_gpus": 1, "higher_is_better": False, "dtype": "bf16 products / f32",
            "data": "synthetic",
            "config": {"workload": f"train_{args.train_steps}_steps", "samples": n,
                       "batch": 512, "network": list(warmstart.WIDTHS)},
            "ms_per_step": dt / args.train_steps * 1e3,
            "loss_first": float(hist[0]), "loss_last": float(hist[-1])}
    print(json.dumps(line), flush=True)


def run_warmstart(args):
    """Learned warm start on the full held-out set: steady states of seeded
    training channels from the batched solver, the network trained on the
    GPU, then held-out channels (length 4W, a seed the training never saw)
    solved to r < tol from the cold, analytic and learned starts, each end
    state against an FP64 reference."""
    import torch
    torch.cuda.set_device(0)
    from paper_2010_01847_gb300 import warmstart
    st = steady_state_study(args.train_instances, args.train_steps, args.instances,
                            min(args.instances, args.reference_instances), args.tol,
                            args.check_every, args.max_steps)
    line = {
        "metric": "time to steady state (r < 1e-8), held-out channels, learned vs cold start",
        "value": st["learned"]["seconds"], "unit": "s", "n_gpus": 1, "higher_is_better": False,
        "dtype": "f32 solve / bf16 network", "data": "synthetic",
        "config": {"workload": f"warm_start_{st['held_out']}_held_out", "tol": args.tol,
                   "check_every": args.check_every,
                   "train_instances": st["train_instances"], "train_steps": args.train_steps,
                   "network": list(warmstart.WIDTHS)},
        "steady_state": st,
    }
    print(json.dumps(line), flush=True)


def main():
    args = parse()
    if args.impl == "reference":
        run_reference(args)
    elif args.workload == "batch":
        run_batch(args)
    elif args.workload == "warmstart":
        run_warmstart(args)
    elif args.workload == "train":
        run_train(args)
    elif args.workload == "d3q14":
        run_d3q14(args)
    elif args.workload == "small":
        run_small(args)
    else:
        run_native(args)


if __name__ == "__main__":
    main()
