#!/usr/bin/env python3
"""Benchmark of the batched FFT-CME integrator on GB300.

One benchmark step = one full integration of the N=512 x 256-instance detuning sweep:
reset the field from a device-resident copy, then 20000 RK4IP steps (h = 5e-4) of every
instance in FP32 (FP32 field, transforms and Kerr term; propagators computed in FP64),
replayed as one CUDA graph.  The metric is mode-steps/s = (sum of N over instances) x RK4IP
steps / time, summed over all ranks (weak scaling: every rank integrates its own 256
instances).

Extra measurements on the same JSON line:
  fp64      the same batch in FP64, and the single-instance N=64 FP64 workload;
  error     FP32 vs FP64 over all 256 instances (full horizon) and GPU vs CPU oracle on the
            oracle's bounded sample;
  roofline  the step kernel against the FP32 ALU peak (152 SMs x 128 lanes x 2 flop x clock);
  e2e       the same metric through the C ABI with host buffers (H2D of the initial field from
            pinned memory and D2H of the power spectrum inside the timed region);
  cpu_baseline  the FP64 CPU oracle (direct O(N^3) sum) on a bounded sample.
  other_workloads  (one GPU) the uneven, octave, N=4096 forward, Strang and Fig. 1 workloads
            and the N=4096 gradient in both precisions, each timed beside the headline.

`--impl reference` times the CPU oracle alone on the same metric (rank 0 only).
"""
from __future__ import annotations

import argparse
import hashlib
import json
import math
import os
import statistics
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "mode-steps/s, batched FP32 FFT-CME RK4IP vs plain FP64, at stated error; % peak"
UNIT = "mode-steps/s"
SMS = 152
FP32_LANES = 128          # FP32 FMA lanes per SM
SM_MAX_MHZ = 2070.0       # maximum SM clock of the part
FP64_NOMINAL_TFLOPS = 1.25
# What the FP64 fractions are of: the library computes FP64 transforms and RK4IP stages in 64-bit
# fixed point, so the FP64-instruction peak is a comparison and not a roof (fractions exceed 1).
FP64_BASIS = ("flop of the algorithm against the FP64-instruction peak; transforms and stages run "
              "in 64-bit fixed point on the integer pipes, so this is a comparison, not a roof")
KERNEL_SOURCES = ["cme_core.cuh", "cme_fixed.cuh", "cme_step.cuh", "cme_launch.cuh", "kern_fp32_rk4ip.cu"]


def flops_per_mode_step(N: int) -> float:
    """Algorithmic FP work of one RK4IP step per mode: 8 complex transforms of length N at
    5 N log2 N flop each, plus 80 flop of Kerr term, pump and Runge-Kutta combination."""
    return 40.0 * math.log2(N) + 80.0


def kernel_source_hash() -> str:
    h = hashlib.sha256()
    for f in KERNEL_SOURCES:
        with open(os.path.join(ROOT, "paper_1307_3428_gb300", "csrc", f), "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()[:16]


# ------------------------------------------------------------------------------ clocks
class ClockSampler:
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.gpu = gpu_index
        self.proc = None
        self.lines = []
        self.thread = None

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.gpu), f"--query-gpu={self.FIELDS}",
                 "--format=csv,noheader,nounits", "-lms", "200"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except (OSError, FileNotFoundError):
            self.proc = None
            return
        self.thread = threading.Thread(target=self._read, daemon=True)
        self.thread.start()
        # the timed region starts only once nvidia-smi is up and sampling: its start-up
        # overlapped the first timed steps of short runs (257 ms for a 0.6 ms step)
        t0 = time.perf_counter()
        while not self.lines and time.perf_counter() - t0 < 5.0 and self.proc.poll() is None:
            time.sleep(0.01)

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def stop(self):
        if self.proc is None:
            return None
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        if self.thread:
            self.thread.join(timeout=2)
        sm, mx, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            parts = [p.strip() for p in ln.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                mx.append(float(parts[2]))
            except ValueError:
                continue
            for n, v in zip(names, parts[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(n)
        if not sm:
            return None
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(mx) if mx else None,
                "samples": len(sm), "reasons": sorted(reasons)}


# ------------------------------------------------------------------------------ distributed
def dist_setup():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1:
        import torch
        import torch.distributed as dist
        backend = "nccl" if torch.cuda.is_available() else "gloo"
        if backend == "nccl":
            torch.cuda.set_device(local)
        dist.init_process_group(backend=backend)
    return world, rank, local


def barrier(world):
    if world > 1:
        import torch.distributed as dist
        dist.barrier()


def max_over_ranks(x: float, world: int) -> float:
    if world == 1:
        return x
    import torch
    import torch.distributed as dist
    dev = "cuda" if dist.get_backend() == "nccl" else "cpu"
    t = torch.tensor([x], dtype=torch.float64, device=dev)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


# ------------------------------------------------------------------------------ oracle leg
def fp32_vs_fp64_errors(f32_parts, f64_parts):
    """Per-instance relative L2 errors of the FP32 result against FP64: of the field D and of
    its power spectrum |D|^2."""
    import numpy as np
    field, power = [], []
    for a, c in zip(f32_parts, f64_parts):
        field.append(float(np.linalg.norm(a - c) / np.linalg.norm(c)))
        pa, pc = np.abs(a) ** 2, np.abs(c) ** 2
        power.append(float(np.linalg.norm(pa - pc) / np.linalg.norm(pc)))
    return field, power


def oracle_sample(target_s: float, sweep_index: int = 128, fixed_steps: int | None = None):
    """Time the FP64 direct-sum oracle on one instance of the sweep for a bounded number of
    RK4IP steps (about target_s seconds); returns (mode-steps/s, steps, seconds, field)."""
    import oracle
    from paper_1307_3428_gb300 import workloads as wl
    inst = wl.sweep512(indices=[sweep_index]).instances[0]
    h = 5e-4
    if fixed_steps is None:
        t0 = time.perf_counter()
        D = oracle.integrate(inst, h, 1, oracle.RK4IP)
        dt1 = time.perf_counter() - t0
        steps = max(1, int(target_s / max(dt1, 1e-6)))
    else:
        steps = fixed_steps
    t0 = time.perf_counter()
    D = oracle.integrate(inst, h, steps, oracle.RK4IP)
    dt = time.perf_counter() - t0
    return inst.N * steps / dt, steps, dt, D


def _oracle_instance_run(job):
    """One process of the all-cores oracle timing: `steps` RK4IP steps of sweep instance
    `index` with the direct-sum oracle as it stands."""
    index, steps = job
    import oracle
    from paper_1307_3428_gb300 import workloads as wl
    inst = wl.sweep512(indices=[index]).instances[0]
    oracle.integrate(inst, 5e-4, steps, oracle.RK4IP)
    return inst.N * steps


def oracle_all_cores(rate1: float, target_s: float):
    """The direct-sum oracle on every host core: one sweep instance per process (a spawn
    pool), each for about target_s seconds at the single-core rate rate1.  Returns
    (mode-steps/s, processes, steps per instance, seconds)."""
    import multiprocessing as mp
    from concurrent.futures import ProcessPoolExecutor
    n = os.cpu_count() or 1
    steps = max(1, int(target_s * rate1 / 512))
    # a worker that dies raises BrokenProcessPool here instead of being replaced forever
    with ProcessPoolExecutor(n, mp_context=mp.get_context("spawn")) as pool:
        list(pool.map(_oracle_instance_run, [(k, 1) for k in range(n)]))   # start-up
        t0 = time.perf_counter()
        work = sum(pool.map(_oracle_instance_run, [(k, steps) for k in range(n)]))
        dt = time.perf_counter() - t0
    return work / dt, n, steps, dt


def fft_engine_sample(target_s: float):
    """The oracle's numpy Eq. 4 engine (the paper's method on the CPU) on the whole
    256-instance sweep, vectorised over the batch, for about target_s seconds."""
    from oracle import fft_engine
    from paper_1307_3428_gb300 import workloads as wl
    w = wl.sweep512()
    fb = fft_engine.Batch(w.instances)
    t0 = time.perf_counter()
    fft_engine.rk4ip(fb, w.h, 2)
    per_step = (time.perf_counter() - t0) / 2
    steps = max(1, int(target_s / max(per_step, 1e-6)))
    t0 = time.perf_counter()
    fft_engine.rk4ip(fb, w.h, steps)
    dt = time.perf_counter() - t0
    return sum(i.N for i in w.instances) * steps / dt, steps, dt


def run_reference(args, world, rank):
    """CPU oracle arm: rank 0 times the oracle as it stands on bounded samples."""
    if rank != 0:
        return 0
    import oracle
    oracle.build()
    total = 0.0
    work = 0.0
    steps_used = None
    for k in range(args.warmup + args.steps):
        rate, steps, dt, _ = oracle_sample(args.ref_seconds, fixed_steps=steps_used)
        steps_used = steps
        if k >= args.warmup:
            total += dt
            work += 512 * steps
    value = work / total
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * total / args.steps,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
        "data": "synthetic",
        "config": {"workload": "sweep_n512_b256 (oracle sample: instance 128, "
                               f"{steps_used} RK4IP steps per bench step)",
                   "engine": "FP64 direct O(N^3) four-wave-mixing sum, C, 1 thread"},
        "cpu_baseline": {"value": value, "unit": UNIT, "cores": 1, "kind": "oracle",
                         "sample": f"1 instance (N=512, sigma index 128) x {steps_used} RK4IP "
                                   "steps per bench step"},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)
    return 0


# ------------------------------------------------------------------------------ adjoint
def run_adjoint(args, world, rank, local):
    """cme_grad on N=4096 x 16 instances, 10000 RK4IP steps, log-spectrum loss against seeded
    sech^2 targets: forward plus the discrete adjoint in FP32, with the library's choice of
    schedule (the stored trajectory where it fits) and with sqrt(n) checkpoints; the FP64
    gradient of the same run, the supported one at this configuration, beside it."""
    import numpy as np
    import torch

    import __graft_entry__
    __graft_entry__.build()
    from paper_1307_3428_gb300 import cme
    from paper_1307_3428_gb300 import workloads as wl

    torch.cuda.set_device(local)
    w = wl.adjoint4096()
    nsteps = args.inner_steps or w.nsteps
    N, B = 4096, len(w.instances)
    T = wl.sech2_target(N, B).reshape(-1)
    insts = [cme.Instance.from_workload(i) for i in w.instances]
    D0 = np.concatenate([i.D0 for i in w.instances])
    d0 = torch.from_numpy(D0.view(np.float64).copy()).cuda()

    flush = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")   # > 129 MB L2

    def timed(prec, n, reps, warmup, sampler=None, budget=-1):
        """Mean device time of `reps` gradients (CUDA events on the batch's stream, L2 flushed
        before each), after `warmup` untimed ones (the first allocates the scratch), and the
        schedule the library took (budget: cme_set_grad_memory)."""
        b = cme.Batch(insts, precision=prec, cluster=args.cluster)
        b.set_grad_memory(budget)
        stream = torch.cuda.ExternalStream(b.stream)
        for _ in range(warmup):
            b.set_state_device(d0.data_ptr())
            b.grad(w.h, n, T)
        ts = []
        if sampler:
            sampler.start()
        for _ in range(reps):
            flush.zero_()
            torch.cuda.synchronize()
            e0 = torch.cuda.Event(enable_timing=True)
            e1 = torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            b.set_state_device(d0.data_ptr())
            g = b.grad(w.h, n, T)              # synchronises
            e1.record(stream)
            e1.synchronize()
            ts.append(e0.elapsed_time(e1) * 1e-3)
        clocks = sampler.stop() if sampler else None
        sched = b.last_grad_schedule
        b.close()
        return sum(ts) / len(ts), g, clocks, sched

    launches0 = cme.kernel_launches()
    t32, g32, clocks, sched32 = timed(cme.FP32, nsteps, args.steps, args.warmup,
                                      ClockSampler(local))
    launches = (cme.kernel_launches() - launches0) // (args.steps + args.warmup)
    # the FP64 gradient of the same workload, full horizon: the supported gradient of this
    # configuration and the reference of the FP32 gradient's error
    t64, g64, _, sched64 = timed(cme.FP64, nsteps, 1, 1)
    mode_steps = N * B * nsteps
    peak = SMS * FP32_LANES * 2 * SM_MAX_MHZ * 1e6 / 1e12

    def grad_flops(sched):
        """Algorithmic work of one gradient: the forward step's 8 transforms of 5 N log2 N flop
        plus ~80 pointwise flop per mode-step, once for the forward pass, once for the backward
        pass (4 vector-Jacobian products of 2 transforms each), and once more for the
        recomputation of the checkpoint schedule."""
        return mode_steps * (2 if sched == "stored" else 3) * (8 * 5 * math.log2(N) + 80)

    flops = grad_flops(sched32)
    achieved = flops / t32 / 1e12
    # the other schedule of the same FP32 gradient, for comparison
    tck, _, _, schedck = timed(cme.FP32, nsteps, 2, 1, budget=0)
    assert schedck == "checkpoint"
    achieved_ck = grad_flops("checkpoint") / tck / 1e12
    rel = lambda a, b: float(np.max(np.abs(np.asarray(a) - np.asarray(b))) /
                             np.max(np.abs(np.asarray(b))))
    line = {
        "metric": "gradient mode-steps/s (forward + discrete adjoint), log-spectrum loss",
        "value": mode_steps / t32, "unit": UNIT, "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": t32 * 1e3, "higher_is_better": True,
        "scaling": "weak",
        "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": {"workload": f"adjoint_n4096_b16: N=4096 x 16, {nsteps} RK4IP steps of "
                               f"h=2e-4, {sched32} schedule, sech^2 log-spectrum targets",
                   "cluster": args.cluster or "library choice",
                   "l2": "flushed between timed steps (256 MiB write)"},
        "clocks": clocks,
        "schedule": sched32,
        "roofline": {"bound": "alu", "achieved": achieved, "peak": peak, "unit": "TFLOP/s",
                     "frac": achieved / peak, "traffic": None,
                     "basis": ("2 x (8 transforms of 5 N log2 N + 80) flop per mode-step: forward "
                               "and backward, the stored trajectory recomputing nothing"
                               if sched32 == "stored" else
                               "3 x (8 transforms of 5 N log2 N + 80) flop per mode-step: forward, "
                               "checkpoint recomputation, backward")},
        "checkpoint_schedule": {
            "what": "the same FP32 gradient with cme_set_grad_memory(0): sqrt(n) checkpoints, "
                    "each segment recomputed on a second stream",
            "value": mode_steps / tck, "ms": tck * 1e3,
            "roofline": {"bound": "alu", "achieved": achieved_ck, "peak": peak,
                         "unit": "TFLOP/s", "frac": achieved_ck / peak,
                         "basis": "3 x (8 transforms of 5 N log2 N + 80) flop per mode-step"}},
        "fp64": {"value": N * B * nsteps / t64, "steps": nsteps, "ms": t64 * 1e3,
                 "schedule": sched64,
                 "roofline": {"bound": "alu", "unit": "TFLOP/s", "peak": FP64_NOMINAL_TFLOPS,
                              "achieved": grad_flops(sched64) / t64 / 1e12,
                              "frac": grad_flops(sched64) / t64 / 1e12 / FP64_NOMINAL_TFLOPS,
                              "basis": FP64_BASIS},
                 "note": "the FP64 gradient is the supported one at this configuration: the FP32 "
                         "gradients of dL/dD2 and dL/dD3 are dominated by noise-floor modes that "
                         "FP32 transforms do not resolve (error.full_horizon)"},
        "error": {"full_horizon": {
            "steps": nsteps,
            "what": "FP32 gradient against the FP64 gradient of the same run: max over the "
                    "batch of |difference| / max |FP64 value|",
            "loss": rel(g32["loss"], g64["loss"]), "d_sigma": rel(g32["d_sigma"], g64["d_sigma"]),
            "d_A_in": rel(g32["d_A_in"], g64["d_A_in"]), "d_D2": rel(g32["d_D2"], g64["d_D2"]),
            "d_D3": rel(g32["d_D3"], g64["d_D3"]), "d_D0": rel(g32["d_D0"], g64["d_D0"])}},
        "gpu_launches": int(launches),
    }
    if rank == 0:
        print(json.dumps(line), flush=True)
    return 0


# ------------------------------------------------------------------------------ large N
# Algorithmic bytes per mode-step of the four-step RK4IP path (FP32, 8 B per complex value):
# per RK stage the row kernel reads Y and writes Z (16 B); the column kernel reads Z and the
# field, and the accumulator S, the propagators E, e1 or e2 as its stage needs them, and writes
# S and Y (stages 0..2: 48, 56, 56 B); the last stage reads Z, D, S, the compensation word and
# e2 and writes D, the compensation word and Y of the next step (64 B).  Constant twiddle-table
# reads are not counted.
LARGE_BYTES_PER_MODE_STEP = 4 * 16 + 48 + 56 + 56 + 64


def measured_peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        with open(path) as fh:
            return json.load(fh), "measured"
    return {"hbm_gbs": 6800.0}, "fallback"


def large_n_roofline(args, sizes, nsteps, kern_ms, cme, alu):
    """HBM and L2 roofline of the large-N (four-step) run: algorithmic bytes per step over the
    device time of a step, against the measured HBM copy bandwidth and the library's L2-resident
    copy bandwidth (cme_l2_peak on 2 x 16 MiB, measured here)."""
    byts = sum(sizes) * LARGE_BYTES_PER_MODE_STEP * nsteps
    achieved = byts / (kern_ms * 1e-3) / 1e9
    peaks, kind = measured_peaks()
    hbm = float(peaks["hbm_gbs"])
    l2 = cme.l2_peak(32 << 20) / 1e9
    traffic = None
    tfile = os.path.join(ROOT, "profiles", "traffic.json")
    if os.path.exists(tfile):
        with open(tfile) as fh:
            ent = json.load(fh).get("large_n_fp32_octave")
        if ent and ent.get("source_hash") == large_source_hash() and not args.radix:
            traffic = ent.get("dram_bytes_per_step")
    return {"bound": "hbm", "achieved": achieved, "peak": hbm, "unit": "GB/s",
            "frac": achieved / hbm, "traffic": traffic,
            "traffic_basis": "ncu dram__bytes_read.sum + dram__bytes_write.sum over the 8 "
                             "kernels of one step (per step, not per launch)",
            "peak_basis": f"MEASURED_PEAKS.json hbm_gbs ({kind})",
            "bytes_per_mode_step": LARGE_BYTES_PER_MODE_STEP,
            "l2": {"achieved": achieved, "peak": l2, "unit": "GB/s", "frac": achieved / l2,
                   "peak_basis": "cme_l2_peak: copies between two L2-resident 16 MiB buffers, "
                                 "this run"},
            "alu": {k: alu[k] for k in ("achieved", "peak", "unit", "frac")},
            "kernel": "large_row_kernel + large_col_kernel (8 per RK4IP step)"}


LARGE_SOURCES = ["cme_core.cuh", "cme_fixed.cuh", "cme_step.cuh", "cme_launch.cuh", "cme_large.cuh",
                 "cme_large_launch.cuh", "kern_large_fp32.cu", "kern_large_fp32_scalar.cu"]


def large_source_hash() -> str:
    h = hashlib.sha256()
    for f in LARGE_SOURCES:
        with open(os.path.join(ROOT, "paper_1307_3428_gb300", "csrc", f), "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()[:16]


# ------------------------------------------------------------------------------ other workloads
def other_workloads(cme, wl, torch, flush, reps: int = 2) -> dict:
    """The other workloads measured beside the headline in the same run (one GPU): each batch on
    the library's default launch plan, one untimed run (graph capture, scratch allocation), then
    `reps` runs timed with CUDA events on the batch's stream, L2 flushed before each.  A workload
    that fails reports its error and leaves the others standing."""
    import types

    import numpy as np
    peak32 = SMS * FP32_LANES * 2 * SM_MAX_MHZ * 1e6 / 1e12
    out = {"how": f"library default plan, 1 untimed run, mean of {reps} timed runs (CUDA events "
                  "on the batch's stream, reset of the field included, L2 flushed before each)"}

    def timed_runs(b, d0, h, n):
        stream = torch.cuda.ExternalStream(b.stream)
        b.set_state_device(d0.data_ptr())
        b.step(h, n)
        b.synchronize()
        ts = []
        for _ in range(reps):
            flush.zero_()
            torch.cuda.synchronize()
            e0 = torch.cuda.Event(enable_timing=True)
            e1 = torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            b.set_state_device(d0.data_ptr())
            b.step(h, n)
            e1.record(stream)
            e1.synchronize()
            ts.append(e0.elapsed_time(e1))
        return statistics.mean(ts)

    def forward(name, w, integ=cme.RK4IP, flop_fn=None, large=False):
        try:
            insts = [cme.Instance.from_workload(i) for i in w.instances]
            b = cme.Batch(insts, precision=cme.FP32, integrator=integ, use_graph=True)
            D0 = np.concatenate([i.D0 for i in w.instances])
            d0 = torch.from_numpy(D0.view(np.float64).copy()).cuda()
            ms = timed_runs(b, d0, w.h, w.nsteps)
            sizes = [i.N for i in w.instances]
            ent = {"workload": w.name, "value": sum(sizes) * w.nsteps / (ms * 1e-3),
                   "unit": UNIT, "ms_per_run": ms, "steps": w.nsteps, "instances": len(sizes),
                   "dtype": "f32", "launch_plan": b.plan(0)}
            if flop_fn is not None:
                f = sum(n * flop_fn(n) for n in sizes) * w.nsteps / (ms * 1e-3) / 1e12
                ent["roofline"] = {"bound": "alu", "achieved": f, "peak": peak32,
                                   "unit": "TFLOP/s", "frac": f / peak32}
            if large:
                alu = ent.pop("roofline")
                ent["roofline"] = large_n_roofline(types.SimpleNamespace(radix=0), sizes,
                                                   w.nsteps, ms, cme, alu)
            b.close()
            out[name] = ent
        except Exception as e:   # context beside the headline: the line stands without it
            out[name] = {"error": f"{type(e).__name__}: {e}"}

    forward("uneven", wl.uneven(), flop_fn=flops_per_mode_step)
    forward("octave", wl.octave(), flop_fn=flops_per_mode_step, large=True)
    forward("forward4096", wl.adjoint4096(), flop_fn=flops_per_mode_step)
    forward("strang_sweep512", wl.sweep512(), integ=cme.STRANG,
            flop_fn=lambda n: 10.0 * math.log2(n) + 40.0)
    forward("fig1", wl.fig1(), integ=cme.STRANG)

    # the gradient workload: N = 4096 x 16, 10000 steps, both precisions, library schedule
    try:
        w = wl.adjoint4096()
        N, B = 4096, len(w.instances)
        T = wl.sech2_target(N, B).reshape(-1)
        insts = [cme.Instance.from_workload(i) for i in w.instances]
        D0 = np.concatenate([i.D0 for i in w.instances])
        d0 = torch.from_numpy(D0.view(np.float64).copy()).cuda()
        for prec, key in ((cme.FP32, "adjoint_fp32"), (cme.FP64, "adjoint_fp64")):
            b = cme.Batch(insts, precision=prec)
            stream = torch.cuda.ExternalStream(b.stream)
            b.set_state_device(d0.data_ptr())
            b.grad(w.h, w.nsteps, T)
            flush.zero_()
            torch.cuda.synchronize()
            e0 = torch.cuda.Event(enable_timing=True)
            e1 = torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            b.set_state_device(d0.data_ptr())
            b.grad(w.h, w.nsteps, T)
            e1.record(stream)
            e1.synchronize()
            ms = e0.elapsed_time(e1)
            sched = b.last_grad_schedule
            b.close()
            f = (N * B * w.nsteps * (2 if sched == "stored" else 3) *
                 (8 * 5 * math.log2(N) + 80) / (ms * 1e-3) / 1e12)
            pk = peak32 if prec == cme.FP32 else FP64_NOMINAL_TFLOPS
            out[key] = {"workload": w.name, "value": N * B * w.nsteps / (ms * 1e-3),
                        "unit": "gradient mode-steps/s", "ms_per_gradient": ms,
                        "steps": w.nsteps, "schedule": sched,
                        "dtype": "f32" if prec == cme.FP32 else "f64",
                        "roofline": {"bound": "alu", "achieved": f, "peak": pk,
                                     "unit": "TFLOP/s", "frac": f / pk,
                                     **({} if prec == cme.FP32 else {"basis": FP64_BASIS})},
                        "timed": "1 untimed gradient, then 1 timed"}
    except Exception as e:
        out["adjoint"] = {"error": f"{type(e).__name__}: {e}"}
    return out


# ------------------------------------------------------------------------------ GPU arm
def run_gpu(args, world, rank, local):
    import numpy as np
    import torch

    import __graft_entry__
    __graft_entry__.build()
    from paper_1307_3428_gb300 import cme
    from paper_1307_3428_gb300 import workloads as wl

    from paper_1307_3428_gb300 import shard

    torch.cuda.set_device(local)
    if args.workload == "sweep512":
        # weak scaling: the global batch is `world` replicas of the sweep with independent
        # noise; each rank integrates its own shard (256 instances) of it
        w = wl.sweep512()
        global_insts = [i for r in range(world)
                        for i in (wl.sweep512(seed_offset=256 * r) if r else w).instances]
    elif args.workload == "uneven":
        w = wl.uneven()
    elif args.workload == "plain64":
        w = wl.plain64()
    elif args.workload == "octave":
        w = wl.octave()
    elif args.workload == "fig1":
        w = wl.fig1()
    elif args.workload == "forward4096":
        w = wl.adjoint4096()   # the gradient workload's instances, forward steps only
    else:
        raise SystemExit(f"unknown workload {args.workload}")
    strang = args.strang or args.workload == "fig1"   # Fig. 1 is a split-step run
    headline = args.workload == "sweep512"
    if not headline:
        global_insts = list(w.instances) * world   # replicas of the whole workload per rank
    sizes = [i.N for i in w.instances]
    N = max(sizes)
    count = len(w.instances)
    nsteps = args.inner_steps or w.nsteps
    mode_steps = sum(sizes) * nsteps

    prec_main = cme.FP64 if args.workload == "plain64" else cme.FP32
    # this rank's shard of the global batch (instances are independent: no exchange while
    # stepping; results cross ranks only through the host gather below)
    sb = shard.ShardedBatch(global_insts, world=world, rank=rank, precision=prec_main,
                            use_graph=True, radix=args.radix, inst_per_cta=args.inst_per_cta,
                            persistent=args.persistent, cluster=args.cluster,
                            integrator=cme.STRANG if strang else cme.RK4IP)
    assert len(sb.local) == count, "one workload's worth of instances per rank"
    w.instances = list(sb.local)
    insts = [cme.Instance.from_workload(i) for i in w.instances]
    b32 = sb.batch
    plan = None
    if args.autotune:
        plan = b32.autotune(w.h, probe_steps=200)
    stream = torch.cuda.ExternalStream(b32.stream)
    D0 = np.concatenate([i.D0 for i in w.instances])
    d0_dev = torch.from_numpy(D0.view(np.float64).copy()).cuda()
    flush = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")   # > 129 MB L2

    def one_step(batch):
        batch.set_state_device(d0_dev.data_ptr())
        batch.step(w.h, nsteps)

    # warm-up (also builds the graph)
    for _ in range(args.warmup):
        one_step(b32)
    torch.cuda.synchronize()

    def timed_loop():
        sampler = ClockSampler(local)
        launches0 = cme.kernel_launches()
        k_ms = []
        barrier(world)
        torch.cuda.synchronize()
        sampler.start()
        t_wall0 = time.perf_counter()
        total_ms = 0.0
        for _ in range(args.steps):
            flush.zero_()                       # evict L2 between timed steps (not timed)
            torch.cuda.synchronize()
            e0 = torch.cuda.Event(enable_timing=True)
            e1 = torch.cuda.Event(enable_timing=True)
            e2 = torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            b32.set_state_device(d0_dev.data_ptr())
            e1.record(stream)
            b32.step(w.h, nsteps)
            e2.record(stream)
            e2.synchronize()
            total_ms += e0.elapsed_time(e2)
            k_ms.append(e1.elapsed_time(e2))
        torch.cuda.synchronize()
        barrier(world)
        wall = time.perf_counter() - t_wall0
        return total_ms, k_ms, wall, sampler.stop(), cme.kernel_launches() - launches0

    total_ms, k_ms, wall, clocks, launches = timed_loop()
    # The clock record cannot show another context time-slicing this GPU.  The library's FMA
    # microbenchmark can: far below the derived FMA peak (here once 21.7 of 80.5 TFLOP/s, with
    # every step 4.8x slow and clocks at their maximum), the timing is repeated once.
    fma_meas = cme.fma_peak(prec_main) / 1e12
    fma_derived = (SMS * FP32_LANES * 2 * SM_MAX_MHZ * 1e6 / 1e12 if prec_main == cme.FP32
                   else FP64_NOMINAL_TFLOPS)
    retimed = False
    if prec_main == cme.FP32 and fma_meas < 0.6 * fma_derived:
        total_ms, k_ms, wall, clocks, launches = timed_loop()
        fma_meas = cme.fma_peak(prec_main) / 1e12
        retimed = True
    step_ms = max_over_ranks(total_ms / args.steps, world)
    value = world * mode_steps / (step_ms * 1e-3)
    # the global batch's final spectra gathered on rank 0, in global instance order
    gathered = sb.spectrum(cme.POWER)
    gather = None
    if rank == 0:
        gather = {"instances": len(global_insts), "modes": int(gathered.size),
                  "all_finite": bool(np.all(np.isfinite(gathered)))}

    # roofline of the step kernel (one graph node per replay)
    kern_ms = statistics.mean(k_ms)
    flops = sum(n * flops_per_mode_step(n) for n in sizes) * nsteps
    if strang:
        flops = sum(n * (10.0 * math.log2(n) + 40.0) for n in sizes) * nsteps
    achieved = flops / (kern_ms * 1e-3) / 1e12
    peak = SMS * FP32_LANES * 2 * SM_MAX_MHZ * 1e6 / 1e12
    traffic = None
    tfile = os.path.join(ROOT, "profiles", "traffic.json")
    if os.path.exists(tfile):
        with open(tfile) as fh:
            tj = json.load(fh)
        ent = tj.get("step_kernel_fp32_n512")
        # the captured kernel must be the one timed here (same sources, same workload shape)
        if (headline and ent and ent.get("source_hash") == kernel_source_hash()
                and not args.radix and not args.strang):
            traffic = ent.get("dram_bytes_per_launch")
    if prec_main == cme.FP64:
        peak = FP64_NOMINAL_TFLOPS
    # fma_meas: the same FMA rate measured by the library's FMA-chain microbenchmark (context:
    # the derived peak above is the denominator)
    roofline = {"bound": "alu", "achieved": achieved, "peak": peak, "unit": "TFLOP/s",
                "frac": achieved / peak, "traffic": traffic,
                "measured_fma_tflops": fma_meas, "frac_of_measured_fma": achieved / fma_meas,
                "kernel": (f"step_kernel<float, 9, {args.radix or 8}, RK4IP>" if headline
                           else f"{args.workload} step kernel(s)"),
                "peak_basis": ("152 SMs x 128 FP32 lanes x 2 flop x 2070 MHz (derived)"
                               if prec_main == cme.FP32 else
                               "GB300 nominal FP64 1.25 TFLOP/s; " + FP64_BASIS)}
    if max(sizes) > 4096 and not strang:
        # The four-step large-N path moves its state, propagators and inter-pass buffers
        # through L2 every step: it is bound by memory, not by the FP32 ALUs.
        roofline = large_n_roofline(args, sizes, nsteps, kern_ms, cme, roofline)

    # FP32 result vs FP64 over the whole batch, full horizon
    fin32 = b32.get_state()
    fp64 = {}
    error = {}
    if headline and not args.skip_fp64:
        b64 = cme.Batch(insts, precision=cme.FP64, use_graph=True)
        one_step(b64)                                 # warm-up / graph build
        torch.cuda.synchronize()
        s64 = torch.cuda.ExternalStream(b64.stream)
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        b64.set_state_device(d0_dev.data_ptr())
        e0.record(s64)
        b64.step(w.h, nsteps)
        e1.record(s64)
        e1.synchronize()
        ms64 = e0.elapsed_time(e1)
        fin64 = b64.get_state()
        errs, errs_p = fp32_vs_fp64_errors(b32.split(fin32), b64.split(fin64))
        # plain single-instance FP64 (N=64, 2000 steps)
        p = wl.plain64()
        bp = cme.Batch([cme.Instance.from_workload(p.instances[0])], precision=cme.FP64,
                       use_graph=True)
        bp.step(p.h, p.nsteps)
        bp.synchronize()
        sp = torch.cuda.ExternalStream(bp.stream)
        pd0 = torch.from_numpy(p.instances[0].D0.view(np.float64).copy()).cuda()
        tp = []
        for _ in range(3):
            e0 = torch.cuda.Event(enable_timing=True)
            e1 = torch.cuda.Event(enable_timing=True)
            bp.set_state_device(pd0.data_ptr())
            e0.record(sp)
            bp.step(p.h, p.nsteps)
            e1.record(sp)
            e1.synchronize()
            tp.append(e0.elapsed_time(e1))
        f_plain = 64 * p.nsteps * flops_per_mode_step(64) / (min(tp) * 1e-3) / 1e12
        f_batch = flops / (ms64 * 1e-3) / 1e12
        fp64 = {
            "batched_value": mode_steps / (ms64 * 1e-3), "batched_ms": ms64,
            "batched_roofline": {"bound": "alu", "achieved": f_batch, "unit": "TFLOP/s",
                                 "peak": FP64_NOMINAL_TFLOPS, "frac": f_batch / FP64_NOMINAL_TFLOPS,
                                 "basis": FP64_BASIS},
            "plain_n64_value": 64 * p.nsteps / (min(tp) * 1e-3), "plain_n64_ms": min(tp),
            "plain_n64_roofline": {
                "bound": "alu", "achieved": f_plain, "unit": "TFLOP/s",
                "peak": FP64_NOMINAL_TFLOPS, "frac": f_plain / FP64_NOMINAL_TFLOPS,
                "basis": "64 modes x 2000 steps x (40 log2 64 + 80) flop; one instance of 32 "
                         "threads: latency of one thread's chain of integer instructions"},
            "unit": UNIT,
            "fp32_speedup_vs_batched_fp64": ms64 / kern_ms,
            "fp32_speedup_vs_plain_fp64": value / world / (64 * p.nsteps / (min(tp) * 1e-3)),
        }
        error = {"fp32_vs_fp64_rel_l2_max": max(errs), "fp32_vs_fp64_rel_l2_median":
                 statistics.median(errs), "instances": len(errs), "bound_fp32": 1e-4,
                 "fp32_vs_fp64_spectrum_rel_l2_max": max(errs_p),
                 "fp32_vs_fp64_spectrum_rel_l2_median": statistics.median(errs_p)}

    # end to end through the C ABI with host buffers
    pinned_in = torch.from_numpy(D0.view(np.float64).copy()).pin_memory()
    host_in = pinned_in.numpy()
    spec = torch.empty(sum(sizes), dtype=torch.float64).pin_memory().numpy()
    import ctypes
    lib = cme.load()
    dp = ctypes.POINTER(ctypes.c_double)
    e2e_steps = max(1, min(args.steps, 5))
    torch.cuda.synchronize()
    barrier(world)
    t0 = time.perf_counter()
    for _ in range(e2e_steps):
        cme._check(lib.cme_set_state(b32.handle, host_in.ctypes.data_as(dp), cme.HOST))
        cme._check(lib.cme_step(b32.handle, w.h, nsteps))
        cme._check(lib.cme_spectrum(b32.handle, -1, cme.POWER, spec.ctypes.data_as(dp)))
    e2e_s = max_over_ranks((time.perf_counter() - t0) / e2e_steps, world)
    e2e = {"value": world * mode_steps / e2e_s, "unit": UNIT,
           "h2d_bytes_per_step": int(host_in.nbytes), "d2h_bytes_per_step": int(spec.nbytes)}

    others = None
    if headline and world == 1 and not args.skip_others:
        others = other_workloads(cme, wl, torch, flush)

    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": step_ms, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": {"workload": (f"sweep_n512_b256: N=512 x {count} instances per GPU, sigma "
                                f"-2..10, A_in=2.5, D2=0.02, {nsteps} RK4IP steps of h=5e-4, "
                                "FP32 field with FP64-derived propagators, one CUDA graph")
                   if headline else f"{w.name}: {w.description}, {nsteps} steps, "
                                    f"{count} instances",
                   "l2": "flushed between timed steps (256 MiB write)",
                   "parallelism": f"replicas x{world}", "global_instances": world * count},
        "roofline": roofline,
        "gpu_launches": int(launches),
        "clocks": clocks,
        "e2e": e2e,
        "fp64": fp64,
        "error": error,
        "wall_s_timed": wall,
        "gather": gather,
    }
    if others is not None:
        line["other_workloads"] = others
    if retimed:
        line["retimed_after_low_fma_rate"] = True
    if plan is not None:
        line["config"]["plan"] = plan
    elif len(set(sizes)) == 1:
        line["config"]["launch_plan"] = b32.plan(0)
    if args.workload == "fig1":
        # the whole ensemble (4 runs of tau~ = 128 pi) in FP64 as well; the paper quotes 54 s
        # for it on a desktop computer (context, not a target)
        b64 = cme.Batch(insts, precision=cme.FP64, integrator=cme.STRANG, use_graph=True)
        one_step(b64)
        torch.cuda.synchronize()
        s64 = torch.cuda.ExternalStream(b64.stream)
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        b64.set_state_device(d0_dev.data_ptr())
        e0.record(s64)
        b64.step(w.h, nsteps)
        e1.record(s64)
        e1.synchronize()
        ms64 = e0.elapsed_time(e1)
        fin64 = b64.get_state()
        errs = [float(np.linalg.norm(a - c) / np.linalg.norm(c))
                for a, c in zip(b32.split(fin32)[:3], b64.split(fin64)[:3])]
        line["fp64"] = {"value": mode_steps / (ms64 * 1e-3), "ensemble_ms": ms64, "unit": UNIT}
        line["error"] = {"fp32_vs_fp64_rel_l2_max_settled": max(errs),
                         "note": "f0 = 4 sqrt(2) is chaotic and left out of the comparison"}
        line["paper_context"] = {"ensemble_s": 54.0, "fp32_ensemble_ms": step_ms,
                                 "what": "Fig. 1 ensemble of four split-step runs on a desktop "
                                         "computer (step size not stated)"}
    if not headline:
        line["dtype"] = "f64" if prec_main == cme.FP64 else "f32"

    if headline and rank == 0 and world == 1 and not args.skip_cpu_baseline:
        rate, steps, dt, Dref = oracle_sample(args.ref_seconds)
        # the GPU on exactly the oracle's sample
        one = cme.Batch([insts[128]], precision=cme.FP32)
        one.step(w.h, steps)
        one64 = cme.Batch([insts[128]], precision=cme.FP64)
        one64.step(w.h, steps)
        e32 = float(np.linalg.norm(one.get_state() - Dref) / np.linalg.norm(Dref))
        e64 = float(np.linalg.norm(one64.get_state() - Dref) / np.linalg.norm(Dref))
        line["cpu_baseline"] = {"value": rate, "unit": UNIT, "cores": 1, "kind": "oracle",
                                "sample": f"1 instance (N=512, sigma index 128) x {steps} RK4IP "
                                          f"steps, FP64 direct O(N^3) sum, {dt:.1f} s"}
        line["error"]["gpu_vs_oracle_sample"] = {"fp32": e32, "fp64": e64, "steps": steps}
        # context beside the single-core baseline: the direct oracle on every host core, and
        # the oracle's numpy Eq. 4 engine (numpy's FFT runs on one thread)
        try:
            r_all, procs, st_all, dt_all = oracle_all_cores(rate, args.ref_seconds)
            all_cores = {
                "value": r_all, "unit": UNIT, "cores": procs, "kind": "oracle",
                "sample": f"{procs} sweep instances, one per process, x {st_all} RK4IP steps, "
                          f"FP64 direct O(N^3) sum, {dt_all:.1f} s"}
        except Exception as e:   # context only: the line stands without it
            all_cores = {"unavailable": f"{type(e).__name__}: {e}"}
        r_fft, st_fft, dt_fft = fft_engine_sample(args.ref_seconds / 2)
        line["cpu_context"] = {
            "direct_oracle_all_cores": all_cores,
            "eq4_engine_one_core": {
                "value": r_fft, "unit": UNIT, "cores": 1, "kind": "oracle (numpy Eq. 4 engine)",
                "sample": f"256 x 512 sweep x {st_fft} RK4IP steps, FP64 numpy.fft, "
                          f"{dt_fft:.1f} s"}}
    if rank == 0:
        print(json.dumps(line), flush=True)
    return 0


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="gpu", choices=["gpu", "reference"])
    ap.add_argument("--inner-steps", type=int, default=0,
                    help="RK4IP steps per benchmark step (default: the workload's 20000)")
    ap.add_argument("--ref-seconds", type=float, default=10.0)
    ap.add_argument("--radix", type=int, default=0, help="field values per thread (0: default)")
    ap.add_argument("--inst-per-cta", type=int, default=0, help="instances per block (0: default)")
    ap.add_argument("--workload", default="sweep512",
                    choices=["sweep512", "uneven", "plain64", "octave", "adjoint", "fig1",
                             "forward4096"],
                    help="sweep512 is the headline workload; the others are secondary records")
    ap.add_argument("--persistent", type=int, default=0, choices=[0, 1, 2])
    ap.add_argument("--cluster", type=int, default=0, choices=[0, 1, 2, 4, 8],
                    help="blocks per instance for N = 2048 / 4096 (0: library choice)")
    ap.add_argument("--autotune", action="store_true")
    ap.add_argument("--strang", action="store_true", help="Strang split step instead of RK4IP")
    ap.add_argument("--skip-fp64", action="store_true")
    ap.add_argument("--skip-cpu-baseline", action="store_true")
    ap.add_argument("--skip-others", action="store_true",
                    help="leave out the other workloads measured beside the headline")
    args = ap.parse_args()
    if args.warmup < 3:
        ap.error("--warmup must be >= 3")
    world, rank, local = dist_setup()
    try:
        if args.impl == "reference":
            return run_reference(args, world, rank)
        if args.workload == "adjoint":
            return run_adjoint(args, world, rank, local)
        return run_gpu(args, world, rank, local)
    finally:
        if world > 1:
            import torch.distributed as dist
            dist.destroy_process_group()


if __name__ == "__main__":
    sys.exit(main())
