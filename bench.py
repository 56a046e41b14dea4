#!/usr/bin/env python3
"""Benchmark of the GPU PIC-MCC time step: particle-steps/s on one GB300 (or N
independent replicas under torchrun), with the HBM roofline fraction of the mover
kernel, the end-to-end rate through the C ABI with host buffers, and the FP64 CPU
oracle timed on the host cores.

Workload (default): the large bounded plasma, 65,536 cells, 1,500 particles per cell
per species, electrons + ions (196,608,000 particles), FP32 particle state, fixed-point
deposit, FP64 integer-exact Poisson solve, elastic + charge-exchange null-collision
MCC, counting sort every 20 steps.  The particle state (4.7 GB) is far larger than
L2, so no L2 flush is needed between steps.

Usage: python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]
"""
from __future__ import annotations

import argparse
import json
import math
import os
import statistics
import subprocess
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

from paper_2404_10270_gb300 import workloads as W  # noqa: E402

METRIC = "particle-steps/s (gather+push+MCC+deposit), FP32 vs FP64 form, % HBM roofline"
UNIT = "particle-steps/s"
# algorithmic bytes per particle-step of the mover (B = 0, constant collision
# frequency): read cell word, off, vx (12 B), write them (12 B) in FP32; read and write
# cell word (4) off (8) vx (8) in FP64.  The id is read only at collision-clock events
# (about one step in 127) and vy/vz only on collisions and wall hits.
MOVER_BYTES = {"f32": 24, "f64": 40}
# FP64 work of the FP64 form per particle-step: gather, one fused multiply-add on the
# node pair; push, one add; move, f + u.  (The add that takes f' - floor(f') is needed
# only by a particle that crossed a cell edge, a few per cent of them: not counted.)
# Peak: 2 FP64 instructions per SM per cycle (ncu's peak_sustained of the dfma pipe on
# this GPU) x 152 SMs x 2.07 GHz.  The form is reported against whichever of the FP64
# pipe and HBM it uses the larger fraction of.
FP64_OPS_PER_PARTICLE = 3
# With B != 0 (Boris) in the x-y plane, as in every workload here: gather 1 (of half the
# acceleration), v + a/2 1, the two cross-product updates 4 x 2 fused multiply-adds, the last
# half step 1, the move 1.
FP64_OPS_PER_PARTICLE_BORIS = 12
FP64_PEAK_INSTR_PER_S = 2 * 152 * 2.07e9
# Mover threads per block of the 196.6 M-particle workload in both forms (the step that
# ends a sort cycle has its own block size, 128): with warps that take chunks of tiles, small
# blocks follow the store most closely (0.761 / 0.764 / 0.779 ms per step at 128 / 256 / 512 in
# FP32 over a sort cycle, 1.52 / 1.55 / 1.63 in FP64).  The subcycled variant and the paper's
# test case keep 256.
LARGE_BLOCK = 128


def peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as fh:
            p = json.load(fh)
        return float(p["hbm_gbs"]), "measured"
    except Exception:
        return 6800.0, "fallback"


def profiled_traffic(kernel: str, precision: str):
    """DRAM bytes per particle of the mover from the committed ncu summary, if one
    matches the current kernel source (else None)."""
    path = os.path.join(ROOT, "profiles", "mover_traffic.json")
    try:
        with open(path) as fh:
            d = json.load(fh)
        ent = d[precision]
        from paper_2404_10270_gb300.build import source_key
        if ent.get("source_key") != source_key():
            return None
        return float(ent["dram_bytes_per_particle"])
    except Exception:
        return None


class Clocks:
    """nvidia-smi sampling of SM clocks and throttle reasons during the timed region."""

    FIELDS = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.samples = []
        self._stop = threading.Event()
        self._t = None

    def _run(self):
        while not self._stop.is_set():
            try:
                out = subprocess.run(["nvidia-smi", "-i", str(self.index),
                                      "--query-gpu=" + self.FIELDS, "--format=csv,noheader,nounits"],
                                     capture_output=True, text=True, timeout=5).stdout.strip()
                if out:
                    self.samples.append([x.strip() for x in out.split(",")])
            except Exception:
                pass
            self._stop.wait(0.2)

    def __enter__(self):
        self._t = threading.Thread(target=self._run, daemon=True)
        self._t.start()
        return self

    def __exit__(self, *exc):
        self._stop.set()
        self._t.join(timeout=10)

    def summary(self):
        if not self.samples:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["unsampled"]}
        sm = [float(s[0]) for s in self.samples if s[0].replace(".", "").isdigit()]
        mx = [float(s[1]) for s in self.samples if s[1].replace(".", "").isdigit()]
        reasons = set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for s in self.samples:
            for name, v in zip(names, s[4:8]):
                if v.lower() == "active":
                    reasons.add(name)
        return {"sm_mhz": statistics.median(sm) if sm else None,
                "sm_max_mhz": max(mx) if mx else None, "reasons": sorted(reasons),
                "samples": len(self.samples)}


class NvmlClocks:
    """NVML (through ctypes) sampling of the SM clock, its maximum and the clock-event
    reasons every few milliseconds during the timed region, so that a region of a few
    tens of milliseconds still gets many samples.  Raises if NVML is unavailable."""

    REASONS = {0x4: "sw_power_cap", 0x8: "hw_slowdown", 0x20: "sw_thermal_slowdown",
               0x40: "hw_thermal_slowdown", 0x80: "hw_power_brake_slowdown"}

    def __init__(self, dev: int, interval_s: float = 0.002):
        import ctypes as C
        self.C = C
        L = C.CDLL("libnvidia-ml.so.1")
        if L.nvmlInit_v2() != 0:
            raise RuntimeError("nvmlInit failed")
        self.L = L
        h = C.c_void_p()
        ok = False
        try:  # the device torch uses, by UUID (CUDA and NVML indices may differ)
            import torch
            u = str(torch.cuda.get_device_properties(dev).uuid)
            u = u if u.startswith("GPU-") else "GPU-" + u
            ok = L.nvmlDeviceGetHandleByUUID(u.encode(), C.byref(h)) == 0
        except Exception:
            ok = False
        if not ok and L.nvmlDeviceGetHandleByIndex_v2(C.c_uint(dev), C.byref(h)) != 0:
            raise RuntimeError("no NVML handle")
        self.h = h
        self.reasons_fn = getattr(L, "nvmlDeviceGetCurrentClocksEventReasons", None) or \
            L.nvmlDeviceGetCurrentClocksThrottleReasons
        mx = C.c_uint()
        self.max_mhz = float(mx.value) if L.nvmlDeviceGetMaxClockInfo(h, 1, C.byref(mx)) == 0 else None
        self.interval = interval_s
        self.samples = []
        self._stop = threading.Event()

    def _one(self):
        C = self.C
        mhz, r = C.c_uint(), C.c_ulonglong()
        if self.L.nvmlDeviceGetClockInfo(self.h, 1, C.byref(mhz)) != 0:
            return
        if self.reasons_fn(self.h, C.byref(r)) != 0:
            r.value = 0
        self.samples.append((float(mhz.value), int(r.value)))

    def _run(self):
        while not self._stop.is_set():
            self._one()
            time.sleep(self.interval)

    def __enter__(self):
        self._one()
        self._t = threading.Thread(target=self._run, daemon=True)
        self._t.start()
        return self

    def __exit__(self, *exc):
        self._stop.set()
        self._t.join(timeout=5)
        self._one()

    def summary(self):
        reasons = set()
        for _, r in self.samples:
            for bit, name in self.REASONS.items():
                if r & bit:
                    reasons.add(name)
        sm = [m for m, _ in self.samples]
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": self.max_mhz,
                "reasons": sorted(reasons), "samples": len(self.samples), "source": "nvml"}


def clock_sampler(dev: int):
    """NVML sampling when the driver's library loads, else nvidia-smi."""
    try:
        return NvmlClocks(dev)
    except Exception:
        return Clocks(dev)


def dist_env():
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return rank, world, local


def oracle_rate(phys: W.Physics, cells: int, seconds: float, seed: int):
    """Oracle p-steps/s on a slice of `cells` cells of the workload (same ppc and
    physics), stepping until `seconds` of CPU time are spent (at least 2 steps)."""
    from oracle.oracle import Oracle
    import dataclasses
    sl = dataclasses.replace(phys, ncells=cells)
    loads = W.initial_load(sl, seed=seed)
    o = Oracle(sl)
    o.load_all(loads)
    o.step(1)  # first field solve and warm caches
    n = sum(len(x) for x in loads)
    t0 = time.perf_counter()
    k = 0
    while True:
        o.step(1)
        k += 1
        el = time.perf_counter() - t0
        if k >= 2 and el >= seconds:
            break
    live = int(o.moments()["live"].sum())
    return (n + live) / 2 * k / el, k, n, el


def run_reference(args):
    rank, world, _ = dist_env()
    if rank != 0:
        return 0
    phys = W.bounded_large()
    cells = args.ref_cells
    rates = []
    n = None
    t_all = time.perf_counter()
    for _ in range(args.warmup):
        oracle_rate(phys, cells, 0.0, seed=1)
    total_ps, total_t = 0.0, 0.0
    for k in range(args.steps):
        r, nsteps, n, el = oracle_rate(phys, cells, 0.0, seed=1 + k)
        total_ps += r * el
        total_t += el
    value = total_ps / total_t
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * total_t / args.steps,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
        "data": "synthetic",
        "config": {"workload": "bounded_large slice: %d of 65536 cells, 1500 ppc/species" % cells,
                   "particles_per_step": n},
        "cpu_baseline": {"value": value, "unit": UNIT, "cores": 1, "kind": "oracle",
                         "sample": "FP64 CPU oracle, each step = 2 time steps of a %d-cell slice "
                                   "(%d particles) of the bounded_large workload" % (cells, n)},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
        "wall_s": time.perf_counter() - t_all,
    }
    print(json.dumps(line), flush=True)
    return 0


def pinned(a: np.ndarray):
    import torch
    t = torch.empty(a.shape, dtype={np.dtype(np.int32): torch.int32, np.dtype(np.float64): torch.float64,
                                     np.dtype(np.float32): torch.float32,
                                     np.dtype(np.uint32): torch.int32}[a.dtype], pin_memory=True)
    v = t.numpy().view(a.dtype)
    v[...] = a
    return t, v


def measure_form(sim, phys, steps, warmup, n_particles, precision_name, rank, world, dev,
                 bytes_per_particle=None, sort_interval=80):
    import torch
    import torch.distributed as dist
    sim.step(warmup)
    # pic_step captures a CUDA graph the first time it meets a window of steps (store copy,
    # place in the sort cycle, length): the warm-up ends on a cycle boundary and runs two
    # whole cycles more, so the timed steps replay graphs captured before the timing (80 is
    # a multiple of every sort interval the autotuner picks; the step count is the
    # handle's, which autotuning steps before this call have advanced)
    K = sort_interval
    done = int(sim.moments(0)["step"])
    sim.step((-done % K) + 2 * K)
    sim.sync()
    physs = phys if isinstance(phys, list) else [phys]

    def live_total():
        return sum(sim.count(i, s) for i, p in enumerate(physs) for s in range(len(p.species)))

    live0 = live_total()
    step0 = int(sim.moments(0)["step"])
    # timed region 1: the steps as pic_step runs them (one CUDA-graph replay per window
    # of steps inside a sort cycle) -> value and ms_per_step
    torch.cuda.synchronize()
    if world > 1:
        dist.barrier()
    start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    with clock_sampler(dev) as clk:
        start.record()
        sim.step(steps)
        end.record()
        torch.cuda.synchronize()
    ms = start.elapsed_time(end)
    live1 = live_total()
    # timed region 2: the same number of steps with a CUDA event pair around every kernel
    # on the library's stream -> per-kernel times and the roofline's launch duration
    sim.profile(True)
    torch.cuda.synchronize()
    if world > 1:
        dist.barrier()
    p0, p1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    p0.record()
    sim.step(steps)
    p1.record()
    torch.cuda.synchronize()
    ms_profiled = p0.elapsed_time(p1)
    mover_n, mover_ms = sim.kernel_time(0)
    field_n, field_ms = sim.kernel_time(1)
    sort_n, sort_ms = sim.kernel_time(2)
    other_n, other_ms = sim.kernel_time(3)
    kernels, _ = sim.kernel_time(4)
    smove_n, smove_ms = sim.kernel_time(5)
    sim.profile(False)
    from paper_2404_10270_gb300.sharding import combine_timing
    ms_max, psteps = combine_timing(ms, (live0 + live1) / 2 * steps, device="cuda")
    hbm, src = peaks()
    bpp = bytes_per_particle or MOVER_BYTES[precision_name]
    per_launch_bytes = bpp * (live0 + live1) / 2
    avg_mover_ms = mover_ms / max(mover_n, 1)
    achieved = per_launch_bytes / (avg_mover_ms * 1e-3) / 1e9
    traffic = profiled_traffic("k_move", precision_name) if bytes_per_particle is None else None
    roof = None
    if precision_name == "f64" and bytes_per_particle is None:
        ach = FP64_OPS_PER_PARTICLE * (live0 + live1) / 2 / (avg_mover_ms * 1e-3)
        pipe = {"achieved": ach, "peak": FP64_PEAK_INSTR_PER_S, "unit": "FP64 instr/s",
                "frac": ach / FP64_PEAK_INSTR_PER_S, "ops_per_particle": FP64_OPS_PER_PARTICLE,
                "peak_source": "derived: 2 FP64 instr/SM/cycle x 152 SMs x 2.07 GHz"}
        if pipe["frac"] > achieved / hbm:
            roof = dict(bound="alu", **pipe, kernel="k_move<double>", avg_launch_ms=avg_mover_ms,
                        hbm={"achieved_GBps": achieved, "frac_of_measured": achieved / hbm,
                             "bytes_per_particle": MOVER_BYTES[precision_name]})
    return {
        "value": psteps / (ms_max * 1e-3),
        "ms_per_step": ms_max / steps,
        "roofline": roof or {"bound": "hbm", "achieved": achieved, "peak": hbm, "unit": "GB/s",
                     "frac": achieved / hbm, "peak_source": src + " (MEASURED_PEAKS.json hbm_gbs)"
                     if src == "measured" else "fallback 6.8 TB/s",
                     "traffic": None if traffic is None else traffic * (live0 + live1) / 2,
                     "kernel": "k_move<%s>" % ("float" if precision_name == "f32" else "double"),
                     "bytes_per_particle": bpp,
                     "avg_launch_ms": avg_mover_ms,
                     **({"fp64_pipe": pipe} if precision_name == "f64" and bytes_per_particle is None
                        else {})},
        "kernel_ms": {"mover": mover_ms, "field": field_ms, "sort": sort_ms, "other": other_ms,
                      "sorting_mover": smove_ms, "mover_launches": mover_n,
                      "sorting_mover_launches": smove_n, "sort_launch_groups": sort_n,
                      "ms_per_step_with_kernel_events": ms_profiled / steps},
        "gpu_launches": kernels,
        "clocks": clk.summary(),
        "live": [live0, live1],
        "first_timed_step": step0,
        # steps of the window where every collision clock tests (multiples of 127)
        "clock_test_steps": [t for t in range(step0, step0 + steps) if t % 127 == 0],
    }


def run_ours(args):
    import torch
    rank, world, local = dist_env()
    torch.cuda.set_device(local)
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl")
    # the library runs on this (non-default) stream; torch's events record on it too
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        return _run_ours(args, stream.cuda_stream, rank, world, local)


def measure_paper_case(args, stream, rank, world, local):
    """The paper's own test case (Section 3, Table 1) in normalized units: a periodic
    plasma of electrons, D+ ions and D neutrals, 100,000 cells x 100 particles per cell
    per species (30M particles), no field solve, electron-neutral elastic, excitation and
    ionization against the neutral particles, which ionization depletes; the neutrals
    move once per 20-step sort cycle.  FP32 and FP64 forms."""
    from paper_2404_10270_gb300 import capi
    phys = W.ionization_case(ncells=args.paper_cells, ppc=100, seed=1 + rank)
    loads = W.initial_load(phys, seed=1 + rank)
    n = sum(len(x) for x in loads)
    # algorithmic bytes per particle-step: e and D+ read/write cell word, offset, vx (24 B
    # in FP32, 40 in FP64) every step; D moves on one step in 20 (the same 24 / 40 B) and
    # is not touched in between (nothing of it changes: its density is kept)
    out = {"workload": "ionization_case: %d cells x 100 ppc x (e, D+, D), periodic, no field, "
                       "elastic + excitation + ionization against the D particles" % args.paper_cells,
           "particles_per_gpu": n}
    for name, prec, full in (("fp32", capi.FP32, 24.0), ("fp64", capi.FP64, 40.0)):
        bpp = (2 * full + full / 20) / 3
        sim = capi.Sim(phys, precision=prec, sort_interval=phys.sort_interval, block=256,
                       stream=stream)
        sim.load_all(loads)
        r = measure_form(sim, phys, max(args.steps, 20), min(args.warmup, 20), n,
                         "f32" if prec == capi.FP32 else "f64", rank, world, local,
                         bytes_per_particle=bpp, sort_interval=phys.sort_interval)
        m = sim.moments(0)
        sim.close()
        out[name] = {"value": r["value"], "ms_per_step": r["ms_per_step"],
                     "roofline": r["roofline"], "neutrals_left": int(m["live"][2])}
    out["unit"] = UNIT
    return out


def measure_batched(args, stream, rank, world, local):
    """The batched ensemble: 512 independent magnetized plasmas of uneven size (cells
    log-uniform in [256, 8192], ppc in [50, 400]; volume source, elastic + ionization +
    charge exchange, Boris push) in one handle, FP32 state.  Block size and sort
    interval are chosen by the library's autotuner, which runs during the untimed
    set-up steps."""
    import concurrent.futures as cf
    from paper_2404_10270_gb300 import capi
    from paper_2404_10270_gb300.sharding import shard_instances
    allphys = W.ensemble(n_instances=args.batched_instances)
    # N GPUs: the instances are partitioned by particle count (no exchange between them)
    mine = shard_instances([p.n_particles() for p in allphys], world)[rank]
    phys = [allphys[i] for i in mine]
    t0 = time.perf_counter()
    with cf.ThreadPoolExecutor(8) as ex:
        loads = list(ex.map(lambda ip: W.initial_load(ip[1], seed=ip[0] + 1),
                            zip(mine, phys)))
    n = sum(len(x) for ld in loads for x in ld)
    sim = capi.Sim(phys, precision=capi.FP32, sort_interval=-1, block=0, stream=stream)
    for i, ld in enumerate(loads):
        sim.load_all(ld, inst=i)
    del loads
    sim.step(args.tune_steps)  # autotuning happens here (or the cached choice is used)
    sim.sync()
    setup = time.perf_counter() - t0
    r = measure_form(sim, phys, args.batched_steps, 5, n, "f32", rank, world, local,
                     bytes_per_particle=40)
    sim.close()
    return {"workload": "ensemble: %d instances, cells log-uniform [256, 8192], ppc [50, 400], "
                        "m_i/m_e {100, 1836}, B angle [0, 89] deg, |B| = 2, volume source, "
                        "elastic + ionization + charge exchange, FP32 state" % len(allphys),
            "scaling": "strong (instances partitioned by particle count over the GPUs)",
            "particles_per_gpu": n, "value": r["value"], "unit": UNIT, "ms_per_step": r["ms_per_step"],
            "steps": args.batched_steps, "roofline": r["roofline"], "gpu_launches": r["gpu_launches"],
            "clocks": r["clocks"], "kernel_ms": r["kernel_ms"], "setup_s": setup,
            "tuning": "block and sort interval by the library autotuner during %d set-up steps"
                      % args.tune_steps}


def measure_small(args, stream):
    """The small bounded plasma (256 cells, 51,200 particles): launch-latency bound; the
    step loop runs as one replayed CUDA graph per sort cycle."""
    import torch
    from paper_2404_10270_gb300 import capi
    phys = W.bounded_small()
    loads = W.initial_load(phys, seed=1)
    out = {}
    for name, prec in (("fp32", capi.FP32), ("fp64", capi.FP64)):
        sim = capi.Sim(phys, precision=prec, sort_interval=20, block=256,
                           stream=stream)
        sim.load_all(loads)
        sim.step(100)
        sim.sync()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        n0 = sum(sim.count(0, s) for s in range(2))
        a.record()
        sim.step(1000)
        b.record()
        torch.cuda.synchronize()
        ms = a.elapsed_time(b)
        n1 = sum(sim.count(0, s) for s in range(2))
        sim.close()
        out[name] = {"value": (n0 + n1) / 2 * 1000 / (ms * 1e-3), "unit": UNIT,
                     "us_per_step": ms * 1e3 / 1000, "steps": 1000}
    out["workload"] = "bounded_small: 256 cells, 100 ppc/species, 51,200 particles, 1000 steps"
    return out


def run_c5(args):
    """The memory-filling ensemble sweep: the batched ensemble scaled to ~150 GB of FP64
    particle state (two copies, 1.5x capacity), run in the FP64 and the FP32 form.  Its
    cpu_baseline leg steps 16 sampled instances with the oracle (timed on one host core),
    and both forms' density, potential and wall-flux errors are taken against those runs."""
    import concurrent.futures as cf
    import torch
    from paper_2404_10270_gb300 import capi
    __import__("__graft_entry__").build()
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        probe = W.ensemble(n_instances=512)
        per = sum(p.n_particles() for p in probe) / 512
        n_inst = int(args.c5_gb * 1e9 / (per * 40 * 1.5 * 2))
        phys = W.ensemble(n_instances=n_inst)
        with cf.ThreadPoolExecutor(16) as ex:
            loads = list(ex.map(lambda ip: W.initial_load(ip[1], seed=ip[0] + 1), enumerate(phys)))
        n = sum(len(x) for ld in loads for x in ld)
        sample = list(range(0, n_inst, max(1, n_inst // 16)))[:16]
        res = {"instances": n_inst, "particles": n, "sampled": sample}
        gpu_moments = {}
        # magnetized movers move cell word, offset and three velocities each way:
        # 2 x (4 + 8 + 24) B in FP64, 2 x (4 + 4 + 12) B in FP32
        for name, prec, bpp in (("fp64", capi.FP64, 72), ("fp32", capi.FP32, 40)):
            sim = capi.Sim(phys, precision=prec, sort_interval=20, block=256,
                           stream=stream.cuda_stream)
            for i, ld in enumerate(loads):
                sim.load_all(ld, inst=i)
            r = measure_form(sim, phys, args.steps, args.warmup, n,
                             "f64" if prec == capi.FP64 else "f32", 0, 1, 0, bytes_per_particle=bpp,
                             sort_interval=20)
            gpu_moments[name] = {i: sim.moments(i) for i in sample}
            sim.close()
            res[name] = {"value": r["value"], "ms_per_step": r["ms_per_step"],
                         "roofline": r["roofline"]}
            if prec == capi.FP64:
                # the FP64 Boris form is bound by the FP64 pipe
                live = sum(r["live"]) / 2
                ach = FP64_OPS_PER_PARTICLE_BORIS * live / (r["roofline"]["avg_launch_ms"] * 1e-3)
                res[name]["roofline_fp64_pipe"] = {
                    "bound": "alu", "achieved": ach, "peak": FP64_PEAK_INSTR_PER_S,
                    "unit": "FP64 instr/s", "frac": ach / FP64_PEAK_INSTR_PER_S,
                    "ops_per_particle": FP64_OPS_PER_PARTICLE_BORIS}
        # cpu_baseline leg: the oracle steps the sampled instances as far as the GPU runs
        # went (the warm-up, the timed steps, as many profiled steps); its moments are the
        # reference for both forms' errors
        total = int(gpu_moments["fp64"][sample[0]]["step"])
        assert all(int(m["step"]) == total for g in gpu_moments.values() for m in g.values())
        ora, psteps, t_cpu = cpu_oracle_instances([phys[i] for i in sample],
                                                  [loads[i] for i in sample], total)
        res["cpu_baseline"] = {"value": psteps / t_cpu, "unit": UNIT, "cores": 1, "kind": "oracle",
                               "sample": "FP64 CPU oracle, %d time steps of the %d sampled instances "
                                         "(%.3g particle-steps, %.1f s)" % (total, len(sample), psteps, t_cpu)}
        for name in ("fp64", "fp32"):
            errs = []
            for i, om in zip(sample, ora):
                g = gpu_moments[name][i]
                dscale = np.abs(om["density"]).max()
                pscale = max(np.abs(om["phi"]).max(), 1e-300)
                errs.append({"inst": i,
                             "density": float(np.abs(g["density"] - om["density"]).max() / dscale),
                             "phi": float(np.abs(g["phi"] - om["phi"]).max() / pscale),
                             "wall_flux": int(np.abs(g["wall_count"] - om["wall_count"]).sum()),
                             "live": int(np.abs(g["live"] - om["live"]).sum())})
            res[name]["errors_vs_oracle_after_%d_steps" % total] = errs
        print(json.dumps({"c5": res}), flush=True)
    return 0


def cpu_oracle_instances(physs, loads, steps):
    """cpu_baseline leg of the ensemble sweep: the FP64 CPU oracle steps each instance
    (one host core); returns their moments, the particle-steps done and the seconds."""
    from oracle.oracle import Oracle
    out, psteps, t = [], 0, 0.0
    for ph, ld in zip(physs, loads):
        o = Oracle(ph)
        o.load_all(ld)
        n0 = sum(len(x.id) for x in ld)
        t0 = time.perf_counter()
        o.step(steps)
        t += time.perf_counter() - t0
        m = o.moments()
        psteps += (n0 + int(np.sum(m["live"]))) / 2 * steps
        out.append(m)
    return out, psteps, t


def _e2e_pass(sim, host, outs, phys, args, world):
    """One end-to-end pass through the public API: load every species from pinned host
    memory, args.steps steps, the moments, every particle read back to pinned host
    memory.  The FP32 form's data travel as float (pic_load_particles_f32: 20 B per
    particle, the ids numbered on the device; pic_get_particles_f32: 24 B with the ids);
    from pinned memory the library's load kernel reads the host arrays itself.
    Returns (seconds, max over ranks; breakdown; moments; bytes read back)."""
    import ctypes as C
    import torch
    from paper_2404_10270_gb300 import capi
    torch.cuda.synchronize()
    if world > 1:
        torch.distributed.barrier()
    t0 = time.perf_counter()
    t_sp = []
    for s, h in enumerate(host):
        # a fresh start: the library numbers the particles itself (the same ids)
        sim.load(0, s, W.Load(*[h[k][1] for k in ("cell", "off", "vx", "vy", "vz")], None))
        t_sp.append(time.perf_counter())
    t_load = time.perf_counter()
    sim.step(args.steps)
    sim.sync()
    t_steps = time.perf_counter()
    mom = sim.moments(0)
    d2h = 0
    for s in range(len(phys.species)):
        o = outs[s]
        got = C.c_int64()
        cap = len(o["cell"])
        f32 = o["off"].dtype == np.float32
        get = capi.lib().pic_get_particles_f32 if f32 else capi.lib().pic_get_particles
        capi._check(get(sim._h, 0, s, cap, *[o[k].ctypes.data for k in
                    ("cell", "off", "vx", "vy", "vz", "id")], None, 0, C.byref(got)), sim._h)
        d2h += got.value * (24 if f32 else 40)
    torch.cuda.synchronize()
    t_end = time.perf_counter()
    parts = {"load_s": t_load - t0, "load_species_s": [b - a for a, b in zip([t0] + t_sp[:-1], t_sp)],
             "steps_s": t_steps - t_load, "read_back_s": t_end - t_steps}
    e2e_t = torch.tensor([t_end - t0], dtype=torch.float64, device="cuda")
    if world > 1:
        torch.distributed.all_reduce(e2e_t, op=torch.distributed.ReduceOp.MAX)
    return float(e2e_t.item()), parts, mom, d2h


def _run_ours(args, stream, rank, world, local):
    import torch
    __import__("__graft_entry__").build()
    from paper_2404_10270_gb300 import capi
    t_setup = time.perf_counter()
    phys = W.bounded_large(ncells=args.cells, ppc=args.ppc, seed=1 + rank)
    loads = W.initial_load(phys, seed=1 + rank)
    n = sum(len(x) for x in loads)
    # pinned host copies of the inputs in double (the loads outside the timed regions)
    host = []
    for ld in loads:
        host.append({k: pinned(getattr(ld, k)) for k in ("cell", "off", "vx", "vy", "vz", "id")})
    # the end-to-end pass's inputs and outputs in pinned host memory, in the FP32 form's
    # own precision (float offsets and velocities; an offset that rounds up to 1 in float
    # is kept just below it), all allocated here, outside every timed region
    host32, outs = [], []
    for ld in loads:
        m = len(ld)
        off32 = np.minimum(ld.off.astype(np.float32), np.float32(1.0) - np.float32(2.0 ** -24))
        host32.append({"cell": pinned(ld.cell), "off": pinned(off32),
                       "vx": pinned(ld.vx.astype(np.float32)), "vy": pinned(ld.vy.astype(np.float32)),
                       "vz": pinned(ld.vz.astype(np.float32))})
        outs.append({k: pinned(np.zeros(m, dt))[1] for k, dt in
                     (("cell", np.int32), ("off", np.float32), ("vx", np.float32),
                      ("vy", np.float32), ("vz", np.float32), ("id", np.uint32))})
    sim = capi.Sim(phys, precision=capi.FP32, sort_interval=args.sort, block=LARGE_BLOCK,
                   stream=stream)
    for s, h in enumerate(host):
        sim.load(0, s, W.Load(*[h[k][1] for k in ("cell", "off", "vx", "vy", "vz", "id")]))
    setup_s = time.perf_counter() - t_setup
    res = measure_form(sim, phys, args.steps, args.warmup, n, "f32", rank, world, local,
                       sort_interval=args.sort)

    # end to end through the public API with host buffers: load from pinned host
    # memory, K steps, read every particle and the moments back to pinned memory; three
    # passes (the host's copy bandwidth varies with other traffic on the shared host),
    # the median is reported and every pass listed
    e2e_passes = []
    for _ in range(3):
        e2e_passes.append(_e2e_pass(sim, host32, outs, phys, args, world))
    e2e_passes.sort(key=lambda x: x[0])
    e2e_s, e2e_parts, mom, d2h = e2e_passes[1]
    e2e_value = n * world * args.steps / e2e_s
    h2d = n * 20  # cell (4 B) and four floats per particle (the ids are numbered on the device)
    assert mom["step"] > 0
    e2e_parts["passes_s"] = [p[0] for p in e2e_passes]

    fp64 = None
    if not args.no_fp64:
        sim.close()
        del sim
        sim64 = capi.Sim(phys, precision=capi.FP64, sort_interval=args.sort, block=LARGE_BLOCK,
                         stream=stream)
        for s, h in enumerate(host):
            sim64.load(0, s, W.Load(*[h[k][1] for k in ("cell", "off", "vx", "vy", "vz", "id")]))
        r64 = measure_form(sim64, phys, max(args.steps // 4, 4), min(args.warmup, 3), n, "f64",
                           rank, world, local, sort_interval=args.sort)
        sim64.close()
        fp64 = {k: r64[k] for k in ("value", "ms_per_step", "roofline", "clocks")}
        fp64["dtype"] = "f64"
    else:
        sim.close()

    # the same workload with the ions subcycled (advanced every 4 steps with 4 dt,
    # deposited every step): every particle still counts once per step
    subcycled = None
    if not args.no_subcycle:
        phys4 = W.bounded_large(ncells=args.cells, ppc=args.ppc, seed=1 + rank)
        phys4.species[1].nstep = 4
        sim4 = capi.Sim(phys4, precision=capi.FP32, sort_interval=args.sort, block=256,
                        stream=stream)
        for s, h in enumerate(host):
            sim4.load(0, s, W.Load(*[h[k][1] for k in ("cell", "off", "vx", "vy", "vz", "id")]))
        r4 = measure_form(sim4, phys4, max(args.steps // 2, 8), min(args.warmup, 4), n, "f32",
                          rank, world, local, sort_interval=args.sort)
        sim4.close()
        subcycled = {"value": r4["value"], "ms_per_step": r4["ms_per_step"],
                     "mover_ms": r4["roofline"]["avg_launch_ms"],
                     "workload": "bounded_large with the ions subcycled: nstep = 4",
                     "unit": UNIT}

    paper = None
    if not args.no_paper:
        paper = measure_paper_case(args, stream, rank, world, local)

    batched = None
    if not args.no_batched:
        batched = measure_batched(args, stream, rank, world, local)
    small = measure_small(args, stream) if rank == 0 and not args.no_small else None

    cpu = None
    if rank == 0 and not args.no_cpu:
        rate, k, ns, el = oracle_rate(phys, args.cpu_cells, args.cpu_seconds, seed=1)
        cpu = {"value": rate, "unit": UNIT, "cores": 1, "kind": "oracle",
               "sample": "FP64 CPU oracle, %d time steps of a %d-cell slice (%d particles, same "
                         "ppc and physics) of the workload, %.1f s" % (k, args.cpu_cells, ns, el)}
    if rank == 0:
        roof = dict(res["roofline"])
        if fp64:  # the FP64 form beside the FP32 one (the metric names both forms)
            r64 = fp64["roofline"]
            roof.update({"fp64_value": fp64["value"], "fp64_ms_per_step": fp64["ms_per_step"],
                         "fp64_bound": r64["bound"], "fp64_frac": r64["frac"],
                         "fp64_hbm_frac": r64["hbm"]["frac_of_measured"] if "hbm" in r64
                         else r64["frac"]})
        line = {
            "metric": METRIC, "value": res["value"], "unit": UNIT, "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": res["ms_per_step"],
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
            "data": "synthetic",
            "config": {"workload": "bounded_large: %d cells x %d ppc x (e, i), m_i/m_e 100, elastic + "
                                   "CX at 0.01, absorbing walls" % (args.cells, args.ppc),
                       "state": "FP32 particles, int64 fixed-point deposit, FP64 field",
                       "particles_per_gpu": n, "cells": args.cells, "sort_interval": args.sort,
                       "parallelism": "replicas" if world > 1 else "single",
                       "l2": "state %.1f GB per GPU > L2 (no flush needed)" % (n * 24 / 1e9),
                       "timing": "value: graph replay (warm-up to a sort-cycle boundary + 2 cycles); "
                                 "roofline: 2nd region, events per kernel",
                       "first_timed_step": res["first_timed_step"],
                       "clock_test_steps_timed": res["clock_test_steps"]},
            "roofline": roof,
            "cpu_baseline": cpu,
            "e2e": {"value": e2e_value, "unit": UNIT, "h2d_bytes_per_step": h2d / args.steps,
                    "d2h_bytes_per_step": d2h / args.steps,
                    "what": "load_f32 (no ids) from pinned host + %d steps + moments + get_f32 "
                            "to pinned host; median of 3" % args.steps,
                    "breakdown": e2e_parts},
            "gpu_launches": res["gpu_launches"],
            "clocks": res["clocks"],
            "kernel_ms": res["kernel_ms"],
            "fp64_form": fp64,
            "subcycled": subcycled,
            "paper_case": paper,
            "batched": batched,
            "small": small,
            "setup_s": setup_s,
        }
        # compact copies of the other forms' and workloads' headline numbers, last on the
        # line so that they are in any tail of the output
        if fp64:
            line["fp64_value"] = fp64["value"]
            line["fp64_frac"] = roof["fp64_frac"]
            line["fp64_bound"] = roof["fp64_bound"]
        if paper:
            for f in ("fp32", "fp64"):
                line["paper_%s_value" % f] = paper[f]["value"]
                line["paper_%s_frac" % f] = paper[f]["roofline"]["frac"]
        if batched:
            line["batched_value"] = batched["value"]
            line["batched_frac"] = batched["roofline"]["frac"]
        if subcycled:
            line["subcycled_value"] = subcycled["value"]
        if small:
            line["small_fp32_us_per_step"] = small["fp32"]["us_per_step"]
        line["fp32_frac"] = res["roofline"]["frac"]
        line["clocks_samples"] = res["clocks"].get("samples")
        print(json.dumps(line), flush=True)
    if world > 1:
        torch.distributed.barrier()
        torch.distributed.destroy_process_group()
    return 0


def profile_case(precision: str, sort_interval: int = 20, steps: int = 6) -> int:
    """The small case the ncu captures use: the bounded_large physics on 16,384 cells
    (49,152,000 particles, state larger than L2), deposit-only launch + `steps` steps.
    The step that ends a sort cycle runs its own kernel (k_move_sort): with
    sort_interval 20 and 20 steps it is the benchmark's sort step, after 19 steps of
    drift."""
    __import__("__graft_entry__").build()
    from paper_2404_10270_gb300 import capi
    phys = W.bounded_large(ncells=16384)
    loads = W.initial_load(phys)
    sim = capi.Sim(phys, precision=capi.FP64 if precision == "f64" else capi.FP32,
                   sort_interval=sort_interval, block=LARGE_BLOCK)
    sim.load_all(loads)
    sim.step(steps)
    sim.sync()
    print("profile case ok", sim.count(0, 0) + sim.count(0, 1))
    sim.close()
    return 0


def profile_ensemble(scale: float) -> int:
    """The small batched case the ncu captures of the magnetized mover use: the 512-instance
    ensemble with every instance's particles per cell scaled by `scale` (0.1: ~5e7
    particles, state larger than L2), deposit-only launch + 6 steps."""
    import concurrent.futures as cf
    __import__("__graft_entry__").build()
    from paper_2404_10270_gb300 import capi
    phys = W.ensemble(n_instances=512, scale=scale)
    with cf.ThreadPoolExecutor(16) as ex:
        loads = list(ex.map(lambda ip: W.initial_load(ip[1], seed=ip[0] + 1), enumerate(phys)))
    sim = capi.Sim(phys, precision=capi.FP32, sort_interval=20, block=256)
    for i, ld in enumerate(loads):
        sim.load_all(ld, inst=i)
    sim.step(6)
    sim.sync()
    print("profile ensemble ok", sum(len(x) for ld in loads for x in ld))
    sim.close()
    return 0


def profile_paper(steps: int) -> int:
    """The paper's test case alone (FP32), for launch lists: load + `steps` steps."""
    __import__("__graft_entry__").build()
    from paper_2404_10270_gb300 import capi
    phys = W.ionization_case()
    sim = capi.Sim(phys, precision=capi.FP32, sort_interval=phys.sort_interval, block=256)
    sim.load_all(W.initial_load(phys))
    sim.step(steps)
    sim.sync()
    print("profile paper case ok", [sim.count(0, s) for s in range(3)])
    sim.close()
    return 0


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=100)
    ap.add_argument("--warmup", type=int, default=20)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--cells", type=int, default=65536)
    ap.add_argument("--ppc", type=int, default=1500)
    ap.add_argument("--sort", type=int, default=20)
    ap.add_argument("--no-fp64", action="store_true")
    ap.add_argument("--no-cpu", action="store_true")
    ap.add_argument("--no-batched", action="store_true")
    ap.add_argument("--no-subcycle", action="store_true")
    ap.add_argument("--no-paper", action="store_true")
    ap.add_argument("--paper-cells", type=int, default=100000)
    ap.add_argument("--no-small", action="store_true")
    ap.add_argument("--c5", action="store_true", help="run the ~150 GB ensemble sweep instead")
    ap.add_argument("--c5-gb", type=float, default=150.0)
    ap.add_argument("--batched-instances", type=int, default=512)
    ap.add_argument("--batched-steps", type=int, default=40)
    ap.add_argument("--tune-steps", type=int, default=300)
    ap.add_argument("--cpu-cells", type=int, default=1024)
    ap.add_argument("--cpu-seconds", type=float, default=10.0)
    ap.add_argument("--ref-cells", type=int, default=256)
    ap.add_argument("--profile-case", action="store_true",
                    help="run the small case the ncu captures use and exit")
    ap.add_argument("--precision", default="f32", choices=["f32", "f64"])
    ap.add_argument("--sort-step", action="store_true",
                    help="with --profile-case: 20 steps, sort every 20 (the last step sorts)")
    ap.add_argument("--profile-paper", type=int, default=0, metavar="STEPS",
                    help="run the paper's test case alone for STEPS steps and exit")
    ap.add_argument("--profile-ensemble", type=float, default=None, metavar="SCALE",
                    help="run the small batched case the ncu captures use and exit")
    args = ap.parse_args()
    if args.profile_case:
        return profile_case(args.precision, 20, 20 if args.sort_step else 6)
    if args.profile_ensemble is not None:
        return profile_ensemble(args.profile_ensemble)
    if args.profile_paper:
        return profile_paper(args.profile_paper)
    if args.c5:
        return run_c5(args)
    if args.warmup < 3:
        args.warmup = 3
    if args.impl == "reference":
        return run_reference(args)
    return run_ours(args)


if __name__ == "__main__":
    sys.exit(main())
