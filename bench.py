#!/usr/bin/env python3
"""Benchmark: facet-updates/s of the LDPM explicit central-difference step on GB300, mixed vs FP64.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference] [--workload NAME]

One "step" is one explicit central-difference step of the whole specimen (facet pass, particle pass
with the half kicks, drift and energy sums).  The default workload is the largest single-GPU
specimen, the confined-compression cube (100 mm, d = 3..6 mm, ~12.5M facets), in mixed precision
(FP32 facet pass, FP64 particle state); the same workload is also measured in FP64, and the
uniaxial-tension cube (50 mm, ~1.8M facets) is reported beside it.  Every arm uses the workload's
fixed time step and times the steps that follow the workload's pre-roll of its loading history and
W warm-up steps.  Where a step's working set is below four times the 129 MB L2, the L2 is flushed (a
512 MB write) before every timed step, outside the timed intervals; above that the K steps run back to
back.  With --gpus N > 1 (torchrun) every rank steps its own replica of the specimen (the explicit
step has no exchange between independent specimens: weak scaling, replicas only).  Prints one JSON
line on rank 0.
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import statistics
import subprocess
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "facet-updates/s per explicit step and % of HBM roofline, mixed vs FP64"
UNIT = "facet-updates/s"

# Algorithmic bytes per facet-update of a layout that stores each facet's frame (I, J, n, m, c_I, A,
# l: 52 B mixed / 96 B FP64), reads and writes the history (t_N, t_M, t_L, e_max: 32 / 64 B), writes
# the facet force (12 / 24 B) and amortises the tetrahedron (ids, shape-function gradients: ~5 / 9 B)
# over its 12 facets: 101 B (mixed) / 193 B (FP64) for the facet pass alone.  The whole step adds the
# force re-read and the CSR gather with its moment arms and the particle state: 178 / 334 B.  The
# headline roofline fractions use these per-unit figures; the library's own layout moves fewer bytes
# (frames rebuilt from the staged positions, per-tetrahedron vertex shares instead of per-facet
# forces), given beside them as the design-byte fractions.  A fraction above 1 on these figures means
# that the pass is faster than that layout's bytes could be moved; the design-byte fraction is the share
# of the memory roofline.
STORED_LAYOUT_BYTES_PER_FACET = {"mixed": {"facet_pass": 101.0, "step": 178.0},
                                 "fp64": {"facet_pass": 193.0, "step": 334.0}}
L2_BYTES = 129e6


# Algorithmic bytes of one facet-pass launch in the library's own layout: values it reads or writes
# once per step.
#   per facet        geometry (arm c_I, area A) 4r, history read + written 8r
#   per tetrahedron  4 particle ids 16 B, its 4 vertex force/moment shares written 24r
#   per particle     the record the pass gathers once: mixed 21 floats (x, u as hi/lo pairs,
#                    theta, v, omega) = 84 B; FP64 15 doubles (x, q, v) = 120 B
def facet_pass_bytes(F: int, T: int, N: int, r: int) -> float:
    return F * 12 * r + T * (16 + 24 * r) + N * (84 if r == 4 else 120)


# Algorithmic bytes of one particle-pass launch in the library's own layout.
#   per tetrahedron  the 4 shares read (24r)
#   per particle     slot table 160 B (40 slot ids, -1 past the row's end; a longer row continues in
#                    the CSR ids, not counted) and row pointer 4 B; q, v read and written 192 B; forces
#                    and energy sums read and written 128 B; inverse masses, BC codes, specimen 64 B;
#                    mixed mode writes the FP32 record 84 B
SLOT_TABLE_BYTES = 160


def gather_pass_bytes(T: int, N: int, r: int) -> float:
    return T * 4 * 6 * r + N * (SLOT_TABLE_BYTES + 4 + 192 + 128 + 64 + (84 if r == 4 else 0))


def kernel_src_hash(kernel: str = "facet_warp_kernel") -> str:
    """Hash of the sources a kernel is compiled from (its translation unit, the shared device header
    and internal layout) and of the build script (its compiler flags shape the kernel): the reverse
    passes live in ldpm_adjoint.cu, every other kernel in ldpm_kernels.cu."""
    unit = "ldpm_adjoint.cu" if kernel.startswith("adjoint_") else "ldpm_kernels.cu"
    h = hashlib.sha256()
    for f in (unit, "ldpm_device.cuh", "ldpm_internal.h"):
        h.update(open(os.path.join(ROOT, "paper_2603_13190_gb300", "csrc", f), "rb").read())
    h.update(open(os.path.join(ROOT, "paper_2603_13190_gb300", "build.py"), "rb").read())
    return h.hexdigest()[:16]


def measured_peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        d = json.load(open(p))
        return float(d["hbm_gbs"]), "measured (MEASURED_PEAKS.json hbm_gbs, copy burst)"
    return 6800.0, "fallback (6.8 TB/s)"


def recorded_traffic(kernel: str, workload: str, prec: str, field: str = "bytes_per_launch"):
    """DRAM bytes (or another recorded count) per launch from a committed ncu summary, valid only for
    the kernel source it was taken from (null otherwise)."""
    p = os.path.join(ROOT, "profiles", "traffic.json")
    if not os.path.exists(p):
        return None
    try:
        d = json.load(open(p))
        e = d.get("%s/%s/%s" % (kernel, workload, prec))
        if e and e.get("kernel_src_hash") == kernel_src_hash(kernel) and field in e:
            return float(e[field])
    except Exception:
        return None
    return None


def fp64_peak_tflops(sm_count: int | None = None, sm_mhz: float | None = None) -> float:
    """FP64 FMA peak derived from the unit counts and clock: SMs x 2 DFMA per cycle x 2 flops x clock
    (GB300: 152 SMs, 2.07 GHz: 1.26 TFLOP/s; the rate ncu reports as
    sm__sass_thread_inst_executed_op_dfma_pred_on.sum.peak_sustained).  The SM count is read from the
    device where there is one, the clock is the sampled maximum SM clock."""
    return (sm_count or 152) * 2 * 2 * (sm_mhz or 2070.0) * 1e6 / 1e12


FP64_PEAK_TFLOPS = fp64_peak_tflops()


def fp64_alu_roofline(workload: str, facet_ms: float, facets: int | None = None, sm_count: int | None = None,
                      sm_mhz: float | None = None):
    """The FP64 facet pass against the FP64 pipe: FP64 flops of one launch (dadd + dmul + 2 dfma,
    counted by ncu on the same kernel source and workload) over the live launch time.  The count
    depends on the loading state (which branch of the law each facet takes: 190 flops per facet on
    the tension cube, 135 on the confined-compression headline), so a workload without its own
    capture reports null rather than another workload's count scaled."""
    fl = recorded_traffic("facet_edge_kernel", workload, "fp64", "fp64_flops_per_launch")
    if fl is None or not facet_ms:
        return None
    peak = fp64_peak_tflops(sm_count, sm_mhz)
    achieved = fl / (facet_ms * 1e-3) / 1e12
    return {"bound": "alu", "achieved": achieved, "peak": peak, "unit": "TFLOP/s",
            "frac": achieved / peak, "flop_per_launch": fl, "flops": "counted on this workload",
            "peak_source": "derived: %d SMs (from the device) x 2 DFMA/cycle x 2 flop x %.2f GHz (sampled maximum SM "
                           "clock); no measured FP64 peak exists for this pool" % (sm_count or 152,
                                                                                    (sm_mhz or 2070.0) / 1e3)}


class ClockSampler:
    """nvidia-smi clocks and throttle reasons sampled during the timed region."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.rows = []
        self.proc = None

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.index), "--query-gpu=" + self.FIELDS,
                                          "--format=csv,noheader,nounits", "-lms", "100"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.thread = threading.Thread(target=self._read, daemon=True)
            self.thread.start()
        except Exception:
            self.proc = None
        return self

    def _read(self):
        for line in self.proc.stdout:
            self.rows.append([c.strip() for c in line.split(",")])

    def __exit__(self, *a):
        if self.proc:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except Exception:
                self.proc.kill()

    def summary(self):
        sm = [float(r[1]) for r in self.rows if len(r) >= 9 and r[1].replace(".", "").isdigit()]
        mx = [float(r[2]) for r in self.rows if len(r) >= 9 and r[2].replace(".", "").isdigit()]
        reasons = set()
        names = ("hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap")
        for r in self.rows:
            if len(r) >= 9:
                for k, nm in enumerate(names):
                    if r[5 + k].lower() == "active":
                        reasons.add(nm)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": sorted(reasons), "samples": len(self.rows)}


def dist_setup(n_gpus: int):
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1:
        import torch.distributed as dist

        import torch

        torch.cuda.set_device(local)
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    return rank, world, local


def barrier_max(world: int, value: float) -> float:
    """Maximum of `value` over the ranks (NCCL reduces device tensors, gloo host tensors)."""
    if world == 1:
        return value
    import torch
    import torch.distributed as dist

    dev = "cpu" if dist.get_backend() == "gloo" else "cuda"
    t = torch.tensor([value], dtype=torch.float64, device=dev)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def job_value(world: int, units_per_rank: float, steps: int, max_ms: float) -> float:
    """Whole-job throughput: the units every rank processed over the slowest rank's time (weak scaling:
    each rank steps its own replica)."""
    return world * units_per_rank * steps / (max_ms * 1e-3)


def barrier(world: int):
    if world > 1:
        import torch.distributed as dist

        dist.barrier()


LAUNCH_MODES = {"pairs": 1, "persistent": 2}


def mode_compare(name, prec, steps, warmup, stream, flush_buf):
    """K timed steps of one workload in each launch mode (same pre-roll and window), launch pairs
    replayed from graphs against one persistent launch per ldpm_step call."""
    import torch

    from paper_2603_13190_gb300 import ldpm

    wl, spec, bc = make_inputs(name)
    r = 4 if prec == "mixed" else 8
    flush = flush_buf if needs_flush(spec.n_facets, spec.n_tets, spec.n_particles, r) else None
    out = {"precision": prec, "facets": spec.n_facets,
           "l2": "flushed before the call of K steps" if flush is not None else "no flush (working set > 4 x L2)"}
    for mode in ("pairs", "persistent"):
        m = ldpm.Model(spec, wl.material, precision=prec, dt=wl.dt, bc=bc, stream=stream)
        ldpm.ldpm_set_launch_mode(m.h, LAUNCH_MODES[mode])
        run_preroll(m, wl.preroll, steps)
        for _ in range(warmup):
            m.step(1)
        stream.synchronize()
        if flush is not None:
            with torch.cuda.stream(stream):
                flush.zero_()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        with torch.cuda.stream(stream):
            a.record(stream)
        m.step(steps)
        with torch.cuda.stream(stream):
            b.record(stream)
        stream.synchronize()
        ms = a.elapsed_time(b)
        out[mode] = {"value": spec.n_facets * steps / (ms * 1e-3), "ms_per_step": ms / steps}
        m.close()
    out["persistent_over_pairs"] = out["persistent"]["value"] / out["pairs"]["value"]
    return out


def make_inputs(workload: str):
    from paper_2603_13190_gb300 import workloads

    wl = workloads.WORKLOADS[workload]
    spec = wl.specimen()
    bc = workloads.workload_bc(workload, spec)
    return wl, spec, bc


def needs_flush(F: int, T: int, N: int, r: int) -> bool:
    """A step whose working set is below four times the L2 could be partly served from L2 across steps:
    flush between timed steps.  Larger ones run back to back."""
    return facet_pass_bytes(F, T, N, r) + gather_pass_bytes(T, N, r) < 4 * L2_BYTES


def run_preroll(model, preroll: int, steps: int):
    """The pre-roll, ending with one call of `steps` steps, so that the CUDA graphs of a later
    ldpm_step(steps) are captured before any timed region."""
    if preroll >= steps > 0:
        model.step(preroll - steps)
        model.step(steps)
    else:
        model.step(preroll)


def time_window(model, torch, stream, flush, steps: int, warmup: int):
    """Device time of `steps` steps (CUDA events on the library's stream), after `warmup` untimed ones.
    With a flush buffer: one step per ldpm_step call, the L2 flushed before each, the per-step
    intervals summed.  Without: one ldpm_step call for all the steps, timed as one interval."""
    for _ in range(warmup):
        if flush is not None:
            with torch.cuda.stream(stream):
                flush.zero_()
        model.step(1)
    stream.synchronize()
    if flush is None:
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        with torch.cuda.stream(stream):
            a.record(stream)
        model.step(steps)
        with torch.cuda.stream(stream):
            b.record(stream)
        stream.synchronize()
        return a.elapsed_time(b)
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(steps)]
    for a, b in ev:
        with torch.cuda.stream(stream):
            flush.zero_()
            a.record(stream)
        model.step(1)
        with torch.cuda.stream(stream):
            b.record(stream)
    stream.synchronize()
    return sum(a.elapsed_time(b) for a, b in ev)


def kernel_split(model, ldpm, torch, stream, flush, steps: int):
    """Per-kernel device times of `steps` more steps: the library's profiling mode launches each
    step's two kernels directly with an event before, between and after them (so the two times add up
    to the step), with the same L2 treatment as the timed window."""
    ldpm.ldpm_profile(model.h, True)
    if flush is None:
        model.step(steps)
    else:
        for _ in range(steps):
            with torch.cuda.stream(stream):
                flush.zero_()
            model.step(1)
    stream.synchronize()
    kms, kcnt = ldpm.ldpm_profile_read(model.h)
    ldpm.ldpm_profile(model.h, False)
    return kms[1] / max(1, kcnt[1]), kms[2] / max(1, kcnt[2])


def hbm_roofline(units_bytes: float, design_bytes: float, ms: float, peak: float, peak_src: str, traffic,
                 what: str):
    """HBM roofline of one launch: achieved = algorithmic bytes (the per-unit figure `what` x units) /
    device time, with the library layout's own bytes beside it."""
    achieved = units_bytes / (ms * 1e-3) / 1e9
    design = design_bytes / (ms * 1e-3) / 1e9
    return {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s", "frac": achieved / peak,
            "traffic": traffic, "algorithmic_bytes_per_launch": units_bytes, "bytes_model": what,
            "frac_design_bytes": design / peak, "design_bytes_per_launch": design_bytes,
            "peak_source": peak_src}


def step_roofline(stored_bytes: float, design_bytes: float, ms: float, peak: float, peak_src: str):
    """HBM roofline of a whole step on the bytes the library's layout moves (frac); the stored-frame
    layout's per-step bytes over the same time (an effective rate, above the peak whenever that layout
    would move more than this one does in the time) beside it."""
    achieved = design_bytes / (ms * 1e-3) / 1e9
    return {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s", "frac": achieved / peak,
            "algorithmic_bytes_per_step": design_bytes, "bytes_model": "design bytes of both passes",
            "frac_stored_layout_bytes": stored_bytes / (ms * 1e-3) / 1e9 / peak,
            "stored_layout_bytes_per_step": stored_bytes, "peak_source": peak_src}


def run_leg(name, wl, spec, bc, prec, steps, warmup, preroll, stream, flush_buf, peak, peak_src, world,
            launch="auto"):
    """One workload in one precision: create (fixed dt; launch "auto": the library's autotuner picks the
    launch shape and mode, else the named mode), pre-roll, warm-up, K timed steps, the per-kernel split
    (from launch pairs on the same state: the persistent kernel has no per-pass split), the rooflines
    and the energy check."""
    import torch

    from paper_2603_13190_gb300 import ldpm

    N, T, F = spec.n_particles, spec.n_tets, spec.n_facets
    r = 4 if prec == "mixed" else 8
    flush = flush_buf if needs_flush(F, T, N, r) else None
    model = ldpm.Model(spec, wl.material, precision=prec, dt=wl.dt, bc=bc, stream=stream, autotune=launch == "auto")
    if launch != "auto":
        ldpm.ldpm_set_launch_mode(model.h, LAUNCH_MODES[launch])
    mode = ldpm.ldpm_launch_mode(model.h)
    run_preroll(model, preroll, steps)
    barrier(world)
    torch.cuda.synchronize()
    tot = barrier_max(world, time_window(model, torch, stream, flush, steps, warmup))
    ldpm.ldpm_set_launch_mode(model.h, LAUNCH_MODES["pairs"])
    facet_ms, gather_ms = kernel_split(model, ldpm, torch, stream, flush, steps)
    energy, _ = model.energy()
    shape = model.launch_shape()
    model.close()
    ms_step = tot / steps
    fb, gb = facet_pass_bytes(F, T, N, r), gather_pass_bytes(T, N, r)
    ref = STORED_LAYOUT_BYTES_PER_FACET[prec]
    kern = "facet_warp_kernel" if prec == "mixed" else "facet_edge_kernel"
    return {
        "workload": name, "precision": prec, "steps": steps, "value": job_value(world, F, steps, tot),
        "ms_per_step": ms_step, "dt_s": wl.dt,
        "launch": {"mode": {v: k for k, v in LAUNCH_MODES.items()}[mode], "by": "autotuner" if launch == "auto" else "set",
                   "tets_per_block": int(shape[0]), "lanes_per_particle": int(shape[1])},
        "l2": ("flushed (512 MB write) before every timed step, outside the timed interval" if flush is not None
               else "working set %.0f MB > 4 x L2 (129 MB): steps back to back, no flush" % ((fb + gb) / 1e6)),
        "timed_window": "steps %d..%d of the loading history (%d untimed pre-roll steps, %d warm-up)" % (
            preroll + warmup, preroll + warmup + steps, preroll, warmup),
        "kernel_ms": {"facet": facet_ms, "gather": gather_ms,
                      "facet_in_step": ms_step * facet_ms / (facet_ms + gather_ms),
                      "gather_in_step": ms_step * gather_ms / (facet_ms + gather_ms),
                      "profiled_step_over_timed_step": (facet_ms + gather_ms) / ms_step,
                      "how": "profiling pass of K more steps as launch pairs: events before, between and after "
                             "each step's two kernels (direct launches), so facet + gather is that pass's step "
                             "time; it exceeds the timed step by the launch gaps that graph replay or the "
                             "persistent launch remove.  *_in_step: the timed step split in the profiled "
                             "shares.  The rooflines use the profiled facet time (the slower, conservative one)"},
        "roofline": hbm_roofline(ref["facet_pass"] * F, fb, facet_ms, peak, peak_src,
                                 recorded_traffic(kern, name, prec),
                                 "%.0f B per facet-update (facet pass of a stored-frame layout)" % ref["facet_pass"]),
        "gather_roofline": hbm_roofline(gb, gb, gather_ms, peak, peak_src, recorded_traffic("gather_kernel", name, prec),
                                        "design bytes (no stored-layout figure for the pass alone)"),
        "step_roofline": step_roofline(ref["step"] * F, fb + gb, ms_step, peak, peak_src),
        "energy_err_pct": float(energy[3]),
        "sizes": {"particles": N, "tets": T, "facets": F},
        # kernels of ours launched in the timed region: two per step as launch pairs; as persistent
        # launches one per ldpm_step call (one call per step when flushing, else one per 4096 steps)
        "gpu_launches": 2 * steps if mode == 1 else (steps if flush is not None else -(-steps // 4096)),
    }


def run_ours(args, rank, world, local):
    import torch

    from paper_2603_13190_gb300 import ldpm, workloads

    torch.cuda.set_device(local)
    wl, spec, bc = make_inputs(args.workload)
    N, T, F = spec.n_particles, spec.n_tets, spec.n_facets
    preroll = wl.preroll if args.preroll is None else args.preroll
    # the oracle's pre-roll and timed window run on a host core meanwhile (a separate process)
    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        cpu = OracleWindow(spec, wl, bc, preroll + args.warmup)
    stream = torch.cuda.Stream()
    flush = torch.empty(512 * 1024 * 1024 // 4, dtype=torch.float32, device="cuda")
    peak, peak_src = measured_peaks()
    sampler = ClockSampler(local) if rank == 0 else None
    if sampler:
        sampler.__enter__()
    mixed = run_leg(args.workload, wl, spec, bc, "mixed", args.steps, args.warmup, preroll, stream, flush, peak,
                    peak_src, world, args.launch)
    fp64 = run_leg(args.workload, wl, spec, bc, "fp64", max(3, args.steps // 4), args.warmup, preroll, stream, flush,
                   peak, peak_src, world, args.launch)
    sms = torch.cuda.get_device_properties(local).multi_processor_count
    extra = {}
    if not args.no_extra and args.workload != "uniaxial_tension":
        # the 1.82M-facet uniaxial-tension cube beside the headline
        w2, s2, b2 = make_inputs("uniaxial_tension")
        extra["uniaxial_tension"] = run_leg("uniaxial_tension", w2, s2, b2, "mixed", args.steps, args.warmup,
                                            w2.preroll, stream, flush, peak, peak_src, world, args.launch)
        del s2
    if not args.no_extra and world == 1:
        # launch pairs against one persistent launch per call, on the small (launch-bound), the 1.82M-facet
        # and the 12.5M-facet specimens
        extra["launch_modes"] = {n: mode_compare(n, p_, max(args.steps, 200) if n == "elastic_vibration" else args.steps,
                                                 args.warmup, stream, flush)
                                 for n, p_ in (("elastic_vibration", "fp64"), ("uniaxial_tension", "mixed"),
                                               (args.workload, "mixed"))}
    if sampler:
        sampler.__exit__()
    clocks = sampler.summary() if sampler else None
    fp64["alu_roofline"] = fp64_alu_roofline(args.workload, fp64["kernel_ms"]["facet"], F, sms,
                                             (clocks or {}).get("sm_max_mhz"))
    # end to end through the C ABI with host buffers: create (H2D of the geometry), K steps each with an
    # energy/reaction read-back (D2H), final state read-back, destroy.
    barrier(world)
    torch.cuda.synchronize()
    K = args.steps
    t0 = time.perf_counter()
    m = ldpm.Model(spec, wl.material, precision="mixed", dt=wl.dt, bc=bc, device=local)
    for _ in range(K):
        m.step(1)
        m.energy()
    q, v, h5, _ = m.get_state()
    m.close()
    torch.cuda.synchronize()
    e2e_s = barrier_max(world, time.perf_counter() - t0)
    # the same calls with the model already created (and its first K steps run): K x (ldpm_step(1) +
    # ldpm_energy read-back), host clock, no state read-back
    m = ldpm.Model(spec, wl.material, precision="mixed", dt=wl.dt, bc=bc, device=local)
    for _ in range(K):
        m.step(1)
        m.energy()
    barrier(world)
    t1 = time.perf_counter()
    for _ in range(K):
        m.step(1)
        m.energy()
    steady_s = barrier_max(world, time.perf_counter() - t1)
    m.close()
    geo_bytes = spec.x.nbytes + spec.diameter.nbytes + spec.tets.nbytes + 3 * 4 * F + spec.facet_vtx.nbytes + \
        bc.mask.nbytes + bc.vel.nbytes + bc.v0.nbytes
    d2h = K * (16 * 8) + q.nbytes + v.nbytes + h5.nbytes
    res = {
        "metric": METRIC, "value": mixed["value"], "unit": UNIT, "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": mixed["ms_per_step"], "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f32+f64", "data": "synthetic",
        "config": {"workload": args.workload, "cube_mm": wl.edge, "d_min_mm": wl.d_min, "d_max_mm": wl.d_max,
                   "particles": N, "tets": T, "facets": F, "precision": "mixed: FP32 facet pass, FP64 particle state",
                   "dt_s": wl.dt, "l2": mixed["l2"], "timed_window": mixed["timed_window"],
                   "launch": mixed["launch"],
                   "parallelism": "replicas" if world > 1 else "single GPU", "seed": wl.seed},
        "roofline": mixed["roofline"],
        "gather_roofline": mixed["gather_roofline"],
        "step_roofline": mixed["step_roofline"],
        "kernel_ms": mixed["kernel_ms"],
        "energy_err_pct": mixed["energy_err_pct"],
        "fp64": {k: fp64[k] for k in ("value", "ms_per_step", "steps", "roofline", "step_roofline", "kernel_ms",
                                      "alu_roofline", "energy_err_pct")},
        "mixed_over_fp64": mixed["value"] / fp64["value"],
        "e2e": {"value": world * F * K / e2e_s, "unit": UNIT, "h2d_bytes_per_step": geo_bytes / K,
                "d2h_bytes_per_step": d2h / K, "seconds": e2e_s,
                "what": "ldpm_create from host arrays, K x (ldpm_step(1) + ldpm_energy read-back), "
                        "ldpm_get_state to host, ldpm_destroy",
                "stepping": {"value": world * F * K / steady_s, "unit": UNIT, "h2d_bytes_per_step": 0,
                             "d2h_bytes_per_step": 16 * 8, "seconds": steady_s,
                             "what": "on a created model (steps K+1..2K from rest): K x (ldpm_step(1) + "
                                     "ldpm_energy read-back of the energies and reactions), host clock"}},
        "gpu_launches": mixed["gpu_launches"],
        "clocks": clocks,
    }
    res.update(extra)
    return res, spec, wl, bc, cpu


def run_batch(args, rank, world, local):
    """Batched workload: 64 random cubes (30-60 mm) of unconfined compression stepped together in
    mixed precision with autotuned launch shapes; compared with the all-FP64 single-specimen path on
    the batch's first specimen, same GPU, same run."""
    import torch

    from paper_2603_13190_gb300 import ldpm, workloads

    torch.cuda.set_device(local)
    t0 = time.perf_counter()
    specs = workloads.batch_specimens(args.batch, seed=1)
    gen_s = time.perf_counter() - t0
    bcs = [workloads.unconfined_compression_bc(sp) for sp in specs]
    mats = [dict(workloads.WORKLOAD_MATERIAL) for _ in specs]
    N = sum(sp.n_particles for sp in specs)
    T = sum(sp.n_tets for sp in specs)
    F = sum(sp.n_facets for sp in specs)
    stream = torch.cuda.Stream()
    flush = torch.empty(512 * 1024 * 1024 // 4, dtype=torch.float32, device="cuda")
    peak, peak_src = measured_peaks()
    t0 = time.perf_counter()
    b = ldpm.Batch(specs, mats, "mixed", bcs=bcs, stream=stream, device=local, autotune=True)
    create_s = time.perf_counter() - t0
    sampler = ClockSampler(local) if rank == 0 else None
    if sampler:
        sampler.__enter__()
    preroll = 200 if args.preroll is None else args.preroll
    fl = flush if needs_flush(F, T, N, 4) else None
    barrier(world)
    torch.cuda.synchronize()
    run_preroll(b, preroll, args.steps)
    tot = barrier_max(world, time_window(b, torch, stream, fl, args.steps, args.warmup))
    facet_ms, gather_ms = kernel_split(b, ldpm, torch, stream, fl, args.steps)
    if sampler:
        sampler.__exit__()
    fb, gb = facet_pass_bytes(F, T, N, 4), gather_pass_bytes(T, N, 4)
    ref = STORED_LAYOUT_BYTES_PER_FACET["mixed"]
    shape = b.launch_shape()
    errs = [float(b.energy(i)[0][3]) for i in range(len(b))]
    b.close()
    # all-FP64 single-specimen path, same GPU: the batch's first specimen
    single = ldpm.Model(specs[0], mats[0], precision="fp64", bc=bcs[0], stream=stream, device=local)
    s0 = specs[0]
    n64 = max(3, args.steps // 4)
    run_preroll(single, preroll, n64)
    ms64 = time_window(single, torch, stream, flush if needs_flush(s0.n_facets, s0.n_tets, s0.n_particles, 8) else None,
                       n64, args.warmup)
    fp64_single = specs[0].n_facets * n64 / (ms64 * 1e-3)
    single.close()
    value = job_value(world, F, args.steps, tot)
    return {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": tot / args.steps, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "f32+f64", "data": "synthetic",
        "config": {"workload": "batched_unconfined_compression", "specimens": len(specs),
                   "edges_mm": [round(sp.edge, 2) for sp in specs[:4]] + ["..."],
                   "particles": N, "tets": T, "facets": F, "particles_min_max": [min(sp.n_particles for sp in specs),
                                                                                 max(sp.n_particles for sp in specs)],
                   "precision": "mixed: FP32 facet pass, FP64 particle state",
                   "launch_shape": {"tets_per_block": shape[0], "lanes_per_particle": shape[1], "by": "autotuner"},
                   "l2": ("flushed (512 MB write) before every timed step, outside the timed interval" if fl is not None
                          else "working set %.1f GB > 4 x L2 (129 MB): steps back to back, no flush" % ((fb + gb) / 1e9)),
                   "timed_window": "steps %d..%d of the loading history (%d untimed pre-roll steps, %d warm-up)" % (
                       preroll + args.warmup, preroll + args.warmup + args.steps, preroll, args.warmup),
                   "dt_s": "per specimen, 0.9 x its critical step (power iteration at create)",
                   "generation_s": round(gen_s, 1), "create_s": round(create_s, 1)},
        "roofline": hbm_roofline(ref["facet_pass"] * F, fb, facet_ms, peak, peak_src, None,
                                 "%.0f B per facet-update (facet pass of a stored-frame layout)" % ref["facet_pass"]),
        "step_roofline": step_roofline(ref["step"] * F, fb + gb, tot / args.steps, peak, peak_src),
        "kernel_ms": {"facet": facet_ms, "gather": gather_ms,
                      "profiled_step_over_timed_step": (facet_ms + gather_ms) / (tot / args.steps)},
        "fp64_single_specimen": {"value": fp64_single, "facets": specs[0].n_facets},
        "batched_mixed_over_fp64_single": value / fp64_single,
        "max_energy_error_pct": max(errs),
        "gpu_launches": 2 * args.steps,
        "clocks": sampler.summary() if sampler else None,
    }


ADJ_METRIC = "adjoint facet-updates/s (forward, recompute and reverse step per facet) and % of HBM roofline"


# Algorithmic bytes of one reverse facet-pass launch (ldpm_adjoint).
#   per facet        geometry 4r, the step's stored history 4r, carried history adjoint read + written
#                    8r, gradient accumulators read + written 8r
#   per tetrahedron  4 particle ids 16 B, its 4 vertex shares written 48r
#   per particle     the forward record of the step (mixed 84 B, FP64 120 B) and the a_f record
#                    (mixed 36 B: hi/lo translation, rotation; FP64 48 B)
def adjoint_facet_bytes(F: int, T: int, N: int, r: int) -> float:
    return F * 24 * r + T * (16 + 48 * r) + N * ((84 + 36) if r == 4 else (120 + 48))


# Algorithmic bytes of one reverse particle-pass launch.
#   per tetrahedron  4 CSR slot ids and the 4 shares read (48r)
#   per particle     row pointer 4 B; Qbar, Ubar read and written 192 B; seed 48 B; inverse masses, BC
#                    codes, specimen 64 B; the a_f record written (mixed 36 B, FP64 48 B)
def adjoint_gather_bytes(T: int, N: int, r: int) -> float:
    return T * 4 * (4 + 12 * r) + N * (4 + 192 + 48 + 64 + (36 if r == 4 else 48))


def run_adjoint(args, rank, world, local):
    """Adjoint workload: one ldpm_adjoint of 5000 steps (mixed precision, checkpoints every 250 steps)
    on the 50 mm tension cube pulled slowly (elastic and pre-peak), gradient of the mean top reaction
    with respect to every facet's E0, alpha, sigma_t.  Device time by CUDA events on the library's
    stream around the call; the per-kernel split from a profiled 250-step call; FP64 on 250 steps."""
    import torch

    from paper_2603_13190_gb300 import ldpm

    torch.cuda.set_device(local)
    wl, spec, bc = make_inputs("adjoint_uniaxial_tension")
    N, T, F = spec.n_particles, spec.n_tets, spec.n_facets
    K, C = wl.steps, 250
    seed = np.zeros((N, 6))
    seed[spec.face_nodes(2, 1), 2] = 1.0
    stream = torch.cuda.Stream()
    peak, peak_src = measured_peaks()
    sampler = ClockSampler(local) if rank == 0 else None
    m = ldpm.Model(spec, wl.material, precision="mixed", dt=wl.dt, bc=bc, stream=stream, device=local)
    dt = m.dt
    start = ldpm.ldpm_save_checkpoint(m.h)
    for _ in range(args.warmup):
        ldpm.ldpm_load_checkpoint(m.h, start)
        m.adjoint(C, seed, C)
    ldpm.ldpm_load_checkpoint(m.h, start)
    if sampler:
        sampler.__enter__()
    barrier(world)
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    with torch.cuda.stream(stream):
        e0.record(stream)
    t0 = time.perf_counter()
    J, gE, ga, gs = m.adjoint(K, seed, C)
    wall = time.perf_counter() - t0
    with torch.cuda.stream(stream):
        e1.record(stream)
    stream.synchronize()
    dev_ms = barrier_max(world, e0.elapsed_time(e1))
    wall = barrier_max(world, wall)
    if sampler:
        sampler.__exit__()
    # kernel split: a profiled call of C steps from the same start
    ldpm.ldpm_load_checkpoint(m.h, start)
    ldpm.ldpm_profile(m.h, True)
    m.adjoint(C, seed, C)
    kms, kcnt = ldpm.ldpm_profile_read(m.h)
    ldpm.ldpm_profile(m.h, False)
    m.close()
    rf_ms, rg_ms = kms[3] / max(1, kcnt[3]), kms[4] / max(1, kcnt[4])
    fb, gb = adjoint_facet_bytes(F, T, N, 4), adjoint_gather_bytes(T, N, 4)
    achieved = fb / (rf_ms * 1e-3) / 1e9
    # FP64 on C steps
    m64 = ldpm.Model(spec, wl.material, precision="fp64", dt=dt, bc=bc, stream=stream, device=local)
    m64.adjoint(16, seed, 16)
    ldpm.ldpm_profile(m64.h, True)
    a0, a1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    with torch.cuda.stream(stream):
        a0.record(stream)
    m64.adjoint(C, seed, C)
    with torch.cuda.stream(stream):
        a1.record(stream)
    stream.synchronize()
    k64, c64 = ldpm.ldpm_profile_read(m64.h)
    m64.close()
    fp64_value = F * C / (a0.elapsed_time(a1) * 1e-3)
    rf64 = k64[3] / max(1, c64[3])
    # the same gradient keeping every step's inputs (no recompute) when they fit in a fraction of the
    # free device memory
    store_all = None
    need = K * (96 * N + 16 * 12 * T) + 4 * (96 * N + 16 * 12 * T)
    free = torch.cuda.mem_get_info()[0]
    if need < 0.7 * free:
        ms_ = ldpm.Model(spec, wl.material, precision="mixed", dt=dt, bc=bc, stream=stream, device=local)
        s0, s1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        try:
            with torch.cuda.stream(stream):
                s0.record(stream)
            ms_.adjoint(K, seed, K)
            with torch.cuda.stream(stream):
                s1.record(stream)
            stream.synchronize()
            store_all = {"value": F * K / (s0.elapsed_time(s1) * 1e-3), "checkpoint_every": K,
                         "device_bytes_for_step_inputs": need}
        except ldpm.LdpmError as e:
            store_all = {"skipped": str(e)}
        ms_.close()
    else:
        store_all = {"skipped": "step inputs of all %d steps (%.0f GB) exceed 70 %% of free memory" % (K, need / 1e9)}
    fb64 = adjoint_facet_bytes(F, T, N, 8)
    value = job_value(world, F, K, dev_ms)
    nseg = (K + C - 1) // C
    return {
        "metric": ADJ_METRIC, "value": value, "unit": "facet-updates/s", "n_gpus": world, "steps": K,
        "warmup": args.warmup, "ms_per_step": dev_ms / K, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f32+f64", "data": "synthetic",
        "config": {"workload": "adjoint_uniaxial_tension", "cube_mm": wl.edge, "particles": N, "tets": T,
                   "facets": F, "steps": K, "checkpoint_every": C, "dt_s": dt,
                   "objective": "time mean of the top-face u_z reaction", "parameters": "E0, alpha, sigma_t per facet",
                   "precision": "mixed: FP32 facet terms, FP64 particle adjoints and gradient totals",
                   "l2": "working set (step inputs of a 250-step segment, 7.9 GB) far above L2; no flush",
                   "warmup": "%d adjoint calls of %d steps" % (args.warmup, C)},
        "objective_J": J, "grad_abs_max": [float(np.abs(x).max()) for x in (gE, ga, gs)],
        "roofline": {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s", "frac": achieved / peak,
                     "traffic": recorded_traffic("adjoint_facet_kernel", "adjoint_uniaxial_tension", "mixed"),
                     "algorithmic_bytes_per_launch": fb, "peak_source": peak_src, "kernel": "adjoint_facet_kernel"},
        "gather_roofline": {"achieved": gb / (rg_ms * 1e-3) / 1e9, "frac": gb / (rg_ms * 1e-3) / 1e9 / peak,
                            "algorithmic_bytes_per_launch": gb},
        "kernel_ms": {"facet": kms[1] / max(1, kcnt[1]), "gather": kms[2] / max(1, kcnt[2]),
                      "reverse_facet": rf_ms, "reverse_gather": rg_ms},
        "fp64": {"value": fp64_value, "steps": C, "reverse_facet_ms": rf64,
                 "reverse_facet_frac": fb64 / (rf64 * 1e-3) / 1e9 / peak},
        "no_recompute": store_all,
        "e2e": {"value": world * F * K / wall, "unit": "facet-updates/s", "h2d_bytes_per_step": seed.nbytes / K,
                "d2h_bytes_per_step": (3 * F * 8 + 8) / K, "seconds": wall,
                "what": "one ldpm_adjoint call: seed from host memory, gradients to host memory"},
        # forward sweep: facet, particle and objective kernels per step; recompute of every segment but
        # the last: facet and particle kernels; reverse: reverse facet and particle kernels; one init,
        # one fold per segment
        "gpu_launches": 3 * K + 2 * (K - (K - (nseg - 1) * C)) + 2 * K + 1 + nseg,
        "clocks": sampler.summary() if sampler else None,
    }


def cpu_baseline_adjoint(spec, wl, bc, dt, budget_s: float = 20.0):
    """The oracle's derivative path as it stands: forward-mode dual numbers carrying 8 parameter
    directions through its FP64 step, single thread, a bounded number of full steps."""
    import oracle

    o = oracle.Oracle(spec, wl.material, dt, bc)
    seed = np.zeros((spec.n_particles, 6))
    seed[spec.face_nodes(2, 1), 2] = 1.0
    rng = np.random.default_rng(0)
    d = rng.standard_normal((8, spec.n_facets))
    n, el = 1, 0.0
    while True:
        t0 = time.perf_counter()
        o.tangent(n, seed, dE0=d)
        el = time.perf_counter() - t0
        if el > budget_s / 3 or n >= 8:
            break
        n *= 2
    return {"value": spec.n_facets * n / el, "unit": "facet-updates/s", "cores": 1, "kind": "oracle",
            "sample": "%d steps of the full %d-facet specimen carrying 8 directional derivatives (forward mode, "
                      "%.1f s, single thread); the oracle has no reverse mode" % (n, spec.n_facets, el)}


# One oracle process of the CPU baseline.  argv: repo root, problem file, JSON arguments.  It rebuilds
# the problem, runs the pre-roll (and warm-up) of the loading history, writes the state it reached to
# the state file, and then (single mode) times whole steps until its time budget is spent, or (cores
# mode) reports ready, loads that state, waits for the start line on stdin and times its window.
_ORACLE_WORKER = r"""
import json, sys, time
import numpy as np
sys.path.insert(0, sys.argv[1])
import oracle
from paper_2603_13190_gb300.specimen import Specimen
from paper_2603_13190_gb300.workloads import BoundaryConditions
z = np.load(sys.argv[2])
a = json.loads(sys.argv[3])
spec = Specimen(x=z['x'], diameter=z['diameter'], tets=z['tets'], facet_pi=z['facet_pi'], facet_pj=z['facet_pj'],
                facet_tet=z['facet_tet'], facet_vtx=z['facet_vtx'], edge=a['edge'], d_min=a['d_min'], d_max=a['d_max'])
bc = BoundaryConditions(mask=z['mask'], vel=z['vel'], ramp_time=a['ramp_time'], v0=z['v0'])
o = oracle.Oracle(spec, a['material'], a['dt'], bc)
if a['mode'] == 'single':
    t0 = time.perf_counter()
    o.step(a['preroll'])
    pre_s = time.perf_counter() - t0
    q, v, h5, st = o.get_state()
    np.savez(a['state'], q=q, v=v, h5=h5, step=st)
    n, t0 = 0, time.perf_counter()
    while n < 1 or time.perf_counter() - t0 < a['budget_s']:
        o.step(1)
        n += 1
    print(json.dumps({'steps': n, 'seconds': time.perf_counter() - t0, 'preroll_s': pre_s}), flush=True)
else:
    s = np.load(a['state'])
    o.set_state(s['q'], s['v'], s['h5'], int(s['step']))
    print('ready', flush=True)
    sys.stdin.readline()
    n, t0 = 0, time.perf_counter()
    while n < 1 or time.perf_counter() - t0 < a['budget_s']:
        o.step(1)
        n += 1
    print(json.dumps({'steps': n, 'seconds': time.perf_counter() - t0}), flush=True)
"""


class OracleWindow:
    """The FP64 oracle as it stands, single thread, on the same workload, time step and window as the
    GPU arm: a separate process (started with subprocess, never forked from a process holding a CUDA
    context) runs the pre-roll and warm-up of the loading history while the GPU is measured, then times
    whole steps for about `budget_s`.  The state it reached is kept for the all-cores figure."""

    def __init__(self, spec, wl, bc, preroll: int, budget_s: float = 20.0):
        import tempfile

        self.spec, self.wl, self.bc, self.preroll = spec, wl, bc, preroll
        self.dir = tempfile.TemporaryDirectory(prefix="oracle_window_")
        self.problem = os.path.join(self.dir.name, "problem.npz")
        self.state = os.path.join(self.dir.name, "state.npz")
        np.savez(self.problem, x=spec.x, diameter=spec.diameter, tets=spec.tets, facet_pi=spec.facet_pi,
                 facet_pj=spec.facet_pj, facet_tet=spec.facet_tet, facet_vtx=spec.facet_vtx, mask=bc.mask, vel=bc.vel,
                 v0=bc.v0)
        self.base = {"edge": spec.edge, "d_min": spec.d_min, "d_max": spec.d_max, "ramp_time": bc.ramp_time,
                     "material": dict(wl.material), "dt": wl.dt, "state": self.state}
        a = json.dumps(dict(self.base, mode="single", preroll=preroll, budget_s=budget_s))
        self.proc = subprocess.Popen([sys.executable, "-c", _ORACLE_WORKER, ROOT, self.problem, a], cwd=ROOT,
                                     stdin=subprocess.DEVNULL, stdout=subprocess.PIPE, stderr=subprocess.PIPE,
                                     text=True)

    def result(self, timeout_s: float = 1800.0):
        try:
            out, err = self.proc.communicate(timeout=timeout_s)
            r = json.loads(out.strip().splitlines()[-1])
        except Exception as e:
            if self.proc.poll() is None:
                self.proc.kill()
            return {"value": None, "reason": "%s: %s" % (type(e).__name__, e)}
        return {"value": self.spec.n_facets * r["steps"] / r["seconds"], "unit": UNIT, "cores": 1, "kind": "oracle",
                "sample": "%d explicit steps of the full %d-facet specimen after its %d-step pre-roll and warm-up "
                          "(%.1f s timed, single thread; dt %.4g s, the GPU arm's)"
                          % (r["steps"], self.spec.n_facets, self.preroll, r["seconds"], self.wl.dt)}

    def all_cores(self, budget_s: float = 10.0, max_procs: int = 16):
        """The oracle on all host cores: one single-thread oracle process per core, each starting from
        the pre-rolled state and stepping its own copy of the full specimen over the same time window;
        the value is the sum of their rates (the host's aggregate throughput on independent copies of the
        workload; the oracle itself is not parallelised).  Returns the reason on any failure."""
        cores = os.cpu_count() or 1
        avail_gb = 8.0
        try:  # memory the kernel can hand out without swapping (free pages plus reclaimable cache)
            with open("/proc/meminfo") as mi:
                avail_gb = next(int(l.split()[1]) for l in mi if l.startswith("MemAvailable:")) / 2 ** 20
        except (OSError, StopIteration, ValueError):
            pass
        per_gb = 1.0 + self.spec.n_facets * 500 / 2 ** 30  # interpreter, libraries, the oracle's arrays
        C = int(max(1, min(cores, max_procs, avail_gb // (2 * per_gb))))
        if not os.path.exists(self.state):
            return {"value": None, "reason": "the single-thread oracle process did not reach the window"}
        a = json.dumps(dict(self.base, mode="cores", budget_s=budget_s))
        procs = []
        try:
            for _ in range(C):
                procs.append(subprocess.Popen([sys.executable, "-c", _ORACLE_WORKER, ROOT, self.problem, a], cwd=ROOT,
                                              stdin=subprocess.PIPE, stdout=subprocess.PIPE,
                                              stderr=subprocess.DEVNULL, text=True))
            import select

            deadline = time.monotonic() + 600.0
            for pr in procs:
                left = deadline - time.monotonic()
                if left <= 0 or not select.select([pr.stdout], [], [], left)[0] or \
                        pr.stdout.readline().strip() != "ready":
                    raise RuntimeError("an oracle process did not get ready")
            for pr in procs:
                pr.stdin.write("go\n")
                pr.stdin.flush()
            res = []
            for pr in procs:
                out, _ = pr.communicate(timeout=budget_s + 300)
                res.append(json.loads(out.strip().splitlines()[-1]))
        except Exception as e:  # the GPU figures stand on their own: report why this one is missing
            for pr in procs:
                if pr.poll() is None:
                    pr.kill()
            return {"value": None, "reason": "%s: %s" % (type(e).__name__, e)}
        rate = sum(self.spec.n_facets * r["steps"] / r["seconds"] for r in res)
        steps = [r["steps"] for r in res]
        return {"value": rate, "unit": UNIT, "cores": C, "kind": "oracle",
                "sample": "%d concurrent single-thread oracle processes (%d host cores), each stepping its own copy "
                          "of the full %d-facet specimen from the pre-rolled state for %.0f s (%d-%d steps each); "
                          "sum of their rates" % (C, cores, self.spec.n_facets, budget_s, min(steps), max(steps))}

    def close(self):
        if self.proc.poll() is None:
            self.proc.kill()
        self.dir.cleanup()


def run_reference(args, rank, world):
    """The oracle as the reference arm: same workload, metric and unit, timed on the host cores."""
    if rank != 0:
        return None
    import oracle

    from paper_2603_13190_gb300 import workloads

    wl, spec, bc = make_inputs(args.workload)
    dt = wl.dt  # the workload's fixed step, the one the GPU arm uses
    preroll = wl.preroll if args.preroll is None else args.preroll
    o = oracle.Oracle(spec, wl.material, dt, bc)
    adjoint = args.workload.startswith("adjoint")
    if adjoint:
        # the oracle's derivative path: forward-mode dual numbers carrying 8 parameter directions
        # through one step (it has no reverse mode); the state then moves on by one plain step
        seed = np.zeros((spec.n_particles, 6))
        seed[spec.face_nodes(2, 1), 2] = 1.0
        d = np.random.default_rng(0).standard_normal((8, spec.n_facets))
    o.step(preroll)
    for _ in range(args.warmup):
        o.step(1)
    t = []
    for _ in range(args.steps):
        t0 = time.perf_counter()
        if adjoint:
            o.tangent(1, seed, dE0=d)
            t.append(time.perf_counter() - t0)
            o.step(1)
        else:
            o.step(1)
            t.append(time.perf_counter() - t0)
    tot = sum(t)
    val = spec.n_facets * args.steps / tot
    what = ("%%d steps each carrying 8 directional derivatives (forward mode), after %d pre-roll and %%d warm-up "
            "steps, single thread" if adjoint else
            "%%d full explicit steps after %d pre-roll and %%d warm-up steps, single thread") % preroll
    return {"impl": "reference", "metric": ADJ_METRIC if adjoint else METRIC, "value": val, "unit": UNIT,
            "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": 1e3 * tot / args.steps, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": args.workload, "cube_mm": wl.edge, "d_min_mm": wl.d_min, "d_max_mm": wl.d_max,
                       "particles": spec.n_particles, "tets": spec.n_tets, "facets": spec.n_facets,
                       "precision": "FP64 oracle", "dt_s": dt, "seed": wl.seed,
                       "timed_window": "steps %d..%d of the loading history (%d untimed pre-roll steps, %d warm-up)" % (
                           preroll + args.warmup, preroll + args.warmup + args.steps, preroll,
                           args.warmup)},
            "cpu_baseline": {"value": val, "unit": UNIT, "kind": "oracle", "cores": 1,
                             "sample": what % (args.steps, args.warmup)},
            "e2e": {"value": val, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}


def counters(args):
    """Algorithmic bytes of each kernel of the workload: what the formulas above count per facet,
    tetrahedron and particle, and the totals of one launch and one step, in both precisions."""
    from paper_2603_13190_gb300 import workloads

    if args.workload == "batched_unconfined_compression":
        specs = workloads.batch_specimens(args.batch, seed=1)
    else:
        specs = [workloads.WORKLOADS[args.workload].specimen()]
    N = sum(sp.n_particles for sp in specs)
    T = sum(sp.n_tets for sp in specs)
    F = sum(sp.n_facets for sp in specs)
    out = {"workload": args.workload, "specimens": len(specs), "particles": N, "tets": T, "facets": F,
           "per_unit": {
               "facet_pass": {"per_facet": "geometry 4R + history read and written 8R",
                              "per_tet": "16 B ids + 4 vertex shares of 6R",
                              "per_particle": "gathered record, 84 B mixed / 120 B FP64"},
               "particle_pass": {"per_tet": "4 slot ids (4 B) + 4 shares read (6R)",
                                 "per_particle": "row 4 B, q/v 192 B, forces and energy sums 128 B, constants "
                                                 "64 B, FP32 record written 84 B (mixed)"},
               "reverse_facet_pass": {"per_facet": "geometry 4R, history 4R, carried adjoint 8R, gradient "
                                                   "accumulators 8R",
                                      "per_tet": "16 B ids + 4 vertex shares of 12R",
                                      "per_particle": "forward record + a_f record, 120 B mixed / 168 B FP64"},
               "reverse_particle_pass": {"per_tet": "4 slot ids + 4 shares read (12R)",
                                         "per_particle": "row 4 B, Qbar/Ubar 192 B, seed 48 B, constants 64 B, "
                                                         "a_f record written 36 B mixed / 48 B FP64"}},
           "R": {"mixed": 4, "fp64": 8}}
    for prec, r in (("mixed", 4), ("fp64", 8)):
        fb, gb = facet_pass_bytes(F, T, N, r), gather_pass_bytes(T, N, r)
        afb, agb = adjoint_facet_bytes(F, T, N, r), adjoint_gather_bytes(T, N, r)
        out[prec] = {"facet_pass_bytes": fb, "particle_pass_bytes": gb, "step_bytes": fb + gb,
                     "reverse_facet_pass_bytes": afb, "reverse_particle_pass_bytes": agb,
                     "adjoint_step_bytes": 2 * (fb + gb) + afb + agb,
                     "step_bytes_per_facet": (fb + gb) / F}
    return out


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=40)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", default="ours", choices=("ours", "reference"))
    ap.add_argument("--workload", default="confined_compression",
                    choices=("uniaxial_tension", "confined_compression", "elastic_vibration",
                             "batched_unconfined_compression", "adjoint_uniaxial_tension"))
    ap.add_argument("--batch", type=int, default=64, help="specimens of the batched workload")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-extra", action="store_true",
                    help="skip the uniaxial-tension line and the launch-mode comparison beside the headline")
    ap.add_argument("--launch", choices=("auto", "pairs", "persistent"), default="auto",
                    help="launch mode of the timed legs: the library's autotuner (default) or a fixed one")
    ap.add_argument("--preroll", type=int, default=None,
                    help="untimed steps of the loading history before the warm-up (default: the workload's own, "
                         "enough for the loading wave to cross the specimen, so that the timed window sees every "
                         "facet strained rather than the law's zero-strain path)")
    ap.add_argument("--counters", action="store_true",
                    help="print the algorithmic bytes of each kernel for the workload (per-unit figures and "
                         "totals per launch and per step) and exit; no GPU is used")
    ap.add_argument("--ncu-case", choices=("mixed", "fp64", "adjoint"), default=None,
                    help="profiling target: create the workload (its fixed dt), run the pre-roll, "
                         "then between profiler start and stop 4 steps with plain launches (adjoint: one "
                         "8-step ldpm_adjoint, checkpoints every 4 steps, on the adjoint workload in mixed "
                         "precision) and exit; nothing is timed")
    args = ap.parse_args()
    if args.counters:
        print(json.dumps(counters(args)), flush=True)
        return
    if args.ncu_case:
        from paper_2603_13190_gb300 import ldpm

        import torch

        # the captured launches come after the pre-roll: run ncu with --profile-from-start off
        if args.ncu_case == "adjoint":
            wl, spec, bc = make_inputs("adjoint_uniaxial_tension")
            m = ldpm.Model(spec, wl.material, precision="mixed", dt=wl.dt, bc=bc, graph_chunk=-1)
            m.step(200 if args.preroll is None else args.preroll)
            m.sync()
            seed = np.zeros((spec.n_particles, 6))
            seed[spec.face_nodes(2, 1), 2] = 1.0
            torch.cuda.profiler.start()
            m.adjoint(8, seed, 4)
        else:
            wl, spec, bc = make_inputs(args.workload)
            m = ldpm.Model(spec, wl.material, precision=args.ncu_case, dt=wl.dt or 2e-7, bc=bc, graph_chunk=-1)
            if args.launch != "auto":
                ldpm.ldpm_set_launch_mode(m.h, LAUNCH_MODES[args.launch])
            m.step(wl.preroll if args.preroll is None else args.preroll)
            m.sync()
            torch.cuda.profiler.start()
            m.step(4)
        m.sync()
        torch.cuda.profiler.stop()
        m.close()
        print("ncu case done: F=%d" % spec.n_facets)
        return
    if args.warmup < 3:
        args.warmup = 3
    if args.impl == "reference":
        rank = int(os.environ.get("RANK", "0"))
        world = int(os.environ.get("WORLD_SIZE", "1"))
        res = run_reference(args, rank, world)
        if res is not None:
            print(json.dumps(res), flush=True)
        return
    rank, world, local = dist_setup(args.gpus)
    if args.workload == "adjoint_uniaxial_tension":
        res = run_adjoint(args, rank, world, local)
        if rank == 0:
            if world == 1 and not args.no_cpu_baseline:
                from paper_2603_13190_gb300 import workloads

                wl = workloads.WORKLOADS["adjoint_uniaxial_tension"]
                spec = wl.specimen()
                res["cpu_baseline"] = cpu_baseline_adjoint(spec, wl, workloads.workload_bc(wl.name, spec),
                                                           res["config"]["dt_s"])
            print(json.dumps(res), flush=True)
        if world > 1:
            import torch.distributed as dist

            dist.destroy_process_group()
        return
    if args.workload == "batched_unconfined_compression":
        res = run_batch(args, rank, world, local)
        if rank == 0:
            print(json.dumps(res), flush=True)
        if world > 1:
            import torch.distributed as dist

            dist.destroy_process_group()
        return
    res, spec, wl, bc, cpu = run_ours(args, rank, world, local)
    if rank == 0:
        if cpu is not None:
            try:
                res["cpu_baseline"] = cpu.result()
                res["cpu_all_cores"] = cpu.all_cores()
            finally:
                cpu.close()
        print(json.dumps(res), flush=True)
    if world > 1:
        import torch.distributed as dist

        dist.destroy_process_group()


if __name__ == "__main__":
    main()
