"""Benchmark of the fused D3Q27 CHM-MRT stream-collide step on GB300.

Workload: pulsatile (Womersley) pipe flow, radius 28 in a 64x64x256 box periodic along z,
tau 0.55, Womersley number 4, sinusoidal body force of amplitude 1e-5 -- 632,832 fluid cells.
One benchmark step = one lattice Boltzmann time step over every fluid cell (one launch of the
fused kernel).  The headline runs the faster of the two pull schemes the method admits, the
esoteric twist (in place, state 100 MB) and A-B (two population arrays, 190 MB), each with its
autotuned launch configuration; the line names the scheme and the other one is a variant.
Before every timed step, outside the timed region, the L2 cache is flushed by writing a 512 MB
buffer and then reading another 512 MB buffer (so that the flush's own dirty lines are written
back before the step starts): every step streams its populations from HBM into a clean, cold L2
(the twist's FP32 state fits in the 129 MB L2, A-B's does not: the line says which).  The
larger-than-L2 anchor, the seeded synthetic aneurysm at 512^3 (FP32 twist state 215 MB), is
timed back to back and reported as its own roofline object.  Variants: FP16 / BF16 storage, the
other scheme, the SRT / TRT operators, 16 batched aneurysms (graph of launches, persistent launch, and 16
sequential runs), and the coarse grid + learned corrector comparison (errors and wall times of
fine, coarse and coarse + corrector runs, and the plain resolution of equal error).

Metric: fluid MLUPS (million fluid-cell updates per second) and the fraction of the HBM roofline
achieved with the algorithmic 27 reads + 27 writes per update (216 B in FP32, 108 B in
FP16/BF16): `frac` against the measured copy bandwidth, `frac_of_8tbs` against the metric's
8 TB/s.

Arms:
  default            the CUDA library (this repository), FP32 storage as the headline, FP16 and
                     BF16 storage, the other scheme and the classical SRT and TRT operators
                     (second-order equilibrium) as variants; plus an end-to-end figure through
                     the public API with host buffers, and the FP64 oracle timed on the host
                     cores.
  --impl reference   the FP64 CPU oracle alone on the same workload (bounded sample: the
                     one-layer z-slab, exact for this z-invariant flow), on the host cores.
Multi-GPU (torchrun): each rank runs an independent replica of the workload (weak scaling);
value = total updates of all ranks / max time over ranks.
"""
import argparse
import json
import os
import statistics
import subprocess
import sys
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

WORKLOAD = "womersley_pipe_64x64x256_R28_Wo4_tau0.55"
METRIC = "fluid MLUPS, D3Q27 CHM-MRT fused stream-collide (% of HBM roofline: measured copy peak and 8 TB/s)"
BYTES_PER_VALUE = {"fp32": 4, "fp16": 2, "bf16": 2}
NOMINAL_HBM_GBS = 8000.0  # the metric's roofline denominator (bytes per fluid-cell update over 8 TB/s)
# DRAM bytes per launch (ncu dram__bytes_read.sum + dram__bytes_write.sum, one capture of the
# kernel named, --clock-control none) of the step kernel, keyed by (workload, storage, launch
# configuration); reported only for the configuration the bench runs, None for any other.  An
# entry is removed whenever the kernel it was taken on changes.
K_STEP_TRAFFIC = {
    ("womersley", "fp32", "ab", "256x3"): (120_867_328, "k_step<fp32, A-B, 4 bricks, 3 CTAs/SM, default rates, no links> (89.77 MB read, 31.10 MB written)"),
    ("womersley", "fp32", "ab", "128x7"): (120_340_992, "k_step<fp32, A-B, 2 bricks, 7 CTAs/SM, default rates, no links> (89.81 MB read, 30.53 MB written)"),
    ("womersley", "fp32", "ab", "128x6"): (121_096_704, "k_step<fp32, A-B, 2 bricks, 6 CTAs/SM, default rates, no links> (89.82 MB read, 31.28 MB written)"),
    ("womersley", "fp32", "ab", "128x8"): (120_348_160, "k_step<fp32, A-B, 2 bricks, 8 CTAs/SM, default rates, no links> (89.79 MB read, 30.55 MB written)"),
    ("womersley", "fp32", "ab", "128x10"): (122_133_760, "k_step<fp32, A-B, 2 bricks, 10 CTAs/SM, default rates, no links> (89.72 MB read, 32.42 MB written)"),
    ("womersley", "fp32", "esoteric", "256x3"): (97_949_184, "k_step<fp32, twist, 4 bricks, 3 CTAs/SM, default rates, parity 1, no links> (82.82 MB read, 15.13 MB written)"),
    ("womersley", "fp32", "esoteric", "128x7"): (98_066_432, "k_step<fp32, twist, 2 bricks, 7 CTAs/SM, default rates, parity 1, no links> (82.82 MB read, 15.25 MB written)"),
    ("womersley", "fp32", "esoteric", "128x6"): (97_976_576, "k_step<fp32, twist, 2 bricks, 6 CTAs/SM, default rates, parity 1, no links> (82.83 MB read, 15.14 MB written)"),
    ("womersley", "fp32", "esoteric", "128x8"): (98_131_968, "k_step<fp32, twist, 2 bricks, 8 CTAs/SM, default rates, parity 1, no links> (82.81 MB read, 15.32 MB written)"),
    ("womersley", "fp32", "esoteric", "128x10"): (101_006_080, "k_step<fp32, twist, 2 bricks, 10 CTAs/SM, default rates, parity 1, no links> (82.98 MB read, 18.03 MB written)"),
    ("womersley", "fp32", "esoteric", "pipe128x6"): (95_522_816, "k_step_et_pipe<fp32, 2 bricks, 6 CTAs/SM, persistent> (79.98 MB read, 15.54 MB written)"),
    ("womersley", "fp32", "esoteric", "2c128x4"): (98_055_424, "k_step2<fp32, 4 bricks, 4 CTAs/SM> (82.85 MB read, 15.20 MB written)"),
    ("womersley", "fp32", "esoteric", "2c128x3"): (97_840_128, "k_step2<fp32, 4 bricks, 3 CTAs/SM> (82.86 MB read, 14.98 MB written)"),
    ("aneurysm512", "fp32", "esoteric", "256x3"): (247_981_312, "k_step<fp32, twist, 4 bricks, 3 CTAs/SM, default rates, parity 1, 3 link rounds> (166.84 MB read, 81.14 MB written)"),
    ("aneurysm512", "fp32", "esoteric", "128x7"): (253_959_424, "k_step<fp32, twist, 2 bricks, 7 CTAs/SM, default rates, parity 1, 3 link rounds> (167.02 MB read, 86.94 MB written)"),
    ("aneurysm512", "fp32", "esoteric", "128x6"): (248_123_136, "k_step<fp32, twist, 2 bricks, 6 CTAs/SM, default rates, parity 1, 3 link rounds> (166.84 MB read, 81.28 MB written)"),
    ("aneurysm512", "fp32", "esoteric", "128x8"): (248_439_040, "k_step<fp32, twist, 2 bricks, 8 CTAs/SM, default rates, parity 1, 3 link rounds> (166.81 MB read, 81.63 MB written)"),
    ("aneurysm512", "fp32", "esoteric", "128x10"): (271_365_888, "k_step<fp32, twist, 2 bricks, 10 CTAs/SM, default rates, parity 1, 3 link rounds> (167.36 MB read, 104.01 MB written)"),
    ("aneurysm512", "fp32", "esoteric", "pipe128x6"): (242_021_120, "k_step_et_pipe<fp32, 2 bricks, 6 CTAs/SM, persistent> (159.48 MB read, 82.54 MB written)"),
    ("aneurysm512", "fp32", "esoteric", "2c128x4"): (246_262_272, "k_step2<fp32, 4 bricks, 4 CTAs/SM> (165.11 MB read, 81.16 MB written)"),
    ("aneurysm512", "fp32", "esoteric", "2c128x3"): (246_018_816, "k_step2<fp32, 4 bricks, 3 CTAs/SM> (165.18 MB read, 80.84 MB written)"),
}


def dist_env():
    return int(os.environ.get("RANK", 0)), int(os.environ.get("WORLD_SIZE", 1)), int(os.environ.get("LOCAL_RANK", 0))


def measured_peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            p = json.load(f)
        return float(p["hbm_gbs"]), "measured"
    except Exception:
        return 6800.0, "fallback"


def run_oracle_sample(seconds, threads=None):
    """The FP64 oracle on the workload's one-layer z-slab (2472 fluid cells), advanced in
    chunks until `seconds` of CPU work have passed; returns (MLUPS, threads, description)."""
    import oracle
    from paper_2101_11107_gb300 import inputs as I

    if threads:
        oracle.set_threads(threads)
    g = I.womersley_pipe()
    slab = g.mask[:1].copy()
    c = oracle.Case(slab, periodic=g.periodic, tau=g.tau, gamp=g.gamp, gomega=g.gomega)
    c.step(5)
    n = 0
    t0 = time.perf_counter()
    while time.perf_counter() - t0 < seconds:
        c.step(20)
        n += 20
    dt = time.perf_counter() - t0
    nf = c.nfluid
    return nf * n / dt / 1e6, oracle.get_threads(), f"{n} steps of the 64x64x1 z-slab ({nf} fluid cells), {dt:.1f} s"


class ClockSampler:
    """nvidia-smi clock / throttle sampling during the timed region."""

    QUERY = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index):
        self.gpu = gpu_index
        self.proc = None

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.gpu), f"--query-gpu={self.QUERY}",
                                          "--format=csv,noheader,nounits", "-lms", "100"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except Exception:
            self.proc = None
        time.sleep(0.3)
        return self

    def __exit__(self, *a):
        self.out = ""
        if self.proc is not None:
            time.sleep(0.2)
            self.proc.terminate()
            try:
                self.out, _ = self.proc.communicate(timeout=5)
            except Exception:
                self.proc.kill()

    def summary(self):
        sm, smax, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in (self.out or "").splitlines():
            f = [x.strip() for x in line.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                smax = float(f[2])
            except ValueError:
                continue
            for name, v in zip(names, f[5:9]):
                if v.lower() == "active":
                    reasons.add(name)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": smax, "reasons": ["unavailable"], "samples": 0}
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": smax, "reasons": sorted(reasons), "samples": len(sm)}


def flush_l2(flush, clean):
    flush.add_(1)        # evicts the domain's lines (writes 512 MB)
    clean.sum()          # evicts the flush's dirty lines (reads 512 MB), so L2 starts clean


def time_steps(dom, steps, warmup, flush, stream, clean=None):
    """Per-step CUDA-event times (ms) of `steps` single-step launches, L2 flushed before each."""
    import torch

    dom.step(warmup)
    torch.cuda.synchronize()
    starts = [torch.cuda.Event(enable_timing=True) for _ in range(steps)]
    ends = [torch.cuda.Event(enable_timing=True) for _ in range(steps)]
    for k in range(steps):
        flush_l2(flush, clean)
        starts[k].record(stream)
        dom.step(1)
        ends[k].record(stream)
    torch.cuda.synchronize()
    return [s.elapsed_time(e) for s, e in zip(starts, ends)]


def batched_variant(steps, flush, clean, stream):
    """Sixteen seeded synthetic aneurysms (box edges drawn from 96..192 in steps of 16, distinct
    inflow waveforms), FP16 storage, esoteric twist: `steps` steps of all of them through one
    batched launch per step replayed as CUDA graphs, against the same steps as 16 sequential
    per-domain runs.  L2 is flushed before each timed run."""
    import numpy as np
    import torch
    from paper_2101_11107_gb300 import inputs as I
    from paper_2101_11107_gb300 import lbm

    rng = np.random.default_rng(2024)
    edges = [int(96 + 16 * rng.integers(0, 7)) for _ in range(16)]
    geoms = [I.aneurysm(300 + k, edge=e, wave_seed=400 + k) for k, e in enumerate(edges)]
    doms = [lbm.Domain.from_geometry(g, storage="fp16") for g in geoms]
    nf = sum(d.info()["n_fluid"] for d in doms)
    for d in doms:
        d.autotune(10)
    graph_steps = 50
    batch = lbm.Batch(doms, graph_steps=graph_steps)
    best, _ = batch.autotune(10)
    batch.step(graph_steps)  # capture + warm-up
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    flush_l2(flush, clean)
    e0.record(stream)
    batch.step(steps)
    e1.record(stream)
    torch.cuda.synchronize()
    t_batch = e0.elapsed_time(e1)
    for d in doms:
        d.step(5)
    flush_l2(flush, clean)
    e0.record(stream)
    for d in doms:
        d.step(steps)
    e1.record(stream)
    torch.cuda.synchronize()
    t_seq = e0.elapsed_time(e1)
    # the same batch as one persistent cooperative launch per graph chunk (grid barrier between
    # steps)
    batch.set_persistent(True, 1.0)
    batch.step(graph_steps)  # capture + warm-up
    batch.sync()
    flush_l2(flush, clean)
    e0.record(stream)
    batch.step(steps)
    e1.record(stream)
    torch.cuda.synchronize()
    batch.sync()
    t_pers = e0.elapsed_time(e1)
    batch.close()
    for d in doms:
        d.close()
    return {"domains": len(doms), "edges": edges, "fluid_cells": nf, "steps": steps,
            "batched_graph_mlups": nf * steps / (t_batch * 1e-3) / 1e6,
            "persistent_graph_mlups": nf * steps / (t_pers * 1e-3) / 1e6,
            "sequential_mlups": nf * steps / (t_seq * 1e-3) / 1e6,
            "speedup": t_seq / t_batch, "batched_ms": t_batch, "persistent_ms": t_pers, "sequential_ms": t_seq,
            "launch_config": lbm.LAUNCH_CONFIG_NAMES[best], "graph_steps": graph_steps}


def large_variant(stream, steps=100):
    """The seeded synthetic aneurysm at 512^3 (working set larger than L2), FP32 and FP16
    storage, twist, autotuned, timed back to back (one CUDA-event pair around `steps` steps):
    each step streams a state larger than L2, so no flush is needed between steps."""
    import torch
    from paper_2101_11107_gb300 import inputs as I
    from paper_2101_11107_gb300 import lbm

    g = I.aneurysm(11, edge=512)
    out = {}
    for storage in ("fp32", "fp16"):
        dom = lbm.Domain.from_geometry(g, storage=storage)
        best, _ = dom.autotune(10)
        info = dom.info()
        nf = info["n_fluid"]
        dom.step(10)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        e0.record(stream)
        dom.step(steps)
        e1.record(stream)
        torch.cuda.synchronize()
        ms = e0.elapsed_time(e1) / steps
        bytes_alg = 2 * 27 * BYTES_PER_VALUE[storage] * nf
        l2 = torch.cuda.get_device_properties(torch.cuda.current_device()).L2_cache_size
        out[f"aneurysm512_{storage}"] = {
            "ms_per_step": ms, "mlups": nf / (ms * 1e-3) / 1e6, "fluid_cells": nf,
            "algorithmic_bytes_per_launch": bytes_alg,
            "achieved_gbs": bytes_alg / (ms * 1e-3) / 1e9, "device_bytes": info["device_bytes"],
            "working_set_over_l2": info["device_bytes"] / l2, "launch_config": lbm.LAUNCH_CONFIG_NAMES[best],
            "timing": "back to back (working set larger than L2)"}
        dom.close()
    return out


def corrector_variant(test_seeds=(200, 201, 202, 203), compare_edges=(144, 160)):
    """The coarse grid + learned corrector comparison (synthetic aneurysms, fine 256^3 / coarse
    128^3, Re 300, 32 training geometries, corrector trained on the GPU with 4 rounds of in-loop
    data), evaluated on held-out geometries: relative L2 error of u against the restricted fine
    run, wall times of the fine, plain coarse and coarse + corrector runs (CUDA events, one
    geometry at a time), and the resolution at which the plain solver reaches coarse +
    corrector's error with its wall time (plain runs at intermediate resolutions)."""
    from paper_2101_11107_gb300 import corrector_study as S

    t0 = time.perf_counter()
    summary, _ = S.run(fine_edge=256, period_f=4000, reynolds=300.0, train_seeds=list(range(100, 132)),
                       test_seeds=list(test_seeds), periods=3, samples_per_period=10, train_steps=4000, lr=1e-3,
                       apply_every=50, workers=16, log=lambda m: None, dagger_rounds=4,
                       compare_edges=tuple(compare_edges))
    keys = ("err_plain_mean", "err_corrected_mean", "err_output_corrected_mean", "si_plain_mean",
            "si_corrected_mean", "wall_fine_s", "wall_coarse_s", "wall_coarse_corrector_s", "train_s")
    out = {k: summary[k] for k in keys}
    out.update({"test_geometries": len(test_seeds), "training_geometries": 32, "equal_error": summary["equal_error"],
                "study_wall_s": time.perf_counter() - t0,
                "fallbacks": sum(r["fallback_at_step"] is not None for r in summary["per_geometry"])})
    return out


def max_over_ranks(x: float, device=None) -> float:
    """The maximum of x over all ranks of the initialised process group (x itself with one rank)."""
    import torch
    import torch.distributed as dist

    if not (dist.is_available() and dist.is_initialized()) or dist.get_world_size() == 1:
        return x
    t = torch.tensor([x], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def replica_throughput(world: int, cells_per_rank: int, steps: int, max_ms: float) -> float:
    """Whole-job MLUPS of `world` independent replicas that each advanced `cells_per_rank` cells
    `steps` times, timed by the slowest rank (max_ms for all steps)."""
    return world * cells_per_rank * steps / (max_ms * 1e-3) / 1e6


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=200)
    ap.add_argument("--warmup", type=int, default=10)
    ap.add_argument("--impl", default="gb300", choices=["gb300", "reference"])
    ap.add_argument("--cpu-seconds", type=float, default=12.0)
    ap.add_argument("--no-variants", action="store_true")
    args = ap.parse_args()
    rank, world, local = dist_env()

    if args.impl == "reference":
        if rank != 0:
            return
        per = max(0.2, min(20.0, 150.0 / max(1, args.steps + args.warmup)))
        for _ in range(args.warmup):
            run_oracle_sample(per)
        vals = []
        desc = ""
        thr = 1
        for _ in range(args.steps):
            v, thr, desc = run_oracle_sample(per)
            vals.append(v)
        value = statistics.mean(vals)
        line = {"impl": "reference", "metric": METRIC, "value": value, "unit": "MLUPS", "n_gpus": args.gpus,
                "steps": args.steps, "warmup": args.warmup, "ms_per_step": per * 1000.0, "higher_is_better": True,
                "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
                "config": {"workload": WORKLOAD, "storage": "fp64 (oracle)", "sample": "64x64x1 z-slab"},
                "cpu_baseline": {"value": value, "unit": "MLUPS", "cores": thr, "kind": "oracle", "sample": desc},
                "e2e": {"value": value, "unit": "MLUPS", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
        print(json.dumps(line), flush=True)
        return

    import torch

    if world > 1:
        import torch.distributed as dist
        torch.cuda.set_device(local)
        dist.init_process_group("nccl")
    else:
        torch.cuda.set_device(0)
    dev = torch.device("cuda", torch.cuda.current_device())
    import __graft_entry__
    from paper_2101_11107_gb300 import build as lib_build

    if rank == 0:
        __graft_entry__.build()
    if world > 1:
        torch.distributed.barrier()
    lib_build.build()
    from paper_2101_11107_gb300 import inputs as I
    from paper_2101_11107_gb300 import lbm

    stream = torch.cuda.current_stream(dev)
    flush = torch.zeros(512 * 1024 * 1024 // 4, dtype=torch.float32, device=dev)
    clean = torch.zeros(512 * 1024 * 1024 // 4, dtype=torch.float32, device=dev)
    g = I.womersley_pipe()
    hbm_peak, peak_kind = measured_peaks()

    results = {}
    clocks = None
    # the headline runs the faster of the two pull schemes the method admits -- the esoteric twist
    # (in place) and A-B (two arrays) -- each with its autotuned launch configuration, chosen by a
    # 20-step cold timing (rank 0's choice on every rank); the other is reported as a variant
    cand = {}
    for scheme in ("esoteric", "ab"):
        dom = lbm.Domain.from_geometry(g, storage="fp32", scheme=scheme)
        best, tune = dom.autotune(20)
        pre_ms = statistics.mean(time_steps(dom, 20, 3, flush, stream, clean))
        cand[scheme] = (dom, best, tune, pre_ms)
    head = min(cand, key=lambda k: cand[k][3])
    if world > 1:
        choice = [head]
        torch.distributed.broadcast_object_list(choice, src=0)
        head = choice[0]
    head_key = "fp32" if head == "esoteric" else "fp32_ab"
    variants = [("fp32", "esoteric", "chm"), ("fp32", "ab", "chm")]
    if not args.no_variants:
        variants += [("fp16", "esoteric", "chm"), ("bf16", "esoteric", "chm"), ("fp32", "esoteric", "srt2"),
                     ("fp32", "esoteric", "trt2")]
    for storage, scheme, collision in variants:
        key = storage if scheme == "esoteric" else f"{storage}_{scheme}"
        if collision != "chm":
            key += "_" + collision
        if storage == "fp32" and collision == "chm":
            dom, best, tune, _ = cand[scheme]
        else:
            dom = lbm.Domain.from_geometry(g, storage=storage, scheme=scheme, collision=collision)
            best, tune = dom.autotune(20)
        info = dom.info()
        nf = info["n_fluid"]
        if key == head_key:
            sampler = ClockSampler(local)
            if world > 1:
                torch.distributed.barrier()
            torch.cuda.synchronize()
            with sampler:
                t0 = time.perf_counter()
                times = time_steps(dom, args.steps, args.warmup, flush, stream, clean)
                wall = time.perf_counter() - t0
            clocks = sampler.summary()
            fp32_times = times
            if world > 1:
                torch.cuda.synchronize()
                torch.distributed.barrier()
        else:
            times = time_steps(dom, args.steps, args.warmup, flush, stream, clean)
        ms = statistics.mean(times)
        bytes_alg = 2 * 27 * BYTES_PER_VALUE[storage] * nf
        results[key] = {"ms_per_step": ms, "mlups": nf / (ms * 1e-3) / 1e6, "fluid_cells": nf,
                        "algorithmic_bytes_per_launch": bytes_alg,
                        "achieved_gbs": bytes_alg / (ms * 1e-3) / 1e9, "scheme": scheme, "collision": collision,
                        "launch_config": lbm.LAUNCH_CONFIG_NAMES[best],
                        "autotune_ms_back_to_back": {k: round(v, 5) for k, v in tune.items()},
                        "device_bytes": info["device_bytes"], "slots": info["n_slots"]}
        if key != head_key:
            dom.close()
        else:
            main_dom = dom

    main = results[head_key]
    total_ms = max_over_ranks(sum(fp32_times), dev)
    value = replica_throughput(world, main["fluid_cells"], args.steps, total_ms)

    # end to end through the public API, host buffers: upload the initial macroscopic state from
    # pinned host memory, advance 200 steps, read rho and u back to pinned host memory
    inner = 200
    nz, ny, nx = g.mask.shape
    nbox = nx * ny * nz
    rho_h = torch.ones(nbox, dtype=torch.float32).pin_memory().numpy().reshape(nz, ny, nx)
    u_h = torch.zeros(3 * nbox, dtype=torch.float32).pin_memory().numpy().reshape(3, nz, ny, nx)
    rho_o = torch.empty(nbox, dtype=torch.float32).pin_memory().numpy()
    u_o = torch.empty(3 * nbox, dtype=torch.float32).pin_memory().numpy()
    L = lbm.load_library()
    import ctypes
    e2e_steps = max(3, min(10, args.steps // 20))
    main_dom.init_equilibrium(rho_h, u_h)
    main_dom.step(inner)
    L.lbm_get_macroscopic(main_dom._h, ctypes.c_void_p(rho_o.ctypes.data), ctypes.c_void_p(u_o.ctypes.data), 1, 0)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for _ in range(e2e_steps):
        main_dom.init_equilibrium(rho_h, u_h)
        main_dom.step(inner)
        st = L.lbm_get_macroscopic(main_dom._h, ctypes.c_void_p(rho_o.ctypes.data),
                                   ctypes.c_void_p(u_o.ctypes.data), 1, 0)
        assert st == 0
    torch.cuda.synchronize()
    e2e_s = (time.perf_counter() - t0) / e2e_steps
    e2e_val = world * main["fluid_cells"] * inner / e2e_s / 1e6

    batch_result = None if args.no_variants else batched_variant(200, flush, clean, stream)
    large_result = None if args.no_variants else large_variant(stream)
    corrector_result = None if (args.no_variants or world > 1) else corrector_variant()

    cpu = None
    if rank == 0 and world == 1:
        v, thr, desc = run_oracle_sample(args.cpu_seconds)
        cpu = {"value": v, "unit": "MLUPS", "cores": thr, "kind": "oracle", "sample": desc}
        # the same oracle on one core, a shorter sample
        v1, _, desc1 = run_oracle_sample(max(1.0, args.cpu_seconds / 3), threads=1)
        run_oracle_sample(0.0, threads=thr)  # back to all cores
        cpu["single_core"] = {"value": v1, "unit": "MLUPS", "cores": 1, "sample": desc1}

    if rank != 0:
        return
    achieved = main["achieved_gbs"]
    l2_bytes = torch.cuda.get_device_properties(dev).L2_cache_size
    traffic, traffic_kernel = K_STEP_TRAFFIC.get(("womersley", "fp32", head, main["launch_config"]), (None, None))
    fits = bool(main["device_bytes"] <= l2_bytes)
    line = {
        "metric": METRIC, "value": value, "unit": "MLUPS", "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": main["ms_per_step"], "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": {"workload": WORKLOAD, "storage": "fp32 deviations",
                   "scheme": "esoteric twist (in place)" if head == "esoteric" else "A-B (two population arrays)",
                   "scheme_choice": {"rule": "faster of the two pull schemes, each autotuned, by a 20-step cold timing",
                                     "cold_ms_20_steps": {k: round(v[3], 5) for k, v in cand.items()}},
                   "launch_config": main["launch_config"], "fluid_cells": main["fluid_cells"],
                   "box": [nx, ny, nz],
                   "l2": "flushed before every timed step (512 MB write, then 512 MB read: cold, clean L2)",
                   "state_bytes": main["device_bytes"], "l2_bytes": l2_bytes,
                   "state_fits_in_l2": fits,
                   "parallelism": "replicas" if world > 1 else "single GPU",
                   "bytes_per_update_algorithmic": 216, "wall_s_timed_loop": wall},
        "roofline": {"bound": "hbm", "achieved": achieved, "peak": hbm_peak, "unit": "GB/s",
                     "frac": achieved / hbm_peak, "frac_of_8tbs": achieved / NOMINAL_HBM_GBS,
                     "traffic": traffic,
                     "traffic_unit": "DRAM bytes per launch (ncu dram__bytes_read.sum + dram__bytes_write.sum) of "
                                     + (traffic_kernel or "no capture of this launch configuration"),
                     "peak_kind": peak_kind + " copy bandwidth (hbm_gbs); frac_of_8tbs: the metric's 8 TB/s",
                     "note": ("the FP32 state of this workload fits in L2; the larger-than-L2 anchor is "
                              "roofline_larger_than_l2") if fits else
                             "the state of this workload (two population arrays) is larger than L2"},
        "cpu_baseline": cpu,
        "e2e": {"value": e2e_val, "unit": "MLUPS", "h2d_bytes_per_step": 16 * nbox, "d2h_bytes_per_step": 16 * nbox,
                "inner_lbm_steps": inner,
                "note": "per e2e step: upload of rho, u from pinned host memory, 200 lattice steps back to back "
                        "(no L2 flush between them, unlike the device-timed value), read-back of rho, u"},
        "gpu_launches": args.steps,
        "clocks": clocks,
        "variants": {k: {kk: (round(vv, 4) if isinstance(vv, float) else vv) for kk, vv in r.items()}
                     for k, r in results.items()},
    }
    for k, r in results.items():
        line["variants"][k]["roofline_frac"] = round(r["achieved_gbs"] / hbm_peak, 4)
        line["variants"][k]["roofline_frac_of_8tbs"] = round(r["achieved_gbs"] / NOMINAL_HBM_GBS, 4)
    if batch_result is not None:
        bb = 2 * 27 * 2 * batch_result["fluid_cells"] * batch_result["steps"] / (batch_result["batched_ms"] * 1e-3) / 1e9
        batch_result["achieved_gbs"] = bb
        batch_result["roofline_frac"] = round(bb / hbm_peak, 4)
        batch_result["roofline_frac_of_8tbs"] = round(bb / NOMINAL_HBM_GBS, 4)
        line["variants"]["batch16_aneurysm_fp16"] = batch_result
    if corrector_result is not None:
        line["variants"]["coarse_corrector_aneurysm256"] = corrector_result
    if large_result is not None:
        for k, r in large_result.items():
            r["roofline_frac"] = round(r["achieved_gbs"] / hbm_peak, 4)
            r["roofline_frac_of_8tbs"] = round(r["achieved_gbs"] / NOMINAL_HBM_GBS, 4)
            line["variants"][k] = r
        big = large_result["aneurysm512_fp32"]
        t_big, k_big = K_STEP_TRAFFIC.get(("aneurysm512", "fp32", "esoteric", big["launch_config"]), (None, None))
        line["roofline_larger_than_l2"] = {
            "workload": "synthetic aneurysm 512^3 (seed 11), FP32 storage, esoteric twist, back to back",
            "bound": "hbm", "achieved": big["achieved_gbs"], "peak": hbm_peak, "unit": "GB/s",
            "frac": big["achieved_gbs"] / hbm_peak, "frac_of_8tbs": big["achieved_gbs"] / NOMINAL_HBM_GBS,
            "traffic": t_big,
            "traffic_unit": "DRAM bytes per launch (ncu) of " + (k_big or "no capture of this launch configuration"),
            "state_bytes": big["device_bytes"], "l2_bytes": l2_bytes, "launch_config": big["launch_config"]}
    print(json.dumps(line), flush=True)


if __name__ == "__main__":
    main()
