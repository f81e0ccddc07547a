"""Benchmark of the HVOX transform pair on one GB300 (or N replicas under torchrun).

A step is one sky->vis and one vis->sky transform of the LOFAR-like workload
(HEALPix nside=256, 30 deg cap: 52,812 pixels; 300 antennas, 4 earth-rotation steps,
8 channels: 1,435,200 baselines) at eps = 1e-9 (FP64-accuracy path). The metric is
(N_pix + N_vis) per transform, two transforms per step, divided by the step time.

value:   device-resident inputs, CUDA events per step on the plan's stream, L2 flushed
         (256 MiB write) before every step outside the timed window.
e2e:     the same step through the C ABI with pinned HOST buffers (the library copies
         host->device and device->host inside the call), wall clock.
roofline: the dominant kernel's live CUDA-event time over the timed region.
secondary: the same step at eps = 1e-6 (FP32 path).
plain_fp64: the same step at eps = 1e-9 in the plain form (FP64 arithmetic in every
         kernel, no graph): the comparison the mixed-precision path has to win.
config3: the SKA-Low-like workload (1,470,612 px x 4,186,112 baselines) at eps = 1e-6,
         chunked (NUFFT sub-problems + direct sums), with a serial profiled pass that
         times every kernel alone for the spreading, interpolation and direct rooflines.
sparse_sky: 500 pixels of interest in the 10 km field x 237,705 baselines at eps = 1e-6.
peaks:   throughput probes run live on this GPU (FP32/FP64 FMA, shared-memory atomics,
         L1 loads) for the denominators the driver's measured peaks do not hold.
serving: a seeded request stream served with continuous batching against the plain
         FP64 one-at-a-time form (p50/p99 latency, throughput).
cpu_baseline: the FP64 oracle on this host's cores, on a bounded sample of outputs.

python bench.py [--gpus N] [--steps K] [--warmup W] [--impl reference] [--eps E]
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

METRIC = "3D NUFFT-3 (pix+vis)/s at ε=1e-6/1e-9, served vs plain; p50/p99 ms"
UNIT = "(pix+vis)/s"
WORKLOAD = ("LOFAR-like: HEALPix nside=256 30deg cap (52,812 px) x 300 antennas log-radial 50 m-100 km, "
            "4 hour angles x 8 channels (1,435,200 baselines); step = sky->vis + vis->sky")
FP32_PEAK_FLOPS = 152 * 128 * 2 * 2.07e9  # FP32 FMA pipes x 2 flops x max SM clock
FLOPS_PER_PAIR = 16.0                      # algorithmic flops per (pixel, baseline) pair


def dist_env():
    return int(os.environ.get("RANK", "0")), int(os.environ.get("WORLD_SIZE", "1")), int(os.environ.get("LOCAL_RANK", "0"))


def max_over_ranks(x: float, world: int, device: str = "cuda") -> float:
    """The largest x over all ranks (a timed region ends when the slowest replica does)."""
    if world <= 1:
        return x
    import torch
    import torch.distributed as dist
    t = torch.tensor([x], device=device, dtype=torch.float64)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def whole_job_rate(units_per_rank_step: float, steps: int, seconds: float, world: int) -> float:
    """Units processed by all replicas per second of the slowest replica (weak scaling)."""
    return world * units_per_rank_step * steps / seconds


WORKLOADS = {
    1: "HEALPix nside=32 45deg cap (1,740 px) x 200 antennas in a 1 km disk (19,900 baselines)",
    2: WORKLOAD,
    3: ("SKA-Low-like: HEALPix nside=1024 40deg cap (1,470,612 px) x 512 antennas (Gaussian core + arms), "
        "32 hour angles (4,186,112 baselines); step = sky->vis + vis->sky"),
}


def load_workload(n_vis=None, config=2, core_radius=0.0, radius_km=0.0, sparse=0):
    import numpy as np
    from hvox_inputs import configs
    if radius_km > 0:  # telescope-radius sweep (Table 3 setups), optionally a sparse sky
        return configs.radius_sweep(radius_km, sparse_pixels=sparse)
    w = configs.CONFIGS[config]()
    if core_radius > 0:  # dense core only: baselines with |(u, v)| <= core_radius wavelengths
        w.uvw = np.ascontiguousarray(w.uvw[np.hypot(w.uvw[:, 0], w.uvw[:, 1]) <= core_radius])
    if n_vis:  # leading baselines only (smaller case for profiler captures)
        w.uvw = w.uvw[:n_vis].copy()
    return w


# ---------------------------------------------------------------------------- CPU oracle

def oracle_rate(w, target_s: float, seed: int = 0):
    """Time the oracle on a seeded sample of outputs; returns (pairs/s, seconds, sample text)."""
    import numpy as np
    import oracle
    from hvox_inputs import configs
    vis = configs.visibilities_cn(2, w.n_vis)
    rng = np.random.default_rng(1234 + seed)
    # calibration
    kv = np.sort(rng.choice(w.n_vis, 16, replace=False))
    kp = np.sort(rng.choice(w.n_pix, 2, replace=False))
    t0 = time.perf_counter()
    oracle.sky2vis(w.pix, w.uvw, w.sky, sample=kv)
    oracle.vis2sky(w.pix, w.uvw, vis, sample=kp)
    dt = max(time.perf_counter() - t0, 1e-3)
    rate0 = (len(kv) * w.n_pix + len(kp) * w.n_vis) / dt
    pairs_target = rate0 * target_s
    n_v = int(max(16, min(w.n_vis, pairs_target / 2 / w.n_pix)))
    n_p = int(max(2, min(w.n_pix, pairs_target / 2 / w.n_vis)))
    kv = np.sort(rng.choice(w.n_vis, n_v, replace=False))
    kp = np.sort(rng.choice(w.n_pix, n_p, replace=False))
    t0 = time.perf_counter()
    oracle.sky2vis(w.pix, w.uvw, w.sky, sample=kv)
    oracle.vis2sky(w.pix, w.uvw, vis, sample=kp)
    dt = time.perf_counter() - t0
    pairs = n_v * w.n_pix + n_p * w.n_vis
    sample = (f"{n_v} baselines (each summed over all {w.n_pix} pixels) + {n_p} pixels (each over all "
              f"{w.n_vis} baselines), FP64 direct sums; extrapolated to the full step by pair count")
    return pairs / dt, dt, sample


def cpu_baseline(w, target_s: float = 12.0):
    import oracle
    rate, dt, sample = oracle_rate(w, target_s)
    step_s = 2.0 * w.n_pix * w.n_vis / rate
    return {"value": 2.0 * (w.n_pix + w.n_vis) / step_s, "unit": UNIT, "cores": oracle.num_threads(),
            "kind": "oracle", "sample": sample, "sample_seconds": round(dt, 2)}


def run_reference(args):
    rank, world, _ = dist_env()
    if rank != 0:
        return 0
    w = load_workload()
    import oracle
    per_step = []
    sample = ""
    sampled_s = 0.0
    for i in range(args.warmup + args.steps):
        rate, dt, sample = oracle_rate(w, 4.0, seed=i)
        if i >= args.warmup:
            per_step.append(2.0 * w.n_pix * w.n_vis / rate)
            sampled_s += dt
    step_s = statistics.mean(per_step)
    value = 2.0 * (w.n_pix + w.n_vis) / step_s
    # Each "step" is a bounded sample of the full step's outputs: ms_per_step is the full
    # step's time extrapolated from the sampled rate by pair count, not a time that ran.
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": 0, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": step_s * 1e3, "ms_per_step_extrapolated": True,
            "timing": (f"each step times the oracle on a bounded sample of outputs ({sampled_s / args.steps:.2f} s "
                       f"run per step, {sampled_s:.1f} s over the {args.steps} timed steps); value and ms_per_step "
                       "are extrapolated to the full step by pixel-baseline pair count"),
            "sampled_seconds_total": round(sampled_s, 2),
            "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": WORKLOAD, "eps": args.eps, "n_pix": w.n_pix, "n_vis": w.n_vis},
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": oracle.num_threads(), "kind": "oracle",
                             "sample": sample},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)
    return 0


# ---------------------------------------------------------------------------- clocks

class ClockSampler:
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.proc = None
        self.path = os.path.join("/tmp", f"hvox_clocks_{os.getpid()}.csv")

    def start(self):
        try:
            self.f = open(self.path, "w")
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.index), f"--query-gpu={self.FIELDS}",
                                          "--format=csv,noheader,nounits", "-lms", "200"], stdout=self.f,
                                         stderr=subprocess.DEVNULL)
        except (OSError, FileNotFoundError):
            self.proc = None

    def stop(self):
        if self.proc is None:
            return None
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        self.f.close()
        sm, mx, reasons = [], 0.0, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in open(self.path):
            parts = [p.strip() for p in line.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                mx = max(mx, float(parts[2]))
            except ValueError:
                continue
            for n, v in zip(names, parts[5:9]):
                if v.lower() == "active":
                    reasons.add(n)
        os.unlink(self.path)
        if not sm:
            return None
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": mx, "reasons": sorted(reasons), "samples": len(sm)}


# ---------------------------------------------------------------------------- GPU arm

def time_steps(plan, I, V, steps, flush, per_direction=None):
    """Device time (ms) of each step (sky -> vis then vis -> sky); per_direction, if a
    list, receives (sky -> vis ms, vis -> sky ms) per step from an event between them."""
    import torch
    times = []
    for _ in range(steps):
        flush.zero_()
        s, m, e = (torch.cuda.Event(enable_timing=True) for _ in range(3))
        s.record()
        plan.synthesize(I)
        m.record()
        plan.analyze(V)
        e.record()
        times.append((s, m, e))
    torch.cuda.synchronize()
    if per_direction is not None:
        per_direction.extend((s.elapsed_time(m), m.elapsed_time(e)) for s, m, e in times)
    return [s.elapsed_time(e) for s, m, e in times]


def serving_study():
    """Served (continuous batching, mixed precision) vs plain (FP64, one job at a time) on
    the same seeded request stream, as it arrives (latency) and all present at t = 0
    (throughput, not bound by the arrival rate); and a larger served stream run twice.
    Latency = completion - arrival; throughput = sum of (N_pix + N_vis) over requests /
    makespan; tail_ms splits the slowest 1 % into plan wait, slot wait and device time."""
    from hvox_inputs import configs
    from paper_2306_06007_gb300.serve import Server
    out = {}
    small = configs.config5_requests(100, rate_hz=50.0, n_min=1e3, n_max=3e4, seed_offset=11)
    for name, kw in (("served", {"max_inflight": 8}), ("plain", {"plain": True})):
        for realtime, suffix in ((True, ""), (False, "_saturated")):
            srv = Server(**kw)
            rep = srv.run(small, realtime=realtime)
            srv.close()
            out[name + suffix] = rep.summary()
    out["stream"] = ("100 requests, Poisson 50/s, N_pix and N_vis log-uniform [1e3, 3e4] (HEALPix caps <= 40 deg; "
                     "config-2/3 layouts), eps uniform {1e-4, 1e-6, 1e-9}, S or A; *_saturated: the same "
                     "requests all present at t = 0")
    big = configs.config5_requests(400, rate_hz=50.0, n_min=1e4, n_max=2e5, seed_offset=12)
    for run in (1, 2):
        srv = Server(max_inflight=8)
        rep = srv.run(big, realtime=True)
        srv.close()
        out[f"served_large_run{run}"] = rep.summary()
    out["stream_large"] = "400 requests, Poisson 50/s, N log-uniform [1e4, 2e5], otherwise as above; run twice"
    return out


def probe_peaks():
    """Live throughput probes on this GPU (libhvox_peaks.so): FP32 / FP64 FMA flop/s,
    shared-memory float atomicAdd/s and L1 load bytes/s; None if the probe is missing."""
    import ctypes
    path = os.path.join(ROOT, "paper_2306_06007_gb300", "libhvox_peaks.so")
    if not os.path.exists(path):
        return None
    lib = ctypes.CDLL(path)
    out = (ctypes.c_double * 6)()
    if lib.hvox_probe_peaks(out) != 0:
        return None
    return {"fp32_flops": out[0], "fp64_flops": out[1], "smem_atomics_per_s": out[2], "l1_load_bytes_per_s": out[3],
            "smem_int_atomics_per_s": out[4], "smem_float_rmw_per_s": out[5],
            "how": "own probe kernels, CUDA events, full occupancy: FMA chains, conflict-free shared float "
                   "atomicAdd, float2 loads from an L1-resident 16 KiB buffer"}


def stage_roofline(info, st, steps, peaks):
    """Per-kernel rooflines of a serial profiled pass (every stage alone on the plan's
    stream, so each stage time is its own launches' device time): spreading against the
    shared-memory atomic rate (2 float atomics per tap: real and imaginary planes),
    interpolation against L1 load bandwidth (one complex grid value per tap), direct sums
    against the FP32 FMA peak (16 flops per pair)."""
    out = {}
    taps_per_step = info["nufft_points"] * info["w"] ** 3  # every NUFFT point spread once and gathered once
    elem = 8.0 if info["precision"] == 1 else 16.0
    for stage in ("spread", "interp", "direct"):
        n = st["launches"][stage]
        ms = st["ms"][stage]
        if n <= 0 or ms <= 0:
            continue
        avg_s = ms * 1e-3 / n
        per_launch = n / steps
        if stage == "direct":
            work = info["direct_pairs"]  # per direction; one launch per direction
            achieved = work * FLOPS_PER_PAIR / avg_s
            peak = peaks["fp32_flops"] if peaks else FP32_PEAK_FLOPS
            out[stage] = {"bound": "alu", "achieved": achieved / 1e12, "peak": peak / 1e12, "unit": "TFLOP/s",
                          "frac": achieved / peak, "traffic": None, "pairs_per_launch": work,
                          "avg_launch_ms": avg_s * 1e3, "pairs_per_s": work / avg_s,
                          "peak_note": "FP32 FMA probe (measured live)" if peaks else "FP32 pipes (derived)"}
            continue
        taps = taps_per_step / per_launch
        if stage == "spread":
            achieved = 2.0 * taps / avg_s
            peak = peaks["smem_atomics_per_s"] if peaks else None
            out[stage] = {"bound": "smem_atomic", "achieved": achieved / 1e12, "peak": peak / 1e12 if peak else None,
                          "unit": "T atomics/s", "frac": achieved / peak if peak else None, "traffic": None,
                          "taps_per_s": taps / avg_s, "avg_launch_ms": avg_s * 1e3, "launches_per_step": per_launch,
                          "peak_note": "conflict-free shared-memory float atomicAdd probe (measured live); taps "
                                       "that miss a CTA's shared tile go to global atomics instead"}
        else:
            achieved = elem * taps / avg_s
            peak = peaks["l1_load_bytes_per_s"] if peaks else None
            out[stage] = {"bound": "l1", "achieved": achieved / 1e12, "peak": peak / 1e12 if peak else None,
                          "unit": "TB/s", "frac": achieved / peak if peak else None, "traffic": None,
                          "taps_per_s": taps / avg_s, "avg_launch_ms": avg_s * 1e3, "launches_per_step": per_launch,
                          "peak_note": "L1-resident float2 load probe (measured live); one complex grid value per tap"}
    return out


def run_gpu(args):
    import numpy as np
    import torch
    import torch.distributed as dist
    import paper_2306_06007_gb300 as hvox
    from hvox_inputs import configs

    rank, world, local = dist_env()
    torch.cuda.set_device(local)
    if world > 1:
        dist.init_process_group("nccl", init_method="env://")
    peaks = probe_peaks()
    flush = torch.empty(64 * 1024 * 1024, dtype=torch.float32, device="cuda")  # 256 MiB > L2

    def measure(w, vis, eps, steps, warmup, with_e2e=False, plain=False, mode=None, serial_steps=0):
        plan = hvox.Plan(w.pix, w.uvw, eps, mode=mode or args.mode, graphs=args.graphs, plain=plain,
                         factor=args.factor if args.factor != "auto" else None, autotune=args.autotune)
        info = plan.info()
        units_per_step = 2.0 * (w.n_pix + w.n_vis)
        I = torch.as_tensor(w.sky, dtype=plan.real_dtype, device="cuda")
        V = torch.as_tensor(vis, dtype=plan.complex_dtype, device="cuda")
        plan.profile(True)  # warm-up runs the profiled form too (its graph is captured there)
        time_steps(plan, I, V, warmup, flush)
        if world > 1:
            dist.barrier()
        torch.cuda.synchronize()
        clocks = ClockSampler(local)
        clocks.start()
        plan.profile(True)
        dirs = []
        ms = time_steps(plan, I, V, steps, flush, dirs)
        st = plan.stats()
        clk = clocks.stop()
        if world > 1:
            dist.barrier()
        total_ms = max_over_ranks(sum(ms), world)
        s2v_ms = max_over_ranks(sum(d[0] for d in dirs), world) / steps
        v2s_ms = max_over_ranks(sum(d[1] for d in dirs), world) / steps
        units = world * (w.n_pix + w.n_vis)
        out = {"plan": plan, "info": info, "ms_per_step": total_ms / steps, "steps": steps, "warmup": warmup,
               "ms_median": max_over_ranks(statistics.median(ms), world),
               "value": whole_job_rate(units_per_step, steps, total_ms * 1e-3, world), "stats": st,
               "clocks": clk,
               "per_direction": {"sky_to_vis_ms": s2v_ms, "vis_to_sky_ms": v2s_ms,
                                 "sky_to_vis_value": units / (s2v_ms * 1e-3),
                                 "vis_to_sky_value": units / (v2s_ms * 1e-3), "unit": UNIT}}
        if serial_steps > 0:
            plan.profile("serial")
            time_steps(plan, I, V, serial_steps, flush)
            out["serial"] = plan.stats()
            out["serial_steps"] = serial_steps
            plan.profile(False)
        if with_e2e:
            Ih = torch.as_tensor(w.sky, dtype=plan.real_dtype).pin_memory()
            Vh = torch.as_tensor(vis, dtype=plan.complex_dtype).pin_memory()
            Vo = torch.empty(w.n_vis, dtype=plan.complex_dtype).pin_memory()
            Io = torch.empty(w.n_pix, dtype=plan.real_dtype).pin_memory()
            for _ in range(max(1, warmup)):
                plan.synthesize(Ih, out=Vo)
                plan.analyze(Vh, out=Io)
            if world > 1:
                dist.barrier()
            t0 = time.perf_counter()
            for _ in range(steps):
                plan.synthesize(Ih, out=Vo)   # host I in, host V out
                plan.analyze(Vh, out=Io)      # host V in, host I out
            el = max_over_ranks(time.perf_counter() - t0, world)
            rb = Ih.element_size()
            out["e2e"] = {"value": whole_job_rate(units_per_step, steps, el, world), "unit": UNIT,
                          "h2d_bytes_per_step": w.n_pix * rb + w.n_vis * 2 * rb,
                          "d2h_bytes_per_step": w.n_vis * 2 * rb + w.n_pix * rb,
                          "ms_per_step": el * 1e3 / steps}
        return out

    def path_dtype(info, eps, plain):
        # Arithmetic of the path: FP64 kernels (plain form), FP32, or for FP64 plans the direct
        # sums' double-float pairs of FP32 (FP64 accuracy on the FP32 pipes, FP64 only once per
        # tile and output; FP64 kernels below eps 1e-9) and the NUFFT sub-problems' FP64 grids.
        if plain:
            return "f64"
        if info["precision"] == 1:
            return "f32"
        kinds = []
        if info["direct_pairs"] > 0:
            kinds.append("f32x2" if eps >= 1e-9 else "f64")
        if info["n_nufft_blocks"] > 0:
            kinds.append("f64")
        return "+".join(dict.fromkeys(kinds)) or "f32x2"

    def summary(m, w, eps, plain=False):
        info = m["info"]
        d = {"eps": eps, "dtype": path_dtype(info, eps, plain), "value": m["value"], "unit": UNIT,
             "ms_per_step": m["ms_per_step"], "ms_median": m["ms_median"], "steps": m["steps"],
             "warmup": m["warmup"], "n_pix": w.n_pix, "n_vis": w.n_vis, "nufft_blocks": info["n_nufft_blocks"],
             "direct_pairs": info["direct_pairs"], "w": info["w"], "upsampfac": info["upsampfac"],
             "plan_seconds": info["plan_seconds"], "per_direction": m["per_direction"], "clocks": m["clocks"],
             "launches_per_step": {k: v / m["steps"] for k, v in m["stats"]["launches"].items()}}
        if "serial" in m:
            ss = m["serial"]
            d["stage_ms_serial"] = {k: v / m["serial_steps"] for k, v in ss["ms"].items()}
            d["stage_note"] = ("stage_ms_serial: one serial profiled step (every stage alone on the plan's stream, "
                               "no lanes or graph) after the timed steps; its stages add up to that step")
            d["roofline"] = stage_roofline(info, ss, m["serial_steps"], peaks)
        return d

    w = load_workload(args.n_vis, args.config, args.core_radius, args.radius_km, args.sparse)
    vis = configs.visibilities_cn(args.config, w.n_vis)
    full_run = not (args.n_vis or args.core_radius or args.radius_km or args.sparse or args.config != 2)
    main = measure(w, vis, args.eps, args.steps, args.warmup, with_e2e=not args.no_e2e, plain=args.plain)
    secondary = measure(w, vis, 1e-6, args.steps, args.warmup) if not args.no_secondary else None  # FP32 path

    st = main["stats"]
    stage_ms = st["ms"]
    dom = max(("direct", "spread", "interp", "fft", "deconv", "permute"), key=lambda k: stage_ms[k])
    launches = max(1, st["launches"][dom])
    avg_s = stage_ms[dom] * 1e-3 / launches
    info = main["info"]
    roofline = None
    if dom == "direct":
        pairs_per_launch = info["direct_pairs"]
        achieved = pairs_per_launch * FLOPS_PER_PAIR / avg_s
        roofline = {"bound": "alu", "achieved": achieved / 1e12, "peak": FP32_PEAK_FLOPS / 1e12,
                    "unit": "TFLOP/s", "frac": achieved / FP32_PEAK_FLOPS, "traffic": None,
                    "kernel": "direct_kernel (one launch per direction and step)",
                    "pairs_per_launch": pairs_per_launch, "avg_launch_ms": avg_s * 1e3,
                    "pairs_per_s": pairs_per_launch / avg_s,
                    "peak_note": "FP32 pipes 152 SMs x 128 lanes x 2 flops x 2.07 GHz (derived)"}
        if peaks:
            roofline["frac_of_probe"] = achieved / peaks["fp32_flops"]
    elif dom in ("spread", "interp"):
        # Every NUFFT point is spread once and interpolated once per step (w^3 taps each),
        # 4 flops per tap (complex value times a real weight, accumulated).
        taps_per_step = info["nufft_points"] * info["w"] ** 3
        taps_per_launch = taps_per_step / (st["launches"][dom] / args.steps)
        achieved = taps_per_launch * 4.0 / avg_s
        roofline = {"bound": "alu", "achieved": achieved / 1e12, "peak": FP32_PEAK_FLOPS / 1e12,
                    "unit": "TFLOP/s", "frac": achieved / FP32_PEAK_FLOPS, "traffic": None,
                    "kernel": dom + " kernels (one launch per NUFFT sub-problem)",
                    "taps_per_s": taps_per_launch / avg_s, "avg_launch_ms": avg_s * 1e3,
                    "peak_note": "FP32 pipes 152 SMs x 128 lanes x 2 flops x 2.07 GHz (derived)"}
    own = sum(st["launches"][k] for k in ("permute", "direct", "spread", "deconv", "interp"))

    line = {"metric": METRIC, "value": main["value"], "unit": UNIT, "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": main["ms_per_step"], "ms_median": main["ms_median"],
            "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": path_dtype(info, args.eps, args.plain),
            "data": "synthetic (seeded HEALPix + layout)",
            "config": {"workload": w.name + "; step = sky->vis + vis->sky" if args.radius_km > 0
                       else WORKLOADS[args.config], "eps": args.eps, "n_pix": w.n_pix, "n_vis": w.n_vis,
                       "mode": args.mode, "core_radius": args.core_radius or None, "graphs": args.graphs,
                       "plain": args.plain,
                       "l2": "flushed before each step (256 MiB write, outside the timed window)",
                       "parallelism": f"{world} replica(s)", "nufft_blocks": info["n_nufft_blocks"],
                       "direct_pairs": info["direct_pairs"], "w": info["w"],
                       "plan_seconds": info["plan_seconds"], "box_ratio": info["box_ratio"],
                       "factor": args.factor, "autotune": args.autotune,
                       "spread_bins": [info["spread_bin_pix"], info["spread_bin_vis"]]},
            "e2e": main.get("e2e"), "roofline": roofline, "gpu_launches": own,
            "stage_ms_per_step": {k: v / args.steps for k, v in stage_ms.items()},
            "per_direction": main["per_direction"],
            "clocks": main["clocks"], "peaks": peaks}
    if secondary is not None:
        line["secondary"] = summary(secondary, w, 1e-6)
        secondary["plan"].close()
    main["plan"].close()
    if full_run and not args.no_plain_line and not args.plain:
        # The plain FP64 form of the same step (the comparison at the same accuracy). Its
        # steps take seconds, so it runs one warm-up and two timed steps.
        pl = measure(w, vis, args.eps, 2, 1, plain=True)
        line["plain_fp64"] = summary(pl, w, args.eps, plain=True)
        line["plain_fp64"]["speedup_of_headline"] = main["value"] / pl["value"]
        pl["plan"].close()
    if full_run and not args.no_config3:
        # SKA-Low-like, chunked: the metric's eps = 1e-6 configuration. A step takes seconds,
        # so it times min(steps, 5) steps after 3 warm-ups, then one serial profiled step.
        w3 = load_workload(config=3)
        vis3 = configs.visibilities_cn(3, w3.n_vis)
        c3 = measure(w3, vis3, 1e-6, min(args.steps, 5), 3, mode="auto", serial_steps=1)
        line["config3"] = summary(c3, w3, 1e-6)
        line["config3"]["workload"] = WORKLOADS[3]
        line["config3"]["l2"] = "flushed before each step (256 MiB write, outside the timed window)"
        line["gpu_launches_config3"] = sum(c3["stats"]["launches"][k]
                                          for k in ("permute", "direct", "spread", "deconv", "interp"))
        c3["plan"].close()
    if full_run and not args.no_sparse:
        # The sparse-sky setup (500 pixels of interest in 5 groups of the 10 km field, all
        # 237,705 baselines): the planner keeps it direct.
        ws = load_workload(radius_km=10.0, sparse=500)
        vs = configs.visibilities_cn(6, ws.n_vis)
        sp = measure(ws, vs, 1e-6, args.steps, args.warmup, mode="auto")
        line["sparse_sky"] = summary(sp, ws, 1e-6)
        line["sparse_sky"]["workload"] = ws.name + "; step = sky->vis + vis->sky"
        sp["plan"].close()
    if rank == 0 and not args.no_serving:
        line["serving"] = serving_study()
    if rank == 0 and not args.no_cpu_baseline:
        line["cpu_baseline"] = cpu_baseline(w)
    if rank == 0:
        print(json.dumps(line), flush=True)
    if world > 1:
        dist.barrier()
        dist.destroy_process_group()
    return 0


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="hvox", choices=["hvox", "reference"])
    ap.add_argument("--eps", type=float, default=1e-9)
    ap.add_argument("--no-secondary", action="store_true")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-serving", action="store_true")
    ap.add_argument("--no-plain-line", action="store_true", help="skip the plain FP64 sub-line")
    ap.add_argument("--no-config3", action="store_true", help="skip the SKA-Low-like eps = 1e-6 sub-line")
    ap.add_argument("--no-sparse", action="store_true", help="skip the sparse-sky sub-line")
    ap.add_argument("--n-vis", type=int, default=0, help="use the first N baselines (profiler captures)")
    ap.add_argument("--config", type=int, default=2, choices=[1, 2, 3],
                    help="workload (2, the LOFAR-like case, is the benchmark; 1 and 3 for studies)")
    ap.add_argument("--mode", default="auto", choices=["auto", "nufft", "direct"])
    ap.add_argument("--radius-km", type=float, default=0.0,
                    help="study: telescope-radius sweep workload (0.1, 0.3, 1, 3, 10, 30 or 100 km)")
    ap.add_argument("--sparse", type=int, default=0, help="study: keep this many sky pixels (sparse sky)")
    ap.add_argument("--plain", action="store_true",
                    help="study: the plain FP64 form (FP64 arithmetic in every kernel, no graph)")
    ap.add_argument("--graphs", type=int, default=0, choices=[-1, 0, 1],
                    help="CUDA graphs: 0 for plans with NUFFT sub-problems, 1 always, -1 never")
    ap.add_argument("--factor", default="auto", choices=["auto", "pixels", "baselines"],
                    help="study: force a factored evaluation (one box spanning the other set)")
    ap.add_argument("--autotune", action="store_true", help="plan with the measured bin-size autotuner")
    ap.add_argument("--core-radius", type=float, default=0.0,
                    help="keep only baselines with |(u, v)| <= R wavelengths (dense-core study)")
    args = ap.parse_args()
    if args.warmup < 3:
        args.warmup = 3
    if args.impl == "reference":
        return run_reference(args)
    return run_gpu(args)


if __name__ == "__main__":
    sys.exit(main())
