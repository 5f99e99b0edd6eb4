#!/usr/bin/env python3
"""Throughput of contour-guided demons registration (CG-DIR) on GB300.

One step = one whole registration (Algorithm A over the pyramid: restriction,
UROI, every level's iterations, prolongation) of the pelvic CT-to-CBCT-like
synthetic case: 512 x 512 x 160 float32 CT, 6 structure masks, 3 levels with
100 / 50 / 25 iterations, FIXED stopping (the largest single-GPU workload).
Metric: voxel-iterations/s = sum over levels of (voxels x iterations) per
step / step time.  The same JSON line carries the 256 x 256 x 96
head-and-neck case as a secondary key, under "batched" the uneven-size mix
of 32 registrations run as one batch with FP16 image storage against plain
FP32 registrations one at a time, and under "e2e" the same registration
through the public API from pinned host buffers, copies included (two in
flight through cgdir_submit / cgdir_wait, and one at a time through
cgdir_register).

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl cgdir|reference]

N > 1 runs under torchrun as independent replicas (one case per rank, no
collective on the data path; a barrier brackets the timed region).  The
reference arm times the FP64 CPU oracle on the host cores on a bounded
sample of the same workload.  Rank 0 prints one JSON line.
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import statistics
import subprocess
import sys
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "voxel-iters/s and p50/p99 latency per registration, batched vs plain FP32"
UNIT = "voxel-iter/s"
# single-registration workloads (--workload): the pelvic CT-to-CBCT-like case
# (default) and the head-and-neck case; both are built on the GPU (host
# generation of 42 M voxels takes minutes) and copied to the host for the
# end-to-end leg and the oracle
WORKLOADS = {"pelvis512": {"name": "pelvis512", "levels": 3, "iters": [100, 50, 25]},
             "headneck256": {"name": "headneck256", "levels": 3, "iters": [100, 50, 25]}}
WORKLOAD = dict(WORKLOADS["pelvis512"])
# bounded sample of the workload for the CPU oracle: the central SAMPLE_SLICES
# axial slices of the same case, the same pyramid and iterations (the oracle
# takes about a minute for the whole 512 x 512 x 160 registration)
SAMPLE_SLICES = 16
FORCE_BYTES_PER_VOXEL = {True: 35, False: 33}   # contour terms on / off, FP32 images
FORCE_BYTES_PER_VOXEL_16 = {True: 31, False: 29}   # the same with 16-bit images
SMOOTH_BYTES_PER_VOXEL = 24                       # Gaussian of a 3-component field: read 12, write 12


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="cgdir", choices=["cgdir", "reference"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--only", choices=["force", "smooth", "compose", "iterate"], default=None,
                    help="profiling aid: launch only the named kernel (via the C ABI primitive) "
                         "on the workload's full-resolution inputs, W + K times, and print its "
                         "CUDA-event time")
    ap.add_argument("--shape", default=None,
                    help="with --only: nz,ny,nx of the inputs (the workload's case resampled)")
    ap.add_argument("--mode", default="single", choices=["single", "batch", "serve"],
                    help="single: one registration per step (default); batch: 32 cases of "
                         "uneven sizes in one graph launch, FP16 images, against plain FP32 one "
                         "at a time; serve: Poisson arrivals of the same mix at 1-64 requests/s "
                         "under a 160 GB device budget, p50/p99 latency against plain FP32 one at "
                         "a time")
    ap.add_argument("--batch-n", type=int, default=32, help="cases in the batch / serving mix")
    ap.add_argument("--workload", default="pelvis512", choices=sorted(WORKLOADS),
                    help="single-registration workload (default: the 512x512x160 pelvic case)")
    ap.add_argument("--no-secondary", action="store_true",
                    help="single: skip the head-and-neck secondary key and the batched comparison")
    ap.add_argument("--batch-passes", type=int, default=2,
                    help="single: timed passes of the batched comparison (after one warm-up pass)")
    ap.add_argument("--storage", default="f32", choices=["f32", "f16", "bf16"],
                    help="image storage type of the registration (arithmetic stays FP32)")
    ap.add_argument("--rates", default="8,16,24,32", help="serve: arrival rates (requests/s)")
    ap.add_argument("--requests", type=int, default=200, help="serve: requests per rate")
    ap.add_argument("--inflight", type=int, default=0,
                    help="serve: requests on the GPU at most (0: the measured saturation point)")
    ap.add_argument("--inflight-candidates", type=lambda v: [int(x) for x in v.split(",")],
                    default=[1, 2, 3, 4, 6, 8], help="serve: caps tried for the saturation point")
    ap.add_argument("--tuning-out", default=None,
                    help="single: write the autotuned per-level schedule to this JSON file")
    ap.add_argument("--tuning-in", default=None,
                    help="single: load the per-level schedule from this JSON file instead of tuning "
                         "(e.g. under a profiler, whose per-launch overhead would skew the tuner)")
    return ap.parse_args()


def dist_env():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return world, rank, local


def replica_case_index(rank: int) -> int:
    """Replicas only: every rank registers its own case (seeded by its rank);
    no data crosses ranks."""
    return rank


def reduce_max(value: float, device=None) -> float:
    """Max over ranks of a per-rank time (the only collective of a run)."""
    import torch
    import torch.distributed as dist
    if not (dist.is_available() and dist.is_initialized()) or dist.get_world_size() == 1:
        return float(value)
    t = torch.tensor([value], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def whole_job_value(world: int, vox_iters_per_step: int, steps: int, max_total_ms: float) -> float:
    """voxel-iterations of all ranks / the slowest rank's time."""
    return world * vox_iters_per_step * steps / (max_total_ms / 1e3)


def workload_config(case, n_gpus, storage="f32", wl=None):
    wl = wl or WORKLOAD
    nz, ny, nx = case.shape
    img = {"f32": "float32", "f16": "float16", "bf16": "bfloat16"}[storage]
    return {"workload": f"{wl['name']}: {nx}x{ny}x{nz} {img} CT, {case.k} uint8 structure "
                        f"masks, {wl['levels']}-level pyramid "
                        f"{'/'.join(map(str, wl['iters']))} iterations, FIXED stop",
            "shape_zyx": [nz, ny, nx], "masks": case.k, "levels": wl["levels"],
            "iters": wl["iters"], "lambda": case.lam[0], "sigma": 1.0,
            "l2": "flushed between timed steps (256 MiB write)",
            "parallelism": f"replicas x{n_gpus}"}


class HostCase:
    """Host copies of a case built on the device (float32 images, uint8 masks
    [k, nz, ny, nx]), plus its structure parameters."""

    def __init__(self, dc):
        self.static, self.moving = dc.static.cpu().numpy(), dc.moving.cpu().numpy()
        self.static_masks, self.moving_masks = dc.static_masks.cpu().numpy(), dc.moving_masks.cpu().numpy()
        self.shape, self.k, self.lam, self.signs = tuple(dc.shape), dc.k, dc.lam, dc.signs


def build_case(torch, name, index, dev):
    """One case of a single-registration workload, built on the device:
    (device case with images and masks, host copies)."""
    import phantom
    dc = phantom.make_case_device(name, index=index, device=dev)
    dc.u_gt = dc.body = None
    host = HostCase(dc)
    torch.cuda.empty_cache()
    return dc, host


def oracle_cores():
    import oracle
    return oracle.num_threads()


def oracle_sample(host):
    """The oracle's bounded sample of a case: its central SAMPLE_SLICES axial
    slices, the same structures and signs."""
    nz = host.shape[0]
    z0 = max(0, (nz - SAMPLE_SLICES) // 2)
    z1 = min(nz, z0 + SAMPLE_SLICES)
    return (host.static[z0:z1], host.moving[z0:z1], host.static_masks[:, z0:z1], host.moving_masks[:, z0:z1])


def time_oracle_sample(host):
    """One registration of the bounded sample by the FP64 CPU oracle:
    (voxel-iterations, seconds)."""
    import oracle
    import phantom
    S, M, SM, MM = oracle_sample(host)
    t0 = time.perf_counter()
    oracle.register(S, M, SM, MM, levels=WORKLOAD["levels"], iters=WORKLOAD["iters"], lam=host.lam,
                    sign=host.signs, stop_mode=oracle.STOP_FIXED)
    dt = time.perf_counter() - t0
    return phantom.voxel_iters(S.shape, WORKLOAD["levels"], WORKLOAD["iters"]), dt


def sample_desc(host):
    import phantom
    S = oracle_sample(host)[0]
    nz, ny, nx = S.shape
    vi = phantom.voxel_iters(S.shape, WORKLOAD["levels"], WORKLOAD["iters"])
    return (f"the central {nz} axial slices of the same case ({nx}x{ny}x{nz}), same structures, pyramid "
            f"and iterations {'/'.join(map(str, WORKLOAD['iters']))} ({vi / 1e6:.1f} M voxel-iters per run, "
            f"set-up included)")


# --------------------------------------------------------------------------- #
class ClockSampler:
    """nvidia-smi clock / throttle samples every 200 ms while running."""
    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_id: str):
        self.gpu_id = gpu_id
        self.proc = None
        self.lines = []

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--query-gpu={self.Q}", "--format=csv,noheader,nounits",
                 "-lms", "200", "-i", self.gpu_id], stdout=subprocess.PIPE,
                stderr=subprocess.DEVNULL, text=True)
        except OSError:
            self.proc = None
        time.sleep(0.3)
        return self

    def __exit__(self, *exc):
        if self.proc is not None:
            time.sleep(0.25)
            self.proc.terminate()
            try:
                out, _ = self.proc.communicate(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()
                out, _ = self.proc.communicate()
            self.lines = [l for l in out.splitlines() if l.strip()]

    def summary(self):
        if not self.lines:
            return None
        sm, mx, reasons, power = [], 0.0, set(), []
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for l in self.lines:
            f = [x.strip() for x in l.split(",")]
            try:
                sm.append(float(f[1]))
                mx = max(mx, float(f[2]))
                power.append(float(f[3]))
            except (ValueError, IndexError):
                continue
            for name, v in zip(names, f[5:9]):
                if v.lower() == "active":
                    reasons.add(name)
        if not sm:
            return None
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": mx, "reasons": sorted(reasons),
                "samples": len(sm), "power_w_max": max(power) if power else None}


def gpu_uuid(torch, dev):
    try:
        u = torch.cuda.get_device_properties(dev).uuid
        s = str(u)
        return s if s.startswith("GPU-") else "GPU-" + s
    except Exception:
        return str(dev)


def measured_peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        with open(p) as f:
            d = json.load(f)
        return float(d["hbm_gbs"]), "measured (MEASURED_PEAKS.json hbm_gbs, copy burst)"
    return 6800.0, "fallback 6.8 TB/s"


def sigma_default(kw):
    """True when the registration smooths with sigma = 1 voxel (the profiled radius)."""
    return kw.get("sigma_fluid", 1.0) == 1.0 and kw.get("sigma_diff", 1.0) == 1.0


def traffic_record(kernel, workload, sources):
    """DRAM bytes per launch of a kernel from its committed ncu summary
    (profiles/<kernel>_<workload>.md), if it was taken on the current kernel
    sources (else None)."""
    path = os.path.join(ROOT, "profiles", f"{kernel}_{workload}.md")
    if not os.path.exists(path):
        return None
    sha, traffic = None, None
    for line in open(path):
        if line.startswith("- kernel sources sha1"):
            sha = line.split(":", 1)[1].strip()
        if line.startswith("- dram bytes per launch (full size):"):
            traffic = float(line.split(":", 1)[1].strip())
    return traffic if (sha == sources_sha1(sources) and traffic) else None


FORCE_SOURCES = ("kernels_force.cu", "warp_corners.cuh")
SMOOTH_SOURCES = ("kernels_smooth.cu", "tma.cuh")


def sources_sha1(files):
    h = hashlib.sha1()
    for f in files:
        h.update(open(os.path.join(ROOT, "paper_1301_0970_gb300", "csrc", f), "rb").read())
    return h.hexdigest()


# --------------------------------------------------------------------------- #
def run_reference(args):
    """The FP64 oracle on the host cores, on a bounded sample of the workload
    per step (rank 0 only; the GPU, where present, only builds the inputs)."""
    world, rank, _ = dist_env()
    if rank != 0:
        return 0
    import torch
    WORKLOAD.update(WORKLOADS[getattr(args, "workload", "pelvis512")])
    dev = torch.device("cuda", 0) if torch.cuda.is_available() else torch.device("cpu")
    dc, host = build_case(torch, WORKLOAD["name"], 0, dev)
    del dc
    times, vi = [], 0
    for i in range(args.warmup + args.steps):
        vi, dt = time_oracle_sample(host)
        if i >= args.warmup:
            times.append(dt)
    value = vi * len(times) / sum(times)
    cores = oracle_cores()
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT,
            "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": 1e3 * sum(times) / len(times), "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": workload_config(host, 1),
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": cores, "kind": "oracle",
                             "sample": sample_desc(host)},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)
    return 0


def time_registrations(torch, cg, ctx, dc, kw, steps, warmup, flush, stream, barrier=lambda: None,
                       profile_levels=None):
    """Register the device-resident case `steps` times after `warmup` untimed
    runs, L2 flushed before each; CUDA events on the context stream around
    each registration.  Returns (per-step ms, kernels launched, clock summary,
    per-kernel profile of the timed steps)."""
    S, M = dc["S"], dc["M"]
    for _ in range(warmup):
        ctx.register(S, M, dc["SM"], dc["MM"], dvf_out=dc["dvf"], **kw)
    torch.cuda.synchronize()
    if profile_levels is not None:
        ctx.profile([cg.CGDIR_K_FORCE, cg.CGDIR_K_SMOOTH_U], levels=profile_levels)
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(steps)]
    barrier()
    torch.cuda.synchronize()
    launches0 = cg.launch_count()
    with ClockSampler(gpu_uuid(torch, stream.device)) as clk:
        for i in range(steps):
            flush.zero_()
            ev[i][0].record(stream)
            ctx.register(S, M, dc["SM"], dc["MM"], dvf_out=dc["dvf"], **kw)
            ev[i][1].record(stream)
        torch.cuda.synchronize()
    launches = cg.launch_count() - launches0
    barrier()
    prof = None
    if profile_levels is not None:
        prof = ctx.profile_read()
        ctx.profile([])
    return [a.elapsed_time(b) for a, b in ev], launches, clk.summary(), prof


def device_case(torch, dc, host, img_t, dev):
    """Device inputs of one registration in the storage type, and its DVF buffer."""
    return {"S": dc.static.to(img_t), "M": dc.moving.to(img_t),
            "SM": list(dc.static_masks.unbind(0)), "MM": list(dc.moving_masks.unbind(0)),
            "dvf": torch.empty((3,) + host.shape, dtype=torch.float32, device=dev)}


def secondary_headneck(torch, cg, dev, flush, stream, steps, warmup):
    """The 256 x 256 x 96 head-and-neck case (FP32), autotuned, timed like
    the headline workload: a secondary key of the line."""
    import numpy as np
    import phantom
    wl = WORKLOADS["headneck256"]
    dc, host = build_case(torch, wl["name"], 0, dev)
    d = device_case(torch, dc, host, torch.float32, dev)
    kw = dict(levels=wl["levels"], iters=wl["iters"], lam=host.lam, sign=host.signs,
              stop_mode=cg.CGDIR_STOP_FIXED, storage_dtype=cg.CGDIR_F32)
    with cg.Context(dev.index) as ctx:
        ctx.autotune(host.shape, host.k, wl["levels"], storage_dtype=cg.CGDIR_F32)
        ms, _, _, _ = time_registrations(torch, cg, ctx, d, kw, steps, warmup, flush, stream)
    vi = phantom.voxel_iters(host.shape, wl["levels"], wl["iters"])
    return {"value": vi * len(ms) / (sum(ms) / 1e3), "unit": UNIT, "ms_per_step": float(np.mean(ms)),
            "latency_ms": {"p50": float(np.percentile(ms, 50)), "p99": float(np.percentile(ms, 99))},
            "steps": steps, "config": workload_config(host, 1, "f32", wl)}


def run_cgdir(args):
    import numpy as np
    import torch

    import paper_1301_0970_gb300 as cg
    import phantom

    world, rank, local = dist_env()
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    WORKLOAD.update(WORKLOADS[args.workload])
    dc, host = build_case(torch, WORKLOAD["name"], replica_case_index(rank), dev)
    L, iters = WORKLOAD["levels"], WORKLOAD["iters"]
    vox_iters = phantom.voxel_iters(host.shape, L, iters)
    N = int(np.prod(host.shape))
    img_t = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}[args.storage]
    img_code = {"f32": cg.CGDIR_F32, "f16": cg.CGDIR_F16, "bf16": cg.CGDIR_BF16}[args.storage]
    d = device_case(torch, dc, host, img_t, dev)
    del dc
    kw = dict(levels=L, iters=iters, lam=host.lam, sign=host.signs, stop_mode=cg.CGDIR_STOP_FIXED,
              storage_dtype=img_code)
    flush = torch.empty(64 * 1024 * 1024, dtype=torch.float32, device=dev)   # 256 MiB > L2

    def barrier():
        if world > 1:
            torch.distributed.barrier()

    ctx = cg.Context(local)
    stream = torch.cuda.current_stream(dev)
    if args.tuning_in:                                    # per-level kernel schedule
        with open(args.tuning_in) as f:
            ctx.load_tuning(json.load(f))
        tuning = ctx.tuning()
    else:
        tuning = ctx.autotune(host.shape, host.k, L, storage_dtype=img_code)
    if args.tuning_out:
        with open(args.tuning_out, "w") as f:
            json.dump(tuning, f)

    # ---- timed region: device-resident inputs, CUDA events on the ctx stream;
    # the roofline's launches are timed too: the force step and the smoothing
    # of u at the finest level
    step_ms, launches, clocks, prof = time_registrations(torch, cg, ctx, d, kw, args.steps, args.warmup, flush,
                                                         stream, barrier, profile_levels=[L - 1])
    total_ms = sum(step_ms)
    max_total_ms = reduce_max(total_ms, dev)
    value = whole_job_value(world, vox_iters, args.steps, max_total_ms)

    # ---- one profiled step with every kernel class timed (breakdown only)
    ctx.profile(list(range(8)))
    flush.zero_()
    ctx.register(d["S"], d["M"], d["SM"], d["MM"], dvf_out=d["dvf"], **kw)
    breakdown = ctx.profile_read()
    ctx.profile([])

    # ---- end to end through the public API from pinned host buffers: every
    # step copies its images and masks in and its DVF out.  Two registrations
    # in flight through cgdir_submit / cgdir_wait, so one step's copies overlap
    # the other's kernels; the synchronous cgdir_register loop is reported
    # beside it ("serial")
    e2e = None
    if not args.no_e2e:
        Sh = torch.from_numpy(host.static).to(img_t).pin_memory()
        Mh = torch.from_numpy(host.moving).to(img_t).pin_memory()
        SMh = [torch.from_numpy(m).pin_memory() for m in host.static_masks]
        MMh = [torch.from_numpy(m).pin_memory() for m in host.moving_masks]
        dvf_hs = [torch.empty((3,) + host.shape, dtype=torch.float32).pin_memory() for _ in range(2)]
        h2d = 2 * N * d["S"].element_size() + 2 * host.k * N
        d2h = 3 * N * 4 + L * (max(iters) + 1) * 8 + 4 * 8 * 4

        def pipelined(steps):
            queue = []
            for i in range(steps):
                if len(queue) == 2:
                    ctx.wait(queue.pop(0))
                queue.append(ctx.submit(Sh, Mh, SMh, MMh, dvf_out=dvf_hs[i % 2], **kw))
            while queue:
                ctx.wait(queue.pop(0))

        ctx.register(Sh, Mh, SMh, MMh, dvf_out=dvf_hs[0], **kw)      # warm the host path
        pipelined(4)                                                 # and both slots' graphs
        flush.zero_()
        torch.cuda.synchronize()
        barrier()
        t0 = time.perf_counter()
        pipelined(args.steps)
        t_pipe = reduce_max(time.perf_counter() - t0, dev)
        et = []
        for _ in range(args.steps):
            flush.zero_()
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            ctx.register(Sh, Mh, SMh, MMh, dvf_out=dvf_hs[0], **kw)
            et.append(time.perf_counter() - t0)
        t_ser = reduce_max(sum(et), dev)
        e2e = {"value": whole_job_value(world, vox_iters, args.steps, 1e3 * t_pipe), "unit": UNIT,
               "h2d_bytes_per_step": h2d, "d2h_bytes_per_step": d2h,
               "ms_per_step": 1e3 * t_pipe / args.steps,
               "api": "cgdir_submit / cgdir_wait, 2 registrations in flight, host (pinned) buffers",
               "serial": {"value": whole_job_value(world, vox_iters, args.steps, 1e3 * t_ser),
                          "ms_per_step": 1e3 * t_ser / args.steps,
                          "api": "cgdir_register, one at a time, host (pinned) buffers"}}
        del Sh, Mh, SMh, MMh, dvf_hs

    # ---- roofline of the dominant kernel (largest share of device time in the
    # launch list): the z-march Gaussian at the finest level, two launches per
    # iteration (du and u; the u launch is the one timed here); the force step
    # (its two passes) as a second entry
    peak, peak_src = measured_peaks()
    fine = {p["kernel"]: p for p in prof if p["level"] == L - 1 and p["launches"]}
    fine_variant = next((t["smooth"] for t in tuning if tuple(t["shape"]) == tuple(host.shape)), None)
    roofline, roofline_force = None, None
    if "smooth_u" in fine and fine_variant in ("march", "march32"):
        p = fine["smooth_u"]
        avg_ms = p["total_ms"] / p["launches"]
        bytes_per_launch = SMOOTH_BYTES_PER_VOXEL * N
        achieved = bytes_per_launch / (avg_ms / 1e3) / 1e9
        roofline = {"bound": "hbm", "kernel": "k_smooth_march (z-march Gaussian of u, finest level; the same kernel "
                                              "also smooths du there)",
                    "achieved": achieved, "peak": peak, "unit": "GB/s", "frac": achieved / peak,
                    "traffic": traffic_record("smooth", args.workload, SMOOTH_SOURCES) if sigma_default(kw)
                    else None,
                    "algorithmic_bytes_per_launch": bytes_per_launch, "avg_launch_ms": avg_ms,
                    "launches": p["launches"], "peak_source": peak_src}
    if "force" in fine:
        p = fine["force"]
        avg_ms = p["total_ms"] / p["launches"]
        bytes_per_launch = (FORCE_BYTES_PER_VOXEL if args.storage == "f32" else FORCE_BYTES_PER_VOXEL_16)[True] * N
        achieved = bytes_per_launch / (avg_ms / 1e3) / 1e9
        nx = host.shape[2]
        pass2 = "k_force_pass4" if nx % 4 == 0 else "k_force_pass2" if nx % 2 == 0 else "k_force_pass"
        roofline_force = {"bound": "hbm", "kernel": f"force step = k_warp_pass + {pass2} (finest level, "
                                                    "contour terms on)",
                          "achieved": achieved, "peak": peak, "unit": "GB/s", "frac": achieved / peak,
                          "traffic": traffic_record("force", args.workload, FORCE_SOURCES)
                          if args.storage == "f32" else None,
                          "algorithmic_bytes_per_launch": bytes_per_launch, "avg_launch_ms": avg_ms,
                          "launches": p["launches"], "peak_source": peak_src}
    if roofline is None:
        roofline = roofline_force
    ctx.close()
    del d
    torch.cuda.empty_cache()

    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        vi, dt = time_oracle_sample(host)
        cpu = {"value": vi / dt, "unit": UNIT, "cores": oracle_cores(), "kind": "oracle",
               "sample": sample_desc(host), "seconds": dt}

    secondary, batched = None, None
    if world == 1 and not args.no_secondary:
        secondary = secondary_headneck(torch, cg, dev, flush, stream, args.steps, args.warmup)
        del flush
        torch.cuda.empty_cache()
        batched = batched_comparison(torch, cg, dev, args.batch_n, args.batch_passes, 1)

    if rank == 0:
        lat = sorted(step_ms)
        line = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world,
                "steps": args.steps, "warmup": args.warmup, "ms_per_step": max_total_ms / args.steps,
                "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
                "dtype": "f32" if args.storage == "f32" else f"{args.storage} images, f32 arithmetic",
                "data": "synthetic", "config": workload_config(host, world, args.storage),
                "latency_ms": {"p50": float(np.percentile(lat, 50)), "p99": float(np.percentile(lat, 99)),
                               "per": "registration"},
                "e2e": e2e, "gpu_launches": int(launches), "roofline": roofline,
                "roofline_force_step": roofline_force,
                "cpu_baseline": cpu, "clocks": clocks,
                "headneck256": secondary, "batched": batched,
                "kernel_breakdown_ms": {f"{p['kernel']}@L{p['level']}": round(p["total_ms"], 4)
                                        for p in breakdown},
                "tuning": [{"shape_zyx": list(t["shape"]), "smooth": t["smooth"],
                            "smooth_zchunk": t["smooth_zchunk"], "force_zchunk": t["force_zchunk"],
                            "force_width": t.get("force_width", 0),
                            "smooth_ms": round(t["smooth_ms"], 4), "force_ms": round(t["force_ms"], 4),
                            "untuned_smooth_ms": round(t["default_smooth_ms"], 4),
                            "untuned_force_ms": round(t["default_force_ms"], 4)} for t in tuning]}
        print(json.dumps(line), flush=True)
    if world > 1:
        torch.distributed.destroy_process_group()
    return 0


# --------------------------------------------------------------------------- #
# the uneven-size mix: batched (one graph launch) and served (Poisson arrivals)
# --------------------------------------------------------------------------- #
MIX = {"seed": 4000, "levels": 3, "iters": [100, 50, 25], "budget_gb": 160}


def build_mix(torch, dev, n):
    """The mix of n cases, built on the device (FP32 images, FP16 copies,
    uint8 masks), each with its voxel-iteration count."""
    import phantom
    cases = []
    for tmpl, index, shp, names in phantom.batch_mix_specs(n, MIX["seed"]):
        c = phantom.make_case_device(tmpl, index, shp, names, device=dev)
        c.u_gt = c.body = None
        cases.append({"S": c.static, "M": c.moving, "S16": c.static.half(), "M16": c.moving.half(),
                      "SM": list(c.static_masks.unbind(0)), "MM": list(c.moving_masks.unbind(0)),
                      "lam": c.lam, "sign": c.signs, "shape": tuple(shp), "k": c.k,
                      "vi": phantom.voxel_iters(shp, MIX["levels"], MIX["iters"])})
        torch.cuda.empty_cache()
    return cases


def mix_request(cg, c, half, dvf=None):
    kw = dict(levels=MIX["levels"], iters=MIX["iters"], lam=c["lam"], sign=c["sign"],
              stop_mode=cg.CGDIR_STOP_FIXED, storage_dtype=cg.CGDIR_F16 if half else cg.CGDIR_F32)
    d = dict(static=c["S16"] if half else c["S"], moving=c["M16"] if half else c["M"],
             static_masks=c["SM"], moving_masks=c["MM"], **kw)
    if dvf is not None:
        d["dvf_out"] = dvf
    return d


def mix_config(cases):
    shapes = sorted({c["shape"] for c in cases})
    return {"workload": f"batch_mix{len(cases)}: {len(cases)} registrations, sizes drawn uniformly "
                        f"from {{128x128x64, 256x256x96, 384x384x128, 512x512x160}}, 2-8 uint8 masks, "
                        f"bumps <= 10 voxels, 3-level pyramid 100/50/25, FIXED stop",
            "shapes_zyx": [list(s) for s in shapes], "cases": len(cases),
            "voxel_iters_total": int(sum(c["vi"] for c in cases)),
            "l2": "inputs larger than L2 (several GB per pass)", "parallelism": "replicas x1"}


def one_at_a_time(torch, cg, ctx, cases, stream):
    """Plain FP32, one registration after another: per-case times (ms)."""
    out = []
    for c in cases:
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        d = mix_request(cg, c, False)
        a.record(stream)
        ctx.register(d.pop("static"), d.pop("moving"), d.pop("static_masks"), d.pop("moving_masks"), **d)
        b.record(stream)
        out.append((a, b))
    torch.cuda.synchronize()
    return [a.elapsed_time(b) for a, b in out]


def batched_comparison(torch, cg, dev, n, passes, warmup):
    """The uneven-size mix of n cases: plain FP32 registrations one at a time
    against all n in one batched graph launch (FP16 images, and FP32 for
    comparison), on the same GPU and context.  voxel-iter/s of each, the
    multiple over plain FP32, and per-registration latency: for plain runs
    each registration's own CUDA-event time, for a batch the pass time (every
    case completes with the batch)."""
    import numpy as np
    t_build = time.perf_counter()
    cases = build_mix(torch, dev, n)
    t_build = time.perf_counter() - t_build
    total_vi = sum(c["vi"] for c in cases)
    stream = torch.cuda.current_stream(dev)
    res = {}
    with cg.Context(dev.index) as ctx:
        ctx.set_autotune(True)        # each new level shape is tuned at its first registration
        # plain FP32, one at a time (warm-up passes capture every shape's graph)
        for _ in range(max(warmup, 1)):
            one_at_a_time(torch, cg, ctx, cases, stream)
        per, tot = [], []
        with ClockSampler(gpu_uuid(torch, dev)) as clk:
            for _ in range(passes):
                t = one_at_a_time(torch, cg, ctx, cases, stream)
                per += t
                tot.append(sum(t))
        res["plain_f32_one_at_a_time"] = {
            "value": total_vi * len(tot) / (sum(tot) / 1e3), "unit": UNIT, "ms_per_pass": float(np.mean(tot)),
            "latency_ms": {"p50": float(np.percentile(per, 50)), "p99": float(np.percentile(per, 99)),
                           "per": "registration", "samples": len(per)},
            "clocks": clk.summary()}
        # batched: every case in one graph launch
        for half in (True, False):
            outs = [torch.empty((3,) + c["shape"], dtype=torch.float32, device=dev) for c in cases]
            reqs = [mix_request(cg, c, half, o) for c, o in zip(cases, outs)]
            for _ in range(max(warmup, 1)):
                ctx.register_batch(reqs)
            torch.cuda.synchronize()
            ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
                  for _ in range(passes)]
            l0 = cg.launch_count()
            with ClockSampler(gpu_uuid(torch, dev)) as clk:
                for i in range(passes):
                    ev[i][0].record(stream)
                    ctx.register_batch(reqs)
                    ev[i][1].record(stream)
                torch.cuda.synchronize()
            launches = cg.launch_count() - l0
            ms = [a.elapsed_time(b) for a, b in ev]
            res["batch_f16" if half else "batch_f32"] = {
                "value": total_vi * len(ms) / (sum(ms) / 1e3), "unit": UNIT, "ms_per_pass": float(np.mean(ms)),
                "latency_ms": {"p50": float(np.percentile(ms, 50)), "p99": float(np.percentile(ms, 99)),
                               "per": "registration (every case of a batch completes with the batch)"},
                "gpu_launches_per_pass": int(launches // max(passes, 1)), "clocks": clk.summary()}
            del outs, reqs
    plain = res["plain_f32_one_at_a_time"]["value"]
    res["multiple_batch_f16_over_plain_f32"] = res["batch_f16"]["value"] / plain
    res["multiple_batch_f32_over_plain_f32"] = res["batch_f32"]["value"] / plain
    res["config"] = mix_config(cases)
    res["passes"] = passes
    res["build_s"] = round(t_build, 1)
    del cases
    torch.cuda.empty_cache()
    return res


def run_batch(args):
    import torch

    import paper_1301_0970_gb300 as cg

    dev = torch.device("cuda", 0)
    torch.cuda.set_device(dev)
    res = batched_comparison(torch, cg, dev, args.batch_n, args.steps, args.warmup)
    b16 = res["batch_f16"]
    line = {"metric": METRIC, "value": b16["value"], "unit": UNIT, "n_gpus": 1, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": b16["ms_per_pass"], "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f16 images, f32 arithmetic",
            "data": "synthetic", "config": res["config"], "latency_ms": b16["latency_ms"],
            "gpu_launches": int(b16["gpu_launches_per_pass"] * args.steps), "clocks": b16["clocks"],
            "batched": res}
    print(json.dumps(line), flush=True)
    return 0


def serve_trace(rng, rate, n_cases, n=200):
    """Seeded Poisson arrivals at `rate` per second (n requests) and the case
    of each request."""
    import numpy as np
    gaps = rng.exponential(1.0 / rate, size=n)
    return np.cumsum(gaps) - gaps[0], rng.integers(0, n_cases, size=n)


def run_serve(args):
    """Poisson arrivals of the uneven-size mix, served with FP16 images under
    a 160 GB budget: each request is submitted at its arrival (oldest first
    when it has to wait) and runs as soon as fewer than `cap` requests are on
    the GPU, overlapping with them; against plain FP32 registrations one at a
    time, first come first served, on the same arrival trace.  The cap is
    where the GPU saturates: the smallest number of concurrent registrations
    of the mix whose throughput comes within 3 % of the best measured."""
    import numpy as np
    import torch

    import paper_1301_0970_gb300 as cg

    dev = torch.device("cuda", 0)
    torch.cuda.set_device(dev)
    cases = build_mix(torch, dev, args.batch_n)
    rates = [float(r) for r in args.rates.split(",")]
    rng = np.random.Generator(np.random.PCG64(MIX["seed"] + 1))
    traces = {r: serve_trace(rng, r, len(cases), args.requests) for r in rates}

    def served(ctx, arrivals, which, half):
        """Continuous admission, oldest first: submit each request at its
        arrival time, or as soon as the cap / the budget admits it; collect
        completions as they come."""
        lat, inflight, i, n = [], {}, 0, len(arrivals)
        t0 = time.perf_counter()
        t_end = t0
        while i < n or inflight:
            now = time.perf_counter() - t0
            progressed = False
            while i < n and arrivals[i] <= now:
                c = cases[int(which[i])]
                d = mix_request(cg, c, half)
                try:
                    r = ctx.submit(d.pop("static"), d.pop("moving"), d.pop("static_masks"),
                                   d.pop("moving_masks"), **d)
                except cg.CgdirError as e:
                    if e.status != cg.CGDIR_EBUSY:
                        raise
                    break
                inflight[r] = (arrivals[i], c["vi"])
                i += 1
                progressed = True
            for r in list(inflight):
                if ctx.poll(r):
                    ctx.wait(r)
                    t_done = time.perf_counter() - t0
                    a, _ = inflight.pop(r)
                    lat.append(1e3 * (t_done - a))
                    t_end = max(t_end, t0 + t_done)
                    progressed = True
            if not progressed:
                time.sleep(0.0002)
        vi = sum(cases[int(w)]["vi"] for w in which)
        return lat, vi / (t_end - t0)

    def plain(ctx, arrivals, which):
        """One at a time, FP32, first come first served."""
        lat, t0 = [], time.perf_counter()
        for a, w in zip(arrivals, which):
            now = time.perf_counter() - t0
            if now < a:
                time.sleep(a - now)
            d = mix_request(cg, cases[int(w)], False)
            ctx.register(d.pop("static"), d.pop("moving"), d.pop("static_masks"), d.pop("moving_masks"), **d)
            lat.append(1e3 * (time.perf_counter() - t0 - a))
        vi = sum(cases[int(w)]["vi"] for w in which)
        return lat, vi / (time.perf_counter() - t0)

    rows, calib = [], []
    with cg.Context(0, mem_budget_bytes=MIX["budget_gb"] << 30) as sctx, cg.Context(0) as pctx:
        sctx.set_autotune(True)
        pctx.set_autotune(True)
        everyone = (np.zeros(len(cases)), np.arange(len(cases)))
        sctx.set_max_inflight(max(args.inflight_candidates))
        for _ in range(2):                                   # warm-up: slots, buffers, graphs
            served(sctx, *everyone, True)
        for _ in range(2):
            plain(pctx, np.zeros(len(cases)), np.arange(len(cases)))
        # the saturation point: the whole mix at once under each cap
        for cap in args.inflight_candidates:
            sctx.set_max_inflight(cap)
            _, v = served(sctx, *everyone, True)
            calib.append({"cap": cap, "value": v})
        best = max(c["value"] for c in calib)
        cap = args.inflight if args.inflight > 0 else \
            min(c["cap"] for c in calib if c["value"] >= 0.97 * best)
        sctx.set_max_inflight(cap)
        torch.cuda.synchronize()
        l0 = cg.launch_count()
        with ClockSampler(gpu_uuid(torch, dev)) as clk:
            for r in rates:
                arr, which = traces[r]
                ls, vs = served(sctx, arr, which, True)
                lp, vp = plain(pctx, arr, which)
                rows.append({"rate_per_s": r, "requests": len(arr),
                             "served_f16": {"value": vs, "p50_ms": float(np.percentile(ls, 50)),
                                            "p99_ms": float(np.percentile(ls, 99))},
                             "plain_f32": {"value": vp, "p50_ms": float(np.percentile(lp, 50)),
                                           "p99_ms": float(np.percentile(lp, 99))}})
                print(json.dumps(rows[-1]), file=sys.stderr, flush=True)
        launches = cg.launch_count() - l0
    top = max(rows, key=lambda x: x["served_f16"]["value"])
    line = {"metric": METRIC, "value": top["served_f16"]["value"], "unit": UNIT, "n_gpus": 1,
            "steps": len(rates), "warmup": 2, "ms_per_step": None, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f16 images, f32 arithmetic",
            "data": "synthetic", "config": dict(mix_config(cases), budget_gb=MIX["budget_gb"],
                                                 max_inflight=cap, arrivals="Poisson, seeded",
                                                 admission="oldest first, at most max_inflight on the GPU"),
            "latency_ms": {"p50": top["served_f16"]["p50_ms"], "p99": top["served_f16"]["p99_ms"],
                           "per": "registration, arrival to completion", "at_rate": top["rate_per_s"]},
            "gpu_launches": int(launches), "clocks": clk.summary(), "inflight_calibration": calib,
            "rates": rows}
    print(json.dumps(line), flush=True)
    return 0


def run_only_kernel(args):
    """One kernel alone on the full-resolution inputs (u = half the
    ground-truth DVF, contour terms on for the force), for kernel profiling."""
    import numpy as np
    import torch

    import paper_1301_0970_gb300 as cg
    import phantom

    dev = torch.device("cuda", 0)
    WORKLOAD.update(WORKLOADS[args.workload])
    shape = tuple(int(v) for v in args.shape.split(",")) if args.shape else None
    case = phantom.make_case_device(WORKLOAD["name"], shape=shape, device=dev)
    pk = torch.zeros(case.shape, dtype=torch.uint8, device=dev)
    mb, sb = pk.clone(), pk.clone()
    for j in range(case.k):
        mb |= (case.moving_masks[j] != 0).to(torch.uint8) << j
        sb |= (case.static_masks[j] != 0).to(torch.uint8) << j
    I0, T0 = case.moving, case.static
    u = (0.5 * case.u_gt).contiguous()
    del pk
    du = torch.empty_like(u)
    dus = (0.1 * u).contiguous()
    n = int(np.prod(case.shape))
    if args.only == "force":
        fn = lambda ctx: ctx.force(I0, T0, mb, sb, case.lam, case.signs, u, du=du)
        nbytes = FORCE_BYTES_PER_VOXEL[True] * n
    elif args.only == "smooth":
        fn = lambda ctx: ctx.smooth(u, 1.0, out=du)
        nbytes = 24 * n
    elif args.only == "compose":
        fn = lambda ctx: ctx.compose(u, dus, cg.CGDIR_COMPOSE, 0.0, out=du)
        nbytes = 36 * n
    else:   # one whole iteration: force, smoothing + composite update, smoothing
        un = torch.empty_like(u)
        fn = lambda ctx: ctx.iterate(I0, T0, mb, sb, case.lam, case.signs, u, out=un)
        nbytes = 95 * n
    with cg.Context(0) as ctx:
        if args.tuning_in:            # the registration's schedule (e.g. the force z chunk)
            with open(args.tuning_in) as f:
                ctx.load_tuning(json.load(f))
        for _ in range(args.warmup):
            fn(ctx)
        torch.cuda.synchronize()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(args.steps):
            fn(ctx)
        b.record()
        torch.cuda.synchronize()
        ctx.sync()
    ms = a.elapsed_time(b) / args.steps
    print(json.dumps({"kernel": args.only, "shape_zyx": list(case.shape), "avg_ms": ms,
                      "algorithmic_GBps": nbytes / (ms / 1e3) / 1e9}))
    return 0


def main():
    args = parse()
    if args.impl == "reference":
        return run_reference(args)
    if args.only:
        return run_only_kernel(args)
    if args.mode == "batch":
        return run_batch(args)
    if args.mode == "serve":
        return run_serve(args)
    return run_cgdir(args)


if __name__ == "__main__":
    sys.exit(main())
