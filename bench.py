#!/usr/bin/env python
"""Throughput of the NeDF composition render path on GB300.

Workload: 1024 instances of three analytic object types (sphere / torus / box) at random rigid
transforms in [-20, 20]^3, a 1024x1024 pinhole frame, 4 point lights, NeDF 6x128 per type
(trained here on ray-march labels), NeRF 8x256 colour network per type.

A step is one composited frame: Step 1 (NeDF generation: binning, NeDF queries with the
plain-method fallback below confidence 0.9 and 4-step bisection refinement, z-min), Step 2
(deferred shading with 8 NeRF samples per pixel), Step 3 (shadow rays to 4 lights answered by
NeDF queries) and the composite.  Beside it: the plain ray-marching frame on the same GPU, the
depth error of the NeDF frame against a fine ray-march judge, the training throughput, an
end-to-end number through the public API with host buffers, and the FP64 CPU oracle timed on
the host cores.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]
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

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "composited rays/s & ms/frame at 1024², NeDF vs ray-march, same GPU, depth err"
WORKLOAD = ("1024 instances (sphere/torus/box, seed 3, T in [-20,20]^3) at 1024x1024, 4 point lights, "
            "NeDF 6x128 per type trained on ray-march labels, NeRF 8x256 per type, 8 shading samples, "
            "fallback below confidence 0.9, 4 refinement steps with outlier re-answering, confident misses "
            "checked at {mc} chord samples, plain-method re-answers at the labels' 256 steps + 8 bisections")
WORKLOAD_STRESS = ("4096 instances (8 shape types x 512, seed 4, T in [-40,40]^3) at 2048x2048, 8 point lights, "
                   "NeDF 6x128 per type trained on ray-march labels, NeRF 8x256 per type, 8 shading samples, "
                   "fallback below confidence 0.9, 4 refinement steps with outlier re-answering, confident misses "
                   "checked at {mc} chord samples, plain-method re-answers at the labels' 256 steps + 8 bisections")
# the frame's options (the C ABI's nedf_options) and the same options in the oracle's names
FRAME_OPTS = dict(fallback_conf=0.9, refine_steps=4, outlier_resample=1, miss_check=64, march_steps=256,
                  march_bisect=8)
ORACLE_OPTS = dict(fallback_conf=0.9, refine_steps=4, outlier_resample=1, miss_check=64, march_n=256, march_b=8)
NEDF_FLOP = 2 * (78 * 128 + 5 * 128 * 128 + 128 * 2)          # per query, unpadded
# one training ray of the 6 x 128 NeDF: the forward pass, the input gradients of the hidden layers
# (5 x 128 x 128) and of the output layer (2 x 128), and every weight gradient (as the forward)
TRAIN_FLOP = NEDF_FLOP + 2 * (5 * 128 * 128 + 2 * 128) + NEDF_FLOP
# the trained NeDF weights of the 1024-instance workload (the bench's own training schedule, written by
# paper_2308_04669_gb300/data/make_trained_weights.py): the reference arm renders with them, so both arms
# time the same frame
TRAINED_WEIGHTS = os.path.join(ROOT, "paper_2308_04669_gb300", "data", "nedf_thousand_bench.npz")
# DRAM bytes (read + write) per launch of a stage's kernel from an ncu capture of the current
# kernel source on this frame (k_pipe<256, 0, 0>: 11.38 MB for 320,826 hit pixels, scaled to the
# bench frame's 320,655); a stage is absent here once its kernel changed after the capture.
PROFILED_TRAFFIC = {"step2_shade": 11.37e6}
NERF_FLOP = 2 * (90 * 256 + 7 * 256 * 256 + 256 * 3)          # per sample, unpadded
# the paper's intersection network: head 1008 -> 256, 16 residual blocks of two 256 x 256 layers,
# tails 256 -> 65 and 256 -> 128; per query, unpadded
CLS_FLOP = 2 * (1008 * 256 + 32 * 256 * 256 + 256 * (65 + 128))


def stage_means(r, render, frames, flush):
    """Mean milliseconds of the stages, and of the NeDF engine launches alone, over frames of their own (a
    profiled frame runs its stages one after another; the timed frames run as a user's do)."""
    r.set_profiling(True)
    for _ in range(2):
        render()
    stages, engines = {}, {}
    for _ in range(frames):
        flush.zero_()
        render()
        for k, v in r.stage_times().items():
            stages[k] = stages.get(k, 0.0) + v / frames
        for k, v in r.engine_times().items():
            engines[k] = engines.get(k, 0.0) + v / frames
    r.set_profiling(False)
    return stages, engines


def peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        d = json.load(open(p))
        return d, "measured"
    return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0, "bf16_tflops_sustained": 1700.0, "sm_max_mhz": 2070.0}, "fallback"


class ClockSampler:
    """nvidia-smi clocks and throttle reasons sampled every 200 ms while running."""

    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.proc = None

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--id={self.index}", f"--query-gpu={self.Q}",
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except OSError:
            self.proc = None
        return self

    def __exit__(self, *a):
        self.lines = []
        if self.proc is not None:
            self.proc.terminate()
            try:
                out, _ = self.proc.communicate(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()
                out, _ = self.proc.communicate()
            self.lines = [l for l in out.splitlines() if l.strip()]

    def summary(self):
        sm, mx, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for l in getattr(self, "lines", []):
            f = [x.strip() for x in l.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                mx = float(f[2])
            except ValueError:
                continue
            for n, v in zip(names, f[5:9]):
                if v.lower() == "active":
                    reasons.add(n)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": mx, "reasons": [], "samples": 0}
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": mx, "reasons": sorted(reasons), "samples": len(sm)}


def dist_setup(n_gpus):
    """One process per GPU (torchrun's RANK / WORLD_SIZE / LOCAL_RANK): NCCL on GPUs, gloo on a
    host without one (the multi-process tests).  Frames are independent, so ranks only meet in
    the barriers around the timed region and in the max over ranks."""
    import torch
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1:
        import torch.distributed as dist
        if torch.cuda.is_available():
            torch.cuda.set_device(local)
            dist.init_process_group("nccl")
        else:
            dist.init_process_group("gloo")
    elif torch.cuda.is_available():
        torch.cuda.set_device(0)
    return rank, world, local


def barrier(world):
    if world > 1:
        import torch.distributed as dist
        dist.barrier()


def allmax(x, world):
    if world == 1:
        return x
    import torch
    import torch.distributed as dist
    t = torch.tensor([x], dtype=torch.float64, device="cuda" if dist.get_backend() == "nccl" else "cpu")
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def job_value(n_pixels, frame_ms_max, world):
    """Whole-job composited rays/s: every rank renders one frame per step, the slowest rank's
    frame time bounds the step."""
    return world * n_pixels / (frame_ms_max * 1e-3)


# ------------------------------------------------------------------------------------------------
# the oracle on the host cores (cpu_baseline and the reference arm)
# ------------------------------------------------------------------------------------------------
def oracle_rate(scene, nedf_weights, target_s, threads, seed=11):
    """Pixels per second of the FP64 oracle on this host: seeded pixel batches of the same frame
    until target_s seconds have been spent."""
    import oracle
    oracle.build()
    osc = oracle.OracleScene(scene, nedf_override=nedf_weights)
    from paper_2308_04669_gb300 import scenegen as sg
    n, done, secs, batch = 0, 0, 0.0, 256
    while secs < target_s and done < scene.W * scene.H:
        px = sg.pixel_subset(scene.W, scene.H, batch, seed + n)
        t0 = time.perf_counter()
        oracle.render(osc, px=px, alt=False, n_threads=threads, **ORACLE_OPTS)
        secs += time.perf_counter() - t0
        done += len(px)
        n += 1
        batch = min(batch * 2, 8192)
    return done / secs, done, secs


def run_reference(args):
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    from paper_2308_04669_gb300 import scenegen as sg
    sc = sg.thousand_scene()
    threads = os.cpu_count() or 1
    per_step_s = max(1.0, 60.0 / max(1, args.steps + args.warmup))
    import oracle
    oracle.build()
    w_ref = reference_weights(sc)
    osc = oracle.OracleScene(sc, nedf_override=w_ref)
    # calibrate a per-step pixel sample that takes about per_step_s on the host cores
    t0 = time.perf_counter()
    oracle.render(osc, px=sg.pixel_subset(sc.W, sc.H, 256, 99), alt=False, n_threads=threads, **ORACLE_OPTS)
    n = int(max(64, 256 * per_step_s / max(time.perf_counter() - t0, 1e-3)))
    for w in range(args.warmup):
        oracle.render(osc, px=sg.pixel_subset(sc.W, sc.H, n, 200 + w), alt=False, n_threads=threads, **ORACLE_OPTS)
    t0 = time.perf_counter()
    for k in range(args.steps):
        oracle.render(osc, px=sg.pixel_subset(sc.W, sc.H, n, 300 + k), alt=False, n_threads=threads, **ORACLE_OPTS)
    dt = time.perf_counter() - t0
    value = n * args.steps / dt
    ms_frame = 1000.0 * sc.W * sc.H / value
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": "rays/s", "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms_frame, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": WORKLOAD.format(mc=args.miss_check), "W": sc.W, "H": sc.H,
                       "instances": sc.n_inst, "lights": len(sc.lights), "sample_px_per_step": n,
                       "oracle": "FP64, same scene, options and trained NeDF weights"},
            "cpu_baseline": {"value": value, "unit": "rays/s", "cores": threads, "kind": "oracle",
                             "sample": f"{n} seeded pixels of the 1024x1024 frame per step, all 1024 instances, "
                                       + ("the trained NeDF weights of the bench's schedule" if w_ref else
                                          "untrained NeDF weights (no trained-weights file)")
                                       + "; ms_per_step extrapolates to the full frame"},
            "e2e": {"value": value, "unit": "rays/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)




def reference_weights(sc):
    """The committed trained NeDF weights of the 1024-instance workload (per type, FP32), or None."""
    if not os.path.exists(TRAINED_WEIGHTS):
        return None
    z = np.load(TRAINED_WEIGHTS)
    w = {t: z[f"type{t}"].astype(np.float64) for t in range(len(sc.types))}
    if any(w[t].shape != sc.types[t].nedf_w.shape for t in w):
        return None
    return w


# ------------------------------------------------------------------------------------------------
# our arm
# ------------------------------------------------------------------------------------------------
def train_types(r, scene, steps, batch, n_rays, log, stream, peak_tflops):
    """The learned part on the GPU: each type's training set (n_rays plain-method labels), then
    `steps` Adam steps of `batch` rays per type.  Device time from CUDA events on the stream."""
    import hashlib
    import torch
    t0 = time.perf_counter()
    for t in range(len(scene.types)):
        r.make_labels(t, n_rays, 2 + t, 256, 8)
    torch.cuda.synchronize()
    t_labels = time.perf_counter() - t0
    losses = []
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    t0 = time.perf_counter()
    e0.record(stream)
    for t in range(len(scene.types)):
        first = r.train_step(t, batch, 1e-3, want_loss=True)
        for s in range(steps - 2):
            r.train_step(t, batch, 1e-3)
        last = r.train_step(t, batch, 1e-3, want_loss=True)
        losses.append((first, last))
    e1.record(stream)
    torch.cuda.synchronize()
    t_train = time.perf_counter() - t0
    dev_s = e0.elapsed_time(e1) * 1e-3
    rays_s = len(scene.types) * steps * batch / dev_s
    tflops = rays_s * TRAIN_FLOP / 1e12
    w = np.concatenate([r.get_nedf_weights(t, scene.types[t].nedf_w.shape[0]) for t in range(len(scene.types))])
    log["train"] = {"types": len(scene.types), "steps_per_type": steps, "batch": batch,
                    "label_rays_per_type": n_rays, "label_s": round(t_labels, 3),
                    "ms_per_step": round(1e3 * dev_s / (len(scene.types) * steps), 4),
                    "train_rays_per_s": round(rays_s, 1), "wall_s": round(t_train, 2),
                    "flop_per_ray": TRAIN_FLOP, "tflops": round(tflops, 2),
                    "roofline": {"bound": "tensor", "achieved": round(tflops, 2), "peak": peak_tflops,
                                 "unit": "TFLOP/s", "frac": round(tflops / peak_tflops, 4)},
                    "loss_first_last": [[round(a, 5), round(b, 5)] for a, b in losses],
                    "weights_sha256": hashlib.sha256(w.astype(np.float32).tobytes()).hexdigest()}


def fp8_frame(sc, r, stream, jdepth, jids, peak_bf16, args, frames=20):
    """The same frame with every hidden layer but the first in E4M3 (per-layer scales), rendered
    with the trained weights of `r` (BF16 training) and the same options: frame time, stages, the
    engines against the FP8 peak, and the all-pixel depth error against the same judge."""
    import copy
    import torch
    from paper_2308_04669_gb300 import native
    n = sc.W * sc.H
    w_tr = [r.get_nedf_weights(t, sc.types[t].nedf_w.shape[0]) for t in range(len(sc.types))]
    sc8 = copy.copy(sc)
    sc8.types = [copy.copy(t) for t in sc.types]
    for t, w in zip(sc8.types, w_tr):
        t.nedf_w = w
    r8 = native.renderer_for(sc8, precision=native.PREC_FP8, stream=stream)
    o8 = r8.get_options()
    for k, v in FRAME_OPTS.items():
        setattr(o8, k, v)
    r8.set_options(o8)
    cam, lights = r8.camera(sc.eye, sc.target, sc.fov_deg), r8.lights(sc.lights)
    sched = r8.autotune(cam, lights, reps=2) if not args.no_autotune else None
    depth = torch.empty(n, device="cuda")
    ids = torch.empty(n, dtype=torch.int32, device="cuda")
    out = torch.empty(n, 4, device="cuda")
    flush = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")
    for _ in range(3):
        r8.render(cam, lights, depth, ids, None, None, out)
    st = r8.render(cam, lights, depth, ids, None, None, out, stats=True)
    torch.cuda.synchronize()
    tot = 0.0
    for _ in range(frames):
        flush.zero_()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        r8.render(cam, lights, depth, ids, None, None, out)
        e1.record(stream)
        torch.cuda.synchronize()
        tot += e0.elapsed_time(e1)
    ms = tot / frames
    stages, engines = stage_means(r8, lambda: r8.render(cam, lights, depth, ids, None, None, out), frames, flush)
    both = (ids != -1) & (jids != -1)
    err = (depth.double() - jdepth.double()).abs()[both]
    peak8 = 2.0 * peak_bf16
    eng = {}
    for k, pairs in (("step1_nedf", st.primary_pairs), ("step3_nedf", st.shadow_pairs)):
        if engines.get(k, 0) > 0:
            tf = pairs * NEDF_FLOP / (engines[k] * 1e-3) / 1e12
            eng[k] = {"engine_ms": round(engines[k], 4), "engine_tflops": round(tf, 1), "engine_frac_fp8": round(tf / peak8, 3)}
    shade_tf = st.hit_pixels * 8 * NERF_FLOP / (stages["step2_shade"] * 1e-3) / 1e12
    r8.close()
    return {"ms_per_frame": ms, "rays_per_s": n / (ms * 1e-3),
            "stage_ms": {k: round(v, 4) for k, v in stages.items()}, "engines": eng,
            "step2_shade": {"tflops": round(shade_tf, 1), "frac_fp8": round(shade_tf / peak8, 3)},
            "fallback_pairs": st.fallback_pairs,
            "depth_err": {"mean_over_rb": float(err.mean()), "p99_over_rb": float(torch.quantile(err.float(), 0.99)),
                          "id_agreement": float((ids == jids)[both].double().mean()),
                          "pixels_both_hit": int(both.sum())},
            "schedule": sched,
            "peak_basis": "fp8 dense = bf16 dense measured (burst) x 2 (nominal 4.5 / 2.25 PFLOP/s)",
            "note": "hidden layers after the first in E4M3 with per-layer scales, FP32 accumulation; the BF16 frame's trained weights and options; same judge"}


def classifier_frame(sc, stream, cam, lights, args, frames=5):
    """The workload's instances, lights and NeRF colour networks with every type's NeDF replaced
    by the paper's classifier network (seeded weights): frame time and the NeDF engines alone."""
    import copy
    import torch
    from paper_2308_04669_gb300 import native
    from paper_2308_04669_gb300 import scenegen as sg
    n = sc.W * sc.H
    scc = copy.copy(sc)
    scc.types = []
    for i, t in enumerate(sc.types):
        tc = sg.make_type(t.kind, 1, i, 0, 0, rb=t.rb, params=t.params, nedf_arch=sg.ARCH_CLASSIFIER)
        tc.nerf_hidden, tc.nerf_width, tc.nerf_w, tc.albedo = t.nerf_hidden, t.nerf_width, t.nerf_w, t.albedo
        scc.types.append(tc)
    rc = native.renderer_for(scc, precision=native.PREC_BF16, stream=stream)
    oc = rc.get_options()
    for k, v in FRAME_OPTS.items():
        setattr(oc, k, v)
    # untrained weights: their confidence means nothing, and most of their misses are wrong
    oc.fallback_conf, oc.outlier_resample, oc.miss_check = 0.0, 0, 0
    rc.set_options(oc)
    cam, lights = rc.camera(sc.eye, sc.target, sc.fov_deg), rc.lights(sc.lights)
    cls_sched = rc.autotune(cam, lights, reps=2) if not args.no_autotune else None
    depth = torch.empty(n, device="cuda")
    ids = torch.empty(n, dtype=torch.int32, device="cuda")
    out = torch.empty(n, 4, device="cuda")
    flush = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")
    for _ in range(2):
        rc.render(cam, lights, depth, ids, None, None, out)
    stc = rc.render(cam, lights, depth, ids, None, None, out, stats=True)
    torch.cuda.synchronize()
    ev_c = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(frames)]
    for a, b in ev_c:
        flush.zero_()
        a.record(stream)
        rc.render(cam, lights, depth, ids, None, None, out)
        b.record(stream)
    torch.cuda.synchronize()
    ms_c = sum(a.elapsed_time(b) for a, b in ev_c) / len(ev_c)
    stg_c, eng_c = stage_means(rc, lambda: rc.render(cam, lights, depth, ids, None, None, out), len(ev_c), flush)
    pk_c, pk_kind_c = peaks()
    pairs_c = {"step1_nedf": stc.primary_pairs, "step3_nedf": stc.shadow_pairs}
    eng = {}
    for k, np_ in pairs_c.items():
        if eng_c.get(k):
            tf = np_ * CLS_FLOP / (eng_c[k] * 1e-3) / 1e12
            eng[k] = {"engine_ms": round(eng_c[k], 4), "pairs": int(np_), "engine_tflops": round(tf, 1),
                      "engine_frac": round(tf / pk_c["bf16_tflops"], 3)}
    rc.close()
    return {"ms_per_frame": ms_c, "rays_per_s": n / (ms_c * 1e-3), "flop_per_query": CLS_FLOP,
            "engines": eng, "stage_ms": {k: round(v, 4) for k, v in stg_c.items()},
            "hit_pixels": int(stc.hit_pixels), "schedule": cls_sched,
            "peak_basis": f"bf16 dense, {pk_kind_c} (burst)",
            "note": "same instances, lights and NeRF colour networks; every type's NeDF is the paper's "
                    "classifier network with seeded random weights; no confidence fallback"}


def run_ours(args):
    import torch
    from paper_2308_04669_gb300 import build as nbuild
    rank, world, local = dist_setup(args.gpus)
    if rank == 0 or True:
        nbuild.build()
    barrier(world)
    from paper_2308_04669_gb300 import native
    from paper_2308_04669_gb300 import scenegen as sg

    sc = sg.thousand_scene() if args.scene == "thousand" else sg.stress_scene()
    workload = (WORKLOAD if args.scene == "thousand" else WORKLOAD_STRESS).format(mc=args.miss_check)
    n_li = len(sc.lights)
    stream = torch.cuda.Stream()            # a non-default stream: frames are CUDA-graph captured
    torch.cuda.set_stream(stream)
    if args.cls_only:                       # the classifier frame alone (profiling)
        if rank == 0:
            print(json.dumps({"classifier_frame": classifier_frame(sc, stream, None, None, args, frames=args.steps)}),
                  flush=True)
        return
    prec = {"fp32": native.PREC_FP32, "bf16": native.PREC_BF16, "fp8": native.PREC_FP8}[args.precision]
    r = native.renderer_for(sc, precision=prec, stream=stream)
    log = {}
    if args.train_steps > 0:
        train_types(r, sc, args.train_steps, args.train_batch, args.label_rays, log, stream, peaks()[0]["bf16_tflops"])
        if args.train_only:                 # the learned part alone (profiling)
            r.close()
            if rank == 0:
                print(json.dumps({"train_only": True, **log}), flush=True)
            return
        ref_w = reference_weights(sc) if args.scene == "thousand" else None
        if ref_w is not None:
            log["train"]["same_weights_as_reference_arm"] = all(
                np.array_equal(ref_w[t].astype(np.float32), r.get_nedf_weights(t, sc.types[t].nedf_w.shape[0]))
                for t in range(len(sc.types)))
    o = r.get_options()
    for k, v in FRAME_OPTS.items():
        setattr(o, k, v)
    r.set_options(o)
    cam, lights = r.camera(sc.eye, sc.target, sc.fov_deg), r.lights(sc.lights)
    n = sc.W * sc.H
    dev = "cuda"
    # the library's autotuner picks the tensor-core kernels' schedule on this frame (untimed)
    schedule = None
    if args.schedule and prec != native.PREC_FP32:        # a fixed schedule (reproducible profiles)
        r.set_schedule([int(x) for x in args.schedule.split(",")])
        schedule = {"fixed": r.get_schedule()}
    elif prec != native.PREC_FP32 and not args.no_autotune:
        schedule = r.autotune(cam, lights, reps=2)
    depth = torch.empty(n, device=dev)
    ids = torch.empty(n, dtype=torch.int32, device=dev)
    out = torch.empty(n, 4, device=dev)
    flush = torch.empty(256 << 20, dtype=torch.uint8, device=dev)     # > 129 MB L2
    for _ in range(args.warmup):
        r.render(cam, lights, depth, ids, None, None, out)
    st = r.render(cam, lights, depth, ids, None, None, out, stats=True)
    torch.cuda.synchronize()
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(args.steps)]
    barrier(world)
    torch.cuda.synchronize()
    with ClockSampler(local) as clk:
        t_wall = time.perf_counter()
        for k in range(args.steps):
            flush.zero_()                                   # L2 flushed between timed frames (untimed)
            ev[k][0].record(stream)
            r.render(cam, lights, depth, ids, None, None, out)
            ev[k][1].record(stream)
        torch.cuda.synchronize()
        t_wall = time.perf_counter() - t_wall
    barrier(world)
    frame_ms = sum(a.elapsed_time(b) for a, b in ev) / args.steps
    frame_ms_max = allmax(frame_ms, world)
    stage_ms, engine_ms = stage_means(r, lambda: r.render(cam, lights, depth, ids, None, None, out), args.steps, flush)
    engine_ms = {k: v for k, v in engine_ms.items() if v > 0}                # the NeDF engine launches alone
    clocks = clk.summary()

    if args.frames_only:
        r.close()
        if rank == 0:
            print(json.dumps({"frames_only": True, "schedule": schedule, "ms_per_frame": frame_ms, "rays_per_s": n / (frame_ms * 1e-3),
                              "stage_ms": stage_ms, "engine_ms": engine_ms, "primary_pairs": st.primary_pairs, "shadow_pairs": st.shadow_pairs,
                              "hit_pixels": st.hit_pixels, "fallback_pairs": st.fallback_pairs}), flush=True)
        return

    # ---- depth error against a fine ray-march judge ------------------------------------------
    o2 = r.get_options()
    saved = (o2.depth_source, o2.march_steps, o2.march_bisect)
    o2.depth_source, o2.march_steps, o2.march_bisect = 1, 1024, 24
    r.set_options(o2)
    jdepth = torch.empty(n, device=dev)
    jids = torch.empty(n, dtype=torch.int32, device=dev)
    r.render(cam, lights, jdepth, jids, None, None, None)
    (o2.depth_source, o2.march_steps, o2.march_bisect) = saved
    r.set_options(o2)
    torch.cuda.synchronize()
    both = (ids != -1) & (jids != -1)
    err = (depth.double() - jdepth.double()).abs()[both] / 1.0       # r_b = 1, s = 1: world = local
    same = both & (ids == jids)
    err_same = (depth.double() - jdepth.double()).abs()[same]
    edges = [0.0, 1e-4, 3e-4, 1e-3, 3e-3, 1e-2, 3e-2, 1e-1, 3e-1, 1.0, float("inf")]
    hist = torch.histogram(err_same.cpu(), bins=torch.tensor(edges, dtype=torch.float64))[0] if err_same.numel() else None
    derr = {"mean_over_rb": float(err.mean()) if err.numel() else None,
            "median_over_rb": float(err.median()) if err.numel() else None,
            "p99_over_rb": float(torch.quantile(err.float(), 0.99)) if err.numel() else None,
            "pixels_both_hit": int(both.sum()),
            "id_agreement": float((ids == jids)[both].double().mean()) if err.numel() else None,
            "mean_over_rb_same_id": float(err_same.mean()) if err_same.numel() else None,
            "p99_over_rb_same_id": float(torch.quantile(err_same.float(), 0.99)) if err_same.numel() else None,
            "histogram_same_id": {"edges_over_rb": edges[:-1] + ["inf"],
                                  "counts": [int(c) for c in hist]} if hist is not None else None,
            "hit_mask_agreement": float(((ids != -1) == (jids != -1)).double().mean())}

    # ---- plain ray-march frame on the same GPU ------------------------------------------------
    march = {}
    mrgba = torch.empty(n, 4, device=dev)
    for es, key in [(1, "early_stop"), (0, "dense")]:
        if not es and not args.march_dense:
            continue
        try:
            r.render_march(cam, 128, es, mrgba)
            torch.cuda.synchronize()
            reps = 1
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            for _ in range(reps):
                r.render_march(cam, 128, es, mrgba)
            e1.record(stream)
            torch.cuda.synchronize()
            ms = e0.elapsed_time(e1) / reps
            march[key] = {"ms_per_frame": ms, "rays_per_s": n / (ms * 1e-3), "samples_per_pair": 128}
        except native.NedfError as e:
            march[key] = {"unavailable": str(e)}

    # ---- the same frame with Step-2 outlier resampling ("rs": pixels whose sample densities are
    # all below 1 re-rendered by the plain method, 128 samples per pair), as the paper times it ----
    rs = None
    if not args.no_resample:
        o_keep = r.get_options()
        o_rs = r.get_options()
        o_rs.shade_resample, o_rs.shade_sigma_min = 128, 1.0
        r.set_options(o_rs)
        for _ in range(2):
            r.render(cam, lights, depth, ids, None, None, out)
        st_rs = r.render(cam, lights, depth, ids, None, None, out, stats=True)
        torch.cuda.synchronize()
        ev_rs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(5)]
        for a, b in ev_rs:
            flush.zero_()
            a.record(stream)
            r.render(cam, lights, depth, ids, None, None, out)
            b.record(stream)
        torch.cuda.synchronize()
        ms_rs = sum(a.elapsed_time(b) for a, b in ev_rs) / len(ev_rs)
        rs = {"ms_per_frame": ms_rs, "rays_per_s": n / (ms_rs * 1e-3), "resampled_pixels": int(st_rs.resampled_pixels),
              "samples_per_pair": 128, "sigma_min": 1.0}
        # the paper's order: no Step-1 refinement or re-answering, Step 2's density test instead
        o_rs.refine_steps, o_rs.outlier_resample = 0, 0
        r.set_options(o_rs)
        for _ in range(2):
            r.render(cam, lights, depth, ids, None, None, out)
        st_nr = r.render(cam, lights, depth, ids, None, None, out, stats=True)
        torch.cuda.synchronize()
        for a, b in ev_rs:
            flush.zero_()
            a.record(stream)
            r.render(cam, lights, depth, ids, None, None, out)
            b.record(stream)
        torch.cuda.synchronize()
        ms_nr = sum(a.elapsed_time(b) for a, b in ev_rs) / len(ev_rs)
        o_rs.shade_resample = 0
        r.set_options(o_rs)
        for a, b in ev_rs:
            flush.zero_()
            a.record(stream)
            r.render(cam, lights, depth, ids, None, None, out)
            b.record(stream)
        torch.cuda.synchronize()
        ms_wo = sum(a.elapsed_time(b) for a, b in ev_rs) / len(ev_rs)
        rs["without_refinement"] = {"rs_ms_per_frame": ms_nr, "wo_rs_ms_per_frame": ms_wo,
                                    "resampled_pixels": int(st_nr.resampled_pixels)}
        r.set_options(o_keep)

    # ---- buffer reuse while one instance is dragged: the other objects' work frozen, edit frames
    # redo only what the moved instance changes (the paper's interactive manipulation mode) -------
    edit = None
    if not args.no_edit:
        r.render(cam, lights, depth, ids, None, None, out)
        torch.cuda.synchronize()
        idv = ids.cpu().numpy().view(np.uint32)
        won = np.bincount(idv[idv != 0xFFFFFFFF], minlength=sc.n_inst)
        e_inst = int(np.argmax(won))                      # the instance covering the most pixels
        r.begin_edit(cam, lights, e_inst)
        T_edit = sc.inst_T.copy()
        ev_ed = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(10)]
        for k, (a, b) in enumerate(ev_ed):
            T_edit[e_inst] = sc.inst_T[e_inst] + np.float32(0.05) * np.float32(k + 1)   # dragged along x, y, z
            r.set_instances(sc.inst_type, sc.inst_R, T_edit, sc.inst_s)
            flush.zero_()
            a.record(stream)
            r.render_edit(depth, ids, None, None, out)
            b.record(stream)
        torch.cuda.synchronize()
        ms_edit = sum(a.elapsed_time(b) for a, b in ev_ed[2:]) / (len(ev_ed) - 2)   # first two capture the graph
        r.end_edit()
        r.set_instances(sc.inst_type, sc.inst_R, sc.inst_T, sc.inst_s)
        edit = {"ms_per_frame": ms_edit, "whole_frame_ms": frame_ms, "speedup": frame_ms / ms_edit,
                "instance": e_inst, "pixels_won": int(won[e_inst]),
                "note": "device time of render_edit; set_instances (host upload) between frames is not timed"}

    # ---- the same scene with the paper's classifier intersection network on every type --------
    cls = None
    if prec == native.PREC_BF16 and not args.no_cls:
        cls = classifier_frame(sc, stream, cam, lights, args)

    # ---- the same frame with the FP32 CUDA-core networks (reference precision) -----------------
    fp32 = None
    if prec != native.PREC_FP32 and not args.no_fp32:
        r32 = native.renderer_for(sc, precision=native.PREC_FP32, stream=stream)
        w_tr = [r.get_nedf_weights(t, sc.types[t].nedf_w.shape[0]) for t in range(len(sc.types))]
        import copy
        sc32 = copy.copy(sc)
        sc32.types = [copy.copy(t) for t in sc.types]
        for t, w in zip(sc32.types, w_tr):
            t.nedf_w = w
        r32.load_scene(sc32)
        o32 = r32.get_options()
        for k, v in FRAME_OPTS.items():
            setattr(o32, k, v)
        r32.set_options(o32)
        r32.render(cam, lights, depth, ids, None, None, out)
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        for _ in range(3):
            r32.render(cam, lights, depth, ids, None, None, out)
        e1.record(stream)
        torch.cuda.synchronize()
        fp32 = {"ms_per_frame": e0.elapsed_time(e1) / 3, "rays_per_s": n / (e0.elapsed_time(e1) / 3 * 1e-3)}
        r32.close()

    # ---- the same frame with E4M3 hidden layers (the precision ladder's next rung) ------------
    fp8 = None
    if prec == native.PREC_BF16 and not args.no_fp8:
        fp8 = fp8_frame(sc, r, stream, jdepth, jids, peaks()[0]["bf16_tflops"], args)

    # ---- end to end through the public API with host buffers ---------------------------------
    host_out = torch.empty(n, 4, dtype=torch.float32, pin_memory=True)
    inst_args = (sc.inst_type, sc.inst_R, sc.inst_T, sc.inst_s)
    for _ in range(2):
        r.set_instances(*inst_args)
        r.render_host(cam, lights, out=host_out.data_ptr())
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for _ in range(args.steps):
        r.set_instances(*inst_args)                          # H2D: this step's instance records
        r.render_host(cam, lights, out=host_out.data_ptr())  # D2H: the composited frame
    e2e_s = (time.perf_counter() - t0) / args.steps
    h2d = sc.n_inst * 56 + 16 * 0
    d2h = n * 16

    # ---- roofline of the dominant kernel ------------------------------------------------------
    pk, pk_kind = peaks()
    P1, P3, Hv = st.primary_pairs, st.shadow_pairs, st.hit_pixels
    flops = {"step1_nedf": P1 * NEDF_FLOP, "step2_shade": Hv * sc.n_shade * NERF_FLOP, "step3_nedf": P3 * NEDF_FLOP}
    dom = max(flops, key=lambda k: stage_ms.get(k, 0.0))
    achieved = flops[dom] / (stage_ms[dom] * 1e-3) / 1e12
    # every MLP stage against the same peak (the NeDF stages also hold their deferred plain-method pairs)
    mlp_stages = {k: {"tflops": round(f / (stage_ms[k] * 1e-3) / 1e12, 1), "ms": round(stage_ms[k], 4)}
                  for k, f in flops.items() if stage_ms.get(k)}
    if prec == native.PREC_FP32:
        peak = 152 * 128 * 2 * pk.get("sm_max_mhz", 2070.0) * 1e6 / 1e12
        roof = {"bound": "alu", "achieved": achieved, "peak": peak, "unit": "TFLOP/s", "frac": achieved / peak,
                "traffic": None, "kernel": dom,
                "peak_basis": "FP32 FMA: 152 SMs x 128 lanes x 2 FLOP x max SM clock (CUDA-core path)"}
    elif prec == native.PREC_BF16:
        peak = pk["bf16_tflops"]
        roof = {"bound": "tensor", "achieved": achieved, "peak": peak, "unit": "TFLOP/s", "frac": achieved / peak,
                "traffic": PROFILED_TRAFFIC.get(dom), "kernel": dom, "peak_basis": f"bf16 dense, {pk_kind} (burst)"}
    else:
        # E4M3 hidden layers: the BF16 peak x the nominal FP8 / BF16 ratio (4.5 / 2.25 PFLOP/s); the
        # first layer (BF16) is a few per cent of the FLOPs, so this peak is a slight overstatement
        peak = pk["bf16_tflops"] * 2.0
        roof = {"bound": "tensor", "achieved": achieved, "peak": peak, "unit": "TFLOP/s", "frac": achieved / peak,
                "traffic": None, "kernel": dom,
                "peak_basis": f"fp8 dense = bf16 dense {pk_kind} (burst) x 2 (nominal 4.5 / 2.25 PFLOP/s)"}
    for k in mlp_stages:
        mlp_stages[k]["frac"] = round(mlp_stages[k]["tflops"] / roof["peak"], 3)
        if k in engine_ms:                 # the engine kernel alone (CUDA events around its launch)
            t = flops[k] / (engine_ms[k] * 1e-3) / 1e12
            mlp_stages[k].update(engine_ms=round(engine_ms[k], 4), engine_tflops=round(t, 1),
                                 engine_frac=round(t / roof["peak"], 3))

    # ---- CPU baseline: the oracle on the host cores ------------------------------------------
    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu:
        w_tr = {t: r.get_nedf_weights(t, sc.types[t].nedf_w.shape[0]).astype(np.float64)
                for t in range(len(sc.types))}
        threads = os.cpu_count() or 1
        rate, npx, secs = oracle_rate(sc, w_tr, args.cpu_seconds, threads)
        rate1, npx1, secs1 = oracle_rate(sc, w_tr, max(2.0, args.cpu_seconds / 3), 1, seed=71)
        cpu = {"value": rate, "unit": "rays/s", "cores": threads, "kind": "oracle",
               "sample": f"{npx} seeded pixels of the same {sc.W}x{sc.H} frame (same trained weights, all {sc.n_inst} "
                         f"instances, {n_li} lights), {secs:.1f} s on {threads} threads",
               "single_core": {"value": rate1, "unit": "rays/s", "cores": 1,
                               "sample": f"{npx1} seeded pixels, {secs1:.1f} s on 1 thread"}}
    r.close()

    value = job_value(n, frame_ms_max, world)
    line = {"metric": METRIC, "value": value, "unit": "rays/s", "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": frame_ms_max, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": {"fp32": "f32", "bf16": "bf16", "fp8": "e4m3 (first layer bf16)"}[args.precision],
            "data": "synthetic",
            "config": {"workload": workload, "W": sc.W, "H": sc.H, "instances": sc.n_inst, "lights": n_li,
                       "l2": "flushed between timed frames (256 MiB write, outside the timed events)",
                       "parallelism": f"replicas x{world} (one frame per GPU)"},
            "roofline": roof, "cpu_baseline": cpu,
            "e2e": {"value": world * n / e2e_s, "unit": "rays/s", "h2d_bytes_per_step": h2d, "d2h_bytes_per_step": d2h},
            "gpu_launches": int(st.kernel_launches) * args.steps,
            "clocks": clocks,
            "frame": {"ms": frame_ms, "total_rays_per_s": n * (1 + n_li) / (frame_ms * 1e-3),
                      "primary_pairs": P1, "shadow_pairs": P3, "hit_pixels": Hv, "fallback_pairs": st.fallback_pairs,
                      "fallback_rate": st.fallback_pairs / max(1, P1 + P3), "mlp_stages": mlp_stages,
                      "stage_ms": {k: round(v, 4) for k, v in stage_ms.items()}, "wall_s": t_wall},
            "fp32_frame": fp32,
            "fp8_frame": fp8,
            "rs_frame": rs,
            "edit_frame": edit,
            "classifier_frame": cls,
            "march_frame": march,
            "speedup_vs_march": {k: v["ms_per_frame"] / frame_ms for k, v in march.items() if "ms_per_frame" in v},
            "depth_err": derr, "schedule": schedule, **log}
    if rank == 0:
        print(json.dumps(line), flush=True)
    if world > 1:
        import torch.distributed as dist
        dist.destroy_process_group()


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=120, help="timed frames (the paper averages 120)")
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--precision", default="bf16", choices=["fp32", "bf16", "fp8"])
    ap.add_argument("--scene", default="thousand", choices=["thousand", "stress"],
                    help="thousand: the metric's 1024-instance 1024^2 frame; stress: 4096 instances at 2048^2, 8 lights")
    ap.add_argument("--train-steps", type=int, default=20000, help="Adam steps per type (the workload's 20k)")
    ap.add_argument("--train-batch", type=int, default=65536)
    ap.add_argument("--label-rays", type=int, default=1 << 22, help="plain-method labelled rays per type (2^22)")
    ap.add_argument("--miss-check", type=int, default=64, help="chord samples that verify a confident NeDF miss")
    ap.add_argument("--cpu-seconds", type=float, default=12.0)
    ap.add_argument("--no-cpu", action="store_true")
    ap.add_argument("--no-fp32", action="store_true")
    ap.add_argument("--no-fp8", action="store_true", help="skip the E4M3 frame beside the BF16 one")
    ap.add_argument("--no-autotune", action="store_true", help="keep the default tensor-core schedule")
    ap.add_argument("--no-resample", action="store_true", help="skip the frame with Step-2 outlier resampling")
    ap.add_argument("--no-edit", action="store_true", help="skip the buffer-reuse (edit) frames")
    ap.add_argument("--no-cls", action="store_true", help="skip the classifier-network frames")
    ap.add_argument("--cls-only", action="store_true", help="only the classifier-network frame (for profiling)")
    ap.add_argument("--schedule", default="", help="fixed stage bytes per tensor-core kernel (shade, march colour, "
                    "Step-1 NeDF, Step-3 NeDF, query), comma-separated; skips the autotuner")
    ap.add_argument("--no-march-dense", dest="march_dense", action="store_false",
                    help="skip the dense 128-sample ray-march frame (timed by default beside the early-stop one)")
    ap.add_argument("--train-only", action="store_true",
                    help="only the labels and training steps of the learned part (profiling runs)")
    ap.add_argument("--frames-only", action="store_true",
                    help="timed frames only: no judge, ray-march, FP32, e2e or CPU legs (profiling runs)")
    args = ap.parse_args()
    if args.warmup < 3:
        args.warmup = 3
    FRAME_OPTS["miss_check"] = ORACLE_OPTS["miss_check"] = args.miss_check
    if args.impl == "reference":
        run_reference(args)
    else:
        run_ours(args)


if __name__ == "__main__":
    main()
