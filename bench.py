"""Benchmark: one online frame of the geometry core per step.

A step is the whole hot path for one frame: temporal depth refinement of all
input views, the confidence-weight map, TSDF fusion with zero-crossing
extraction into the target view, and the per-view forward splat (clear,
scatter, resolve with the guided mask).  The workload is 8 input views at
1920x1080 (2x4 rig, 10 cm spacing) fused into one 1920x1080 target, D = 128
samples on [0.3, 8] m, mu = 0.04 m, synthetic seeded scene.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl gvs|reference]

Under torchrun each rank runs its own frames (replicas, weak scaling); rank 0
prints one JSON line.  `--impl reference` times the FP64 CPU oracle on a
bounded sample of the same workload (rank 0 only).
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import tempfile
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "target-view Mpix/s (TSDF fuse+splat, 8x1080p inputs, D=128); fwd+bwd Mpix/s; % HBM peak"
WORKLOAD = "headline_8x1080p"
RING = 4                 # distinct frames resident in HBM, cycled step by step
OPS_PER_SAMPLE_VIEW = 20  # algorithmic FP32 instructions per (sample, view) of the fusion loop


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=200)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", default="gvs", choices=["gvs", "reference"])
    ap.add_argument("--e2e-steps", type=int, default=60)
    ap.add_argument("--no-clocks", action="store_true")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--only-form", default=None, choices=sorted(FORM_CLASSES),
                    help="time one form of the 8x1080p frame alone (for profiling) and print its ms per step")
    return ap.parse_args()


def dist_env():
    return int(os.environ.get("RANK", 0)), int(os.environ.get("LOCAL_RANK", 0)), int(os.environ.get("WORLD_SIZE", 1))


def measured_peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        with open(p) as f:
            d = json.load(f)
        return d.get("hbm_gbs", 6800.0), "measured", d
    return 6800.0, "fallback", {}


# ------------------------------------------------------------------ clocks --

class ClockSampler:
    """nvidia-smi clock / throttle sampling while the timed region runs."""
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int, enabled: bool = True):
        self.proc = None
        self.path = None
        self.gpu = gpu_index
        if not enabled:
            return
        try:
            fd, self.path = tempfile.mkstemp(suffix=".csv")
            os.close(fd)
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(gpu_index), f"--query-gpu={self.FIELDS}",
                                          "--format=csv,noheader,nounits", "-lms", "100"],
                                         stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
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
        rows = []
        for line in open(self.path):
            parts = [x.strip() for x in line.split(",")]
            if len(parts) < 9:
                continue
            try:
                rows.append((float(parts[1]), float(parts[2]), parts[5:9]))
            except ValueError:
                continue
        os.unlink(self.path)
        if not rows:
            return None
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for _, _, r in rows for i, v in enumerate(r) if v.lower().startswith("active")})
        return {"sm_mhz": statistics.median(r[0] for r in rows), "sm_max_mhz": max(r[1] for r in rows),
                "reasons": reasons, "samples": len(rows)}


# ------------------------------------------------------------------ inputs --

def render_frames(w, frames):
    from synth import rgba_to_u32
    out = []
    for t in frames:
        rgb, d = w.render_inputs(t)
        out.append((rgba_to_u32(rgb), d))
    return out


# --------------------------------------------------------------- GPU path --

def tune_fusion(w, depth0, ws, tgt, half, fused, cross):
    """The fusion's bundle shape for a workload, picked by the library's autotuner on its
    first frame (every variant gives the same bits; only the time differs).  Returns
    (variant, {variant: ms}); the choice is cached per device and workload."""
    from paper_2505_18932_gb300 import autotune, gvs
    N, H, W = depth0.shape
    mapped = []

    def runner(v):  # called only when the choice is not cached
        if not mapped:
            gvs.weight_map(depth0, w.mu, ws=ws, map_half=half)
            mapped.append(True)
        return lambda: gvs.fuse_depth_from_map(w.inputs, ws, (N, H, W), tgt, w.num_samples, w.z_near, w.z_far,
                                               w.mu, fused=fused, crossing=cross, map_half=half, variant=v)
    shape = {"views": (N, H, W), "target": (tgt.width, tgt.height), "D": w.num_samples,
             "z": (w.z_near, w.z_far), "mu": w.mu, "map_half": half}
    return autotune.choose(shape, runner, candidates=autotune.variants_for(N, tgt.width * tgt.height, H * W))


class Pipeline:
    """Device buffers and the per-frame call sequence through the C ABI."""

    def __init__(self, w, frames_np, device, half=False):
        import torch
        from paper_2505_18932_gb300 import gvs
        self.torch, self.gvs, self.w, self.half = torch, gvs, w, half
        self.tgt = w.targets[0]
        N = len(w.inputs)
        H, W = w.inputs[0].height, w.inputs[0].width
        Ht, Wt = self.tgt.height, self.tgt.width
        self.N, self.H, self.W, self.Ht, self.Wt = N, H, W, Ht, Wt
        self.rgba = [torch.from_numpy(c.view(np.int32)).to(device) for c, _ in frames_np]
        dt = torch.float16 if half else torch.float32
        self.depth = [torch.from_numpy(d).to(device).to(dt) for _, d in frames_np]
        self.state = self.depth[0].clone()
        self.mask = torch.empty((N, H, W), dtype=torch.uint8, device=device)
        self.fused = torch.empty((Ht, Wt), dtype=torch.float32, device=device)
        self.cross = torch.empty((Ht, Wt), dtype=torch.int16, device=device)
        self.ws_fuse = gvs.workspace(gvs.fuse_workspace_bytes(N, W, H), device)
        # two z-buffers: two views per scatter/resolve pass (measured fastest; four overflow L2)
        self.ws_splat = gvs.workspace(2 * gvs.splat_workspace_bytes(N, Wt, Ht), device)
        shape = (N, Ht, Wt)
        self.outs = {"winner": torch.empty(shape, dtype=torch.int32, device=device),
                     "warped_rgba": torch.empty(shape, dtype=torch.int32, device=device),
                     "warped_depth": torch.empty(shape, dtype=torch.float32, device=device),
                     "alpha": torch.empty(shape, dtype=torch.uint8, device=device),
                     "guided": torch.empty(shape, dtype=torch.uint8, device=device)}
        self.variant, self.tune_ms = self.tune()

    def tune(self):
        return tune_fusion(self.w, self.depth[0], self.ws_fuse, self.tgt, self.half, self.fused, self.cross)

    def step(self, i, events=None):
        """Frame i of the ring: refine -> fuse -> splat.  `events`: 4 CUDA events bracketing the stages."""
        w, gvs = self.w, self.gvs
        cur, prev = i % len(self.rgba), (i - 1) % len(self.rgba)
        if events:
            events[0].record()
        gvs.refine_depth(self.rgba[cur], self.rgba[prev], self.depth[cur], self.state, self.mask, tau=w.tau)
        if events:
            events[1].record()
        gvs.fuse_depth(w.inputs, self.state, self.tgt, w.num_samples, w.z_near, w.z_far, w.mu,
                       fused=self.fused, crossing=self.cross, ws=self.ws_fuse, map_half=self.half,
                       variant=self.variant)
        if events:
            events[2].record()
        gvs.forward_splat(w.inputs, self.state, self.rgba[cur], self.tgt, fused=self.fused, mu_guide=w.mu,
                          outputs=self.outs, ws=self.ws_splat)
        if events:
            events[3].record()

    def launches_per_step(self):
        # refine (vector kernel + tail), weight map + two bound-pyramid kernels, fuse,
        # splat clear + scatter/resolve per group of views
        slots = max(1, min(self.N, self.ws_splat.numel() // (self.Ht * self.Wt * 8)))
        groups = (self.N + slots - 1) // slots
        n_refine = 1 + (1 if (self.N * self.H * self.W) % 4 else 0)
        return n_refine + 3 + 1 + 1 + 2 * groups


class SoftRefine:
    """The paper's soft difference mask and blend (Sec. 3.2, Eq. 1-2 as printed: the mask at
    quarter resolution, 3x3 max-pooled, bilinearly upsampled, D' = M D + (1 - M) D'_prev)
    over the 8 input views of a frame, the state updated in place."""

    def __init__(self, w, frames_np, device):
        import torch
        from paper_2505_18932_gb300 import gvs
        self.gvs, self.w, self.half = gvs, w, False
        self.rgba = [torch.from_numpy(c.view(np.int32)).to(device) for c, _ in frames_np]
        self.depth = [torch.from_numpy(d).to(device) for _, d in frames_np]
        self.state = self.depth[0].clone()
        N, H, W = self.state.shape
        self.ws = gvs.workspace(gvs.load().gvs_refine_soft_workspace_bytes(N, W, H), device)
        self.alg_bytes = N * H * W * (4 + 4 + 4 + 4 + 4)  # both colours, the new depth, the state read and written

    def step(self, i, events=None):
        cur, prev = i % len(self.rgba), (i - 1) % len(self.rgba)
        self.gvs.refine_depth_soft(self.rgba[cur], self.rgba[prev], self.depth[cur], self.state, ws=self.ws)


class VideoStream(Pipeline):
    """A video as a stream: every frame resident in HBM, each refined against the one
    before it (the last wraps to the first) and fused and splatted into that frame's own
    target camera (the video's target moves)."""

    def step(self, i, events=None):
        self.tgt = self.w.targets_at(i % len(self.rgba))[0]
        super().step(i, events)


def algorithmic_fuse(cross_np, D, K):
    """Sample-views the method evaluates: every sample up to the crossing's second
    bracket (s + 2), all D where there is no crossing, times K views."""
    s = cross_np.astype(np.int64)
    n = np.where(s >= 0, np.minimum(s + 2, D), D)
    return int(n.sum()) * K


def alg_bytes(N, H, W, Ht, Wt):
    """Compulsory HBM bytes of one step (each input read once, each output written once)."""
    px, tpx = N * H * W, Ht * Wt
    refine = px * (4 + 4 + 4 + 4) + px * (4 + 1)
    wmap = px * 4 + px * 8
    fuse = px * 8 + tpx * (4 + 2)
    splat = px * (4 + 4) + tpx * N * (4 + 4 + 4 + 1 + 1) + tpx * 4
    return {"refine": refine, "weight_map": wmap, "fuse": fuse, "splat": splat}


def rank_frames(rank):
    """Frames streamed by one rank: disjoint across ranks (replicas, weak scaling)."""
    return [rank * RING + t for t in range(RING)]


def max_over_ranks(value, world, device):
    """Largest per-rank time: the job finishes when the slowest rank does."""
    if world <= 1:
        return value
    import torch
    import torch.distributed as dist
    t = torch.tensor([float(value)], device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def run_gvs(args, rank, local_rank, world):
    import torch
    import torch.distributed as dist
    from synth import configs

    torch.cuda.set_device(local_rank)
    device = torch.device("cuda", local_rank)
    w = configs.headline_8x1080p()
    # each rank streams its own frames (weak scaling)
    frames = rank_frames(rank)
    frames_np = render_frames(w, frames)
    pipe = Pipeline(w, frames_np, device)
    stream = torch.cuda.current_stream()

    def flush_barrier():
        if world > 1:
            dist.barrier()
        torch.cuda.synchronize()

    for i in range(max(3, args.warmup)):
        pipe.step(i)
    torch.cuda.synchronize()

    K = args.steps
    ev = [[torch.cuda.Event(enable_timing=True) for _ in range(4)] for _ in range(K)]
    clocks = ClockSampler(local_rank, enabled=(rank == 0 and not args.no_clocks))
    time.sleep(0.25 if clocks.proc else 0.0)
    flush_barrier()
    t_start = torch.cuda.Event(enable_timing=True)
    t_end = torch.cuda.Event(enable_timing=True)
    wall0 = time.perf_counter()
    t_start.record(stream)
    for i in range(K):
        pipe.step(i + 1, ev[i])
    t_end.record(stream)
    flush_barrier()
    wall = time.perf_counter() - wall0
    clk = clocks.stop()
    total_ms = t_start.elapsed_time(t_end)
    stage = {"refine": [], "fuse": [], "splat": []}
    for e in ev:
        stage["refine"].append(e[0].elapsed_time(e[1]))
        stage["fuse"].append(e[1].elapsed_time(e[2]))
        stage["splat"].append(e[2].elapsed_time(e[3]))
    total_ms = max_over_ranks(total_ms, world, device)

    # fuse-only kernel duration for the roofline: time the fusion stage alone, weight map excluded
    fuse_kernel_ms = time_fuse_kernel(pipe, K=min(K, 50))
    crosses = []
    for r in range(RING):
        pipe.step(r)
        torch.cuda.synchronize()
        crosses.append(pipe.cross.cpu().numpy())
    units = statistics.mean(algorithmic_fuse(c, w.num_samples, pipe.N) for c in crosses)
    holes = statistics.mean(float((c < 0).mean()) for c in crosses)

    e2e = run_e2e(pipe, frames_np, args.e2e_steps) if args.e2e_steps > 0 else None
    forms = {"f16_storage": form_line("f16_storage", w, time_form(Pipeline(w, frames_np, device, half=True),
                                                                  steps=min(K, 100)),
                                      "refine + weight map + fuse + splat with FP16 depth and half2 map")}
    forms["fwd_bwd"] = form_line("fwd_bwd", w, time_form(FwdBwd(w, frames_np[:2], device).capture(),
                                                         steps=min(K, 30)),
                                 "fuse + differentiable splat forward, 0.8 L1 + 0.1 L_Depth, both adjoints; "
                                 "one CUDA graph per frame")
    forms["fwd_bwd_eager"] = form_line("fwd_bwd_eager", w, time_form(FwdBwd(w, frames_np[:2], device),
                                                                     steps=min(K, 30)),
                                       "the same step launched op by op from Python (autograd)")
    forms["fwd_bwd_torch_loss"] = form_line(
        "fwd_bwd_torch_loss", w, time_form(FwdBwd(w, frames_np[:2], device, library_loss=False).capture(),
                                           steps=min(K, 30)),
        "the same step with the blend and the loss written as torch operations on the splat's outputs "
        "(one CUDA graph per frame): the per-view upstream gradients are materialised")
    w256 = type(w)(**{**w.__dict__, "num_samples": 256})
    p256 = Pipeline(w256, frames_np, device)
    f256 = form_line("headline_d256", w256, time_form(p256, steps=min(K, 100)),
                     "the benchmark's frame with D = 256 samples (spacing 3.0 cm < mu: no holes): refine, weight "
                     "map, fusion, splat of the 8 views")
    p256.step(1)
    torch.cuda.synchronize()
    f256["coverage"] = round(float((p256.cross >= 0).float().mean()), 4)
    forms["headline_d256"] = f256
    sr = SoftRefine(w, frames_np, device)
    forms["soft_mask_refine"] = form_line("soft_mask_refine", w, time_form(sr, steps=min(K, 100)),
                                          "the paper's soft difference mask and blend (Sec. 3.2, Eq. 1-2: quarter "
                                          "resolution, 3x3 max-pool, bilinear) over the 8 views; refinement only")
    forms["soft_mask_refine"]["hbm_frac"] = round(
        sr.alg_bytes / (forms["soft_mask_refine"]["ms_per_step"] * 1e-3) / 1e9 / measured_peaks()[0], 4)
    forms["temporal_online"] = form_line("temporal_online", w, time_form(TemporalOnline(w, frames_np, device),
                                                                         steps=min(K, 100)),
                                         "refine + splat + temporal weight + fusion with the previous output "
                                         "(Supplement A.2) + guided mask, fixed novel viewpoint")
    forms["gauss_render"] = form_line("gauss_render", w, time_form(GaussRender(w, frames_np, device),
                                                                   steps=min(K, 20)),
                                      "8 views rendered separately with pixel-sized Gaussians, alpha-composited "
                                      "front to back (Supplement A.3, 3DGS rules); render only")
    forms["network_frame_k4"] = form_line("network_frame_k4", w, time_form(NetworkFrame(w, frames_np, device),
                                                                           steps=min(K, 20)),
                                          "K = 4 closest views: refine, fusion, splat, network input (bf16), "
                                          "4-level U-Net with random weights (cuDNN, bf16), Eq. 4-5 blend")
    forms["sphere_trace_fusion"] = sphere_form(w, frames_np, device, steps=min(K, 20))
    forms["mixed_precision_16x1080p_stereo"] = mixed_form(device, steps=min(K, 10))
    forms.update(time_batched(device, steps=min(K, 20)))
    wd = configs.diff_640x360()
    w1 = configs.plain_320x240()
    forms["cfg1_plain_320x240"] = form_line(
        "cfg1_plain_320x240", w1, time_form(Pipeline(w1, render_frames(w1, range(RING)), device), steps=min(K, 100)),
        "4 x 320x240 inputs on a 30 degree arc, D = 64 on [0.5, 5]: refine, weight map, fusion, splat of the 4 views")
    w2 = configs.video_8x720p()
    forms["cfg2_video_8x720p"] = form_line(
        "cfg2_video_8x720p", w2, time_form(Pipeline(w2, render_frames(w2, range(RING)), device), steps=min(K, 100)),
        "one frame of the 8 x 1280x720 video (2x4 rig, sphere moving 1 cm per frame), D = 128: refine, weight map, "
        "fusion, splat of the 8 views")
    forms["cfg2_video_stream_30f"] = form_line(
        "cfg2_video_stream_30f", w2,
        time_form(VideoStream(w2, render_frames(w2, range(w2.n_frames)), device), steps=min(K, 3 * w2.n_frames)),
        f"the {w2.n_frames}-frame 8 x 1280x720 video as a stream, all frames in HBM: per frame refine against the "
        "previous frame, weight map, fusion and splat of the 8 views into that frame's (moving) target; "
        "ms_per_step is per frame")
    frd = render_frames(wd, [0, 1])
    forms["fwd_bwd_640x360"] = form_line("fwd_bwd_640x360", wd,
                                         time_form(FwdBwd(wd, frd, device).capture(), steps=min(K, 50)),
                                         "the differentiable workload: 4 x 640x360, D = 96, forward + backward; "
                                         "one CUDA graph per frame")
    forms["fwd_bwd_640x360_eager"] = form_line("fwd_bwd_640x360_eager", wd,
                                               time_form(FwdBwd(wd, frd, device), steps=min(K, 50)),
                                               "the same step launched op by op from Python (autograd)")

    if rank != 0:
        return
    tpx = pipe.Ht * pipe.Wt
    ms_per_step = total_ms / K
    value = world * tpx / (ms_per_step * 1e-3) / 1e6
    hbm_peak, peak_src, peaks = measured_peaks()
    sm_max = peaks.get("sm_max_mhz", 2070.0)
    alu_peak = device_sms() * 128 * sm_max * 1e6 / 1e12  # T lane-ops/s
    ab = alg_bytes(pipe.N, pipe.H, pipe.W, pipe.Ht, pipe.Wt)
    step_bytes = sum(ab.values())
    fuse_bytes = ab["fuse"]
    st_ms = {k: statistics.median(v) for k, v in stage.items()}
    counters = recorded_counters(pipe.variant)
    stage_time = {"refine": st_ms["refine"], "weight_map": st_ms["fuse"] - fuse_kernel_ms, "fuse": fuse_kernel_ms,
                  "splat": st_ms["splat"]}
    by_stage = {k: {"alg_bytes": ab[k], "ms": round(t, 4), "gbs": round(ab[k] / (t * 1e-3) / 1e9, 1),
                    "frac": round(ab[k] / (t * 1e-3) / 1e9 / hbm_peak, 4)} for k, t in stage_time.items()}
    line = {
        "metric": METRIC, "value": round(value, 3), "unit": "target Mpix/s", "n_gpus": world, "steps": K,
        "warmup": max(3, args.warmup), "ms_per_step": round(ms_per_step, 4), "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": {"workload": w.name, "inputs": f"{pipe.N}x{pipe.W}x{pipe.H}", "target": f"{pipe.Wt}x{pipe.Ht}",
                   "num_samples": w.num_samples, "z_range": [w.z_near, w.z_far], "mu": w.mu, "tau": w.tau,
                   "l2": f"inputs > L2: {RING}-frame ring, {round((pipe.N * pipe.H * pipe.W * 16) / 1e6)} MB read per step",
                   "parallelism": f"replicas{world}", "fuse_variant": pipe.variant,
                   "fuse_autotune_ms": {str(v): round(t, 4) for v, t in pipe.tune_ms.items()}},
        "stage_ms": {k: round(statistics.median(v), 4) for k, v in stage.items()},
        "hbm": {"alg_bytes_per_step": step_bytes, "achieved_gbs": round(step_bytes / (ms_per_step * 1e-3) / 1e9, 1),
                "peak_gbs": hbm_peak, "frac": round(step_bytes / (ms_per_step * 1e-3) / 1e9 / hbm_peak, 4),
                "peak_source": peak_src, "by_stage": by_stage,
                "note": "weight_map = fusion stage minus the fusion kernel (the map and its two bound kernels); "
                        "the map's 49-tap stencil and the fusion march are FP32-issue bound, refine and splat "
                        "move memory"},
        "roofline": fuse_roofline(units, fuse_kernel_ms, counters, alu_peak, sm_max, holes, fuse_bytes, hbm_peak,
                                  device_sms()),
        "e2e": e2e,
        "forms": forms,
        "gpu_launches": pipe.launches_per_step() * K,
        "clocks": clk,
        "wall_s": round(wall, 3),
    }
    if not args.no_cpu_baseline and world == 1:
        line["cpu_baseline"] = cpu_baseline(w, frames_np, gpu_values={
            "plain_320x240": forms["cfg1_plain_320x240"]["value"],
            "diff_640x360_fwd_bwd": forms["fwd_bwd_640x360"]["value"],
            "video_8x720p": forms["cfg2_video_8x720p"]["value"],
            "mixed_16x1080p": forms["mixed_precision_16x1080p_stereo"]["value"]})
    print(json.dumps(line), flush=True)


def fuse_roofline(units, kernel_ms, counters, alu_peak, sm_max, holes, fuse_bytes, hbm_peak, sms):
    """Roofline of the dominant kernel, the fusion march: bound by FP32 instruction issue.
    achieved = executed warp instructions x 32 lanes / the kernel's live CUDA-event time, so
    frac <= 1 by construction (one warp instruction per cycle per SM sub-partition); the
    instruction count is the committed ncu record's (null when the kernel's sources changed
    since).  The algorithmic figure of the uniform march (sample-views up to each ray's
    crossing x 20 instructions) is reported beside it: the march proves most of those
    samples crossing-free without evaluating them, so it is a speed-up, not an efficiency."""
    inst = counters.get("warp_instructions") if counters else None
    achieved = inst * 32 / (kernel_ms * 1e-3) / 1e12 if inst else None
    alg = units * OPS_PER_SAMPLE_VIEW / (kernel_ms * 1e-3) / 1e12
    return {"kernel": "fuse_kernel", "bound": "alu",
            "achieved": round(achieved, 3) if achieved else None, "peak": round(alu_peak, 2),
            "unit": "T FP32 lane-instructions/s", "frac": round(achieved / alu_peak, 4) if achieved else None,
            "traffic": counters["dram_bytes_per_launch"] if counters else None,
            "kernel_ms": round(kernel_ms, 4), "warp_instructions_per_launch": inst,
            "ncu_issue_active": counters.get("issue_active_frac") if counters else None,
            "peak_source": f"{sms} SMs x 128 FP32 lanes x {sm_max:.0f} MHz (measured max SM clock; "
                           "one warp instruction per cycle per SM sub-partition)",
            "algorithmic": {"units_per_launch": units, "ops_per_unit": OPS_PER_SAMPLE_VIEW,
                            "lane_ops_per_s_T": round(alg, 3),
                            "speedup_vs_uniform_march": round(units * OPS_PER_SAMPLE_VIEW / (inst * 32), 3)
                            if inst else None,
                            "note": "sample-views of the uniform D-sample march up to each ray's crossing (all D "
                                    "where none) x 20 FP32 instructions; the march skips provably crossing-free "
                                    "runs, so this can exceed the issue peak"},
            "hole_fraction": round(holes, 4), "hbm_alg_bytes": fuse_bytes,
            "hbm_frac": round(fuse_bytes / (kernel_ms * 1e-3) / 1e9 / hbm_peak, 4)}


class FwdBwd:
    """One training-style step on a frame: fused depth and differentiable splat forward,
    the loss 0.8 L1(blend, ground truth) + 0.1 L_Depth (Sec. 3.3, uniform blend weights),
    and both adjoints back to the input depths and colours."""

    def __init__(self, w, frames_np, device, library_loss=True):
        import torch
        from paper_2505_18932_gb300 import gvs
        self.torch, self.gvs, self.w = torch, gvs, w
        self.library_loss = library_loss
        self.tgt = w.targets[0]
        self.depth = [torch.from_numpy(d).to(device) for _, d in frames_np]
        self.color = [torch.from_numpy(np.ascontiguousarray(c).view(np.uint8).reshape(c.shape + (4,))).to(device)
                      .float().div_(255.0) for c, _ in frames_np]
        gts = []
        for t in range(len(frames_np)):
            rgb, _ = w.render_target_gt(self.tgt, t)
            gts.append((torch.from_numpy(np.ascontiguousarray(rgb[..., :3], np.float32)).to(device) / 255.0).contiguous())
        self.gt = gts
        self.cfg = dict(num_samples=w.num_samples, z_near=w.z_near, z_far=w.z_far, mu=w.mu)
        self.half = False
        self.graphs = None
        N, H, W = self.depth[0].shape
        shape_t = (self.tgt.height, self.tgt.width)
        self.cfg["variant"], _ = tune_fusion(w, self.depth[0], gvs.workspace(gvs.fuse_workspace_bytes(N, W, H), device),
                                             self.tgt, False, torch.empty(shape_t, device=device),
                                             torch.empty(shape_t, dtype=torch.int16, device=device))

    def step(self, i, events=None):
        if self.graphs is not None:
            self.graphs[i % len(self.graphs)].replay()
            return
        self._step(i % len(self.depth))

    def capture(self):
        """One CUDA graph per frame of the ring: forward, loss and both adjoints replayed as one
        launch (the same kernels; the graph removes the per-launch host cost)."""
        torch = self.torch
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            for r in range(len(self.depth)):
                self._step(r)
        torch.cuda.current_stream().wait_stream(side)
        torch.cuda.synchronize()
        graphs = []
        for r in range(len(self.depth)):
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g):
                self._step(r)
            graphs.append(g)
        torch.cuda.synchronize()
        self.graphs = graphs
        return self

    def _step(self, cur):
        torch, gvs, w = self.torch, self.gvs, self.w
        d = self.depth[cur].detach().requires_grad_(True)
        c = self.color[cur].detach().requires_grad_(True)
        fused, _ = gvs.FuseDepth.apply(d, w.inputs, self.tgt, self.cfg)
        if self.library_loss:
            # splat, blend, loss and the per-pixel upstream gradient in the library
            loss = gvs.SoftSplatBlendLoss.apply(d, c, fused, w.inputs, self.tgt, self.gt[cur], {"mu_band": w.mu})
            loss.backward()
            self.last = (d.grad, c.grad, loss.detach())
            return
        color, wdepth, alpha = gvs.SoftSplat.apply(d, c, w.inputs, self.tgt, {"mu_band": w.mu})
        asum = alpha.sum(0, dtype=torch.float32)
        valid = asum > 0
        inv = 1.0 / asum.clamp_min(1.0)
        # alpha is 0 or 1 and the splat's colour and depth are 0 wherever it is 0, so the
        # alpha-weighted sums over the views are plain sums (the same values, and the
        # gradient reaching an uncovered pixel is ignored by the splat's adjoint).
        # RGBA planes with A = 0 blend to A = 0: blend all four, drop A after the sum.
        blend = color.sum(0)[..., :3] * inv.unsqueeze(-1)
        l1 = ((blend - self.gt[cur]).abs().sum(-1) * valid).sum() / (3.0 * valid.sum().clamp_min(1))
        dblend = wdepth.sum(0) * inv
        dvalid = valid & (fused > 0)
        ldepth = ((fused - dblend).abs() * dvalid).sum() / (len(w.inputs) * dvalid.numel())
        loss = 0.8 * l1 + 0.1 * ldepth
        loss.backward()
        self.last = (d.grad, c.grad, loss.detach())


def time_form(pipe, steps):
    """ms per step of another form of the same workload (events around `steps` steps)."""
    import torch
    for i in range(3):
        pipe.step(i)
    torch.cuda.synchronize()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    a.record()
    for i in range(steps):
        pipe.step(i + 1)
    b.record()
    torch.cuda.synchronize()
    return {"ms_per_step": round(a.elapsed_time(b) / steps, 4), "steps": steps,
            "storage": "depth f16, (d, w) map half2, FP32 arithmetic" if pipe.half else "f32"}


class TemporalOnline:
    """The online video loop with the temporal term, for a fixed novel viewpoint:
    refine (binary masks) -> weight map -> splat (winners) -> temporal weight ->
    fusion with the previous output as an extra input -> guided mask."""

    def __init__(self, w, frames_np, device, library_loss=True):
        import torch
        from paper_2505_18932_gb300 import gvs
        self.torch, self.gvs, self.w = torch, gvs, w
        self.library_loss = library_loss
        self.half = False
        self.tgt = w.targets[0]
        self.rgba = [torch.from_numpy(c.view(np.int32)).to(device) for c, _ in frames_np]
        self.depth = [torch.from_numpy(d).to(device) for _, d in frames_np]
        self.state = self.depth[0].clone()
        N, H, W = self.depth[0].shape
        self.mask = torch.empty((N, H, W), dtype=torch.uint8, device=device)
        self.map = gvs.workspace(gvs.fuse_workspace_bytes(N, W, H), device)
        self.tf = gvs.TemporalFusion(w.inputs, self.tgt, w.num_samples, w.z_near, w.z_far, w.mu, device=device)

    def step(self, i, events=None):
        w, gvs = self.w, self.gvs
        cur, prev = i % len(self.rgba), (i - 1) % len(self.rgba)
        gvs.refine_depth(self.rgba[cur], self.rgba[prev], self.depth[cur], self.state, self.mask, tau=w.tau)
        self.tf.step(self.state, self.rgba[cur], self.mask, ws_map=self.map)


class GaussRender:
    """The paper's own forward render: every input view rendered into the target with
    pixel-sized Gaussians, alpha-composited (8 views, per frame of the ring)."""

    def __init__(self, w, frames_np, device):
        import torch
        from paper_2505_18932_gb300 import gvs
        self.gvs, self.w, self.half = gvs, w, False
        self.tgt = w.targets[0]
        self.rgba = [torch.from_numpy(c.view(np.int32)).to(device) for c, _ in frames_np]
        self.depth = [torch.from_numpy(d).to(device) for _, d in frames_np]
        N, H, W = self.depth[0].shape
        shape = (N, self.tgt.height, self.tgt.width)
        self.color = torch.empty(shape + (4,), dtype=torch.float32, device=device)
        self.out_depth = torch.empty(shape, dtype=torch.float32, device=device)
        self.ws = gvs.workspace(gvs.gauss_splat_workspace_bytes(W, H, self.tgt.width, self.tgt.height), device)

    def step(self, i, events=None):
        cur = i % len(self.rgba)
        self.gvs.gauss_splat(self.w.inputs, self.depth[cur], self.rgba[cur], self.tgt, color=self.color,
                             depth=self.out_depth, ws=self.ws)


class NetworkFrame:
    """The paper's whole per-frame path with K = 4 closest views: refine, fusion and splat of
    those views, the network input (bf16), the blending U-Net with seeded random weights
    (cuDNN convolutions, bf16) and the Eq. 4-5 blend with L_Depth."""

    def __init__(self, w, frames_np, device, K=4):
        import torch
        from paper_2505_18932_gb300 import gvs
        from paper_2505_18932_gb300.blendnet import BlendUNet
        self.torch, self.gvs, self.w, self.half = torch, gvs, w, False
        self.tgt = w.targets[0]
        self.sel = gvs.select_views(w.inputs, self.tgt, K)
        self.cams = [w.inputs[i] for i in self.sel]
        self.pipe = Pipeline(type(w)(**{**w.__dict__, "inputs": self.cams}), [(c[self.sel], d[self.sel])
                                                                               for c, d in frames_np], device)
        # channels-last convolutions (NHWC, 15 % faster than NCHW for this network at 1080p)
        self.net = BlendUNet(K).to(device).to(torch.bfloat16).eval().to(memory_format=torch.channels_last)
        Ht, Wt = self.tgt.height, self.tgt.width
        self.feats = torch.empty((9 * K + 1, Ht, Wt), dtype=torch.bfloat16, device=device)
        self.image = torch.empty((3, Ht, Wt), dtype=torch.float32, device=device)
        self.L = torch.empty((), dtype=torch.float64, device=device)

    def step(self, i, events=None):
        p, gvs, torch = self.pipe, self.gvs, self.torch
        p.step(i)
        gvs.blend_features(self.cams, self.tgt, p.outs["warped_rgba"], p.outs["warped_depth"], p.outs["alpha"],
                           p.fused, out=self.feats)
        with torch.no_grad():
            wk, wbg, ibg = self.net(self.feats[None].contiguous(memory_format=torch.channels_last))
        gvs.blend(p.outs["warped_rgba"], p.outs["alpha"], p.outs["warped_depth"], p.fused, wk, wbg, ibg,
                  image=self.image, l_depth=self.L)


class SphereTrace:
    """The paper's own raymarch (0.8 s steps, three bisections) over the same refined depths,
    in place of the uniform D-sample march: refine -> sphere-traced fusion (map included)."""

    def __init__(self, w, frames_np, device):
        import torch
        from paper_2505_18932_gb300 import gvs
        self.gvs, self.w, self.half = gvs, w, False
        self.pipe = Pipeline(w, frames_np, device)
        self.fused = torch.empty((w.targets[0].height, w.targets[0].width), dtype=torch.float32, device=device)
        self.evals = torch.empty_like(self.fused, dtype=torch.int32)

    def step(self, i, events=None):
        p, w = self.pipe, self.w
        cur, prev = i % len(p.rgba), (i - 1) % len(p.rgba)
        self.gvs.refine_depth(p.rgba[cur], p.rgba[prev], p.depth[cur], p.state, p.mask, tau=w.tau)
        self.gvs.fuse_depth_sphere(w.inputs, p.state, p.tgt, w.z_near, w.z_far, w.mu, fused=self.fused,
                                   evals=self.evals, ws=p.ws_fuse)


def sphere_form(w, frames_np, device, steps):
    """Time the sphere-traced fusion and compare its depth with the uniform march on one frame."""
    import torch
    st = SphereTrace(w, frames_np, device)
    f = time_form(st, steps)
    p = st.pipe
    p.step(1)
    st.step(1)
    torch.cuda.synchronize()
    a, b = st.fused, p.fused
    both = (a > 0) & (b > 0)
    agree = ((a - b).abs() <= w.mu) & both
    # the uniform march with a sample spacing below mu (D = 256: 3.0 cm against mu = 4 cm) has no holes
    fine = FineUniform(w, frames_np, device, 256)
    ff = time_form(fine, steps)
    fine.step(1)
    torch.cuda.synchronize()
    c = fine.fused
    both_f = (a > 0) & (c > 0)
    agree_f = ((a - c).abs() <= w.mu) & both_f
    return {**form_line("sphere_trace_fusion", w, f, "refine + Supplement A.1 raymarch (0.8 s steps, three "
                                                      "bisections) instead of the uniform march; no splat"),
            "evals_per_ray": round(float(st.evals.float().mean()), 2),
            "coverage": round(float((a > 0).float().mean()), 4),
            "uniform_coverage": round(float((b > 0).float().mean()), 4),
            "agree_within_mu_where_both": round(float(agree.sum() / both.sum().clamp(min=1)), 4),
            "uniform_d256": {"ms_per_step": ff["ms_per_step"], "coverage": round(float((c > 0).float().mean()), 4),
                             "agree_with_sphere_within_mu": round(float(agree_f.sum() / both_f.sum().clamp(min=1)), 4),
                             "note": "refine + uniform march with D = 256 (spacing below mu, no holes)"}}


class FineUniform:
    """refine -> uniform-march fusion with another sample count (no splat)."""

    def __init__(self, w, frames_np, device, D):
        from paper_2505_18932_gb300 import gvs
        self.gvs, self.w, self.D, self.half = gvs, w, D, False
        self.pipe = Pipeline(w, frames_np, device)
        self.fused = self.pipe.fused

    def step(self, i, events=None):
        p, w = self.pipe, self.w
        cur, prev = i % len(p.rgba), (i - 1) % len(p.rgba)
        self.gvs.refine_depth(p.rgba[cur], p.rgba[prev], p.depth[cur], p.state, p.mask, tau=w.tau)
        self.gvs.fuse_depth(w.inputs, p.state, p.tgt, self.D, w.z_near, w.z_far, w.mu, fused=p.fused,
                            crossing=p.cross, ws=p.ws_fuse)


class MixedScale:
    """Mixed precision at scale: 16 inputs at 1920x1080 (4x4 rig), depth stored as FP16 and
    the (d, w) map as half2, colour for the differentiable splat as bfloat16, D = 192,
    a stereo pair of targets.  Per step: refine, one weight map, fusion into both targets,
    the hard splat and the differentiable colour splat of all 16 views into both."""

    def __init__(self, w, frames_np, device, half=True):
        import torch
        from paper_2505_18932_gb300 import gvs
        self.torch, self.gvs, self.w, self.half = torch, gvs, w, half
        ddt = torch.float16 if half else torch.float32
        cdt = torch.bfloat16 if half else torch.float32
        self.rgba = [torch.from_numpy(c.view(np.int32)).to(device) for c, _ in frames_np]
        self.depth = [torch.from_numpy(d).to(device).to(ddt) for _, d in frames_np]
        # packed RGBA8 -> [N, H, W, 4] in [0, 1]
        self.color = [torch.from_numpy(np.ascontiguousarray(c).view(np.uint8).reshape(c.shape + (4,))).to(device)
                      .to(torch.float32).div_(255.0).to(cdt) for c, _ in frames_np]
        self.state = self.depth[0].clone()
        N, H, W = self.depth[0].shape
        self.N, self.H, self.W = N, H, W
        self.mask = torch.empty((N, H, W), dtype=torch.uint8, device=device)
        self.ws = gvs.workspace(gvs.fuse_workspace_bytes(N, W, H), device)
        self.tg = w.targets
        Ht, Wt = self.tg[0].height, self.tg[0].width
        self.fused = [torch.empty((Ht, Wt), dtype=torch.float32, device=device) for _ in self.tg]
        self.cross = [torch.empty((Ht, Wt), dtype=torch.int16, device=device) for _ in self.tg]
        self.ws_splat = gvs.workspace(2 * gvs.splat_workspace_bytes(N, Wt, Ht), device)
        self.ws_soft = gvs.workspace(gvs.soft_splat_workspace_bytes(N, Wt, Ht), device)
        self.outs = [None] * len(self.tg)
        self.soft = [None] * len(self.tg)
        self.variant, _ = tune_fusion(w, self.state, self.ws, self.tg[0], half, self.fused[0], self.cross[0])

    def step(self, i, events=None):
        w, gvs = self.w, self.gvs
        cur, prev = i % len(self.rgba), (i - 1) % len(self.rgba)
        gvs.refine_depth(self.rgba[cur], self.rgba[prev], self.depth[cur], self.state, self.mask, tau=w.tau)
        gvs.weight_map(self.state, w.mu, ws=self.ws, map_half=self.half)
        for t, tgt in enumerate(self.tg):
            gvs.fuse_depth_from_map(w.inputs, self.ws, (self.N, self.H, self.W), tgt, w.num_samples, w.z_near,
                                    w.z_far, w.mu, fused=self.fused[t], crossing=self.cross[t], map_half=self.half,
                                    variant=self.variant)
            self.outs[t] = gvs.forward_splat(w.inputs, self.state, self.rgba[cur], tgt, fused=self.fused[t],
                                             mu_guide=w.mu, outputs=self.outs[t], ws=self.ws_splat)
            self.soft[t] = gvs.soft_splat(w.inputs, self.state, self.color[cur], tgt, mu_band=w.mu,
                                          outputs=self.soft[t], ws=self.ws_soft)


def _err_stats(x):
    x = np.asarray(x, np.float64)
    if x.size == 0:
        return {"n": 0}
    return {"median": float(np.median(x)), "p99": float(np.percentile(x, 99)), "max": float(x.max()), "n": int(x.size)}


def mixed_form(device, steps, pixels=2048):
    """Time the mixed-precision form, then compare one frame of it with the FP64 oracle run on
    the original FP32 depths and uint8 colours (the total error: storage rounding included).
    Fused depth at `pixels` seeded target pixels of each target (relative error where both find
    a crossing, and the crossing-index agreement); for the first target the hard splat over the
    whole frame (winner agreement, warped-depth relative error where the winners agree) and the
    differentiable colour at `pixels` seeded target pixels of every view (absolute error of the
    worst channel where both cover the pixel)."""
    import torch
    import oracle
    from synth import configs
    w = configs.mixed_16x1080p()
    fr = render_frames(w, [0, 1])
    lo = MixedScale(w, fr, device, half=True)
    f = time_form(lo, steps)
    lo.state.copy_(lo.depth[0])
    lo.step(1)
    torch.cuda.synchronize()
    (c0, d0), (c1, d1) = fr
    rgba = lambda c: np.ascontiguousarray(c).view(np.uint8).reshape(c.shape + (4,))
    state, _ = oracle.refine_depth(rgba(c1), rgba(c0), d1, d0, w.tau)
    rng = np.random.default_rng(5)
    threads = os.cpu_count() or 1
    acc = {}
    for t, tgt in enumerate(w.targets):
        pix = np.stack([rng.integers(0, tgt.width, pixels), rng.integers(0, tgt.height, pixels)], 1).astype(np.int32)
        rf = oracle.fuse_depth(w.inputs, state, tgt, w.num_samples, w.z_near, w.z_far, w.mu, pixels=pix,
                               threads=threads)
        g = lo.fused[t].cpu().numpy()[pix[:, 1], pix[:, 0]].astype(np.float64)
        gi = lo.cross[t].cpu().numpy()[pix[:, 1], pix[:, 0]]
        both = (gi >= 0) & (rf["index"] >= 0)
        e = {"fused_depth_rel_err": _err_stats(np.abs(g[both] - rf["depth"][both]) / rf["depth"][both]),
             "crossing_index_agree": round(float((gi == rf["index"]).mean()), 6), "pixels": pixels}
        if t == 0:
            hard = oracle.forward_splat(w.inputs, state, c1, tgt, mu_guide=w.mu, fused=np.zeros((tgt.height, tgt.width)))
            gw = lo.outs[0]["winner"].cpu().numpy()
            same = (gw == hard["winner"]) & (gw >= 0)
            gd = lo.outs[0]["warped_depth"].cpu().numpy().astype(np.float64)
            hd = hard["warped_depth"].astype(np.float64)
            e["splat_winner_agree"] = round(float((gw == hard["winner"]).mean()), 6)
            e["warped_depth_rel_err"] = _err_stats(np.abs(gd[same] - hd[same]) / hd[same])
            soft = oracle.soft_splat(w.inputs, state, rgba(c1).astype(np.float64) / 255.0, tgt, mu_band=w.mu)
            gc = lo.soft[0]["color"].float().cpu().numpy()[:, pix[:, 1], pix[:, 0], :3].astype(np.float64)
            ga = lo.soft[0]["alpha"].cpu().numpy()[:, pix[:, 1], pix[:, 0]]
            oc = soft["color"][:, pix[:, 1], pix[:, 0], :3]
            oa = soft["alpha"][:, pix[:, 1], pix[:, 0]]
            cov = (ga > 0) & (oa > 0)
            e["soft_colour_abs_err"] = _err_stats(np.abs(gc - oc).max(axis=-1)[cov])
            e["soft_colour_within_1e-3"] = round(float((np.abs(gc - oc).max(axis=-1)[cov] <= 1e-3).mean()), 6)
        acc[f"target{t}"] = e
    tpx = sum(t.width * t.height for t in w.targets)
    return {**f, "value": round(tpx / (f["ms_per_step"] * 1e-3) / 1e6, 3), "unit": "target Mpix/s",
            "workload": w.name, "storage": "depth f16, map half2, colour bf16; FP32 arithmetic",
            "vs_fp64_oracle": acc,
            "note": "16 x 1920x1080 inputs, stereo pair of targets, D = 192: refine, map, fusion, hard splat and "
                    "differentiable colour splat of all views into both targets; errors against the FP64 oracle on "
                    "the original FP32 depths and uint8 colours (storage rounding included; the kernels' own "
                    "arithmetic is held to the FP32 bar in the precision tests)"}


def time_batched(device, steps):
    """The serving-style workload (8 x 1280x720 inputs, 16 targets of four sizes, 2 frames):
    the CUDA-graph BatchPlan (fusion in shared launches, autotuned variant) against the
    same work through the single-view API, launched eagerly item by item."""
    import torch
    from paper_2505_18932_gb300 import batch, gvs
    from synth import configs
    w = configs.batched_16_targets()
    fr = render_frames(w, [0, 1, 2])
    rgba = [torch.from_numpy(c.view(np.int32)).to(device) for c, _ in fr]
    dep = [torch.from_numpy(d).to(device) for _, d in fr]
    plan = batch.BatchPlan(w.inputs, w.targets, rgba[1:], dep[1:], w.num_samples, w.z_near, w.z_far, w.mu,
                           tau=w.tau, rgba_prev=rgba[0], state0=dep[0], variant=None, graph=True)
    graph_ms = _event_ms(plan.run, steps)
    # the same launch sequence without the graph: refine, maps, shared fusion launches, 32 splats
    same_ms = _event_ms(plan._run_eager, steps)

    def per_item():
        # refine and maps as the plan runs them, then one fusion call per (frame, target) item
        for f in range(plan.F):
            prev_state = plan.state0 if f == 0 else plan.states[f - 1]
            plan.states[f].copy_(prev_state)
            gvs.refine_depth(plan.rgba[f], plan.rgba_prev if f == 0 else plan.rgba[f - 1], plan.depth[f],
                             plan.states[f], plan.masks[f], tau=w.tau)
            gvs.weight_map(plan.states[f], w.mu, ws=plan.maps[f])
        for f in range(plan.F):
            for n, t in enumerate(plan.targets):
                gvs.fuse_depth_from_map(w.inputs, plan.maps[f], plan.shape, t, w.num_samples, w.z_near, w.z_far,
                                        w.mu, fused=plan.fused[f][n], crossing=plan.cross[f][n], variant=plan.variant)
                gvs.forward_splat(w.inputs, plan.states[f], plan.rgba[f], t, fused=plan.fused[f][n], mu_guide=w.mu,
                                  outputs=plan.splat[f][n], ws=plan.ws_splat)
    eager_ms = _event_ms(per_item, steps)
    px = plan.target_pixels()
    return {"batched_graph": {"ms_per_step": round(graph_ms, 4), "steps": steps, "workload": w.name,
                              "value": round(px / (graph_ms * 1e-3) / 1e6, 3), "unit": "target Mpix/s",
                              "variant": plan.variant, "autotune_ms": plan.timings,
                              "launches_per_step": plan.launches_per_run(),
                              "note": "2 frames x 16 targets (640x360 .. 1920x1080): refine + maps + shared fusion "
                                      "launches + 32 splats, replayed as one CUDA graph"},
            "batched_eager_same_launches": {"ms_per_step": round(same_ms, 4), "steps": steps, "workload": w.name,
                                            "value": round(px / (same_ms * 1e-3) / 1e6, 3), "unit": "target Mpix/s",
                                            "note": "the graph's launch sequence issued eagerly"},
            "batched_eager_per_item": {"ms_per_step": round(eager_ms, 4), "steps": steps, "workload": w.name,
                                       "value": round(px / (eager_ms * 1e-3) / 1e6, 3), "unit": "target Mpix/s",
                                       "note": "the same work through the single-view API: refine and maps per "
                                               "frame, then one fusion call and one splat call per item, no graph"}}


def _event_ms(fn, steps, warmup=3):
    import torch
    for _ in range(warmup):
        fn()
    torch.cuda.synchronize()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    a.record()
    for _ in range(steps):
        fn()
    b.record()
    torch.cuda.synchronize()
    return a.elapsed_time(b) / steps


def form_line(name, w, f, note):
    tpx = w.targets[0].width * w.targets[0].height
    return {**f, "value": round(tpx / (f["ms_per_step"] * 1e-3) / 1e6, 3), "unit": "target Mpix/s",
            "workload": w.name, "note": note}


def recorded_counters(variant, kernel_file="fuse_kernel_traffic.txt"):
    """The committed ncu record of the roofline kernel (DRAM bytes per launch, issue-active
    fraction, warp instructions), or None when the kernel's sources changed since or the
    record is of another bundle shape than the one timed."""
    import hashlib
    path = os.path.join(ROOT, "profiles", kernel_file)
    if not os.path.exists(path):
        return None
    with open(path) as f:
        rec = json.load(f)
    h = hashlib.sha256()
    for src in rec["source_files"]:
        with open(os.path.join(ROOT, src), "rb") as f:
            h.update(f.read())
    return rec if h.hexdigest() == rec["source_sha256"] and rec.get("variant", 0) == variant else None


def device_sms():
    import torch
    return torch.cuda.get_device_properties(torch.cuda.current_device()).multi_processor_count


def time_fuse_kernel(pipe, K):
    """Average duration of the fusion kernel alone (weight map already in the workspace),
    via the two-stage entry points, CUDA events on the launching stream."""
    import torch
    from paper_2505_18932_gb300 import gvs
    w = pipe.w
    durs = []
    for i in range(K + 3):
        cur = i % len(pipe.rgba)
        gvs.weight_map(pipe.depth[cur], w.mu, ws=pipe.ws_fuse)
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        gvs.fuse_depth_from_map(w.inputs, pipe.ws_fuse, (pipe.N, pipe.H, pipe.W), pipe.tgt, w.num_samples,
                                w.z_near, w.z_far, w.mu, fused=pipe.fused, crossing=pipe.cross,
                                variant=pipe.variant)
        b.record()
        if i >= 3:
            durs.append((a, b))
    torch.cuda.synchronize()
    return statistics.mean(a.elapsed_time(b) for a, b in durs)


def run_e2e(pipe, frames_np, steps):
    """Same metric through the public API with host buffers: per step the new
    frame (colour + depth) goes host->device and the fused depth plus the warped
    views come back device->host, all inside the timed region.  Copies run on
    their own streams, double-buffered, so frame i+1's upload and frame i-1's
    download overlap frame i's kernels."""
    import torch
    R = len(frames_np)
    assert R >= 4, "the input ring needs the frame being uploaded, the current and the previous one"
    host_in = [(torch.from_numpy(c.view(np.int32)).pin_memory(), torch.from_numpy(d).pin_memory())
               for c, d in frames_np]
    names = ["warped_rgba", "warped_depth", "alpha", "guided"]
    outs = [{n: torch.empty_like(pipe.outs[n]) for n in pipe.outs} for _ in range(2)]
    fused = [torch.empty_like(pipe.fused) for _ in range(2)]
    cross = [torch.empty_like(pipe.cross) for _ in range(2)]
    host_out = [{n: torch.empty(pipe.outs[n].shape, dtype=pipe.outs[n].dtype).pin_memory() for n in names}
                for _ in range(2)]
    host_fused = [torch.empty(pipe.fused.shape, dtype=torch.float32).pin_memory() for _ in range(2)]
    dev_rgba = [torch.empty_like(x) for x in pipe.rgba]
    dev_depth = [torch.empty_like(x) for x in pipe.depth]
    h2d = host_in[0][0].numel() * 4 + host_in[0][1].numel() * 4
    d2h = sum(host_out[0][n].numel() * host_out[0][n].element_size() for n in names) + host_fused[0].numel() * 4
    comp = torch.cuda.current_stream()
    up, down = torch.cuda.Stream(), torch.cuda.Stream()
    ev = lambda: torch.cuda.Event()
    ev_up, ev_comp, ev_down = {}, {}, {}
    saved = (pipe.rgba, pipe.depth, pipe.outs, pipe.fused, pipe.cross)
    pipe.rgba, pipe.depth = dev_rgba, dev_depth

    def upload(i):
        if i - R + 1 in ev_comp:  # slot i % R was last read, as the previous frame, by frame i - R + 1
            up.wait_event(ev_comp[i - R + 1])
        with torch.cuda.stream(up):
            dev_rgba[i % R].copy_(host_in[i % R][0], non_blocking=True)
            dev_depth[i % R].copy_(host_in[i % R][1], non_blocking=True)
            ev_up[i] = ev()
            ev_up[i].record(up)

    def compute(i):
        comp.wait_event(ev_up[i])
        if i - 2 in ev_down:  # output set i % 2 is free once frame i - 2 is downloaded
            comp.wait_event(ev_down[i - 2])
        pipe.outs, pipe.fused, pipe.cross = outs[i % 2], fused[i % 2], cross[i % 2]
        pipe.step(i)
        ev_comp[i] = ev()
        ev_comp[i].record(comp)

    def download(i):
        down.wait_event(ev_comp[i])
        with torch.cuda.stream(down):
            host_fused[i % 2].copy_(fused[i % 2], non_blocking=True)
            for n in names:
                host_out[i % 2][n].copy_(outs[i % 2][n], non_blocking=True)
            ev_down[i] = ev()
            ev_down[i].record(down)

    def run(first, n):
        upload(first)
        upload(first + 1)
        for i in range(first, first + n):
            compute(i)
            if i + 2 < first + n:
                upload(i + 2)
            download(i)

    for i in range(R):  # fill every device slot once
        upload(i)
    run(R, 4)
    torch.cuda.synchronize()
    ev_up.clear(); ev_comp.clear(); ev_down.clear()
    first = 2 * R
    a = torch.cuda.Event(enable_timing=True)
    b = torch.cuda.Event(enable_timing=True)
    a.record(up)
    run(first, steps)
    b.record(down)
    torch.cuda.synchronize()
    ms = a.elapsed_time(b) / steps
    # the same copies with no kernels between them, on the same two streams: the
    # host link's bound on this step
    start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    start.record(comp)
    up.wait_stream(comp)
    down.wait_stream(comp)
    for i in range(steps):
        with torch.cuda.stream(up):
            dev_rgba[i % R].copy_(host_in[i % R][0], non_blocking=True)
            dev_depth[i % R].copy_(host_in[i % R][1], non_blocking=True)
        with torch.cuda.stream(down):
            host_fused[i % 2].copy_(fused[i % 2], non_blocking=True)
            for n in names:
                host_out[i % 2][n].copy_(outs[i % 2][n], non_blocking=True)
    comp.wait_stream(up)
    comp.wait_stream(down)
    end.record(comp)
    torch.cuda.synchronize()
    copy_ms = start.elapsed_time(end) / steps
    pipe.rgba, pipe.depth, pipe.outs, pipe.fused, pipe.cross = saved
    return {"value": round(pipe.Ht * pipe.Wt / (ms * 1e-3) / 1e6, 3), "unit": "target Mpix/s",
            "h2d_bytes_per_step": int(h2d), "d2h_bytes_per_step": int(d2h), "ms_per_step": round(ms, 4),
            "overlap": "uploads, kernels and downloads on three streams, double-buffered",
            "copies_alone_ms_per_step": round(copy_ms, 4),
            "link_gbs": round((h2d + d2h) / (copy_ms * 1e-3) / 1e9, 1),
            "of_copy_bound": round(copy_ms / ms, 3)}


# ------------------------------------------------------------ CPU oracle --

ORACLE_SAMPLE_PIXELS = 8192  # target pixels per bounded oracle step (4 source rows of 1080 in every view)


def _crop_rows(cams, rows):
    return [c.__class__(**{**c.__dict__, "height": rows}) for c in cams]


def oracle_sample_step(w, frames_np, i, n_pixels, seed, threads):
    """One bounded step of the FP64 oracle on frame i of the ring: every stage on the same
    fraction f of the frame.  Fusion on n_pixels random target pixels of each target
    (f = n_pixels / (Wt Ht)); refinement and the splat on a band of round(f H) source rows of
    every view.  Returns (seconds, f, {stage: seconds}).  Fusion uses `threads` threads; the
    oracle's refinement and splat are single-threaded."""
    import oracle
    cur, prev = frames_np[i % len(frames_np)], frames_np[(i - 1) % len(frames_np)]
    H = w.inputs[0].height
    tgts = w.targets_at(0)
    Wt, Ht = tgts[0].width, tgts[0].height
    f = n_pixels / (Wt * Ht)
    band = max(1, int(round(H * f)))
    f = band / H  # the same fraction everywhere: the band fixes it
    n_pixels = max(1, int(round(f * Wt * Ht)))
    rgba_t = cur[0].view(np.uint8).reshape(cur[0].shape + (4,))[:, :band]
    rgba_p = prev[0].view(np.uint8).reshape(prev[0].shape + (4,))[:, :band]
    t0 = time.perf_counter()
    oracle.refine_depth(np.ascontiguousarray(rgba_t), np.ascontiguousarray(rgba_p),
                        np.ascontiguousarray(cur[1][:, :band]), np.ascontiguousarray(prev[1][:, :band]), w.tau)
    t1 = time.perf_counter()
    rng = np.random.default_rng(seed)
    for tgt in tgts:
        pix = np.stack([rng.integers(0, tgt.width, n_pixels), rng.integers(0, tgt.height, n_pixels)],
                       1).astype(np.int32)
        oracle.fuse_depth(w.inputs, cur[1], tgt, w.num_samples, w.z_near, w.z_far, w.mu, pixels=pix,
                          threads=threads)
    t2 = time.perf_counter()
    crop = _crop_rows(w.inputs, band)
    for tgt in tgts:
        oracle.forward_splat(crop, np.ascontiguousarray(cur[1][:, :band]), np.ascontiguousarray(cur[0][:, :band]),
                             tgt, mu_guide=w.mu, fused=np.zeros((tgt.height, tgt.width)))
    t3 = time.perf_counter()
    return t3 - t0, f, {"refine": t1 - t0, "fuse": t2 - t1, "splat": t3 - t2}


def oracle_full_plain(w, threads):
    """Full frame of a single-target workload: fusion of every target pixel and the splat of
    every source pixel (no refinement: one frame)."""
    import oracle
    rgb, d = w.render_inputs(0)
    tgt = w.targets[0]
    t0 = time.perf_counter()
    r = oracle.fuse_depth(w.inputs, d, tgt, w.num_samples, w.z_near, w.z_far, w.mu, threads=threads)
    t1 = time.perf_counter()
    oracle.forward_splat(w.inputs, d, np.ascontiguousarray(rgb).view(np.uint32)[..., 0], tgt, mu_guide=w.mu,
                         fused=r["depth"])
    t2 = time.perf_counter()
    return t2 - t0, {"fuse": t1 - t0, "splat": t2 - t1}


def oracle_full_fwd_bwd(w, threads):
    """Full frame of the differentiable workload: fusion and its adjoint, the differentiable
    colour splat and its adjoint (upstream gradients of ones)."""
    import oracle
    rgb, d = w.render_inputs(0)
    tgt = w.targets[0]
    col = rgb.astype(np.float64) / 255.0
    t0 = time.perf_counter()
    oracle.fuse_depth(w.inputs, d, tgt, w.num_samples, w.z_near, w.z_far, w.mu, threads=threads)
    t1 = time.perf_counter()
    oracle.fuse_depth_grad(w.inputs, d, tgt, w.num_samples, w.z_near, w.z_far, w.mu,
                           np.ones((tgt.height, tgt.width)))
    t2 = time.perf_counter()
    ss = oracle.soft_splat(w.inputs, d, col, tgt, mu_band=w.mu)
    oracle.soft_splat_grad(w.inputs, d, col, tgt, np.ones(ss["color"].shape), np.ones(ss["depth"].shape),
                           mu_band=w.mu)
    t3 = time.perf_counter()
    return t3 - t0, {"fuse": t1 - t0, "fuse_adjoint": t2 - t1, "soft_splat_fwd_bwd": t3 - t2}


def _mpix(px, s):
    return round(px / s / 1e6, 6)


def cpu_baseline(w, frames_np, gpu_values=None, budget_s=8.0):
    """The FP64 oracle as it stands, timed on this host's cores: the headline on bounded
    samples (every stage on the same fraction of the frame, measured, not projected), and
    whole frames of the 4 x 320x240 workload and of the 4 x 640x360 differentiable workload,
    each at 1 thread and at all cores (only the oracle's fusion is threaded)."""
    from synth import configs
    threads = os.cpu_count() or 1
    n_pixels = ORACLE_SAMPLE_PIXELS
    tpx = w.targets[0].width * w.targets[0].height
    out = {"kind": "oracle", "unit": "target Mpix/s", "cores": threads, "nproc": threads,
           "threads_by_stage": {"refine": 1, "fuse": threads, "fuse_adjoint": 1, "splat": 1, "soft_splat": 1}}
    head = {}
    for th in (threads, 1):
        spent, steps, px, stages = 0.0, 0, 0.0, {}
        i = 1
        while spent < (budget_s if th == threads else budget_s / 4) and steps < 40:
            s, f, st = oracle_sample_step(w, frames_np, i, n_pixels, seed=i, threads=th)
            spent += s
            px += f * tpx
            steps += 1
            i += 1
            for k, v in st.items():
                stages[k] = stages.get(k, 0.0) + v
        head[f"threads_{th}"] = {"value": _mpix(px, spent), "measured_s": round(spent, 3), "steps": steps,
                                 "fraction_per_step": round(f, 6),
                                 "stage_s": {k: round(v, 3) for k, v in stages.items()}}
    out["value"] = head[f"threads_{threads}"]["value"]
    out["headline"] = head
    out["sample"] = (f"{w.name}: per step every stage on the same fraction ({head[f'threads_{threads}']['fraction_per_step']:.4f}) "
                     f"of one frame: refinement and splat on a band of source rows of each view, fusion on as many "
                     f"random target pixels; value = target pixels processed / measured seconds")
    full = {}
    for name, fn, wl in (("plain_320x240", oracle_full_plain, configs.plain_320x240()),
                         ("diff_640x360_fwd_bwd", oracle_full_fwd_bwd, configs.diff_640x360())):
        px = wl.targets[0].width * wl.targets[0].height
        rec = {}
        for th in (1, threads):
            s, st = fn(wl, th)
            rec[f"threads_{th}"] = {"value": _mpix(px, s), "s": round(s, 3),
                                    "stage_s": {k: round(v, 3) for k, v in st.items()}}
        if gpu_values and name in gpu_values:
            rec["gpu_value"] = gpu_values[name]
        full[name] = rec
    out["full_frames"] = full
    # one frame of the 8 x 720p video and of the 16 x 1080p stereo workload, on bounded samples
    sampled = {}
    for name, wl in (("video_8x720p", configs.video_8x720p()), ("mixed_16x1080p", configs.mixed_16x1080p())):
        fr = render_frames(wl, [0, 1])
        px_frame = sum(t.width * t.height for t in wl.targets_at(0))
        rec = {}
        for th in (1, threads):
            s, f, st = oracle_sample_step(wl, fr, 1, 4096, seed=7, threads=th)
            rec[f"threads_{th}"] = {"value": _mpix(f * px_frame, s), "s": round(s, 3), "fraction": round(f, 5),
                                    "stage_s": {k: round(v, 3) for k, v in st.items()}}
        if gpu_values and name in gpu_values:
            rec["gpu_value"] = gpu_values[name]
        sampled[name] = rec
    out["sampled_frames"] = sampled
    return out


def run_reference(args, rank, world):
    """The FP64 oracle on this host's cores, on the benchmark's workload and metric: each step
    is one bounded sample of a frame (every stage on the same fraction; see oracle_sample_step),
    the same sample as the GPU arm's cpu_baseline (about half a second per step on 8 cores)."""
    if rank != 0:
        return
    from synth import configs
    w = configs.headline_8x1080p()
    frames_np = render_frames(w, list(range(RING)))
    threads = os.cpu_count() or 1
    # the same bounded sample per step as the cpu_baseline of the GPU arm, so that the two agree
    n_pixels = ORACLE_SAMPLE_PIXELS
    tpx = w.targets[0].width * w.targets[0].height
    for i in range(max(3, args.warmup)):
        oracle_sample_step(w, frames_np, i + 1, n_pixels, seed=i, threads=threads)
    t0 = time.perf_counter()
    px, f = 0.0, 0.0
    for i in range(args.steps):
        _, f, _ = oracle_sample_step(w, frames_np, i + 1, n_pixels, seed=100 + i, threads=threads)
        px += f * tpx
    wall = time.perf_counter() - t0
    ms = wall * 1e3 / max(args.steps, 1)
    value = px / wall / 1e6
    line = {"impl": "reference", "metric": METRIC, "value": round(value, 6), "unit": "target Mpix/s", "n_gpus": world,
            "steps": args.steps, "warmup": max(3, args.warmup), "ms_per_step": round(ms, 3),
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": w.name, "inputs": "8x1920x1080", "target": "1920x1080",
                       "num_samples": w.num_samples, "parallelism": "cpu",
                       "step": f"a bounded sample: {f:.5f} of a frame in every stage",
                       "projected_ms_per_full_frame": round(ms / max(f, 1e-12), 1)},
            "cpu_baseline": {"value": round(value, 6), "unit": "target Mpix/s", "cores": threads, "kind": "oracle",
                             "threads_by_stage": {"refine": 1, "fuse": threads, "splat": 1},
                             "sample": (f"per step every stage on the same fraction ({f:.5f}) of one frame: "
                                        "refinement and splat on a band of source rows of each view, fusion on as "
                                        "many random target pixels; value = target pixels processed / measured "
                                        "seconds")},
            "e2e": {"value": round(value, 6), "unit": "target Mpix/s", "h2d_bytes_per_step": 0,
                    "d2h_bytes_per_step": 0},
            "wall_s": round(wall, 3)}
    print(json.dumps(line), flush=True)


FORM_CLASSES = ("plain", "f16_storage", "fwd_bwd", "fwd_bwd_640x360", "gauss_render", "network_frame_k4",
                "sphere_trace_fusion", "temporal_online", "soft_mask_refine", "batched", "mixed")


def run_only_form(args):
    """One form alone: max(3, warmup) untimed steps, then `steps` steps between CUDA events.
    Builds nothing but that form (no other workload is rendered or put on the device), so a
    profiler capture of one of its kernels sees only its own launches.  `plain` is the
    benchmark's own 8 x 1080p frame (refine -> weight map -> fuse -> splat)."""
    import torch
    from synth import configs
    device = torch.device("cuda", 0)
    name = args.only_form
    if name == "batched":
        from paper_2505_18932_gb300 import batch
        w = configs.batched_16_targets()
        fr = render_frames(w, [0, 1, 2])
        rgba = [torch.from_numpy(c.view(np.int32)).to(device) for c, _ in fr]
        dep = [torch.from_numpy(d).to(device) for _, d in fr]
        plan = batch.BatchPlan(w.inputs, w.targets, rgba[1:], dep[1:], w.num_samples, w.z_near, w.z_far, w.mu,
                               tau=w.tau, rgba_prev=rgba[0], state0=dep[0], variant=None, graph=True)
        ms = _event_ms(plan.run, args.steps, warmup=max(3, args.warmup))
    elif name == "mixed":
        w = configs.mixed_16x1080p()
        form = MixedScale(w, render_frames(w, [0, 1]), device, half=True)
        frame = iter(range(1, 1 << 30))
        ms = _event_ms(lambda: form.step(next(frame)), args.steps, warmup=max(3, args.warmup))
    else:
        w = configs.diff_640x360() if name == "fwd_bwd_640x360" else configs.headline_8x1080p()
        frames_np = render_frames(w, [0, 1] if name.startswith("fwd_bwd") else rank_frames(0))
        cls = {"plain": Pipeline, "f16_storage": Pipeline, "fwd_bwd": FwdBwd, "fwd_bwd_640x360": FwdBwd,
               "gauss_render": GaussRender, "network_frame_k4": NetworkFrame, "sphere_trace_fusion": SphereTrace,
               "temporal_online": TemporalOnline, "soft_mask_refine": SoftRefine}[name]
        form = cls(w, frames_np, device, half=True) if name == "f16_storage" else cls(w, frames_np, device)
        for i in range(max(3, args.warmup)):
            form.step(i)
        torch.cuda.synchronize()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for i in range(args.steps):
            form.step(i + 1)
        b.record()
        torch.cuda.synchronize()
        ms = a.elapsed_time(b) / max(args.steps, 1)
    print(json.dumps({"form": name, "ms_per_step": round(ms, 4), "steps": args.steps, "workload": w.name}),
          flush=True)


def main():
    args = parse()
    rank, local_rank, world = dist_env()
    if args.only_form:
        run_only_form(args)
        return
    if args.impl == "reference":
        run_reference(args, rank, world)
        return
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl")
    try:
        run_gvs(args, rank, local_rank, world)
    finally:
        if world > 1:
            import torch.distributed as dist
            dist.destroy_process_group()


if __name__ == "__main__":
    main()
