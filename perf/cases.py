"""Performance cases of the geometry core: what a program that uses this library has it do.

Every case goes through the public binding (`paper_2505_18932_gb300.gvs` and `.batch`) on seeded
synthetic RGB-D frames made on the GPU: planes and a sphere seen by a rig of calibrated cameras,
smooth 8-bit textures with sensor noise, depth noise of 2 mm and blocks of rejected (0) depth, as
an estimator with a consistency check leaves them.  A frame and the one before it differ by the
sphere's motion (1 cm) and by the noise.

`kind` names the path:
  frame     the online frame: binary refinement, TSDF fusion into the target, splat of all views
  train     a training step: fusion, differentiable splat and Sec. 3.3's loss, both adjoints
  warp      the differentiable splat alone, forward and backward, upstream gradients per view
  temporal  the online frame with the paper's soft mask and the temporal TSDF term
  gauss     the alpha-composited render of pixel-sized Gaussians
  sphere    the paper's sphere-tracing raymarch
  network   the blending network's input planes and the blend of its outputs
  batch     many targets and two frames as one captured plan
"""
import math
from dataclasses import dataclass

import numpy as np
import torch

from paper_2505_18932_gb300 import gvs
from paper_2505_18932_gb300.batch import BatchPlan

TAU, NOISE = 0.03, 0.002
WEIGHT_CONST, WINDOW = 0.001, 7


def _case(name, kind, views, width, height, t_width=None, t_height=None, samples=128, rig="grid", depth="f32",
          color="f32", targets=""):
    c = {"kind": kind, "views": views, "width": width, "height": height, "t_width": t_width or width,
         "t_height": t_height or height, "samples": samples, "rig": rig, "depth": depth, "color": color,
         "targets": targets}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest online frame: four cameras on an arc, where latency and launches count
        _case("frame_4x320x240", "frame", 4, 320, 240, samples=64, rig="arc"),
        # an online frame whose width, height and view count divide by nothing
        _case("frame_5x961x541", "frame", 5, 961, 541, 859, 487, samples=96),
        # the headline frame: eight 1080p cameras into a 1080p view
        _case("frame_8x1080p", "frame", 8, 1920, 1080),
        # the largest frame, stored in half precision: a 4 x 4 rig of 1080p cameras
        _case("frame_f16_16x1080p", "frame", 16, 1920, 1080, samples=192, depth="f16"),
        # a training step at the size of small training crops
        _case("train_4x640x360", "train", 4, 640, 360, samples=96, rig="arc"),
        # a training step on whole 1080p frames
        _case("train_8x1080p", "train", 8, 1920, 1080),
        # differentiable warping of half depth and bfloat16 colour inside a larger model, odd sizes
        _case("warp_bf16_6x1279x719", "warp", 6, 1279, 719, 1151, 863, depth="f16", color="bf16"),
        # the online loop with temporal consistency at 720p
        _case("temporal_8x720p", "temporal", 8, 1280, 720),
        # the paper's own forward render of the four closest views
        _case("gauss_4x720p", "gauss", 4, 1280, 720),
        # the paper's own raymarch, four views
        _case("sphere_4x960x540", "sphere", 4, 960, 540),
        # the planes around the blending network at the paper's evaluation size, bfloat16
        _case("network_4x1352x1014", "network", 4, 1352, 1014, color="bf16"),
        # serving: two frames of eight 720p cameras into four viewers' targets
        _case("batch_2x4_8x720p", "batch", 8, 1280, 720, targets="640x360,960x540,1280x720,1920x1080"),
    ]


def draw(rng):
    def size(lo, hi):
        w = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        return w, max(16, int(round(w * rng.choice([9 / 16, 3 / 4, rng.uniform(0.5, 0.8)]))) if w <= 1440 else w * 9 // 16)

    kind = rng.choice(["frame", "frame", "train", "train", "warp", "temporal", "gauss", "sphere", "network", "batch"])
    lo, hi, vmin, vmax = {"frame": (200, 1920, 2, 8), "train": (200, 1920, 2, 8), "warp": (200, 1280, 2, 8),
                          "temporal": (320, 1280, 2, 8), "gauss": (160, 1280, 2, 4), "sphere": (160, 960, 2, 6),
                          "network": (240, 1352, 2, 4), "batch": (320, 1280, 2, 8)}[kind]
    w, h = size(lo, hi)
    tw, th = (w, h) if kind == "network" or rng.random() < 0.5 else size(lo, hi)
    views = rng.randint(vmin, vmax)
    depth = rng.choice(["f32", "f32", "f16"]) if kind in ("frame", "warp", "gauss") else "f32"
    if kind == "frame" and depth == "f16":
        views = rng.randint(vmin, 16)
    color = rng.choice(["f32", "bf16"]) if kind in ("warp", "network") else "f32"
    targets = ""
    if kind == "batch":
        targets = ",".join("%dx%d" % size(320, 1440) for _ in range(rng.randint(2, 4)))
    return _case(None, kind, views, w, h, tw, th, samples=rng.choice([64, 96, 128, 192]),
                 rig=rng.choice(["grid", "arc"]), depth=depth, color=color, targets=targets)


# -- inputs ------------------------------------------------------------------------------------------
@dataclass
class Camera:
    """x_cam = R x_world + t; pixel centres at integer coordinates, y down, z forward."""
    width: int
    height: int
    fx: float
    fy: float
    cx: float
    cy: float
    R: np.ndarray
    t: np.ndarray


def _camera(w, h, centre, R=None):
    f = (w / 2.0) / math.tan(math.radians(30.0))
    R = np.eye(3) if R is None else R
    return Camera(w, h, f, f, (w - 1) / 2.0, (h - 1) / 2.0, R, -R @ np.asarray(centre, np.float64))


def _arc_camera(w, h, degrees, radius=2.0):
    a = math.radians(degrees)
    c = np.array([radius * math.sin(a), 0.0, -radius * math.cos(a)])
    z = -c / np.linalg.norm(c)
    x = np.cross([0.0, -1.0, 0.0], z)
    x /= np.linalg.norm(x)
    return _camera(w, h, c, np.stack([x, np.cross(z, x), z]))


def _setup(case, seed):
    """Cameras, target(s), scene and method parameters; the target's place follows the seed."""
    rng = np.random.default_rng(seed)
    n, w, h = case["views"], case["width"], case["height"]
    sizes = [tuple(int(v) for v in s.split("x")) for s in case["targets"].split(",")] if case["targets"] else \
        [(case["t_width"], case["t_height"])]
    if case["rig"] == "arc":
        cams = [_arc_camera(w, h, d) for d in np.linspace(-15, 15, n)]
        targets = [_arc_camera(*s, rng.uniform(-4, 4)) for s in sizes]
        planes = [(0, 0, 1, 1.5), (0, 1, 0, 0.8), (1, 0, 0, -1.2)]
        ball = (0.1 + rng.uniform(-0.1, 0.1), rng.uniform(-0.1, 0.1), 0.2, 0.35)
        z_near, z_far, mu = 0.5, 5.0, 0.05
    else:
        cols = min(4, max(2, (n + 1) // 2))
        rows = -(-n // cols)
        cams = [_camera(w, h, ((i % cols - (cols - 1) / 2) * 0.1, (i // cols - (rows - 1) / 2) * 0.1, 0.0))
                for i in range(n)]
        targets = [_camera(*s, (rng.uniform(-0.1, 0.1), rng.uniform(-0.04, 0.04), 0.0)) for s in sizes]
        planes = [(0, 0, 1, 6.0), (0, 1, 0, 1.2), (1, 0, 0, -2.0)]
        ball = (-0.15 + rng.uniform(-0.3, 0.3), rng.uniform(-0.2, 0.2), 2.0, 0.3)
        z_near, z_far, mu = 0.3, 8.0, 0.04
    waves = rng.normal(size=(4, 4)) * [6.0, 6.0, 6.0, 0.0] + [0, 0, 0, 1.0] * rng.uniform(0, 6.28, (4, 1))
    cfg = dict(num_samples=case["samples"], z_near=z_near, z_far=z_far, mu=mu)
    return cams, targets, (planes, ball, waves), cfg


def _trace(scene, cam, shift=0.0):
    """(z-depth [H, W], colour [H, W, 3] in [0, 1]) of the nearest plane or the sphere moved by `shift`."""
    planes, (bx, by, bz, br), waves = scene
    dev = "cuda"
    y, x = torch.meshgrid(torch.arange(cam.height, device=dev, dtype=torch.float32),
                          torch.arange(cam.width, device=dev, dtype=torch.float32), indexing="ij")
    r = torch.stack([(x - cam.cx) / cam.fx, (y - cam.cy) / cam.fy, torch.ones_like(x)], -1)
    o = torch.tensor(-cam.R.T @ cam.t, device=dev, dtype=torch.float32)
    r = r @ torch.tensor(cam.R, device=dev, dtype=torch.float32)
    best, tint = torch.full_like(x, 50.0), torch.zeros_like(x)
    for n, (a, b, c, e) in enumerate(planes):
        nv = torch.tensor([a, b, c], device=dev, dtype=torch.float32)
        s = (e - o @ nv) / (r @ nv)
        hit = (s > 0.01) & (s < best)
        best, tint = torch.where(hit, s, best), torch.where(hit, torch.full_like(x, n * 0.9), tint)
    oc = o - torch.tensor([bx + shift, by, bz], device=dev, dtype=torch.float32)
    a, b, c = (r * r).sum(-1), (r * oc).sum(-1), (oc * oc).sum() - br * br
    disc = b * b - a * c
    s = (-b - disc.clamp(min=0).sqrt()) / a
    hit = (disc > 0) & (s > 0.01) & (s < best)
    best, tint = torch.where(hit, s, best), torch.where(hit, torch.full_like(x, 4.0), tint)
    p = o + best[..., None] * r
    wv = torch.tensor(waves, device=dev, dtype=torch.float32)
    f = torch.sin(p @ wv[:, :3].T + wv[:, 3] + tint[..., None])
    col = 0.5 + 0.22 * f[..., :3] + 0.18 * f[..., 3:]
    return best, col.clamp(0.02, 0.98)


def _gen(seed, salt):
    return torch.Generator("cuda").manual_seed((int(seed) * 1000003 + salt) % (1 << 62))


def _noise(shape, gen):
    return torch.randn(shape, generator=gen, device="cuda")


def _frame(scene, cams, seed, salt, shift, dtype):
    """One frame of every view: packed RGBA8 int32 [N, H, W], depth [N, H, W], float colour [N, H, W, 4]."""
    rgba, depths, colors = [], [], []
    for k, cam in enumerate(cams):
        g = _gen(seed, 100 * salt + k)
        z, col = _trace(scene, cam, shift)
        z = z + NOISE * _noise(z.shape, g)
        h, w = z.shape
        holes = torch.rand((h + 15) // 16, (w + 15) // 16, generator=g, device="cuda") < 0.005
        holes = holes.repeat_interleave(16, 0).repeat_interleave(16, 1)[:h, :w]
        depths.append(torch.where(holes, torch.zeros_like(z), z).to(dtype))
        col = (col + (1.0 / 255.0) * _noise(col.shape, g)).clamp(0, 1)
        b = (col * 255 + 0.5).to(torch.int32)
        rgba.append(b[..., 0] | (b[..., 1] << 8) | (b[..., 2] << 16) | (-1 << 24))
        colors.append(torch.cat([col, torch.ones_like(col[..., :1])], -1))
    return torch.stack(rgba), torch.stack(depths), torch.stack(colors)


def _inputs(case, seed):
    cams, targets, scene, cfg = _setup(case, seed)
    dt = torch.float16 if case["depth"] == "f16" else torch.float32
    cdt = torch.bfloat16 if case["color"] == "bf16" else torch.float32
    kind, t = case["kind"], targets[0]
    rgba, depth, col = _frame(scene, cams, seed, 1, 0.0, dt)
    x = dict(cams=cams, targets=targets, target=t, cfg=cfg, rgba=rgba, depth=depth)
    if kind in ("frame", "temporal", "batch"):
        x["rgba_prev"], x["state"], _ = _frame(scene, cams, seed, 2, -0.01, dt)
    if kind == "batch":
        x["rgba2"], x["depth2"], _ = _frame(scene, cams, seed, 3, 0.01, dt)
    g = _gen(seed, 7)
    N, ht, wt = len(cams), t.height, t.width
    if kind in ("train", "warp"):
        x["color"] = col.to(cdt)
    if kind == "train":
        gt = _trace(scene, t)[1]
        x["gt"] = (gt + (1.0 / 255.0) * _noise(gt.shape, g)).contiguous()
    if kind == "warp":
        x["g_color"] = _noise((N, ht, wt, 4), g) * 1e-3
        x["g_depth"] = _noise((N, ht, wt), g) * 1e-4
    if kind == "temporal":  # the loop in full swing: the last fused depth and its weights
        z = _trace(scene, t, -0.01)[0]
        x["prev"] = {"prev": z + 0.5 * NOISE * _noise(z.shape, g),
                     "w_tmp_prev": 10.0 * torch.rand((ht, wt), generator=g, device="cuda"),
                     "w_view_prev": N * torch.rand((ht, wt), generator=g, device="cuda")}
    if kind == "network":
        z, gt = _trace(scene, t)
        x["fused"] = z + 0.5 * NOISE * _noise(z.shape, g)
        x["warped_depth"] = (z + NOISE * _noise((N, ht, wt), g)).contiguous()
        x["alpha"] = (torch.rand((N, ht, wt), generator=g, device="cuda") < 0.93).to(torch.uint8)
        b = ((gt + (2.0 / 255.0) * _noise((N, ht, wt, 3), g)).clamp(0, 1) * 255 + 0.5).to(torch.int32)
        x["warped_rgba"] = (b[..., 0] | (b[..., 1] << 8) | (b[..., 2] << 16) | (-1 << 24)) * x["alpha"]
        x["warped_depth"] *= x["alpha"]
        for n, sh in (("w", (N, ht, wt)), ("w_bg", (ht, wt)), ("i_bg", (3, ht, wt))):
            x[n] = torch.sigmoid(_noise(sh, g)).to(cdt)
    return x


def prepare(case, seed):
    x = _inputs(case, seed)
    kind, cams, t = case["kind"], x["cams"], x["target"]
    N, H, W = x["depth"].shape
    x["kind"], x["f16"] = kind, case["depth"] == "f16"
    # what an online program allocates once and keeps: the map, two z-buffers and its outputs
    if kind in ("frame", "temporal", "sphere"):
        x["ws_map"] = gvs.workspace(gvs.fuse_workspace_bytes(N, W, H))
    if kind == "frame":
        sh = (N, t.height, t.width)
        x["mask"] = torch.empty((N, H, W), dtype=torch.uint8, device="cuda")
        x["fused"] = torch.empty(sh[1:], dtype=torch.float32, device="cuda")
        x["crossing"] = torch.empty(sh[1:], dtype=torch.int16, device="cuda")
        x["ws_splat"] = gvs.workspace(2 * gvs.splat_workspace_bytes(N, t.width, t.height))
        x["out"] = {n: torch.empty(sh, dtype=d, device="cuda") for n, d in
                    (("winner", torch.int32), ("warped_rgba", torch.int32), ("warped_depth", torch.float32),
                     ("alpha", torch.uint8), ("guided", torch.uint8))}
    if kind == "temporal":
        x["mask"] = torch.empty((N, H, W), dtype=torch.float32, device="cuda")
        x["loop"] = gvs.TemporalFusion(cams, t, **x["cfg"])
        x["loop"].load_state_dict(x["prev"])
    if kind == "gauss":
        x["ws"] = gvs.workspace(gvs.gauss_splat_workspace_bytes(W, H, t.width, t.height))
    if kind in ("train", "warp"):
        x["depth"].requires_grad_()
        x["color"].requires_grad_()
    if kind == "batch":
        x["plan"] = BatchPlan(cams, x["targets"], [x["rgba"], x["rgba2"]], [x["depth"], x["depth2"]],
                              **x["cfg"], tau=TAU, rgba_prev=x["rgba_prev"], state0=x["state"], variant=0)
    return x


# -- the passes --------------------------------------------------------------------------------------
def run(s):
    return _RUN[s["kind"]](s, **s["cfg"])


def _run_frame(s, mu, **cfg):
    gvs.refine_depth(s["rgba"], s["rgba_prev"], s["depth"], s["state"], s["mask"], tau=TAU)
    gvs.fuse_depth(s["cams"], s["state"], s["target"], mu=mu, fused=s["fused"], crossing=s["crossing"],
                   ws=s["ws_map"], map_half=s["f16"], **cfg)
    out = gvs.forward_splat(s["cams"], s["state"], s["rgba"], s["target"], fused=s["fused"], mu_guide=mu,
                            outputs=s["out"], ws=s["ws_splat"])
    return dict(out, state=s["state"], mask=s["mask"], fused=s["fused"], crossing=s["crossing"])


def _run_train(s, mu, **cfg):
    fused, _ = gvs.FuseDepth.apply(s["depth"], s["cams"], s["target"], dict(cfg, mu=mu))
    loss = gvs.SoftSplatBlendLoss.apply(s["depth"], s["color"], fused, s["cams"], s["target"], s["gt"],
                                        {"mu_band": mu})
    gd, gc = torch.autograd.grad(loss, (s["depth"], s["color"]))
    return {"loss": loss, "fused": fused, "grad_depth": gd, "grad_color": gc}


def _run_warp(s, mu, **cfg):
    color, depth, alpha = gvs.SoftSplat.apply(s["depth"], s["color"], s["cams"], s["target"], {"mu_band": mu})
    gd, gc = torch.autograd.grad((color, depth), (s["depth"], s["color"]), (s["g_color"], s["g_depth"]))
    return {"color": color, "depth": depth, "alpha": alpha, "grad_depth": gd, "grad_color": gc}


def _run_temporal(s, **cfg):
    gvs.refine_depth_soft(s["rgba"], s["rgba_prev"], s["depth"], s["state"], s["mask"])
    fused, crossing, sp, w_tmp = s["loop"].step(s["state"], s["rgba"], s["mask"], ws_map=s["ws_map"])
    return dict(sp, state=s["state"], mask=s["mask"], fused=fused, crossing=crossing, w_tmp=w_tmp,
                w_view=s["loop"].w_view_prev)


def _run_gauss(s, **cfg):
    color, depth = gvs.gauss_splat(s["cams"], s["depth"], s["rgba"], s["target"], ws=s["ws"])
    return {"color": color, "depth": depth}


def _run_sphere(s, z_near, z_far, mu, **cfg):
    fused, evals = gvs.fuse_depth_sphere(s["cams"], s["depth"], s["target"], z_near, z_far, mu, ws=s["ws_map"])
    return {"fused": fused, "evals": evals}


def _run_network(s, **cfg):
    features = gvs.blend_features(s["cams"], s["target"], s["warped_rgba"], s["warped_depth"], s["alpha"],
                                  s["fused"], dtype=s["w"].dtype)
    image, l_depth = gvs.blend(s["warped_rgba"], s["alpha"], s["warped_depth"], s["fused"], s["w"], s["w_bg"],
                               s["i_bg"])
    return {"features": features, "image": image, "l_depth": l_depth}


def _run_batch(s, **cfg):
    p = s["plan"]
    p.run()
    return {"states": p.states, "fused": p.fused, "crossing": p.cross, "splat": p.splat}


_RUN = {"frame": _run_frame, "train": _run_train, "warp": _run_warp, "temporal": _run_temporal, "gauss": _run_gauss,
        "sphere": _run_sphere, "network": _run_network, "batch": _run_batch}


def work(case):
    """Each input read once and each output written once; the operations of the confidence window
    (4 per neighbour), of two samples per ray and view (20 each) and of a source pixel's projection (30)."""
    kind, n = case["kind"], case["views"]
    p = n * case["width"] * case["height"]
    sizes = [s.split("x") for s in case["targets"].split(",")] if case["targets"] else \
        [(case["t_width"], case["t_height"])]
    t = sum(int(a) * int(b) for a, b in sizes)
    db = 2 if case["depth"] == "f16" else 4
    cb = 2 if case["color"] == "bf16" else 4
    fuse, win = 40 * n * t, 4 * WINDOW * WINDOW * p
    if kind == "frame":
        return {"bytes": p * (9 + 3 * db) + 6 * t + 14 * n * t, "flops": win + fuse + 30 * p}
    if kind == "train":
        return {"bytes": p * (4 + 16) * 2 + 16 * t + 4, "flops": 3 * win + 3 * fuse + 120 * p}
    if kind == "warp":
        return {"bytes": p * (db + 4 * cb) * 2 + n * t * (16 + 4 + 1 + 16 + 4), "flops": 120 * p}
    if kind == "temporal":
        return {"bytes": p * (12 + 3 * db) + t * (12 + 18) + 14 * n * t, "flops": win + fuse + 60 * p}
    if kind == "gauss":
        return {"bytes": p * (db + 4) + 20 * n * t, "flops": 60 * p + 20 * 25 * p}
    if kind == "sphere":
        return {"bytes": p * db + 8 * t, "flops": win + 5 * fuse}
    if kind == "network":
        return {"bytes": t * ((9 * n + 1) * cb + 9 * n + 4 + (n + 4) * cb + 12) + 8, "flops": t * 40 * n}
    return {"bytes": 2 * (p * 20 + 6 * t + 14 * n * t) + p * 4, "flops": 2 * (win + fuse + 30 * p)}


# -- the same in 64 bits -----------------------------------------------------------------------------
_F = torch.float64


def _xform(to, frm):
    """depth * (M [i j 1]) + b: homogeneous pixel coordinates in `to` of a pixel of `frm`."""
    k_to = np.array([[to.fx, 0, to.cx], [0, to.fy, to.cy], [0, 0, 1.0]])
    k_from = np.array([[frm.fx, 0, frm.cx], [0, frm.fy, frm.cy], [0, 0, 1.0]])
    q = to.R @ frm.R.T
    return k_to @ q @ np.linalg.inv(k_from), k_to @ (to.t - q @ frm.t)


def _grid(h, w):
    y, x = torch.meshgrid(torch.arange(h, device="cuda", dtype=_F), torch.arange(w, device="cuda", dtype=_F),
                          indexing="ij")
    return x, y


def _rays(to, frm):
    M, b = _xform(to, frm)
    x, y = _grid(frm.height, frm.width)
    return [M[r, 0] * x + M[r, 1] * y + M[r, 2] for r in range(3)], b


def _f32(v):
    return float(np.float32(v))


def _variation(d, mu):
    """nu of one view, summed over the window; differentiable in d (an invalid neighbour counts mu^2)."""
    h, w = d.shape
    r, m2 = WINDOW // 2, mu * mu
    ok = d > 0
    yi = torch.arange(h, device="cuda")
    xi = torch.arange(w, device="cuda")
    nu = torch.zeros_like(d)
    for dy in range(-r, r + 1):
        for dx in range(-r, r + 1):
            rows, cols = (yi + dy).clamp(0, h - 1), (xi + dx).clamp(0, w - 1)
            n = d[rows][:, cols]
            e = (d - n).square().clamp(max=m2)
            nu = nu + torch.where(ok[rows][:, cols], e, torch.full_like(e, m2))
    return nu


def _omega_of(nu, d):
    n = nu / (WINDOW * WINDOW)
    w = torch.where(n > 0, WEIGHT_CONST * n.clamp(min=1e-300).rsqrt(), torch.ones_like(n)).clamp(max=1.0)
    return torch.where(d > 0, w, torch.zeros_like(w))


def _omega(depth, mu):
    return torch.stack([_omega_of(_variation(d, mu), d) for d in depth])


class _Views:
    """The fused signed distance of a set of views at given depths along the target's rays."""

    def __init__(self, cams, target, depth, omega, mu):
        self.depth, self.omega, self.mu = depth.flatten(1), omega.flatten(1), mu
        self.rays = [_rays(c, target) for c in cams]
        self.rays = [([a.flatten() for a in r], b) for r, b in self.rays]
        self.w, self.h = cams[0].width, cams[0].height

    def at(self, z, sel=None):
        S, W = 0.0, 0.0
        for k, (a, b) in enumerate(self.rays):
            a = a if sel is None else [v[sel] for v in a]
            hx, hy, hz = (z * a[r] + b[r] for r in range(3))
            ok = hz > 1e-6
            hs = torch.where(ok, hz, torch.ones_like(hz))
            u, v = torch.round(hx.detach() / hs.detach()), torch.round(hy.detach() / hs.detach())
            ok = ok & (u >= 0) & (u < self.w) & (v >= 0) & (v < self.h)
            i = torch.where(ok, v * self.w + u, torch.zeros_like(u)).long()
            sdf = (self.depth[k][i] - hz) / self.mu
            om = torch.where(ok & (sdf >= -1), self.omega[k][i], torch.zeros_like(sdf))
            S, W = S + om * sdf.clamp(-1, 1), W + om
        return S, W


def _march(views, samples, z_near, z_far, mu, prev=None, w_tmp=None):
    """(fused, first sample of the crossing or -1, the views' weight at the crossing), flat."""
    zn, zf = _f32(z_near), _f32(z_far)
    dz = (zf - zn) / (samples - 1)
    n = views.rays[0][0][0].numel()
    out = [torch.zeros(n, dtype=_F, device="cuda") for _ in range(2)]
    index = torch.full((n,), -1, dtype=torch.long, device="cuda")
    last = None
    for s in range(samples):
        z = torch.full((n,), zn + s * dz, dtype=_F, device="cuda")
        S, Wv = views.at(z)
        W = Wv
        if prev is not None:
            sdf = (prev - z) / mu
            om = torch.where((prev > 0) & (sdf >= -1), w_tmp, torch.zeros_like(sdf))
            S, W = S + om * sdf.clamp(-1, 1), W + om
        if last is not None:
            S0, W0, V0 = last
            hit = (index < 0) & (W0 > 0) & (W > 0) & (S0 > 0) & (S <= 0)
            f = torch.where(hit, S0 / torch.where(hit, S0 - S, torch.ones_like(S)), torch.zeros_like(S))
            out[0] = torch.where(hit, zn + (s - 1) * dz + dz * f, out[0])
            out[1] = torch.where(hit, V0 + f * (Wv - V0), out[1])
            index = torch.where(hit, torch.full_like(index, s - 1), index)
        last = (S, W, Wv)
    return out[0], index, out[1]


def _exact_fuse(x, depth, target, omega=None, **more):
    c = x["cfg"]
    mu = _f32(c["mu"])
    views = _Views(x["cams"], target, depth, _omega(depth, mu) if omega is None else omega, mu)
    return [v.view(target.height, target.width) for v in
            _march(views, c["num_samples"], c["z_near"], c["z_far"], mu, **more)]


def _footprint(cam, target, d):
    """Splat geometry of one view, flat over its source pixels: x, y, z, half-width, valid."""
    m, c = _rays(target, cam)
    hx, hy, hz = (d * m[r] + c[r] for r in range(3))
    ok = ((d > 0) & (hz > 1e-6)).flatten()
    hz = torch.where(hz > 1e-6, hz, torch.ones_like(hz))
    hw = (0.5 * (target.fx / cam.fx) * (d / hz)).clamp(0.5, 2.0)
    return (hx / hz).flatten(), (hy / hz).flatten(), hz.flatten(), hw.flatten(), ok


def _pairs(cam, target, d):
    """(source, target) index pairs of one view's footprints."""
    x, y, z, hw, ok = _footprint(cam, target, d)
    lx, ly, hx, hy = torch.ceil(x - hw), torch.ceil(y - hw), torch.floor(x + hw), torch.floor(y + hw)
    q, p = [], []
    for dy in range(5):
        for dx in range(5):
            i, j = lx + dx, ly + dy
            s = (ok & (i <= hx) & (j <= hy) & (i >= 0) & (j >= 0) & (i < target.width) & (j < target.height)).nonzero()[:, 0]
            q.append(s)
            p.append((j[s] * target.width + i[s]).long())
    return torch.cat(q), torch.cat(p), z


def _exact_splat_depth(x, depth, target):
    out = []
    for cam, d in zip(x["cams"], depth):
        q, p, z = _pairs(cam, target, d)
        zb = torch.full((target.width * target.height,), math.inf, dtype=_F, device="cuda")
        zb.scatter_reduce_(0, p, z[q], "amin")
        out.append(torch.where(torch.isinf(zb), torch.zeros_like(zb), zb).view(target.height, target.width))
    return torch.stack(out)


def _refined(x):
    def bytes_of(v):
        return torch.stack([(v >> (8 * c)) & 255 for c in range(3)], -1)

    m = (bytes_of(x["rgba"]) - bytes_of(x["rgba_prev"])).abs().amax(-1) > int(255 * TAU)
    return torch.where(m, x["depth"], x["state"])


def _exact_frame(x):
    st = _refined(x).to(_F)
    return {"state": st, "fused": _exact_fuse(x, st, x["target"])[0], "warped_depth": _exact_splat_depth(x, st, x["target"])}


def _soft_colors(x, k, d, c, target):
    """Differentiable splat of view k in 64 bits: colour [P, 4], depth [P], covered [P]."""
    cam, mu = x["cams"][k], _f32(x["cfg"]["mu"])
    P = target.width * target.height
    xs, ys, zs, hw, _ = _footprint(cam, target, d)
    q, p, z = _pairs(cam, target, d.detach())
    zb = torch.full((P,), math.inf, dtype=_F, device="cuda").scatter_reduce_(0, p, z[q], "amin")
    keep = z[q] <= zb[p] + mu
    q, p = q[keep], p[keep]
    i, j = (p % target.width).to(_F), (p // target.width).to(_F)
    sg = hw[q] / 2
    g = torch.exp(-((xs[q] - i).square() + (ys[q] - j).square()) / (2 * sg.square()))
    wsum = torch.zeros(P, dtype=_F, device="cuda").index_add(0, p, g)
    col = torch.zeros(P, 3, dtype=_F, device="cuda").index_add(0, p, g[:, None] * c.reshape(-1, 4)[q, :3])
    cov = torch.isfinite(zb)
    col = col / torch.where(cov, wsum, torch.ones_like(wsum))[:, None]
    win = z[q] == zb[p]
    src = torch.full((P,), z.numel(), dtype=torch.long, device="cuda").scatter_reduce_(0, p[win], q[win], "amin")
    src = torch.where(cov, src, torch.zeros_like(src))  # equal depths: the lower source index
    dep = torch.where(cov, zs[src], torch.zeros_like(wsum))
    return torch.cat([col, torch.zeros_like(col[:, :1])], 1), dep, cov


def _exact_warp(x):
    t = x["target"]
    out = {"color": [], "depth": [], "grad_depth": [], "grad_color": []}
    for k in range(len(x["cams"])):
        d = x["depth"][k].to(_F).requires_grad_()
        c = x["color"][k].to(_F).requires_grad_()
        col, dep, _ = _soft_colors(x, k, d, c, t)
        gd, gc = torch.autograd.grad((col, dep), (d, c), (x["g_color"][k].reshape(-1, 4).to(_F), x["g_depth"][k].flatten().to(_F)))
        for n, v in (("color", col.detach().view(t.height, t.width, 4)), ("depth", dep.detach().view(t.height, t.width)),
                     ("grad_depth", gd), ("grad_color", gc)):
            out[n].append(v)
    return {n: torch.stack(v) for n, v in out.items()}


def _exact_train(x):
    t, mu = x["target"], _f32(x["cfg"]["mu"])
    P, K = t.width * t.height, len(x["cams"])
    depth, color, gt = x["depth"].to(_F), x["color"].to(_F), x["gt"].to(_F).reshape(-1, 3)
    omega = _omega(depth, mu)
    fused, index, _ = _exact_fuse(x, depth, t, omega)
    with torch.no_grad():
        soft = [_soft_colors(x, k, depth[k], color[k], t) for k in range(K)]
    I = [s[0][:, :3].clone().requires_grad_() for s in soft]
    D = [s[1].clone().requires_grad_() for s in soft]
    F = fused.flatten().clone().requires_grad_()
    a = [s[2].to(_F) for s in soft]
    A = sum(a)
    on, An = A > 0, A.clamp(min=1.0)
    B = sum(ak[:, None] * Ik for ak, Ik in zip(a, I)) / An[:, None]
    l1 = ((B - gt).abs() * on[:, None]).sum() / (3 * on.sum())
    Db = sum(ak * Dk for ak, Dk in zip(a, D)) / An
    ld = ((F - Db).abs() * (on & (F.detach() > 0))).sum() / (K * P)
    loss = _f32(0.8) * l1 + _f32(0.1) * ld
    grads = torch.autograd.grad(loss, I + D + [F])
    gI, gD, gF = grads[:K], grads[K:2 * K], grads[-1]
    # the fusion's adjoint: through the two samples around each crossing, then through the weights
    c = x["cfg"]
    zn, dz = _f32(c["z_near"]), (_f32(c["z_far"]) - _f32(c["z_near"])) / (c["num_samples"] - 1)
    sel = (index.flatten() >= 0).nonzero()[:, 0]
    s0 = index.flatten()[sel].to(_F)
    d, om = depth.clone().requires_grad_(), omega.clone().requires_grad_()
    views = _Views(x["cams"], t, d, om, mu)
    S0, S1 = (views.at(zn + (s0 + n) * dz, sel)[0] for n in (0, 1))
    g_depth, g_omega = torch.autograd.grad((dz * S0 / (S0 - S1)), (d, om), gF[sel])
    g_depth, g_color = [v for v in g_depth], []
    for k in range(K):
        d = depth[k].clone().requires_grad_()
        g_depth[k] = g_depth[k] + torch.autograd.grad(_omega_of(_variation(d, mu), d.detach()), d, g_omega[k])[0]
        d, cl = depth[k].clone().requires_grad_(), color[k].clone().requires_grad_()
        col, dep, _ = _soft_colors(x, k, d, cl, t)
        gd, gc = torch.autograd.grad((col[:, :3], dep), (d, cl), (gI[k], gD[k]))
        g_depth[k] = g_depth[k] + gd
        g_color.append(gc)
    return {"loss": loss.detach(), "fused": fused, "grad_depth": torch.stack(g_depth), "grad_color": torch.stack(g_color)}


def _soft_refined(x, beta=0.6, lam=0.7):
    """(state, mask) of the soft refinement: quarter-resolution means, 3 x 3 max-pool, bilinear."""
    beta, lam = _f32(beta), _f32(lam)

    def bytes_of(v):
        return torch.stack([(v >> (8 * c)) & 255 for c in range(3)], -1)

    diff = (bytes_of(x["rgba"]) - bytes_of(x["rgba_prev"])).abs().amax(-1).to(_F) / 255.0
    N, H, W = diff.shape
    qh, qw = -(-H // 4), -(-W // 4)
    pad = torch.nn.functional.pad(diff, (0, 4 * qw - W, 0, 4 * qh - H))
    one = torch.nn.functional.pad(torch.ones_like(diff), (0, 4 * qw - W, 0, 4 * qh - H))
    cell = lambda v: v.view(N, qh, 4, qw, 4).sum((2, 4))  # noqa: E731
    m = (cell(pad) / cell(one) / lam + beta).clamp(max=1.0)
    m = torch.nn.functional.max_pool2d(m[:, None], 3, 1, 1)[:, 0]
    xs, ys = ((torch.arange(n, device="cuda", dtype=_F) + 0.5) / 4 - 0.5 for n in (W, H))
    xs, ys = xs.clamp(0, qw - 1), ys.clamp(0, qh - 1)
    x0, y0 = xs.floor().long(), ys.floor().long()
    x1, y1 = (x0 + 1).clamp(max=qw - 1), (y0 + 1).clamp(max=qh - 1)
    fx, fy = xs - x0, (ys - y0)[:, None]
    top = m[:, y0][:, :, x0] * (1 - fx) + m[:, y0][:, :, x1] * fx
    bot = m[:, y1][:, :, x0] * (1 - fx) + m[:, y1][:, :, x1] * fx
    m = top * (1 - fy) + bot * fy
    new, old = x["depth"].to(_F), x["state"].to(_F)
    st = m * new + (1 - m) * old
    st = torch.where(old > 0, st, new)
    return torch.where(new > 0, st, old), m


def _exact_temporal(x):
    t = x["target"]
    st, mask = _soft_refined(x)
    P = t.width * t.height
    M = torch.full((P,), -1.0, dtype=_F, device="cuda")
    warped = []
    for k, cam in enumerate(x["cams"]):
        q, p, z = _pairs(cam, t, st[k])
        zb = torch.full((P,), math.inf, dtype=_F, device="cuda").scatter_reduce_(0, p, z[q], "amin")
        win = z[q] == zb[p]
        M.scatter_reduce_(0, p[win], mask[k].flatten()[q[win]], "amax")
        warped.append(torch.where(torch.isinf(zb), torch.zeros_like(zb), zb).view(t.height, t.width))
    M = torch.where(M < 0, torch.ones_like(M), M)
    prev = {n: v.to(_F).flatten() for n, v in x["prev"].items()}
    w_tmp = ((prev["w_tmp_prev"] + prev["w_view_prev"]) * (1 - M).clamp(min=0)).clamp(max=15.0)
    fused, _, w_view = _exact_fuse(x, st, t, prev=prev["prev"], w_tmp=w_tmp)
    return {"state": st, "mask": mask, "w_tmp": w_tmp.view(t.height, t.width), "warped_depth": torch.stack(warped),
            "fused": fused, "w_view": w_view}


def _exact_gauss(x, scale=0.5, cap=8):
    t = x["target"]
    P = t.width * t.height
    colors, depths = [], []
    for k, cam in enumerate(x["cams"]):
        d = x["depth"][k].to(_F)
        X, Y, Z, _, ok = _footprint(cam, t, d)
        s2 = (scale * (t.fx / cam.fx) * d.flatten() / Z).square()
        a, b, q = (X - t.cx) / t.fx, (Y - t.cy) / t.fy, t.fy / t.fx
        sxx, sxy, syy = s2 * (1 + a * a) + 0.3, s2 * q * a * b, s2 * q * q * (1 + b * b) + 0.3
        det, mid = sxx * syy - sxy * sxy, 0.5 * (sxx + syy)
        r = torch.ceil(3 * (mid + (mid * mid - det).clamp(min=0.1).sqrt()).sqrt()).clamp(max=cap)
        i0, j0 = torch.ceil(X - r), torch.ceil(Y - r)
        rank = torch.empty_like(Z, dtype=torch.long)
        rank[torch.sort(Z, stable=True)[1]] = torch.arange(Z.numel(), device="cuda")
        src, pix, al = [], [], []
        n = 2 * int(r[ok].max().item()) + 1 if bool(ok.any()) else 0
        for dj in range(n):
            for di in range(n):
                i, j = i0 + di, j0 + dj
                dx, dy = X - i, Y - j
                alpha = torch.exp(-0.5 * (syy * dx * dx - 2 * sxy * dx * dy + sxx * dy * dy) / det).clamp(max=0.99)
                s = (ok & (i <= X + r) & (j <= Y + r) & (i >= 0) & (j >= 0) & (i < t.width) & (j < t.height) &
                     (alpha >= 1 / 255)).nonzero()[:, 0]
                src.append(s)
                pix.append((j[s] * t.width + i[s]).long())
                al.append(alpha[s])
        src, pix, al = torch.cat(src), torch.cat(pix), torch.cat(al)
        order = torch.sort(pix * Z.numel() + rank[src])[1]
        src, pix, al = src[order], pix[order], al[order]
        lt = torch.log1p(-al)
        run = torch.cumsum(lt, 0)
        first = torch.ones_like(pix, dtype=torch.bool)
        first[1:] = pix[1:] != pix[:-1]
        base = (run - lt)[first][torch.cumsum(first.long(), 0) - 1]
        after = torch.exp(run - base)
        use = after >= 1e-4
        src, pix, wgt = src[use], pix[use], (al * torch.exp(run - lt - base))[use]
        v = x["rgba"][k].flatten()[src]
        c = torch.stack([((v >> (8 * n)) & 255).to(_F) / 255 for n in range(3)] + [torch.ones_like(wgt), Z[src]], 1)
        acc = torch.zeros(P, 5, dtype=_F, device="cuda").index_add_(0, pix, c * wgt[:, None])
        colors.append(acc[:, :4].reshape(t.height, t.width, 4))
        depths.append(torch.where(acc[:, 3] > 0, acc[:, 4] / acc[:, 3].clamp(min=1e-300), acc[:, 3]).view(t.height, t.width))
    return {"color": torch.stack(colors), "depth": torch.stack(depths)}


def _exact_sphere(x, max_steps=1024, min_frac=0.0625):
    c, t = x["cfg"], x["target"]
    mu, zf = _f32(c["mu"]), _f32(c["z_far"])
    depth = x["depth"].to(_F)
    views = _Views(x["cams"], t, depth, _omega(depth, mu), mu)
    P = t.width * t.height
    out = torch.zeros(P, dtype=_F, device="cuda")
    sel = torch.arange(P, device="cuda")
    z = torch.full((P,), _f32(c["z_near"]), dtype=_F, device="cuda")
    pz, ps, pw = z, torch.zeros_like(z), torch.zeros_like(z)
    for _ in range(max_steps):
        live = z <= zf
        sel, z, pz, ps, pw = (v[live] for v in (sel, z, pz, ps, pw))
        if not sel.numel():
            break
        S, W = views.at(z, sel)
        hit = (pw > 0) & (W > 0) & (ps > 0) & (S <= 0)
        if bool(hit.any()):
            lo, hi, hs = pz[hit], z[hit], sel[hit]
            for _ in range(3):
                m = 0.5 * (lo + hi)
                Sm, Wm = views.at(m, hs)
                front = (Wm > 0) & (Sm > 0)
                lo, hi = torch.where(front, m, lo), torch.where(front, hi, m)
            out[hs] = 0.5 * (lo + hi)
            sel, z, S, W = (v[~hit] for v in (sel, z, S, W))
        frac = torch.where(W > 0, (S / W.clamp(min=1e-300)).clamp(min=min_frac), torch.ones_like(S))
        pz, ps, pw = z, S, W
        z = z + 0.8 * mu * frac
    return {"fused": out.view(t.height, t.width)}


def _exact_network(x):
    t, K = x["target"], len(x["cams"])
    h, w = t.height, t.width
    rgb = torch.stack([((x["warped_rgba"] >> (8 * c)) & 255).to(_F) / 255 for c in range(3)], 1)
    D, dk, al = x["fused"].to(_F), x["warped_depth"].to(_F), x["alpha"].to(_F)
    u, v = _grid(h, w)
    ray = torch.stack([(u - t.cx) / t.fx, (v - t.cy) / t.fy, torch.ones_like(u)], 0)
    p = ray * D
    normal = torch.zeros_like(p)
    cross = torch.cross(p[:, 1:-1, 2:] - p[:, 1:-1, :-2], p[:, 2:, 1:-1] - p[:, :-2, 1:-1], dim=0)
    good = (D[1:-1, 1:-1] > 0) & (D[1:-1, 2:] > 0) & (D[1:-1, :-2] > 0) & (D[2:, 1:-1] > 0) & (D[:-2, 1:-1] > 0)
    size = cross.square().sum(0).sqrt()
    facing = torch.where((cross * p[:, 1:-1, 1:-1]).sum(0) > 0, -1.0, 1.0)
    normal[:, 1:-1, 1:-1] = torch.where(good & (size > 0), facing * cross / size.clamp(min=1e-300), torch.zeros_like(cross))
    rt = ray / ray.square().sum(0).sqrt()
    nd, rd, dist, axis = [], [], [], []
    for cam in x["cams"]:
        centre = t.R @ (-cam.R.T @ cam.t) + t.t
        dv = p - torch.tensor(centre, device="cuda", dtype=_F)[:, None, None]
        dv = dv / dv.square().sum(0).sqrt()
        zero = torch.zeros_like(D)
        nd.append(torch.where(D > 0, (normal * dv).sum(0), zero))
        rd.append(torch.where(D > 0, (rt * dv).sum(0), zero))
        dist.append(torch.full_like(D, float(np.linalg.norm(centre))))
        axis.append(torch.full_like(D, float(cam.R[2] @ t.R[2])))
    features = torch.cat([rgb.reshape(3 * K, h, w), dk, al, D[None], torch.stack(nd + rd + dist + axis)], 0)
    wk, bg, ib = x["w"].to(_F) * al, x["w_bg"].to(_F), x["i_bg"].to(_F)
    W = wk.sum(0)
    den = torch.where(W > 0, W, torch.ones_like(W))
    fg = torch.where(W > 0, (rgb * wk[:, None]).sum(0) / den, torch.zeros_like(ib))
    db = torch.where(W > 0, (dk * wk).sum(0) / den, torch.zeros_like(W))
    return {"features": features, "image": (1 - bg) * fg + bg * ib, "l_depth": (D - db).abs().sum() / (h * w * K)}


def _exact_batch(x):
    s1 = _refined(x)
    s2 = _refined(dict(rgba=x["rgba2"], rgba_prev=x["rgba"], depth=x["depth2"], state=s1))
    out = {"states": [s1.to(_F), s2.to(_F)], "fused": [], "splat": []}
    for st in out["states"]:
        om = _omega(st, _f32(x["cfg"]["mu"]))
        out["fused"].append([_exact_fuse(x, st, t, om)[0] for t in x["targets"]])
        out["splat"].append([{"warped_depth": _exact_splat_depth(x, st, t)} for t in x["targets"]])
    return out


_EXACT = {"frame": _exact_frame, "train": _exact_train, "warp": _exact_warp, "temporal": _exact_temporal,
          "gauss": _exact_gauss, "sphere": _exact_sphere, "network": _exact_network, "batch": _exact_batch}


def exact(case, seed):
    return _EXACT[case["kind"]](_inputs(case, seed))
