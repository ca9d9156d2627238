"""The march's slab tests on rigs where the ray coefficients vary over a bundle: views rolled,
pitched and yawed up to 80 degrees, views whose camera plane cuts the target's rays, views that
look away, one-pixel-wide bundles and very few samples, against the FP64 oracle's full march
(the crossing index exactly; see gpu_util for the depth rule)."""
import numpy as np
import pytest
import torch

from gpu_util import compare_fused, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gvs():
    assert torch.cuda.is_available()
    from paper_2505_18932_gb300 import gvs as g
    g.load()
    return g


def _rot(roll, pitch, yaw):
    r, p, y = np.radians([roll, pitch, yaw])
    rz = np.array([[np.cos(r), -np.sin(r), 0], [np.sin(r), np.cos(r), 0], [0, 0, 1]])
    rx = np.array([[1, 0, 0], [0, np.cos(p), -np.sin(p)], [0, np.sin(p), np.cos(p)]])
    ry = np.array([[np.cos(y), 0, np.sin(y)], [0, 1, 0], [-np.sin(y), 0, np.cos(y)]])
    return rz @ rx @ ry


def _rig(n, w, h, seed):
    """Views around the arc scene: the first two upright, the others turned further and further;
    the fourth stands in front of the target camera and the sixth looks away from the scene."""
    from synth import camera_at
    from synth.configs import arc_cameras
    rng = np.random.default_rng(seed)
    cams = arc_cameras(w, h, np.linspace(-10, 10, n).tolist())
    out = cams[:2]
    for k in range(2, n):
        turn = 80.0 * (k - 1) / n
        R = _rot(rng.uniform(-1, 1) * turn, rng.uniform(-0.3, 0.3) * turn, rng.uniform(-0.3, 0.3) * turn) @ cams[k].R
        c = np.array(cams[k].centre)
        if k == 3:
            c = c * 0.4          # between the target camera and the surface
        if k == 5:
            R = _rot(0, 0, 170.0) @ cams[k].R
        out.append(camera_at(w, h, c, R))
    return out


@pytest.mark.parametrize("n,size,samples,variants", [
    (3, (61, 47), 64, (0,)), (4, (61, 47), 2, (0,)), (5, (64, 48), 9, (0, 2, 6)), (8, (61, 47), 96, (0, 1, 3, 4, 6)),
    (16, (40, 33), 33, (0, 3, 6)), (17, (40, 33), 64, (0, 6))])
def test_slab_on_turned_views(gvs, oracle_mod, n, size, samples, variants):
    from synth import render
    from synth.configs import _arc_scene, arc_cameras
    w, h = size
    cams = _rig(n, w, h, n)
    sc = _arc_scene(0, 3)
    d = np.stack([render(sc, c, noise_seed=5, noise_sigma=0.002, view_id=k)[1] for k, c in enumerate(cams)])
    tgt = arc_cameras(w + 6, h - 3, [2.5])[0]
    ref = oracle_mod.fuse_depth(cams, d, tgt, samples, 0.5, 5.0, 0.05)
    dd = to_dev(d)
    for v in variants:
        fused, cross = gvs.fuse_depth(cams, dd, tgt, samples, 0.5, 5.0, 0.05, variant=v)
        torch.cuda.synchronize()
        compare_fused(fused, cross, ref)
