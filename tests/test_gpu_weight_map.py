"""The stored (depth, weight) map pixel by pixel at every window, storage type and rounding, on
sizes whose last blocks of 32 x 64 pixels are partial."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

WINDOWS = range(1, 16, 2)
U = 2.0 ** -24


@pytest.fixture(scope="module")
def gvs():
    assert torch.cuda.is_available()
    from paper_2505_18932_gb300 import gvs as g
    g.load()
    return g


def _depths(size, half):
    """Two turned views of the arc scene with rejected, infinite and NaN pixels; as stored."""
    from synth import render
    from synth.configs import _arc_scene, arc_cameras
    w, h = size
    cams = arc_cameras(w, h, [-6.0, 5.0])
    sc = _arc_scene(0, 3)
    d = np.stack([render(sc, c, noise_seed=5, noise_sigma=0.01, view_id=k)[1] for k, c in enumerate(cams)])
    bad = np.random.default_rng(w).random(d.shape) < 0.02
    d[bad] = np.random.default_rng(h).choice([0.0, -1.0, np.inf, np.nan], bad.sum())
    return cams, d.astype(np.float16) if half else d


def _reference(weight, d, mu, window):
    """(depth or 0, weight or 0) of float32 depths d."""
    ok = np.isfinite(d) & (d > 0)
    w = np.zeros(d.shape, np.float64)
    for k, v, u in np.argwhere(ok):
        w[k, v, u] = weight(d[k], u, v, mu, window=window)
    return np.where(ok, d, 0), w


def _stored(m, d, map_half):
    e = m[: d.size * (4 if map_half else 8)].view(torch.float16 if map_half else torch.float32)
    return e.cpu().numpy().reshape(d.shape + (2,))


@pytest.mark.parametrize("window", WINDOWS)
@pytest.mark.parametrize("depth_half,map_half,size", [(False, False, (45, 73)), (True, False, (33, 65)),
                                                      (False, True, (45, 73)), (True, True, (33, 65))])
def test_stored_map(gvs, oracle_mod, window, depth_half, map_half, size):
    """nu sums window^2 squares of once rounded differences with one rounding a term; the root halves
    its relative error; the reciprocal root errs by 2 ulp, the products, 1 / window^2 and the constant
    by half an ulp each.  A half2 map rounds the weight once more."""
    _, d = _depths(size, depth_half)
    mu = float(np.float32(0.05))
    m = gvs.weight_map(torch.from_numpy(d).cuda(), mu, window=window, map_half=map_half)
    torch.cuda.synchronize()
    as_stored = d.astype(np.float16 if map_half else np.float32).astype(np.float32)
    rd, rw = _reference(oracle_mod.weight, as_stored, mu, window)
    got = _stored(m, d, map_half)
    assert np.array_equal(got[..., 0].astype(np.float32), rd.astype(np.float32))
    tol = (0.5 * (window * window + 2) + 7) * U + (2.0 ** -11 if map_half else 0.0)
    assert (rw > 0).mean() > 0.9 and rw.min() == 0.0
    err = np.abs(got[..., 1].astype(np.float64) - rw)
    assert (err <= tol * rw).all(), (err / np.maximum(rw, 1e-30)).max()


@pytest.mark.parametrize("window", WINDOWS)
@pytest.mark.parametrize("depth_half,size", [(False, (45, 73)), (True, (33, 65))])
def test_correctly_rounded_map(gvs, oracle_mod, window, depth_half, size):
    """The map of the sphere-tracing march, left in its workspace, bit for bit."""
    cams, d = _depths(size, depth_half)
    mu = float(np.float32(0.05))
    ws = gvs.workspace(gvs.fuse_workspace_bytes(2, *size))
    gvs.fuse_depth_sphere(cams, torch.from_numpy(d).cuda(), cams[0], 0.5, 5.0, mu, window=window, ws=ws)
    torch.cuda.synchronize()
    rd, rw = _reference(oracle_mod.weight_f32, d.astype(np.float32), mu, window)
    got = _stored(ws, d, False)
    assert np.array_equal(got[..., 0], rd.astype(np.float32))
    assert np.array_equal(got[..., 1].view(np.uint32), rw.astype(np.float32).view(np.uint32))
