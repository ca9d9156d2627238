"""Views seen so obliquely that a slab of samples spans 128 pixels and more: the free-space test then
falls back on the bounds of the whole view."""
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


def _oblique(K, size):
    """K views 15 to 25 degrees beside the target, with some rejected depth."""
    from synth import render
    from synth.configs import _arc_scene, arc_cameras
    cams = arc_cameras(*size, list(np.linspace(-25, -15, K)) if K > 1 else [-18.0])
    sc = _arc_scene(0, 3)
    d = np.stack([render(sc, c, noise_seed=5, noise_sigma=0.002, view_id=k)[1] for k, c in enumerate(cams)])
    d[:, 40:48, 60:90] = 0.0
    return cams, d, arc_cameras(96, 64, [2.0])[0]


@pytest.mark.parametrize("K", [1, 3, 17])
def test_whole_view_bounds(gvs, K):
    """The map's last section: smallest and largest valid depth of each view."""
    size = (300, 170)
    _, d, _ = _oblique(K, size)
    d[0] = np.where(np.arange(d[0].size).reshape(d[0].shape) % 7 == 0, np.nan, d[0])
    if K > 1:
        d[1] = 0.0  # no valid depth at all
    m = gvs.weight_map(to_dev(d), 0.05)
    torch.cuda.synchronize()
    start = gvs.fuse_workspace_bytes(K, *size) - -(-K * 16 // 256) * 256
    g = m[start: start + K * 16].view(torch.float32).cpu().numpy().reshape(K, 4)
    for k in range(K):
        ok = d[k][np.isfinite(d[k]) & (d[k] > 0)]
        if ok.size:
            assert g[k, 0] == ok.min() and g[k, 1] == ok.max(), k
        else:
            assert g[k, 0] == np.inf and g[k, 1] <= 0, k


@pytest.mark.parametrize("K,samples", [(1, 16), (1, 24), (2, 24), (6, 20), (9, 16), (17, 16)])
def test_fusion(gvs, oracle_mod, K, samples):
    cams, d, tgt = _oblique(K, (320, 240))
    dd = to_dev(d)
    for mu in (0.05, 0.2):
        ref = oracle_mod.fuse_depth(cams, d, tgt, samples, 0.5, 5.0, mu)
        assert (ref["index"] >= 0).mean() > 0.1
        for variant in (0, 1, 3, 6):
            fused, cross = gvs.fuse_depth(cams, dd, tgt, samples, 0.5, 5.0, mu, variant=variant)
            torch.cuda.synchronize()
            compare_fused(fused, cross, ref)


@pytest.mark.parametrize("K", [1, 2, 4, 8, 17])
def test_sphere_march(gvs, oracle_mod, K):
    cams, d, tgt = _oblique(K, (320, 240))
    for mu, frac in ((0.2, 1.0), (0.2, 0.0625), (0.3, 0.25)):
        ref = oracle_mod.fuse_depth_sphere(cams, d, tgt, 0.5, 5.0, mu, min_frac=frac)
        assert (ref["depth"] > 0).mean() > 0.2
        fused, evals = gvs.fuse_depth_sphere(cams, to_dev(d), tgt, 0.5, 5.0, mu, min_frac=frac)
        torch.cuda.synchronize()
        assert np.array_equal(evals.cpu().numpy(), ref["evals"])
        assert np.array_equal(fused.cpu().numpy().view(np.uint32), ref["depth"].view(np.uint32))
