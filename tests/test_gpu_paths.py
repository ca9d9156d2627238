"""Kernel paths at the sizes where they change form or could go wrong: the sphere march's
free-space test on turned views, the Gaussian render's list lengths, the fusion adjoint at
image borders, and the splat over many groups of views on odd sizes."""
import numpy as np
import pytest
import torch

from gpu_util import to_dev, u32
from test_gpu_gauss import _case as gauss_case
from test_gpu_grad import _case as grad_case
from test_gpu_slab import _rig
from test_gpu_slab import test_slab_on_turned_views as turned_views

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gvs():
    assert torch.cuda.is_available()
    from paper_2505_18932_gb300 import gvs as g
    g.load()
    return g


@pytest.mark.parametrize("n,size,mu,steps", [(3, (61, 47), 0.05, 1024), (4, (61, 47), 0.2, 1024), (8, (40, 33), 0.05, 61),
                                             (9, (40, 33), 0.05, 1024), (16, (33, 31), 0.1, 1024), (17, (24, 19), 0.05, 1024)])
def test_sphere_on_turned_views(gvs, oracle_mod, n, size, mu, steps):
    """Views rolled, pitched, yawed, looking away or in front of the target, bit for bit."""
    from synth import render
    from synth.configs import _arc_scene, arc_cameras
    w, h = size
    cams = _rig(n, w, h, n)
    sc = _arc_scene(0, 3)
    d = np.stack([render(sc, c, noise_seed=5, noise_sigma=0.002, view_id=k)[1] for k, c in enumerate(cams)])
    tgt = arc_cameras(w + 6, h - 3, [2.5])[0]
    ref = oracle_mod.fuse_depth_sphere(cams, d, tgt, 0.5, 5.0, mu, max_steps=steps)
    fused, evals = gvs.fuse_depth_sphere(cams, to_dev(d), tgt, 0.5, 5.0, mu, max_steps=steps)
    torch.cuda.synchronize()
    assert np.array_equal(evals.cpu().numpy(), ref["evals"])
    assert np.array_equal(fused.cpu().numpy().view(np.uint32), ref["depth"].view(np.uint32))


@pytest.mark.parametrize("target", [(96, 72), (61, 47), (24, 18), (16, 16)])
def test_gauss_list_lengths(gvs, oracle_mod, target):
    """Lists up to 512 keys, up to 2048 and above (96x72 Gaussians a view in smaller targets)."""
    from synth import configs
    w = configs.tiny(96, 72, 2, 16)
    t = configs.tiny(*target, 2, 16).targets[0]
    gauss_case(gvs, oracle_mod, w, target=t)


@pytest.mark.parametrize("size,window", [((12, 9), 15), ((40, 30), 15), ((12, 9), 9), ((32, 32), 7), ((33, 34), 7), ((65, 31), 5), ((38, 70), 9)])
def test_grad_at_borders(gvs, oracle_mod, size, window):
    from synth import configs
    w = configs.tiny(*size, 3, 96)
    _, d = w.render_inputs(0)
    grad_case(gvs, oracle_mod, w, d, seed=window, window=window)


@pytest.mark.parametrize("target", [(45, 33), (48, 33)])
@pytest.mark.parametrize("slots", [1, 5])
def test_splat_groups_of_views(gvs, target, slots):
    """32 views in groups of 1 (all 32 tags) and 5 equal one group of 32."""
    from synth import configs
    w = configs.tiny(40, 31, 32, 16)
    t = configs.tiny(*target, 2, 16).targets[0]
    rgb, d = w.render_inputs(0)
    dd, rr = to_dev(d), to_dev(u32(rgb))
    n = target[0] * target[1]
    pad = gvs.splat_workspace_bytes(1, *target) - n * 8
    outs = [gvs.forward_splat(w.inputs, dd, rr, t, ws=gvs.workspace(s * n * 8 + pad)) for s in (slots, 32)]
    torch.cuda.synchronize()
    for k in outs[0]:
        assert torch.equal(outs[0][k], outs[1][k]), k
    col = torch.from_numpy(np.ascontiguousarray(rgb, np.float32) / 255.0).cuda()
    one = gvs.soft_splat_workspace_bytes(1, *target)
    soft = [gvs.soft_splat(w.inputs, dd, col, t, ws=gvs.workspace(s * (one + 256))) for s in (slots, 32)]
    torch.cuda.synchronize()
    for k in ("winner", "depth", "alpha"):
        assert torch.equal(soft[0][k], soft[1][k]), k
    # sums of at most a few tens of FP32 terms in another order
    torch.testing.assert_close(soft[0]["wsum"], soft[1]["wsum"], rtol=1e-5, atol=1e-7)
    torch.testing.assert_close(soft[0]["color"], soft[1]["color"], rtol=1e-5, atol=1e-5)


@pytest.mark.parametrize("K", [2, 3, 5, 6, 7, 8, 12])
def test_batch_of_more_items_than_a_launch(gvs, K):
    """17 items of mixed sizes (two launches) and both bundle shapes equal single calls, bit for bit."""
    from synth import configs
    w = configs.tiny(61, 47, K, 40)
    _, d = w.render_inputs(0)
    dd = to_dev(d)
    ws = gvs.weight_map(dd, w.mu)
    sizes = [(61, 47), (24, 18), (97, 33), (8, 70), (1, 1)]
    targets = [configs.tiny(*sizes[i % len(sizes)], 2, 16).targets[0] for i in range(17)]
    new = lambda t, dt: torch.empty((t.height, t.width), dtype=dt, device="cuda")  # noqa: E731
    items = [(ws, t, new(t, torch.float32), new(t, torch.int16)) for t in targets]
    batch = gvs.FuseBatch(w.inputs, items, w.num_samples, w.z_near, w.z_far, w.mu)
    batch.launch()
    torch.cuda.synchronize()
    for _, t, fused, cross in items:
        for variant in (0, 1, 3):
            f, c = gvs.fuse_depth(w.inputs, dd, t, w.num_samples, w.z_near, w.z_far, w.mu, variant=variant)
            assert torch.equal(f, fused) and torch.equal(c, cross)
    batch.close()


@pytest.mark.parametrize("n,size,samples", [(2, (61, 47), 96), (6, (61, 47), 64), (7, (40, 33), 33)])
def test_fuse_of_exact_view_counts(gvs, oracle_mod, n, size, samples):
    """Counts of views with a kernel of their own, on turned views, against the oracle."""
    turned_views(gvs, oracle_mod, n, size, samples, (0, 1, 3))
