"""Splats in several groups of views, against the oracle, on target sizes that reach every form of the
resolves: pixels strided (odd), by fours, by eights and by bulk copies."""
import numpy as np
import pytest
import torch

from gpu_util import to_dev, u32

pytestmark = pytest.mark.gpu

SIZES = [(45, 33), (44, 33), (40, 33), (48, 33)]  # Wt Ht divisible by 1, 4, 8 and 16 only
SLOTS = [1, 3, 7]


@pytest.fixture(scope="module")
def gvs():
    assert torch.cuda.is_available()
    from paper_2505_18932_gb300 import gvs as g
    g.load()
    return g


def _workload(target):
    from synth import configs
    w = configs.tiny(40, 31, 7, 16)
    return w, configs.tiny(*target, 2, 16).targets[0]


@pytest.mark.parametrize("target", SIZES)
@pytest.mark.parametrize("slots", SLOTS)
def test_hard_splat(gvs, oracle_mod, target, slots):
    w, t = _workload(target)
    rgb, d = w.render_inputs(0)
    fused = np.full((t.height, t.width), np.float32(np.median(d)), np.float32)
    ws = gvs.workspace(slots * target[0] * target[1] * 8 + 255)
    out = gvs.forward_splat(w.inputs, to_dev(d), to_dev(u32(rgb)), t, fused=to_dev(fused), mu_guide=0.25, ws=ws)
    torch.cuda.synchronize()
    out = {k: v.cpu().numpy() for k, v in out.items()}
    ref = oracle_mod.forward_splat(w.inputs, d, u32(rgb), t)
    assert np.array_equal(out["winner"], ref["winner"]) and (ref["winner"] < 0).any()
    assert np.array_equal(out["warped_rgba"].view(np.uint32), ref["warped_rgba"])
    assert np.array_equal(out["warped_depth"].view(np.uint32), ref["warped_depth"].view(np.uint32))
    has = ref["winner"] >= 0
    assert np.array_equal(out["alpha"] != 0, has)
    guided = has & (np.abs(ref["warped_depth"] - fused) <= np.float32(0.25))
    assert np.array_equal(out["guided"] != 0, guided) and guided.any() and (has & ~guided).any()


@pytest.mark.parametrize("target", SIZES)
@pytest.mark.parametrize("slots", SLOTS)
def test_differentiable_splat(gvs, oracle_mod, target, slots):
    """Tolerances of the one-group comparison: colour 1e-3, weight sums 1e-5 relative, the rest exact."""
    w, t = _workload(target)
    rgb, d = w.render_inputs(0)
    col = np.ascontiguousarray(rgb, np.float32) / 255.0
    n = target[0] * target[1]
    ws = gvs.workspace(-(-slots * n * 8 // 256) * 256 + slots * n * 16)
    out = gvs.soft_splat(w.inputs, to_dev(d), to_dev(col), t, mu_band=w.mu, ws=ws)
    torch.cuda.synchronize()
    out = {k: v.cpu().numpy() for k, v in out.items()}
    ref = oracle_mod.soft_splat(w.inputs, d, col, t, mu_band=w.mu)
    assert np.array_equal(out["winner"], ref["winner"]) and (ref["winner"] < 0).any()
    assert np.array_equal(out["alpha"], ref["alpha"])
    assert np.array_equal(out["depth"].view(np.uint32), ref["depth"].view(np.uint32))
    assert np.abs(out["color"] - ref["color"]).max() <= 1e-3
    np.testing.assert_allclose(out["wsum"], ref["wsum"], rtol=1e-5, atol=1e-7)


@pytest.mark.parametrize("scale", [1.0, 1.55, 1.7])
@pytest.mark.parametrize("reject", [False, True])
@pytest.mark.parametrize("size", [(161, 157), (227, 222)])
def test_scatter_of_many_pixels(gvs, oracle_mod, scale, reject, size):
    """32 views in one launch (807,000 and 1,612,608 pixels: several per thread) and in a launch per view (one
    per thread), to both sides of the magnification where that changes: as the oracle, bit for bit."""
    from synth import configs
    w = configs.tiny(*size, 32, 16)
    t = configs.tiny(90, 64, 2, 16).targets[0]
    t.fx = t.fy = w.inputs[0].fx * scale
    rgb, d = w.render_inputs(0)
    fused = np.full((64, 90), np.float32(np.median(d)), np.float32)
    for dt in (torch.float32, torch.float16):
        depth = to_dev(d).to(dt)
        ref = oracle_mod.forward_splat(w.inputs, depth.float().cpu().numpy(), u32(rgb), t, mu_guide=0.25,
                                       fused=fused.astype(np.float64), guide_reject=reject)
        for slots in (32, 1):
            out = gvs.forward_splat(w.inputs, depth, to_dev(u32(rgb)), t, fused=to_dev(fused), mu_guide=0.25,
                                    guide_reject=reject, ws=gvs.workspace(slots * 90 * 64 * 8))
            torch.cuda.synchronize()
            assert np.array_equal(out["winner"].cpu().numpy(), ref["winner"])
            assert np.array_equal(out["warped_depth"].cpu().numpy().view(np.uint32), ref["warped_depth"].view(np.uint32))
        assert (ref["winner"] >= 0).any()
