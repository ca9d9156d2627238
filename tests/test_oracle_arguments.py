"""The oracle takes arrays of any floating type and layout: what it converts lives through the call."""
import numpy as np


def test_blend_converts_its_arguments(oracle_mod):
    rng = np.random.default_rng(0)
    K, H, W = 3, 41, 67
    rgba = rng.integers(0, 1 << 32, (K, H, W), dtype=np.uint32)
    alpha = (rng.random((K, H, W)) < 0.7).astype(np.uint8)
    depth, fused = rng.random((K, H, W)).astype(np.float32), rng.random((H, W)).astype(np.float32)
    w, w_bg, i_bg = (rng.random(s).astype(np.float32) for s in ((K, H, W), (H, W), (3, H, W)))
    ref, L = oracle_mod.blend(rgba, alpha, depth, fused, w.astype(np.float64), w_bg.astype(np.float64),
                              i_bg.astype(np.float64))
    for order in ("C", "F"):
        f = lambda a: np.asarray(a, order=order)  # noqa: E731
        got, Lg = oracle_mod.blend(f(rgba), f(alpha.astype(np.int64)), f(depth.astype(np.float64)),
                                   f(fused.astype(np.float64)), f(w), f(w_bg), f(i_bg))
        assert np.array_equal(got, ref) and Lg == L
