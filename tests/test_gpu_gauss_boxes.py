"""The Gaussian render's lists where boxes of 2 x 2 tiles and larger ones meet in one warp."""
import pytest
import torch

from test_gpu_gauss import _case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gvs():
    assert torch.cuda.is_available()
    from paper_2505_18932_gb300 import gvs as g
    g.load()
    return g


@pytest.mark.parametrize("scale_px,max_radius", [(1.0, 8), (2.0, 16), (3.0, 32), (6.0, 32)])
def test_mixed_boxes(gvs, oracle_mod, scale_px, max_radius):
    from synth import configs
    w = configs.tiny(70, 45, 2, 16)
    _case(gvs, oracle_mod, w, target=configs.tiny(130, 70, 2, 16).targets[0], scale_px=scale_px, max_radius=max_radius)
