"""The adjoint from stored ids by 256 or 128 threads per tile (few or many 16 px tiles) and, for faces of
many pixels, with a warp's gradients added up first: the gradients of the re-rasterizing
adjoint, which has one form."""
import dataclasses

import pytest
import torch

import synth
from paper_2204_01386_gb300 import PackedScene, Renderer

pytestmark = pytest.mark.gpu


# (608 tiles are the last for 256 threads; 256 pixels per face the last without sums)
@pytest.mark.parametrize("cfg,W,H", [("config1", 64, 64), ("config1", 287, 285), ("config1", 289, 287), ("config1", 700, 517),
                                     ("config2", 304, 512), ("config2", 320, 512), ("config2", 1180, 1100),
                                     ("config2", 1150, 1150)])
@pytest.mark.parametrize("tile", [16, 32])
def test_forms_agree(cfg, W, H, tile):
    s = getattr(synth, cfg)()
    r = 2.0 / max(W, H)
    s.params = dataclasses.replace(s.params, r=r, sigma=r / 7, delta=r)
    s.views = [synth.View(synth.camera_mvp((0.3, 0.2, 2.9), W, H), 0, W, H)]
    rr = Renderer(PackedScene(s.meshes, "cuda"), s.views, s.params, tile=tile)
    out, ids = rr.forward()
    g = torch.randn(out.shape, device="cuda", generator=torch.Generator(device="cuda").manual_seed(1))
    a = [t.clone() for t in rr.backward(g, ids=ids) if t is not None]
    b = [t for t in rr.backward(g, ids=None, reuse_setup=False) if t is not None]
    # the same layers' terms added up in another order: sums of up to 1e4 FP32 terms of mixed sign
    for x, y in zip(a, b):
        assert (x - y).norm().item() <= 1e-5 * max(y.norm().item(), 1e-30)
    assert (rr.device_status() & ~1) == 0
