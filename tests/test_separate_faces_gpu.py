"""Meshes with more vertices than faces (separate triangles), without stored layer ids: all lists get their layers
in one pass, and the images and gradients are those of passes with ids and of passes without words."""
import numpy as np
import pytest
import torch

import synth
from paper_2204_01386_gb300 import PackedScene, Renderer
from scenes_small import identity_mvp
from test_fronts_gpu import _rel

pytestmark = pytest.mark.gpu


# up to 8 faces on a tile (one pass for any mesh), some tens, and more than a staged chunk of 128
@pytest.mark.parametrize("n,size", [(12, 6.0), (400, 8.0), (3000, 9.0)])
@pytest.mark.parametrize("K,edge", [(1, 0), (3, 0), (5, 2)])
@pytest.mark.parametrize("tile,schedule", [(16, 0), (32, 2)])
def test_separate_triangles(n, size, K, edge, tile, schedule):
    W, H = 97, 70
    g = np.random.default_rng(n)
    p = g.uniform(0, 1, (n, 1, 2)) * (W, H) + g.normal(0, size, (n, 3, 2))
    pos = np.concatenate([2 * p / (W, H) - 1, g.uniform(0.1, 0.9, (n, 3, 1))], 2).reshape(-1, 3).astype(np.float32)
    m = synth.Mesh(pos, np.arange(3 * n, dtype=np.int32).reshape(n, 3), col=g.random(pos.shape).astype(np.float32))
    r = 2.0 / W
    s = synth.Scene("separate", [m], [synth.View(identity_mvp(), 0, W, H)],
                    synth.Params(K=K, r=r, sigma=r / 7, delta=r, edge_mode=edge, shade_mode=0))
    # (3,000 such triangles are more list entries than the default capacity holds)
    r = Renderer(PackedScene(s.meshes, "cuda"), s.views, s.params, tile=tile, schedule=schedule, list_cap=40 * n)
    full, ids = r.forward(store_layers=True)
    grad = torch.randn(full.shape, device="cuda", generator=torch.Generator(device="cuda").manual_seed(3))
    want = [t.clone() for t in r.backward(grad, ids=ids) if t is not None]
    out, _ = r.forward(store_layers=False)
    assert torch.equal(out, full)
    # the same per-layer terms added up in another order: FP32 rounding, far below 1e-5 of the norm
    for reuse in (None, False):
        for a, b in zip([t for t in r.backward(grad, ids=None, reuse_setup=reuse) if t is not None], want):
            assert _rel(a, b) < 1e-5
    assert r.device_status() == 0
