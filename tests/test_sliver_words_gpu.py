"""Faces one FP32 step thin, seen edge-on along the pixel diagonal: their cross products and area are
rounding noise, so pixel centres count as inside them with interpolated depths far outside [0, 1]
(keys of 1/2, 2 and more).  Passes without stored layer ids, whose pixel words hold keys, give what
the passes with layer ids and the adjoint without words give."""
import numpy as np
import pytest
import torch

import synth
from paper_2204_01386_gb300 import PackedScene, Renderer
from scenes_small import identity_mvp
from test_fronts_gpu import _check, _rel

pytestmark = pytest.mark.gpu


def scene(pos, faces, W, **kw):
    pos = np.asarray(pos, np.float32)
    col = np.random.default_rng(4).random(pos.shape).astype(np.float32)
    r = kw.pop("r_px", 2.0) / W
    p = synth.Params(r=r, sigma=r / 7, shade_mode=0, **kw)
    return synth.Scene("slivers", [synth.Mesh(pos, np.asarray(faces, np.int32), col=col)],
                       [synth.View(identity_mvp(), 0, W, W)], p)


def past_two():
    """the sliver and the face of test_layer_key_past_two"""
    m = np.float32(0.19097761809825897)
    a, b = np.float32(-0.7712559700012207), np.float32(0.4108498990535736)
    pos = [(a, a, 0.95), (b, b, 0.96), (m, np.nextafter(m, np.float32(2)), 0.97),
           (38 / 32 - 1, -1.5, 0.5), (38 / 32 - 1, 2.5, 0.5), (-3.0, 0.1, 0.5)]
    return pos, [(0, 1, 2), (3, 4, 5)]


@pytest.mark.parametrize("K", [1, 2, 3])
@pytest.mark.parametrize("tile", [16, 32])
def test_layer_key_past_two(tile, K):
    """A sliver crosses the pixels (32..43)^2 of the diagonal with keys of 5 to 8 (evaluated step by step
    in FP32), behind a face whose edge at x = 38 px puts them inside the edge mask."""
    _check(scene(*past_two(), 64, K=K, delta=8.0 / 64), tile, 1)


def slivers(n, W, seed):
    """n slivers on diagonals y = x + k pixels; the thickness is one FP32 step at the third corner"""
    g = np.random.default_rng(seed)
    pos = []
    for _ in range(n):
        k = np.float32(g.integers(-W // 2, W // 2 + 1) * 2.0 / W)
        a, b = sorted(np.round(g.uniform(-0.95, 0.95, 2) * 2**20) / 2**20)
        m = np.float32(np.round((a + (b - a) * g.uniform(0.2, 0.8)) * 2**20) / 2**20)
        pos += [(a, np.float32(a) + k, 0.93), (b, np.float32(b) + k, 0.96),
                (m, np.nextafter(m + k, np.float32(9)), 0.99)]
    return pos, np.arange(3 * n).reshape(n, 3)


def check_alone(s, tile):
    r = Renderer(PackedScene(s.meshes, "cuda"), s.views, s.params, tile=tile, schedule=1)
    full, _ = r.forward(store_layers=True)
    out, _ = r.forward(store_layers=False)
    assert full.abs().sum().item() > 0
    assert torch.equal(out, full)
    # the forward's words or none: the same layers' terms in another order
    g = torch.randn(out.shape, device="cuda", generator=torch.Generator(device="cuda").manual_seed(3))
    got = [t.clone() for t in r.backward(g, ids=None) if t is not None]
    want = [t for t in r.backward(g, ids=None, reuse_setup=False) if t is not None]
    for x, y in zip(got, want):
        assert _rel(x, y) < 1e-5


@pytest.mark.parametrize("K,edge,r_px", [(1, 0, 1.0), (2, 0, 1.0), (3, 0, 0.5), (2, 2, 1.0)])
@pytest.mark.parametrize("tile,n", [(16, 12), (16, 60), (32, 30)])
def test_slivers_alone(tile, n, K, edge, r_px):
    for seed in range(4):
        check_alone(scene(*slivers(n, 64, seed), 64, K=K, delta=1.0 / 64, r_px=r_px, edge_mode=edge), tile)
