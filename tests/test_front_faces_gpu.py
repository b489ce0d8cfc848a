"""Front fragments from the face table for faces of every box size (a lane's own, a warp's list, bands of
rows shared by all warps), thin and cut ones among them, with edges through pixel centres: the image of a
pass that stores every layer, bit for bit, whatever the room for the list of large faces."""
import numpy as np
import pytest
import torch

import synth
from paper_2204_01386_gb300 import PackedScene, Renderer, binding as B
from scenes_small import identity_mvp

pytestmark = pytest.mark.gpu


def _mesh(W, H, boxes, seed, n=18000, thin=0.3):
    """n triangles with boxes of about `boxes` pixels, corners on a 1/2-pixel grid (a share of them needles,
    some with corners far outside the view), fewer than 24 view pixels per face"""
    g = np.random.default_rng(seed)
    c = np.stack([g.uniform(-4, W + 4, n), g.uniform(-4, H + 4, n)], 1)
    w = np.exp(g.uniform(np.log(0.3), np.log(boxes), n))
    h = np.clip(boxes / w * g.uniform(0.2, 1.2, n), 0.3, 60)
    p = c[:, None, :] + g.uniform(-0.5, 0.5, (n, 3, 2)) * np.stack([w, h], 1)[:, None, :]
    needle = g.random(n) < thin
    p[needle, 2] = p[needle, 0] + (p[needle, 1] - p[needle, 0]) * g.uniform(0, 1, (needle.sum(), 1)) + g.normal(0, 0.02, (needle.sum(), 2))
    far = g.random(n) < 0.02
    p[far, 1] = p[far, 0] + (p[far, 1] - p[far, 0]) * g.uniform(20, 200, (far.sum(), 1))
    snap = g.random(n) < 0.5
    p[snap] = np.round(p[snap] * 2) / 2
    z = g.uniform(0.1, 0.9, (n, 3, 1))
    pos = np.concatenate([2 * p / (W, H) - 1, z], 2).reshape(-1, 3).astype(np.float32)
    return synth.Mesh(pos, np.arange(3 * n, dtype=np.int32).reshape(n, 3), col=g.random(pos.shape).astype(np.float32))


@pytest.mark.parametrize("W,H", [(500, 300), (512, 3), (97, 611)])
@pytest.mark.parametrize("boxes", [8, 64, 256, 1100])
def test_box_sizes(W, H, boxes):
    r = 1.0 / max(W, H)
    m = _mesh(W, H, boxes, W + boxes)
    s = synth.Scene("boxes", [m], [synth.View(identity_mvp(), 0, W, H)], synth.Params(K=2, r=r, sigma=r / 7, delta=r, shade_mode=0))
    ps = PackedScene(s.meshes, "cuda")
    want, _ = Renderer(ps, s.views, s.params).forward(store_layers=True)
    got, _ = Renderer(ps, s.views, s.params).forward(store_layers=False)
    assert torch.equal(got, want)
    # no room in the tile lists, nor in the list of large faces kept in their place
    rr = Renderer(ps, s.views, s.params, list_cap=3)
    got, _ = rr.forward(store_layers=False)
    assert torch.equal(got, want)
    assert rr.device_status() == B.DEV_TILE_OVERFLOW


def test_no_room_for_large_faces_of_several_views():
    """views of unlike meshes, the last one smaller than a warp's share"""
    W = 120
    r = 1.0 / W
    ms = [_mesh(W, W, 300, 1, n=9000), _mesh(W, W, 3000, 2, n=9001), _mesh(W, W, 9000, 3, n=5)]
    views = [synth.View(identity_mvp(), m, W, W) for m in (0, 1, 2, 1, 2)]
    ps = PackedScene(ms, "cuda")
    p = synth.Params(K=3, r=r, sigma=r / 7, delta=r, shade_mode=0)
    want, _ = Renderer(ps, views, p).forward(store_layers=True)
    for cap in (1, 2, 64):
        rr = Renderer(ps, views, p, list_cap=cap)
        got, _ = rr.forward(store_layers=False)
        assert torch.equal(got, want)
