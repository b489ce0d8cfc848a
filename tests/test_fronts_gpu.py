"""Passes without stored layer ids take the layers behind the front one only inside the edge
mask: the image equals the one of a pass that stores every layer, bit for bit, and the
re-rasterizing adjoint (from the forward's words, or on its own) gives the gradients of the
adjoint from stored ids."""
import dataclasses

import numpy as np
import pytest
import torch

import synth
from paper_2204_01386_gb300 import PackedScene, Renderer
from scenes_small import pixel_mesh, pixel_scene

pytestmark = pytest.mark.gpu


def _scene(W, H, views=2, **kw):
    s = synth.config2()
    r = kw.pop("r_px", 2.0) / max(W, H)
    s.params = dataclasses.replace(s.params, r=r, sigma=r / 7, delta=min(r, 8.0 / max(W, H)), **kw)
    s.views = [synth.View(synth.camera_mvp(3.0 * d, W, H), 0, W, H) for d in synth.fibonacci_dirs(views + 1)[:views]]
    return s


def _rel(a, b):
    return (a - b).norm().item() / max(b.norm().item(), 1e-30)


def _check(s, tile, schedule, words=True):
    r = Renderer(PackedScene(s.meshes, "cuda"), s.views, s.params, tile=tile, schedule=schedule)
    full, ids = r.forward(store_layers=True)
    g = torch.randn(full.shape, device="cuda", generator=torch.Generator(device="cuda").manual_seed(3))
    want = [t.clone() for t in r.backward(g, ids=ids) if t is not None]
    out, _ = r.forward(store_layers=False)
    assert torch.equal(out, full)
    # the same per-layer terms (bit for bit) added up in another order: FP32 rounding of sums of
    # some thousands of terms, far below 1e-5 of their norm
    for reuse in ([None, False] if words else [False]):
        got = [t for t in r.backward(g, ids=None, reuse_setup=reuse) if t is not None]
        for a, b in zip(got, want):
            assert _rel(a, b) < 1e-5
    assert r.device_status() == 0


@pytest.mark.parametrize("tile,schedule", [(16, 1), (32, 2)])
@pytest.mark.parametrize("K", [1, 2, 3, 5])
@pytest.mark.parametrize("edge", [0, 1, 2])
def test_images_and_gradients_without_ids(tile, schedule, K, edge):
    _check(_scene(131, 75, K=K, edge_mode=edge), tile, schedule)


@pytest.mark.parametrize("W,H,r_px", [(33, 17, 0.5), (64, 64, 7.0), (31, 1, 1.0), (200, 96, 4.0)])
def test_sizes_and_radii_without_ids(W, H, r_px):
    _check(_scene(W, H, views=1, r_px=r_px), 32, 1)


@pytest.mark.parametrize("texgrad", [1, 2])
def test_texel_gradient_modes_without_ids(texgrad):
    _check(_scene(90, 90, texgrad_mode=texgrad), 16, 1)


@pytest.mark.parametrize("tile", [16, 32])
def test_far_plane_ties_without_ids(tile):
    """Hard fragments at depth exactly 1 (key 1/2) tie with soft ones at distance exactly 0 (a face
    whose edge runs through pixel centres): the smaller face id is in front."""
    W, H = 40, 36
    v = [(4, 4), (20.5, 4), (4, 30), (20.5, 30), (36, 4), (36, 30)]
    f = [(0, 1, 2), (1, 3, 2), (1, 4, 3), (4, 5, 3)]
    for order in ([0, 1, 2, 3], [3, 2, 1, 0]):
        m = pixel_mesh(v, [f[i] for i in order], W, H, z=1.0, col=np.random.default_rng(1).random((6, 3)).astype(np.float32))
        s = pixel_scene(m, W, H, K=3, r=2.0 / W, sigma=0.3 / W, delta=2.0 / W, shade_mode=0)
        _check(s, tile, 1)


@pytest.mark.parametrize("tile,schedule", [(16, 1), (32, 2)])
@pytest.mark.parametrize("K,edge", [(1, 0), (3, 0), (3, 2)])
@pytest.mark.parametrize("W,H", [(257, 193), (1040, 611)])
def test_fronts_from_the_face_table(tile, schedule, K, edge, W, H):
    """Scenes of 32,768 faces and more, small ones beside some that fill the view (their boxes are
    above and below the size that gets warps of its own)."""
    pos, f = synth.icosphere(6)
    g = np.random.default_rng(5)
    big = np.array([[-3, -2, -3], [3, -2, -3], [0, 3, -3], [-0.3, 0.2, 1.3], [0.3, 0.1, 1.3], [0.1, 0.6, 1.2],
                    [-0.05, -0.3, 1.4], [0.05, -0.33, 1.4], [0.0, -0.2, 1.4]], np.float64)
    n = pos.shape[0]
    m = synth.Mesh(np.concatenate([synth.displace(pos, 0.1, 3), big]).astype(np.float32),
                   np.concatenate([f, [[n, n + 1, n + 2], [n + 3, n + 4, n + 5], [n + 6, n + 7, n + 8]]]).astype(np.int32),
                   col=g.random((n + 9, 3)).astype(np.float32))
    r = 2.0 / max(W, H)
    views = [synth.View(synth.camera_mvp(e, W, H), 0, W, H) for e in ((0, 0, 3), (0.5, 0.4, 2.9))]
    s = synth.Scene("front_words", [m], views, synth.Params(K=K, r=r, sigma=r / 7, delta=r, edge_mode=edge))
    _check(s, tile, schedule)


@pytest.mark.parametrize("subdiv", [3, 6])
def test_words_of_an_earlier_setup_are_not_used(subdiv):
    """forward without ids, then moved positions: a rebuilding adjoint and the reusing one after it
    (which finds the rebuilt setup, not the forward's words) agree."""
    W, H = 90, 70
    pos, f = synth.icosphere(subdiv)
    m = synth.Mesh(synth.displace(pos, 0.1, 3).astype(np.float32), f,
                   col=np.random.default_rng(0).random((pos.shape[0], 3)).astype(np.float32))
    r = 2.0 / W
    s = synth.Scene("moved", [m], [synth.View(synth.camera_mvp((0, 0, 3), W, H), 0, W, H)],
                    synth.Params(K=3, r=r, sigma=r / 7, delta=r))
    ps = PackedScene(s.meshes, "cuda")
    rr = Renderer(ps, s.views, s.params)
    out, _ = rr.forward(store_layers=False)
    ps.pos.mul_(0.8)
    g = torch.randn(out.shape, device="cuda", generator=torch.Generator(device="cuda").manual_seed(3))
    want = [t.clone() for t in rr.backward(g, ids=None, reuse_setup=False) if t is not None]
    got = [t for t in rr.backward(g, ids=None) if t is not None]
    for a, b in zip(got, want):
        assert _rel(a, b) < 1e-5
