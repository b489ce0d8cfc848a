"""Tiles with long face lists are worked on by a cluster of CTAs when few tiles hold most of the
work (a dense mesh in a small view).  In a batch of many such views they are not (every tile is
like the others): both forms give the same layers and image, bit for bit."""
import dataclasses

import pytest
import torch

import synth
from paper_2204_01386_gb300 import PackedScene, Renderer, binding as B

pytestmark = pytest.mark.gpu


def _scene(W, H, subdiv=5, **kw):
    pos, f = synth.icosphere(subdiv)
    g = synth.rng(9)
    m = synth.Mesh(synth.displace(pos, 0.1, 4).astype("float32"), f, col=g.random((pos.shape[0], 3)).astype("float32"))
    r = kw.pop("r_px", 2.0) / max(W, H)
    p = synth.Params(r=r, sigma=r / 7, delta=r, **kw)
    return synth.Scene("dense", [m], [synth.View(synth.camera_mvp((0.4, 0.3, 2.9), W, H), 0, W, H)], p)


def _launches(r, **kw):
    c0 = B.load().dressi_launch_count()
    res = r.forward(**kw)
    torch.cuda.synchronize()
    return res, B.load().dressi_launch_count() - c0


def _check(s, tile, schedule, store, copies=200):
    ps = PackedScene(s.meshes, "cuda")
    v = s.views[0]
    n = v.width * v.height
    # room for every entry: past the capacity tiles would take all faces of their view
    cap = 16 * s.meshes[0].faces.shape[0]
    one = Renderer(ps, s.views, s.params, tile=tile, schedule=schedule, list_cap=cap)
    many = Renderer(ps, s.views * copies, s.params, tile=tile, schedule=schedule, list_cap=cap * copies)
    out, ids = one.forward(store_layers=store)
    ref, ref_ids = many.forward(store_layers=store)
    assert torch.equal(out, ref[:n]) and torch.equal(out, ref[-n:])
    if store:
        assert torch.equal(ids, ref_ids[:, :n])
    g = torch.randn(out.shape, device="cuda", generator=torch.Generator(device="cuda").manual_seed(2))
    a = one.backward(g, ids=ids)
    b = Renderer(ps, s.views, s.params, tile=16, schedule=1).backward(g, ids=None if not store else ids)
    for x, y in zip(a, b):
        # the same layers' terms in another order
        assert x is None or (x - y).norm().item() <= 1e-5 * max(y.norm().item(), 1e-30)
    assert one.device_status() == 0 and many.device_status() == 0


@pytest.mark.parametrize("tile,schedule", [(16, 1), (16, 2), (32, 1), (32, 2)])
@pytest.mark.parametrize("K", [1, 3, 5])
@pytest.mark.parametrize("store", [True, False])
def test_long_lists(tile, schedule, K, store):
    _check(_scene(40, 33, K=K), tile, schedule, store)


@pytest.mark.parametrize("edge,r_px", [(1, 7.0), (2, 0.5), (0, 7.0)])
def test_long_lists_edges(edge, r_px):
    for store in (True, False):
        _check(_scene(61, 64, edge_mode=edge, r_px=r_px), 32, 2, store)


# scenes of few tiles share all but short lists among 8, 4 or 2 CTAs, by their number; batches of more
# than 1,216 tiles do not
@pytest.mark.parametrize("W,H,copies", [(90, 66, 45), (200, 150, 10), (300, 250, 5), (420, 400, 2)])
@pytest.mark.parametrize("K", [2, 4])
def test_small_scenes(W, H, copies, K):
    _check(_scene(W, H, K=K), 16, 1, True, copies)
    _check(_scene(W, H, K=K, subdiv=4, edge_mode=1, r_px=5.0), 16, 2, False, copies)


def test_long_lists_normal_map():
    s = synth.config2n()
    r = 2.0 / 20
    s.views = [synth.View(synth.camera_mvp((0.4, 0.3, 2.9), 20, 17), 0, 20, 17)]
    s.params = dataclasses.replace(s.params, r=r, sigma=r / 7, delta=r)
    _check(s, 16, 1, True)


def test_list_capacity_exceeded():
    """A long list past the capacity: the tile takes every face of its view, by the cluster too."""
    s = _scene(40, 33)
    ps = PackedScene(s.meshes, "cuda")
    want, want_ids = Renderer(ps, s.views, s.params, tile=32).forward()
    r = Renderer(ps, s.views, s.params, tile=32, list_cap=3000)
    out, ids = r.forward()
    assert torch.equal(out, want) and torch.equal(ids, want_ids)
    assert r.device_status() == B.DEV_TILE_OVERFLOW
