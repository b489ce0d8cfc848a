"""The setup's launch forms: tables in the vertex transform's parameter (two sizes) or uploaded,
scans and the longest-first order in one block or several kernels.  Whatever the form, a batch's
views equal the same views rendered one by one, bit for bit."""
import ctypes as C
import dataclasses

import numpy as np
import pytest
import torch

import synth
from paper_2204_01386_gb300 import PackedScene, Renderer, binding as B

pytestmark = pytest.mark.gpu


def _views(s, n, W, H):
    s.views = [synth.View(synth.camera_mvp(3.0 * d, W, H), 0, W, H) for d in synth.fibonacci_dirs(n + 1)[:n]]
    r = 2.0 / max(W, H)
    s.params = dataclasses.replace(s.params, r=r, sigma=r / 7, delta=r)
    return s


# a view's table entry is 160 bytes: 1 view takes the small parameter (512 bytes), 2 to 99 the large
# one (16,000 bytes), more the upload
@pytest.mark.parametrize("n", [1, 2, 3, 98, 99, 100, 200])
@pytest.mark.parametrize("cfg", ["config1", "config2"])
def test_batches_equal_single_views(n, cfg):
    s = _views(getattr(synth, cfg)(), n, 24, 20)
    ps = PackedScene(s.meshes, "cuda")
    r = Renderer(ps, s.views, s.params, tile=16, schedule=2)
    out, ids = r.forward()
    for i in sorted({0, 1, n // 2, n - 1} & set(range(n))):
        one, one_ids = Renderer(ps, [s.views[i]], s.params, tile=16, schedule=1).forward()
        sl = slice(480 * i, 480 * (i + 1))
        assert torch.equal(one, out[sl]) and torch.equal(one_ids, ids[:, sl])
    assert r.device_status() == 0


# 16 px tiles: 24,576 scan items are the last that one block takes, 16,384 tiles the last order
@pytest.mark.parametrize("W,H,n", [(2048, 2048, 1), (2048, 2064, 1), (2048, 3056, 1), (2048, 3072, 1), (2048, 3088, 1)])
def test_scans_and_order_at_their_limits(W, H, n):
    s = _views(synth.config1(), n, W, H)
    ps = PackedScene(s.meshes, "cuda")
    want, want_ids = Renderer(ps, s.views, s.params, tile=32, schedule=1).forward()
    tiles = (W // 16) * (H // 16) * n
    order, lengths = (torch.full((tiles,), -1, dtype=torch.int32, device="cuda") for _ in range(2))
    lib = B.load()
    r = Renderer(ps, s.views, s.params, tile=16, schedule=2)
    lib.dressi_set_tile_order_buffer(C.c_void_p(order.data_ptr()), C.c_void_p(lengths.data_ptr()))
    try:
        out, ids = r.forward()
        torch.cuda.synchronize()
    finally:
        lib.dressi_set_tile_order_buffer(None, None)
    assert torch.equal(ids, want_ids)
    assert (out - want).abs().max().item() <= 1e-5   # the forward tolerance between tile sizes
    o, ln = order.cpu().numpy(), lengths.cpu().numpy()
    assert (np.sort(o) == np.arange(tiles)).all()
    assert (np.diff(np.minimum(ln[o], 1023)) <= 0).all() and ln.max() > 0
    assert r.device_status() == 0
