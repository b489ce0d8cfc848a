"""The adjoint's 1 / Q (Q: the sum of the perspective weights) is correctly rounded: a scene in which
every other step of dL/dMVP is exact or one rounded product, compared bit for bit."""
import numpy as np
import pytest
import torch

import synth
from paper_2204_01386_gb300 import PackedScene, Renderer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("store", [True, False])
def test_adjoint_divides_by_the_weights_sum(store):
    # corners at (32, 32), (64, 32), (32, 64) px with w = 1, 3, 3: the areas' ratios are multiples of 1/64,
    # the weights lam / w and their sum Q (corners 0, 2, 1: the record's order) round as below.
    # Corner 0 alone has z != 0 in the object (so dL/dMVP's z column is its share) and lies at clip
    # x = y = 0; it alone is red, and the gradient is of red.
    W = 64
    pos = np.array([[0, 0, 1], [3, 0, 0], [0, 3, 0]], np.float32)
    mvp = np.array([[1, 0, 0, 0], [0, 1, 0, 0], [0, 0, -1, 1.5], [0, 0, -2, 3]], np.float32)
    m = synth.Mesh(pos, np.array([[0, 1, 2]], np.int32), col=np.array([[1, 0, 0], [0, 0, 0], [0, 0, 0]], np.float32))
    r = 2.0 / W
    p = synth.Params(K=1, r=r, sigma=r / 7, delta=r, edge_mode=2, shade_mode=0)
    rr = Renderer(PackedScene([m], "cuda"), [synth.View(mvp.reshape(16), 0, W, W)], p)
    out, ids = rr.forward(store_layers=store)
    img = out.cpu().numpy().reshape(W, W, 4)
    f = np.float32
    checked = 0
    third = f(1) / f(3)
    for y in range(32, 63):
        for x in range(32, 64 - (y - 32) - 1):
            l1, l2 = f((x + 0.5 - 32) / 32), f((y + 0.5 - 32) / 32)
            l0 = f(1 - l1 - l2)
            Q = f(f(l0 + f(l2 * third)) + f(l1 * third))
            b0 = img[y, x, 0]   # the forward's barycentric of corner 0
            assert abs(b0 - l0 / Q) < 1e-6
            g = torch.zeros_like(out)
            g[y * W + x, 0] = 1.0
            gm = rr.backward(g, ids=ids, camera=True)[3]
            want = -f(f(f(f(1) - b0) * f(f(1) / Q)) * l0)
            assert gm[0, 14].item() == want, (x, y)
            checked += 1
    assert checked > 400
