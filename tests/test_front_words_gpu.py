"""Front fragments from the face table where a depth is at or past the far plane: hard keys of exactly 1/2
(ties with soft fragments) and, of slivers whose area is rounding noise, far above it.  The images and
gradients are those of passes that store every layer, bit for bit and to rounding."""
import numpy as np
import pytest

from test_fronts_gpu import _check
from test_sliver_words_gpu import check_alone, past_two, scene, slivers

pytestmark = pytest.mark.gpu


def off_view(pos, faces, n=17000):
    """beside n faces that no pixel sees: enough for the front fragments to come from the face table"""
    g = np.random.default_rng(6)
    far = (np.array([3.0, 3.0, 0.5]) + 0.1 * g.random((3 * n, 3))).astype(np.float32)
    k = len(pos)
    return (np.concatenate([np.asarray(pos, np.float32), far]),
            np.concatenate([np.asarray(faces, np.int32), k + np.arange(3 * n, dtype=np.int32).reshape(n, 3)]))


@pytest.mark.parametrize("K", [1, 2, 3])
@pytest.mark.parametrize("tile", [16, 32])
def test_layer_key_past_two_from_the_face_table(tile, K):
    _check(scene(*off_view(*past_two()), 64, K=K, delta=8.0 / 64), tile, 1)


@pytest.mark.parametrize("K,edge,r_px", [(1, 0, 1.0), (2, 0, 1.0), (3, 0, 0.5), (2, 2, 1.0)])
@pytest.mark.parametrize("tile,n", [(16, 12), (16, 60), (32, 30)])
def test_slivers_from_the_face_table(tile, n, K, edge, r_px):
    for seed in range(4):
        check_alone(scene(*off_view(*slivers(n, 64, seed)), 64, K=K, delta=1.0 / 64, r_px=r_px, edge_mode=edge), tile)


@pytest.mark.parametrize("tile,schedule", [(16, 1), (32, 2)])
@pytest.mark.parametrize("order", [[0, 1, 2, 3], [3, 2, 1, 0]])
def test_far_plane_ties_from_the_face_table(tile, schedule, order):
    """Hard fragments at depth exactly 1 tie with soft ones at distance 0: such tiles are decided from all
    layers, by the forward and by the adjoint, where the front fragments come from the face table."""
    W = 40
    v = [(4, 4), (20.5, 4), (4, 30), (20.5, 30), (36, 4), (36, 30)]
    f = [(0, 1, 2), (1, 3, 2), (1, 4, 3), (4, 5, 3)]
    pos, faces = off_view([(2 * x / W - 1, 2 * y / W - 1, 1.0) for x, y in v], [f[i] for i in order])
    _check(scene(pos, faces, W, K=3, delta=2.0 / W), tile, schedule)
