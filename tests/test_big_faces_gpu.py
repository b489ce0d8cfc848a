"""Parity with the oracle where faces hold more than 256 pixels each: the adjoint from stored ids then adds a
warp's gradients up before it adds them to the corners'."""
import dataclasses

import pytest

import synth
from parity import compare_scene

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile", [16, 32])
def test_big_faces(tile):
    W, H = 300, 280   # 84,000 pixels, 320 faces
    s = synth.config1()
    s.views = [synth.View(synth.camera_mvp((0.3, 0.2, 2.9), W, H), 0, W, H)]
    r = 2.0 / W
    s.params = dataclasses.replace(s.params, r=r, sigma=r / 7, delta=r)
    assert W * H > 256 * s.meshes[0].faces.shape[0]
    st = compare_scene(s, tile=tile)
    assert st["ids_checked"] > 80000
