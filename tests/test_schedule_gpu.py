"""The form of the forward tile kernel that a schedule gets, read off a captured graph: one CTA per tile
where the caller asks for it (schedule 1), clusters of 8, 4 or 2 CTAs for the long lists of scenes of few
tiles otherwise -- with lists long enough that clusters do get tiles -- and the same layers and image."""
import ctypes as C
import re

import numpy as np
import pytest
import torch

import synth
from paper_2204_01386_gb300 import PackedScene, Renderer, binding as B
from test_long_lists_gpu import _scene

pytestmark = pytest.mark.gpu


def _kernels(r, tmp_path, **kw):
    """(name, CTAs per cluster) of the kernels of a forward pass"""
    rt = C.CDLL("libcudart.so.13")
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g):
        r.forward(**kw)
    path = str(tmp_path / "graph.dot")
    assert rt.cudaGraphDebugDotPrint(C.c_void_p(g.raw_cuda_graph()), path.encode(), C.c_uint(1)) == 0
    found = []
    for name, node in re.findall(r"\| (\w+)\\<.*?\n.*?func handle\} \| \{(0x[0-9A-Fa-f]+)", open(path).read()):
        value = (C.c_uint * 16)()
        # attribute 4: the cluster's dimensions
        assert rt.cudaGraphKernelNodeGetAttribute(C.c_void_p(int(node, 16)), C.c_int(4), value) == 0
        found.append((name, int(value[0])))
    return found


def _long_tiles(r, tiles, shortest):
    """the tiles that the list fill calls long, from the inspection hook's list lengths (schedule 2)"""
    order = torch.zeros(tiles, dtype=torch.int32, device="cuda")
    lengths = torch.zeros(tiles, dtype=torch.int32, device="cuda")
    lib = B.load()
    lib.dressi_set_tile_order_buffer(C.c_void_p(order.data_ptr()), C.c_void_p(lengths.data_ptr()))
    try:
        r.forward()
    finally:
        lib.dressi_set_tile_order_buffer(None, None)
    n = lengths.cpu().numpy()
    return int((n > max(shortest, int(n.sum()) // 608 * 2)).sum())


@pytest.mark.parametrize("W,H,subdiv,ctas,shortest", [(90, 66, 5, 8, 96), (200, 150, 5, 4, 96), (300, 250, 5, 2, 96),
                                                      (420, 400, 7, 8, 256)])
@pytest.mark.parametrize("K", [1, 3, 5])
def test_forms_of_the_forward(W, H, subdiv, ctas, shortest, K, tmp_path):
    s = _scene(W, H, subdiv=subdiv, K=K)
    ps = PackedScene(s.meshes, "cuda")
    cap = 16 * s.meshes[0].faces.shape[0]
    tiles = ((W + 15) // 16) * ((H + 15) // 16)
    plain = Renderer(ps, s.views, s.params, tile=16, schedule=1, list_cap=cap)
    want, want_ids = plain.forward()
    names = _kernels(plain, tmp_path, out=want.clone(), ids=want_ids.clone())
    assert [c for n, c in names if "k_tile" in n] == [c for n, c in names if "6k_tileI" in n] and names
    for schedule in (0, 2):
        r = Renderer(ps, s.views, s.params, tile=16, schedule=schedule, list_cap=cap)
        out, ids = r.forward()
        assert torch.equal(out, want) and torch.equal(ids, want_ids)
        names = _kernels(r, tmp_path, out=out, ids=ids)
        assert [c for n, c in names if "k_tile" in n] == [ctas] and any("k_tile_heavy" in n for n, _ in names)
    assert 0 < _long_tiles(r, tiles, shortest) <= 1024
    assert plain.device_status() == 0 and r.device_status() == 0


def test_many_tiles_without_long_lists(tmp_path):
    """more tiles than the GPU has CTAs and no long list: the plain forms for every schedule"""
    s = synth.config2()
    ps = PackedScene(s.meshes, "cuda")
    s.views = [synth.View(synth.camera_mvp((0.4, 0.3, 2.9), 640, 600), 0, 640, 600)]
    for schedule, form in ((0, "6k_tileI"), (1, "6k_tileI"), (2, "k_tile_persistent")):
        r = Renderer(ps, s.views, s.params, tile=16, schedule=schedule)
        out, ids = r.forward()
        assert [form in n for n, _ in _kernels(r, tmp_path, out=out, ids=ids) if "k_tile" in n] == [True]
