"""The grids of the per-face and per-vertex kernels of a ragged batch, read off captured graphs: one long mesh
among many short ones still gets blocks enough for its own length."""
import ctypes as C
import re

import numpy as np
import pytest
import torch

import synth
from paper_2204_01386_gb300 import PackedScene, Renderer

pytestmark = pytest.mark.gpu


def _grids(fn, tmp_path):
    """kernel name -> blocks along x of a captured call"""
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g):
        fn()
    path = str(tmp_path / "graph.dot")
    assert C.CDLL("libcudart.so.13").cudaGraphDebugDotPrint(C.c_void_p(g.raw_cuda_graph()), path.encode(), C.c_uint(1)) == 0
    return {n: eval("(%s,)" % x)[0] for n, x in re.findall(r"\| (\w+)(?:\\<){3}[\\{]*([\d,]+)", open(path).read())}


def test_blocks_for_one_long_mesh_among_many(tmp_path):
    def mesh(subdiv, seed):
        pos, f = synth.icosphere(subdiv)
        g = np.random.default_rng(seed)
        return synth.Mesh(synth.displace(pos, 0.1, seed).astype(np.float32), f,
                          uv=g.random((pos.shape[0], 2)).astype(np.float32), tex=g.random((16, 16, 4)).astype(np.float32))
    meshes = [mesh(1, i) for i in range(200)] + [mesh(7, 7)]   # 80 faces each, and 327,680
    views = [synth.View(synth.camera_mvp((0, 0, 3), 32, 32), i, 32, 32) for i in range(len(meshes))]
    r = Renderer(PackedScene(meshes, "cuda"), views, synth.Params(K=2, r=2 / 32, sigma=0.3 / 32, delta=1 / 32, shade_mode=2))
    out, ids = r.forward()
    grad = torch.randn_like(out)
    res = r.backward(grad, ids=ids)
    fwd = _grids(lambda: r.forward(out=out, ids=ids), tmp_path)
    bwd = _grids(lambda: r.backward(grad, ids=ids, grad_pos=res[0], grad_tex=res[2]), tmp_path)
    faces = meshes[-1].faces.shape[0]
    seen = 0
    for grids, names in ((fwd, ("k_face", "k_bin")), (bwd, ("k_vertex_bwd",))):
        for name in names:
            x = [v for k, v in grids.items() if name in k]
            assert len(x) == 1
            assert x[0] * 256 * 16 >= faces, (name, x)   # sixteen faces a thread at most
            seen += 1
    assert seen == 3
