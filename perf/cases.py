"""Performance cases: the calls that a user of this renderer makes, through its public
entry points (PackedScene, Renderer, render), on seeded synthetic scenes.

A case names a kind of call and its sizes.  The kinds:

  step      one training step: forward with the L2 image loss fused in, then the adjoint, from
            the stored layer ids (``store`` true) or re-rasterizing (checkpointed)
  autograd  the same through ``render`` and torch.autograd, as a PyTorch program writes it
  texfit    texture optimisation of a static geometry: forward from stored layers, loss, adjoint
  view      rendering alone: a preview or an evaluation image, nothing kept for an adjoint

Meshes are displaced spheres (``ico``: an icosphere subdivided ``n`` times; ``uv``: a UV sphere of
``n`` slices and ``m`` stacks; ``mix``: meshes of log-uniform face counts, one view of its own
resolution each), seen from distance 3 with a 45 degree lens; loss targets are images of a
sphere of about the same outline, so that the pixel gradient is dense inside the
silhouette and zero on the background.
"""
import math
import types

import numpy as np
import torch

from paper_2204_01386_gb300 import PackedScene, Renderer, render

DEV = "cuda"
LIGHT = np.full(3, 1.0 / math.sqrt(3.0), np.float32)
BASE = dict(kind="step", mesh="uv", n=64, m=41, views=1, w=256, h=256, tex=512, f16=False, shade=2, K=3, r_px=2.0,
            edge=0, texgrad=0, store=True, camera=False, tile=0, schedule=0)


def _case(name=None, **kw):
    c = dict(BASE, **kw)
    if c["shade"] == 0:
        c["tex"] = 0
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: a 320-face icosphere with vertex colours at 64 x 64 (first contact,
        # unit-sized fits, a step of a small optimisation): launches and latency
        _case("icosphere_64px_step", mesh="ico", n=2, m=0, w=64, h=64, shade=0, r_px=0.0448),
        # one textured view at 256 x 256, the ordinary single-image fit
        _case("textured_256px_step"),
        # the batched multi-view fit: 64 views of 512 x 512, 20,480 faces, 1024^2 texture
        _case("multiview_64x512_step", n=128, m=81, views=64, w=512, h=512, tex=1024, tile=32, schedule=2),
        # a ragged batch: 32 meshes of 1k to 200k faces, 128^2 to 1024^2 views, 512^2 to 2048^2 textures
        _case("ragged_32_step", mesh="mix", n=1000, m=200000, views=32, w=0, h=0, tex=0, tile=32, schedule=2),
        # the largest: 1.31 M faces, 4096^2 FP16 texture, 8 views of 2048^2, checkpointed (no layer ids)
        _case("large_8x2048_checkpointed", mesh="ico", n=8, m=0, views=8, w=2048, h=2048, tex=4096, f16=True,
              store=False, tile=32, schedule=1),
        # texture optimisation of a static geometry, 24 views
        _case("texture_fit_24x512", kind="texfit", n=128, m=81, views=24, w=512, h=512, tex=1024, tile=32, schedule=2),
        # relighting: normal map, with the gradients of the map, the camera and the light
        _case("normal_map_camera_6x384", n=96, m=61, views=6, w=384, h=384, tex=256, shade=3, camera=True),
        # silhouette and colour fit in the manner of SoftRas: blending everywhere, K = 5, wide blur
        _case("softras_K5_16x224_autograd", kind="autograd", mesh="ico", n=4, m=0, views=16, w=224, h=224, shade=0, K=5,
              r_px=7.0, edge=1),
        # bitwise reproducible texel gradients (the texel gather)
        _case("deterministic_texgrad_8x512", n=128, m=81, views=8, w=512, h=512, tex=1024, texgrad=1),
        # the inverse-UV texel gradient on one view of odd size
        _case("inverse_uv_521x337", n=80, m=51, w=521, h=337, tex=512, shade=1, texgrad=2),
        # an evaluation image: one 1280 x 720 view of an 81,920-face mesh, FP16 texture, nothing stored
        _case("render_1280x720", kind="view", mesh="ico", n=6, m=0, w=1280, h=720, tex=2048, f16=True),
        # a checkpointed fit through autograd, where the adjoint re-rasterizes
        _case("checkpointed_4x768_autograd", kind="autograd", n=160, m=101, views=4, w=768, h=768, tex=1024, store=False),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "autograd", "texfit", "view"])
    shade = rng.choice([0, 1, 2, 2, 2, 3])
    if kind == "texfit" and shade == 0:
        shade = 2
    views, r_px, K = _log(rng, 1, 64), rng.choice([0.5, 1.0, 2.0, 2.0, 2.0, 4.0, 7.0]), rng.choice([1, 2, 3, 3, 3, 4, 5])
    # at most the pixels of the multi-view case, fewer where the blur or K make each one dearer
    side = _log(rng, 48, min(2048, int(math.sqrt((16.8e6 if r_px <= 2 and K <= 3 else 3e6) / views))))
    w = max(33, min(2300, int(side * math.sqrt(rng.uniform(0.6, 1.7)))))
    h = max(33, side * side // w)
    bands = _log(rng, 12, min(400, max(24, side // 3)))
    c = dict(kind=kind, shade=shade, views=views, w=w, h=h, mesh="uv", n=max(3, int(bands * 1.57)), m=bands + 1)
    if rng.random() < 0.3:
        c.update(mesh="ico", n=rng.choice([2, 3, 4, 5, 6]), m=0)
    if shade:
        c["tex"] = rng.choice([_log(rng, 64, 2048), 256, 512, 1024])
        c["f16"] = rng.random() < 0.3
        c["texgrad"] = rng.choice([0, 0, 0, 0, 1, 2]) if shade < 3 and kind != "view" else 0
    c["K"], c["r_px"] = K, r_px
    c["edge"] = rng.choice([0, 0, 0, 0, 1, 2])
    c["store"] = rng.random() < 0.65 or kind == "texfit"
    c["camera"] = kind == "step" and rng.random() < 0.2
    c["tile"] = rng.choice([0, 16, 32, 32])
    c["schedule"] = rng.choice([0, 1, 2])
    return _case(**c)


# ----------------------------------------------------------------------------
# inputs, made on the GPU from the seed
# ----------------------------------------------------------------------------

def _outward(pos, f):
    p = pos[f.reshape(-1)].view(-1, 3, 3)
    flip = (torch.linalg.cross(p[:, 1] - p[:, 0], p[:, 2] - p[:, 0]) * p.sum(1)).sum(1) < 0
    return torch.where(flip[:, None], f[:, [0, 2, 1]], f)


def _uv_sphere(slices, stacks):
    """Latitude-longitude sphere, seam and poles duplicated; 2 slices (stacks - 1) faces."""
    i = torch.arange(stacks + 1, device=DEV, dtype=torch.float64)[:, None]
    j = torch.arange(slices + 1, device=DEV, dtype=torch.float64)[None, :]
    th, ph = math.pi * i / stacks, 2 * math.pi * (j % slices) / slices
    pos = torch.stack([torch.sin(th) * torch.cos(ph), torch.cos(th).expand(-1, slices + 1), torch.sin(th) * torch.sin(ph)], -1)
    uv = torch.stack([(j / slices).expand(stacks + 1, -1), (i / stacks).expand(-1, slices + 1)], -1).reshape(-1, 2)
    a = torch.arange(stacks, device=DEV)[:, None].expand(-1, slices)
    v00 = a * (slices + 1) + torch.arange(slices, device=DEV)[None, :]
    v01, v10, v11 = v00 + 1, v00 + slices + 1, v00 + slices + 2
    up, down = torch.stack([v00, v01, v11], -1), torch.stack([v00, v11, v10], -1)
    down = torch.where((a == stacks - 1)[..., None], torch.stack([v00, v01, v10], -1), down)
    quad = torch.stack([up, down], 2).reshape(-1, 3)
    keep = torch.ones(stacks, slices, 2, dtype=torch.bool, device=DEV)
    keep[0, :, 0] = False
    keep[-1, :, 0] = False
    pos = pos.reshape(-1, 3)
    return pos, _outward(pos, quad[keep.reshape(-1)]), uv


def _icosphere(subdiv):
    t = (1.0 + math.sqrt(5.0)) / 2.0
    v = torch.tensor([[-1, t, 0], [1, t, 0], [-1, -t, 0], [1, -t, 0], [0, -1, t], [0, 1, t], [0, -1, -t], [0, 1, -t],
                      [t, 0, -1], [t, 0, 1], [-t, 0, -1], [-t, 0, 1]], dtype=torch.float64, device=DEV)
    v = v / v.norm(dim=1, keepdim=True)
    f = torch.tensor([[0, 11, 5], [0, 5, 1], [0, 1, 7], [0, 7, 10], [0, 10, 11], [1, 5, 9], [5, 11, 4], [11, 10, 2],
                      [10, 7, 6], [7, 1, 8], [3, 9, 4], [3, 4, 2], [3, 2, 6], [3, 6, 8], [3, 8, 9], [4, 9, 5],
                      [2, 4, 11], [6, 2, 10], [8, 6, 7], [9, 8, 1]], device=DEV)
    for _ in range(subdiv):
        nv, nf = v.shape[0], f.shape[0]
        e = torch.cat([f[:, [0, 1]], f[:, [1, 2]], f[:, [2, 0]]])
        lo, hi = e.min(1).values, e.max(1).values
        uk, inv = torch.unique(lo * nv + hi, return_inverse=True)
        mid = v[uk // nv] + v[uk % nv]
        v = torch.cat([v, mid / mid.norm(dim=1, keepdim=True)])
        a, b, c = inv[:nf] + nv, inv[nf:2 * nf] + nv, inv[2 * nf:] + nv
        f = torch.stack([torch.stack([f[:, 0], a, c], 1), torch.stack([f[:, 1], b, a], 1),
                         torch.stack([f[:, 2], c, b], 1), torch.stack([a, b, c], 1)], 1).reshape(-1, 3)
    return v, _outward(v, f)


def _seam_split(pos, f):
    """Spherical UVs; the corners of faces across the seam duplicated with u + 1."""
    u = 0.5 + torch.atan2(pos[:, 2], pos[:, 0]) / (2 * math.pi)
    v = torch.arccos(pos[:, 1].clamp(-1, 1)) / math.pi
    fu = u[f]
    low = ((fu.max(1).values - fu.min(1).values) > 0.5)[:, None] & (fu < 0.5)
    src = f[low]
    f = f.clone()
    f[low] = pos.shape[0] + torch.arange(src.numel(), device=DEV)
    uv = torch.stack([torch.cat([u, u[src] + 1.0]), torch.cat([v, v[src]])], 1)
    return torch.cat([pos, pos[src]]), f, uv


def _displace(pos, gen, amp=0.1, waves=24):
    """Radius 1 + amp * a seeded smooth field of the direction (a few octaves of plane waves)."""
    k = torch.randn(waves, 3, generator=gen, device=DEV, dtype=torch.float64)
    k = k * (2.0 * 2.0 ** (torch.arange(waves, device=DEV) % 3))[:, None]
    ph = torch.rand(waves, generator=gen, device=DEV, dtype=torch.float64) * 2 * math.pi
    a = 0.5 ** (torch.arange(waves, device=DEV) % 3).double()
    s = torch.zeros(pos.shape[0], dtype=torch.float64, device=DEV)
    for i in range(waves):
        s = s + a[i] * torch.sin(pos @ k[i] + ph[i])
    return pos * (1.0 + amp * s / math.sqrt(waves))[:, None]


def _texture(gen, side, f16):
    t = torch.rand(side, side, 4, generator=gen, device=DEV)
    t[..., 3] = 0
    return t.half() if f16 else t


def _normal_map(gen, side, f16):
    x = torch.arange(side, device=DEV) * (2 * math.pi / side)
    c = torch.randn(4, generator=gen, device=DEV) * 0.15
    nx = c[0] * torch.sin(3 * x)[None, :] + c[1] * torch.cos(5 * x)[:, None]
    ny = c[2] * torch.cos(4 * x)[None, :] + c[3] * torch.sin(2 * x)[:, None]
    nx, ny = nx.expand(side, side).clamp(-0.6, 0.6), ny.expand(side, side).clamp(-0.6, 0.6)
    nz = torch.sqrt(1 - nx * nx - ny * ny)
    t = torch.stack([(nx + 1) / 2, (ny + 1) / 2, (nz + 1) / 2, torch.zeros_like(nx)], -1)
    return t.half() if f16 else t


def _mvp(eye, w, h, fovy=45.0, near=0.1, far=10.0):
    f = -eye / np.linalg.norm(eye)
    up = np.array([0.0, 1.0, 0.0]) if abs(f[1]) < 0.999 else np.array([1.0, 0.0, 0.0])
    s = np.cross(f, up)
    s /= np.linalg.norm(s)
    u = np.cross(s, f)
    look = np.eye(4)
    look[0, :3], look[1, :3], look[2, :3] = s, u, -f
    look[:3, 3] = -s @ eye, -u @ eye, f @ eye
    t = 1.0 / math.tan(math.radians(fovy) / 2)
    p = np.zeros((4, 4))
    # the shorter side takes the field of view, so that the whole object is seen
    p[0, 0], p[1, 1] = (t * h / w, -t) if w >= h else (t, -t * w / h)
    p[2, 2], p[2, 3], p[3, 2] = far / (near - far), near * far / (near - far), -1.0
    return (p @ look).astype(np.float32).reshape(16)


def _mesh(case, gen):
    if case["mesh"] == "ico":
        pos, f = _icosphere(case["n"])
        uv = None
        if case["shade"]:
            pos, f, uv = _seam_split(pos, f)
    else:
        pos, f, uv = _uv_sphere(case["n"], case["m"])
    col = torch.rand(pos.shape[0], 3, generator=gen, device=DEV) if case["shade"] == 0 else None
    m = types.SimpleNamespace(pos=_displace(pos, gen).float(), faces=f.int(), col=col,
                              uv=uv.float() if case["shade"] else None, tex=None, ntex=None)
    if case["shade"]:
        m.tex = _texture(gen, case["tex"], case["f16"])
        if case["shade"] == 3:
            m.ntex = _normal_map(gen, case["tex"], case["f16"])
    return m


def _mixed_sizes(case):
    """The ragged batch's sizes: (slices, stacks, resolution, texture side) per mesh, the same for every seed."""
    g, got = np.random.default_rng(1238), []
    for _ in range(case["views"]):
        faces = math.exp(g.uniform(math.log(case["n"]), math.log(case["m"])))
        bands = max(2, int(round(math.sqrt(faces / 4))))
        got.append((max(3, int(round(faces / (2 * bands)))), bands + 1, int(g.choice([128, 256, 512, 1024])),
                    int(g.choice([512, 1024, 2048]))))
    return got


def _inputs(case, seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed))
    g = np.random.default_rng(int(seed))
    if case["mesh"] == "mix":
        sizes = _mixed_sizes(case)
        meshes = [_mesh(dict(case, mesh="uv", n=a, m=b, tex=t), gen) for a, b, _, t in sizes]
        shapes = [(i, r, r) for i, (_, _, r, _) in enumerate(sizes)]
        ref = 512
    else:
        meshes = [_mesh(case, gen)]
        shapes = [(0, case["w"], case["h"])] * case["views"]
        ref = max(case["w"], case["h"])
    n, views, turn = len(shapes), [], g.uniform(0, 2 * math.pi)
    for i, (m, w, h) in enumerate(shapes):
        y = 1 - (2 * i + 1) / n if n > 1 else g.uniform(-0.5, 0.5)
        phi = turn + i * math.pi * (3 - math.sqrt(5))
        rho = math.sqrt(1 - y * y)
        views.append(types.SimpleNamespace(mvp=_mvp(3.0 * np.array([rho * math.cos(phi), y, rho * math.sin(phi)]), w, h),
                                           light=LIGHT, mesh=m, width=w, height=h))
    r = case["r_px"] / ref
    params = types.SimpleNamespace(K=case["K"], r=r, sigma=r / 7, delta=r, gamma=1e-4, edge_mode=case["edge"],
                                   shade_mode=case["shade"], texgrad_mode=case["texgrad"])
    if case["texgrad"] == 2:
        params.uv_jitter = tuple(float(x) for x in g.uniform(-0.5, 0.5, 2))
    target = []
    for _, w, h in shapes:   # a disc of about the outline, in noisy shades
        x = (torch.arange(w, device=DEV) + 0.5 - w / 2)[None, :]
        y = (torch.arange(h, device=DEV) + 0.5 - h / 2)[:, None]
        inside = (x * x + y * y < (0.43 * min(w, h) * float(g.uniform(0.95, 1.05))) ** 2).float()
        t = torch.rand(h, w, 4, generator=gen, device=DEV) * 0.6
        t[..., 3] = 1.0
        target.append((t * inside[..., None]).reshape(-1, 4))
    return meshes, views, params, torch.cat(target)


def prepare(case, seed):
    meshes, views, params, target = _inputs(case, seed)
    scene = PackedScene(meshes, DEV)
    s = types.SimpleNamespace(case=case, scene=scene, target=target, loss=torch.zeros(1, device=DEV))
    s.renderer = Renderer(scene, views, params, tile=case["tile"], schedule=case["schedule"])
    if case["kind"] == "texfit":
        _, s.ids = s.renderer.forward()
    if case["kind"] == "autograd":
        s.pos = scene.pos.clone().requires_grad_()
        s.col = None if scene.col is None else scene.col.clone().requires_grad_()
        s.tex = None if scene.tex is None else scene.tex.clone().requires_grad_()
    return s


def run(s):
    c, r = s.case, s.renderer
    if c["kind"] == "view":
        return {"out": r.forward(store_layers=False)[0]}
    if c["kind"] == "autograd":
        out = render(s.pos, s.col, s.tex, r, c["store"])
        loss = (out - s.target).square().sum()
        leaves = [t for t in (s.pos, s.col, s.tex) if t is not None]
        return {"out": out.detach(), "grads": list(torch.autograd.grad(loss, leaves))}
    if c["kind"] == "texfit":
        out = r.forward_from_layers(s.ids)
        s.loss.zero_()
        grad = r.l2_grad(out, s.target, loss=s.loss)
        gp, _, gt = r.backward(grad, ids=s.ids)
        return {"out": out, "loss": s.loss, "grads": [gp, gt]}
    s.loss.zero_()
    out, ids, grad = r.forward(store_layers=c["store"], target=s.target, loss=s.loss)
    got = r.backward(grad, ids=ids, camera=c["camera"], normal_map=c["shade"] == 3)
    return {"out": out, "ids": ids, "grad": grad, "loss": s.loss, "grads": [t for t in got if t is not None]}


def work(case):
    """Inputs read once, outputs written once; arithmetic of the hard layers of the covered
    pixels (57 % of a view): two layer evaluations of 50, one shaded layer of 110 and, with an
    adjoint, one back-propagated layer of 340 operations."""
    if case["mesh"] == "mix":
        each = [(2 * a * (b - 1), (a + 1) * (b + 1), t * t, r * r) for a, b, r, t in _mixed_sizes(case)]
        faces, verts, texels, px = (sum(x) for x in zip(*each))
    else:
        faces = 20 * 4 ** case["n"] if case["mesh"] == "ico" else 2 * case["n"] * (case["m"] - 1)
        verts = faces // 2 + 2 if case["mesh"] == "ico" else (case["n"] + 1) * (case["m"] + 1)
        texels, px = case["tex"] ** 2, case["views"] * case["w"] * case["h"]
    maps = 2 if case["shade"] == 3 else 1
    texel = 8 if case["f16"] else 16
    back = case["kind"] != "view"
    b = 12 * faces + verts * (24 if case["shade"] == 0 else 20) + texels * texel * maps + 16 * px
    if back:
        # target read; gradients of the positions and colours or texels
        b += 16 * px + verts * (24 if case["shade"] == 0 else 12) + texels * 16 * maps
    if case["kind"] == "step":
        b += 16 * px   # the pixel gradient comes back too
    if case["store"] and case["kind"] in ("step", "texfit"):
        b += 4 * case["K"] * px   # layer ids, written or read
    return {"bytes": b, "flops": 0.57 * px * (210 + (340 if back else 0))}


# ----------------------------------------------------------------------------
# the same results in 64 bits, in plain torch
# ----------------------------------------------------------------------------

def _cross(ax, ay, bx, by):
    return ax * by - ay * bx


class _View:
    """One view in float64: screen corners (sorted lexicographically per face, so that shared
    edges are computed alike), the K nearest layers of every pixel, and their colours."""

    def __init__(self, pos, faces, mvp, W, H, p):
        self.W, self.H, self.p = W, H, p
        S = max(W, H)
        self.r = float(np.float32(float(np.float32(p.r)) * S))
        self.sigma = float(np.float32(p.sigma)) * S
        self.S = S
        self.rho = max(1, int(math.floor(float(np.float32(p.delta)) * S + 0.5)))
        c = torch.cat([pos, torch.ones_like(pos[:, :1])], 1) @ mvp.view(4, 4).t()
        self.iw = 1.0 / c[:, 3]
        self.X = (c[:, 0] * self.iw + 1) * (0.5 * W)
        self.Y = (c[:, 1] * self.iw + 1) * (0.5 * H)
        self.z = c[:, 2] * self.iw
        with torch.no_grad():
            ok = (c[:, 3] > 1e-6) & (self.z >= 0) & (self.z <= 1)
            o = torch.argsort(self.Y[faces], dim=1, stable=True)
            f = torch.gather(faces, 1, o)
            o = torch.argsort(self.X[f], dim=1, stable=True)
            self.f = torch.gather(f, 1, o)
            X, Y = self.X[self.f], self.Y[self.f]
            A2 = _cross(X[:, 1] - X[:, 0], Y[:, 1] - Y[:, 0], X[:, 2] - X[:, 0], Y[:, 2] - Y[:, 0])
            self.live = ok[self.f].all(1) & (A2 != 0)

    def pair(self, fi, px, py, grad=False):
        """Signed distance, hard test, key and screen barycentrics of faces fi at points."""
        with torch.set_grad_enabled(grad):
            v = self.f[fi]
            X, Y = self.X[v], self.Y[v]
            A2 = _cross(X[:, 1] - X[:, 0], Y[:, 1] - Y[:, 0], X[:, 2] - X[:, 0], Y[:, 2] - Y[:, 0])
            s = torch.sign(A2)
            F, d2, t_, lam, inside = [], [], [], [None] * 3, torch.ones_like(s, dtype=torch.bool)
            for i, (a, b, sw) in enumerate(((0, 1, 1.0), (1, 2, 1.0), (0, 2, -1.0))):   # edge 2 runs 2 -> 0
                ex, ey = X[:, b] - X[:, a], Y[:, b] - Y[:, a]
                dx, dy = px - X[:, a], py - Y[:, a]
                c = _cross(ex, ey, dx, dy)
                L2 = ex * ex + ey * ey
                fn = s * sw * c
                lam[(i + 2) % 3] = fn / A2.abs()
                F.append(fn / L2.sqrt())
                t = ((dx * ex + dy * ey) / L2).clamp(0, 1)
                qx, qy = dx - t * ex, dy - t * ey
                d2.append(qx * qx + qy * qy)
                t_.append(t)
                ox, oy = sw * ex, sw * ey
                owns = torch.where(s > 0, (oy < 0) | ((oy == 0) & (ox > 0)), (oy > 0) | ((oy == 0) & (ox < 0)))
                inside &= (fn > 0) | ((fn == 0) & owns)
            F, d2, t_, lam = torch.stack(F, 1), torch.stack(d2, 1), torch.stack(t_, 1), torch.stack(lam, 1)
            e = torch.where(inside, F.argmin(1), d2.argmin(1))[:, None]
            out = torch.gather(d2, 1, e)[:, 0]
            dist = torch.where(inside, torch.gather(F, 1, e)[:, 0], -torch.where(inside, torch.ones_like(out), out).sqrt())
            t = torch.gather(t_, 1, e)[:, 0]
            zero = torch.zeros_like(t)
            e = e[:, 0]
            soft = torch.stack([torch.where(e == 1, zero, 1 - t), torch.where(e == 0, t, torch.where(e == 1, 1 - t, zero)),
                                torch.where(e == 0, zero, t)], 1)
            lam = torch.where(inside[:, None], lam, soft)
            key = torch.where(inside, 0.5 * (lam * self.z[v]).sum(1), 0.5 - 0.5 * dist / self.S)
        return dist, inside, key, lam

    @torch.no_grad()
    def layers(self, most=1 << 23):
        """[K, H W] face per pixel (-1 none) and its hard flag, nearest key first."""
        W, H, K = self.W, self.H, self.p.K
        X, Y = self.X[self.f], self.Y[self.f]
        lim = torch.zeros_like(X[:, 0])
        x0 = torch.maximum(torch.ceil(X.min(1).values - self.r - 0.5), lim).long()
        x1 = torch.minimum(torch.floor(X.max(1).values + self.r - 0.5), lim + W - 1).long()
        y0 = torch.maximum(torch.ceil(Y.min(1).values - self.r - 0.5), lim).long()
        y1 = torch.minimum(torch.floor(Y.max(1).values + self.r - 0.5), lim + H - 1).long()
        n = ((x1 - x0 + 1).clamp(min=0) * (y1 - y0 + 1).clamp(min=0)) * self.live
        ends = torch.cumsum(n, 0)
        total, at = int(ends[-1]), 0
        pix, keys, fs, hs = [], [], [], []
        while at < total:   # the faces whose pairs fill the next block
            f0 = int(torch.searchsorted(ends, at, right=True))
            f1 = max(f0 + 1, int(torch.searchsorted(ends, at + most, right=True)))
            cnt = n[f0:f1]
            fi = torch.repeat_interleave(torch.arange(f0, f0 + cnt.numel(), device=DEV), cnt)
            k = torch.arange(fi.numel(), device=DEV) - (ends[fi] - n[fi] - at)
            w = (x1 - x0 + 1)[fi]
            x, y = x0[fi] + k % w, y0[fi] + k // w
            dist, inside, key, _ = self.pair(fi, x + 0.5, y + 0.5)
            keep = dist >= -self.r
            pix.append((y * W + x)[keep])
            keys.append(key[keep])
            fs.append(fi[keep])
            hs.append(inside[keep])
            at += int(cnt.sum())
        ids = torch.full((K, H * W), -1, dtype=torch.long, device=DEV)
        hard = torch.zeros(K, H * W, dtype=torch.bool, device=DEV)
        if pix:
            pix, keys, fs, hs = (torch.cat(t) for t in (pix, keys, fs, hs))
            o = torch.argsort(keys, stable=True)   # pairs stand in face order: ties go to the smaller face
            o = o[torch.argsort(pix[o], stable=True)]
            pix, fs, hs = pix[o], fs[o], hs[o]
            first = torch.searchsorted(pix, pix)
            rank = torch.arange(pix.numel(), device=DEV) - first
            m = rank < K
            ids[rank[m], pix[m]] = fs[m]
            hard[rank[m], pix[m]] = hs[m]
        return ids, hard

    def mask(self, hard):
        """S^H and the edge mask E of every pixel."""
        SH = hard[0]
        if self.p.edge_mode:
            return SH, torch.full_like(SH, self.p.edge_mode == 1)
        img = SH.view(1, 1, self.H, self.W).float()
        k = 2 * self.rho + 1
        some = torch.nn.functional.max_pool2d(img, k, 1, self.rho) > 0
        gap = torch.nn.functional.max_pool2d(1 - img, k, 1, self.rho) > 0
        return SH, (some & gap).view(-1)


def _bilinear(tex, base, w, h, u, v):
    x, y = u * w - 0.5, v * h - 0.5
    x0, y0 = torch.floor(x.detach()), torch.floor(y.detach())
    fx, fy = (x - x0)[:, None], (y - y0)[:, None]
    xa, ya = x0.long() % w, y0.long() % h
    xb, yb = (xa + 1) % w, (ya + 1) % h
    at = lambda yy, xx: tex[base + yy * w + xx, :3]  # noqa: E731
    return ((1 - fx) * (1 - fy) * at(ya, xa) + fx * (1 - fy) * at(ya, xb) + (1 - fx) * fy * at(yb, xa) + fx * fy * at(yb, xb))


def _exact_view(pos, attr, faces, view, mesh, mvp, light, p, base):
    """RGBA [H W, 4] of one view, differentiable in pos, attr (colours, or texels), mvp, light."""
    V = _View(pos, faces, mvp, view.width, view.height, p)
    ids, hard = V.layers()
    SH, E = V.mask(hard)
    n = view.width * view.height
    want = ids >= 0
    want[0] &= E | SH
    want[1:] &= E
    k, pix = torch.nonzero(want, as_tuple=True)
    fi = ids[k, pix]
    px, py = (pix % view.width) + 0.5, torch.div(pix, view.width, rounding_mode="floor") + 0.5
    dist, _, _, lam = V.pair(fi, px, py, True)
    v = V.f[fi]
    q = lam * V.iw[v]
    b = q / q.sum(1, keepdim=True)
    D = torch.sigmoid(dist / V.sigma)
    if p.shade_mode == 0:
        C = (b[..., None] * attr["col"][v]).sum(1)
    else:
        uvf = mesh.uv.double()
        uv = (b[..., None] * uvf[v]).sum(1)
        th, tw = mesh.tex.shape[:2]
        C = _bilinear(attr["tex"], base, tw, th, uv[:, 0], uv[:, 1])
        if p.shade_mode >= 2:
            P = pos[faces]
            a = torch.linalg.cross(P[:, 1] - P[:, 0], P[:, 2] - P[:, 0])
            m = torch.zeros_like(pos).index_add(0, faces.reshape(-1), a[:, None].expand(-1, 3, -1).reshape(-1, 3))
            l = m.norm(dim=1, keepdim=True)
            nv = m / torch.where(l > 0, l, torch.ones_like(l))
            nn = torch.nn.functional.normalize((b[..., None] * nv[v]).sum(1), dim=1, eps=1e-30)
            if p.shade_mode == 3:
                o = faces[fi]
                e1, e2 = pos[o[:, 1]] - pos[o[:, 0]], pos[o[:, 2]] - pos[o[:, 0]]
                d1, d2 = uvf[o[:, 1]] - uvf[o[:, 0]], uvf[o[:, 2]] - uvf[o[:, 0]]
                det = (d1[:, 0] * d2[:, 1] - d2[:, 0] * d1[:, 1])[:, None]
                Tf = torch.where(det != 0, (e1 * d2[:, 1:] - e2 * d1[:, 1:]) / torch.where(det != 0, det, 1.0), 0.0)
                T = torch.nn.functional.normalize(Tf - nn * (nn * Tf).sum(1, keepdim=True), dim=1, eps=1e-30)
                B = torch.where(det < 0, -1.0, 1.0) * torch.linalg.cross(nn, T)
                t = 2 * _bilinear(attr["ntex"], base, tw, th, uv[:, 0], uv[:, 1]) - 1
                nn = torch.nn.functional.normalize(t[:, :1] * T + t[:, 1:2] * B + t[:, 2:] * nn, dim=1, eps=1e-30)
            C = C * (nn @ light).clamp(min=0)[:, None]
    Dk = torch.zeros(p.K, n, dtype=torch.float64, device=DEV).index_put((k, pix), D)
    Ck = torch.zeros(p.K, n, 3, dtype=torch.float64, device=DEV).index_put((k, pix), C)
    Ds = Dk.sum(0)
    rgb = (Dk[..., None] * Ck).sum(0) / torch.where(Ds > 0, Ds, torch.ones_like(Ds))[:, None]
    alpha = 1 - (1 - Dk).prod(0) if p.K > 1 else Dk[0]
    hardpix = torch.cat([torch.where(SH[:, None], Ck[0], 0.0), SH[:, None].double()], 1)
    return torch.where(E[:, None], torch.cat([rgb, alpha[:, None]], 1), hardpix)


def exact(case, seed):
    meshes, views, params, target = _inputs(case, seed)
    pos = [m.pos.double().requires_grad_() for m in meshes]
    attr = []
    for m in meshes:
        a = {} if m.col is None else {"col": m.col.double().requires_grad_()}
        for name in ("tex", "ntex"):
            t = getattr(m, name)
            if t is not None:
                a[name] = t.double().reshape(-1, 4).requires_grad_()
        attr.append(a)
    back = case["kind"] != "view"
    outs, grads, gm, gl, at = [], [], [], [], 0
    for view in views:
        i = view.mesh
        m = meshes[i]
        mvp = torch.tensor(view.mvp, dtype=torch.float64, device=DEV, requires_grad=True)
        light = torch.tensor(view.light, dtype=torch.float64, device=DEV, requires_grad=True)
        out = _exact_view(pos[i], attr[i], m.faces.long(), view, m, mvp, light, params, 0)
        g = 2 * (out.detach() - target[at:at + out.shape[0]].double())
        if back:
            out.backward(g)
            gm.append(mvp.grad)
            gl.append(light.grad if light.grad is not None else torch.zeros_like(light))
        at += out.shape[0]
        outs.append(out.detach())
        grads.append(g)
    out = torch.cat(outs)
    if not back:
        return {"out": out}
    planar = lambda ts: torch.cat([t.grad for t in ts]).t().contiguous()  # noqa: E731
    got = [planar(pos)]
    if case["shade"] == 0:
        got.append(planar([a["col"] for a in attr]))
    else:
        # the inverse-UV gradient is a sampling rule of its own; an FP16 leaf's gradient is rounded by torch
        rounded = case["f16"] and case["kind"] == "autograd"
        got.append(None if case["texgrad"] == 2 or rounded else torch.cat([a["tex"].grad for a in attr]))
    if case["kind"] == "step":
        if case["camera"]:
            rows = torch.stack(gm)
            rows[:, 8:12] = 0   # depth only orders the layers
            got += [rows, torch.stack(gl)]
        if case["shade"] == 3:
            got.append(torch.cat([a["ntex"].grad for a in attr]))
    # the loss is added up in launch order, its last bits differ from run to run
    res = {"out": out, "ids": None, "grad": torch.cat(grads), "loss": None, "grads": got}
    return {k: v for k, v in res.items() if k in ("out", "grads") or (case["kind"] == "step" and k == "grad")}
