"""The work that programs have this library do, as measurable cases.

A case is one call of a public entry point on one input: whole builds of single
meshes over the sizes of the scenes this repository ships (a few hundred
triangles to 10 million, up to a billion <object, cell> pairs), batched builds,
culled builds, builds from and to host memory, and a burst of rebuild requests
to the serving loop.  The scenes follow the recipes of ``scenes`` drawn with
torch on the device (a 10M-triangle scene takes seconds in numpy), plus a
connected surface with shared vertices in mesh order, the kind of mesh that a
deforming model hands over every frame.

How many cells and pairs a build has depends on its triangles, so that two
random scenes of one size have outputs of different lengths.  A seed therefore
gives every case the same triangles in another order (other object ids, another
memory layout), turned to other axes and in other units (a power of two): all
inputs and outputs differ, their sizes and the work do not.

Every output is a whole number except the grid metadata (origin, far corner and
cells per unit length, float32), which ``exact`` gives in 64 bits.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2403_10647_gb300 as pg

# ---- the cases ---------------------------------------------------------------


def listed():
    return [
        # a handful of props or a physics proxy: launches and host round trips
        {"name": "uniform_tiny", "kind": "build", "scene": "uniform", "n": 1_023, "lam": 2.0},
        # the 100,000-triangle soup that every round of a small program rebuilds
        {"name": "uniform_1e5", "kind": "build", "scene": "uniform", "n": 100_000, "lam": 2.0},
        # a deforming indexed surface (cloth, terrain, skin), rebuilt per frame
        {"name": "surface_1e6", "kind": "build", "scene": "surface", "n": 985_606, "lam": 4.0},
        # crowded cells: 1% of the triangles span thousands of cells
        {"name": "nonhomogeneous_1e6", "kind": "build", "scene": "nonhomogeneous", "n": 1_000_000, "lam": 4.0},
        # the headline scene: a building of 10 million triangles, 2e8 pairs
        {"name": "architectural_1e7", "kind": "build", "scene": "architectural", "n": 10_000_000, "lam": 8.0},
        # the largest rebuild that the serving pool holds: about 1e9 pairs
        {"name": "nonhomogeneous_7e6", "kind": "build", "scene": "nonhomogeneous", "n": 7_300_019, "lam": 4.0},
        # 64 meshes of a scene graph in one call, 1e3 to 2e6 triangles each
        {"name": "batch_64", "kind": "batch", "meshes": 64, "lo": 1_000, "hi": 2_000_000, "lam": 4.0},
        # 64 small meshes in one call: what batching is for
        {"name": "batch_64_small", "kind": "batch", "meshes": 64, "lo": 10, "hi": 20_000, "lam": 4.0},
        # culled grids: where most box pairs are false, and where most are true
        {"name": "cull_nonhomogeneous_1e6", "kind": "cull", "scene": "nonhomogeneous", "n": 1_000_000, "lam": 4.0},
        {"name": "cull_architectural_2e6", "kind": "cull", "scene": "architectural", "n": 2_499_983, "lam": 8.0},
        # a program whose meshes and grids live in (pinned) host memory
        {"name": "host_architectural_1e6", "kind": "host", "scene": "architectural", "n": 1_000_000, "lam": 8.0},
        # a burst of rebuild requests to the serving loop, each with its frame's vertices
        {"name": "serve_burst", "kind": "serve", "meshes": 6, "lo": 10_000, "hi": 1_000_000, "requests": 12},
    ]


def draw(rng):
    """One more case: every kind with its sizes log-uniform over its range."""

    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    lam = rng.choice([1.0, 2.0, 4.0, 8.0])
    kind = rng.choice(["build"] * 6 + ["batch", "batch", "cull", "cull", "host", "serve"])
    if kind == "batch":
        lo = size(10, 2_000)
        hi = lo * size(5, 500)
        return {"kind": kind, "meshes": rng.randint(2, 64), "lo": lo, "hi": hi, "lam": rng.choice([2.0, 4.0])}
    if kind == "serve":
        return {"kind": kind, "meshes": rng.randint(1, 8), "lo": 10_000, "hi": size(20_000, 1_000_000),
                "requests": rng.randint(1, 16)}
    scene = rng.choice(["uniform", "surface", "nonhomogeneous", "architectural"])
    top = {"build": 10_000_000, "cull": 3_000_000, "host": 2_000_000}[kind]
    if scene == "nonhomogeneous":   # a hundred pairs per triangle
        top = min(top, 4_000_000)
        lam = rng.choice([1.0, 2.0, 4.0])
    return {"kind": kind, "scene": scene, "n": size(300, top), "lam": lam}


# ---- scenes ---------------------------------------------------------------------


SCENE_SEED = 20_403   # the triangles of every scene; a case's own seed orders and turns them


class _Draw:
    """Seeded random tensors on one device."""

    def __init__(self, seed, device):
        self.device = device
        self.g = torch.Generator(device=device)
        self.g.manual_seed(int(seed))

    def uniform(self, lo, hi, *shape):
        return torch.rand(*shape, generator=self.g, device=self.device) * (hi - lo) + lo

    def normal(self, *shape):
        return torch.randn(*shape, generator=self.g, device=self.device)

    def loguniform(self, lo, hi, *shape):
        return torch.exp(self.uniform(math.log(lo), math.log(hi), *shape))

    def ints(self, lo, hi, n):
        return torch.randint(lo, hi, (n,), generator=self.g, device=self.device)

    def directions(self, n):
        d = self.normal(n, 3)
        return d / d.norm(dim=1, keepdim=True).clamp_min(1e-12)

    def pick(self, n, k):
        """A mask of n with k random entries set."""
        m = torch.zeros(n, dtype=torch.bool, device=self.device)
        m[self.order(n)[:k]] = True
        return m

    def order(self, n):
        return torch.randperm(n, generator=self.g, device=self.device)


def _soup(o, c, e1, e2):
    """Separate triangles of centroids c and edges e1, e2, in the order that o draws."""
    n = c.shape[0]
    p = o.order(n)
    c, e1, e2 = c[p], e1[p], e2[p]
    v0 = c - (e1 + e2) / 3.0
    verts = torch.stack([v0, v0 + e1, v0 + e2], dim=1).reshape(3 * n, 3).contiguous()
    tris = torch.arange(3 * n, dtype=torch.int32, device=c.device).reshape(n, 3)
    return verts, tris


def _uniform(d, o, n):
    return _soup(o, d.uniform(0.0, 1.0, n, 3), d.uniform(-0.01, 0.01, n, 3), d.uniform(-0.01, 0.01, n, 3))


def _nonhomogeneous(d, o, n):
    """Centroids in a box at the 1M-triangle soup's density, 99% small
    triangles, 1% large."""
    side = 100.0 * (n / 1e6) ** (1.0 / 3.0)
    large = d.pick(n, int(round(0.01 * n)))

    def edges():
        small = torch.exp(d.normal(n) * 0.5 + math.log(0.05))
        return d.directions(n) * torch.where(large, d.uniform(5.0, 40.0, n), small)[:, None]

    return _soup(o, d.uniform(0.0, side, n, 3), edges(), edges())


def _architectural(d, o, n):
    """A building at the 10M-triangle one's density: 5% wall and floor quads
    (indexed, two triangles each), the rest small clutter in Gaussian blobs."""
    f = (n / 1e7) ** (1.0 / 3.0)
    size = torch.tensor([200.0 * f, 50.0 * f, 200.0 * f], device=d.device)
    nquad = int(round(0.025 * n))
    axis = d.ints(0, 3, nquad)
    u, w = (axis + 1) % 3, (axis + 2) % 3
    su = torch.minimum(d.loguniform(0.5, 20.0, nquad), size[u])
    sw = torch.minimum(d.loguniform(0.5, 20.0, nquad), size[w])
    pu, pw = d.uniform(0.0, 1.0, nquad) * (size[u] - su), d.uniform(0.0, 1.0, nquad) * (size[w] - sw)
    plane = d.uniform(0.0, 1.0, nquad) * size[axis]
    corners = torch.zeros(nquad, 4, 3, device=d.device)
    row = torch.arange(nquad, device=d.device)
    for k, (a, b) in enumerate(((0, 0), (1, 0), (1, 1), (0, 1))):
        corners[row, k, axis] = plane
        corners[row, k, u] = pu + a * su
        corners[row, k, w] = pw + b * sw
    corners = corners[o.order(nquad)]
    base = 4 * torch.arange(nquad, dtype=torch.int32, device=d.device)
    fan = torch.tensor([[0, 1, 2], [0, 2, 3]], dtype=torch.int32, device=d.device)
    qtris = (base[:, None, None] + fan).reshape(2 * nquad, 3)
    nclut = n - 2 * nquad
    blobs = max(4, int(round(2000 * n / 1e7)))
    centre = d.uniform(0.0, 1.0, blobs, 3) * size
    c = centre[d.ints(0, blobs, nclut)] + 1.5 * d.normal(nclut, 3)
    c = torch.minimum(c.clamp_min(0.0), size)
    e1 = d.directions(nclut) * d.loguniform(0.01, 0.3, nclut)[:, None]
    e2 = d.directions(nclut) * d.loguniform(0.01, 0.3, nclut)[:, None]
    cverts, ctris = _soup(o, c, e1, e2)
    verts = torch.cat([corners.reshape(4 * nquad, 3), cverts])
    return verts.contiguous(), torch.cat([qtris, ctris + 4 * nquad]).contiguous()


def _surface(d, o, n):
    """n triangles of a wavy sheet of shared vertices, row by row from a row
    that o draws."""
    cols = max(1, int(math.sqrt(n / 2)))
    rows = (n + 2 * cols - 1) // (2 * cols)
    y, x = torch.meshgrid(torch.arange(rows + 1, device=d.device), torch.arange(cols + 1, device=d.device),
                          indexing="ij")
    ph = d.uniform(0.0, 6.28, 4)
    step = 10.0 / cols
    px, py = x * step, y * step
    pz = 0.8 * torch.sin(1.3 * px + ph[0]) * torch.cos(0.9 * py + ph[1]) + 0.2 * torch.sin(4.1 * px + 3.3 * py + ph[2])
    verts = torch.stack([px, py, pz], dim=-1).reshape(-1, 3)
    verts = (verts + 0.1 * step * d.normal(verts.shape[0], 3)).float().contiguous()
    v = (y[:-1, :-1] * (cols + 1) + x[:-1, :-1]).reshape(-1, 1)
    quad = torch.cat([v, v + 1, v + cols + 2, v, v + cols + 2, v + cols + 1], dim=1)
    tris = quad.reshape(-1, 3)[:n].to(torch.int32)
    return verts, tris.roll(2 * cols * int(o.ints(0, rows, 1)), 0).contiguous()


_SCENES = {"uniform": _uniform, "surface": _surface, "nonhomogeneous": _nonhomogeneous,
           "architectural": _architectural}


def _sizes(case):
    """Triangle counts of a batch or pool, spread log-uniformly over its range
    (the golden-ratio sequence: every seed has the same sizes)."""
    m, lo, hi = case["meshes"], math.log(case["lo"]), math.log(case["hi"])
    return [int(round(math.exp(lo + (hi - lo) * ((0.5 + 0.6180339887498949 * k) % 1.0)))) for k in range(m)]


def _turned(o, verts, axes=True):
    """The vertices in other units and, unless told not to, on other axes."""
    if axes:
        verts = verts[:, o.order(3)]
    return (verts * 2.0 ** int(o.ints(-3, 4, 1))).contiguous()


def _meshes(case, seed, device):
    """[(verts, tris, lam)] of a case's meshes."""
    d, o = _Draw(SCENE_SEED, device), _Draw(seed, device)
    kind = case["kind"]
    if kind == "batch":
        parts = [("nonhomogeneous", n, case["lam"]) for n in _sizes(case)]
    elif kind == "serve":   # the pool alternates the two scene kinds
        parts = [("nonhomogeneous", n, 4.0) if k % 2 else ("architectural", n, 8.0)
                 for k, n in enumerate(_sizes(case))]
    else:
        parts = [(case["scene"], case["n"], case["lam"])]
    out = []
    for scene, n, lam in parts:
        verts, tris = _SCENES[scene](d, o, n)
        # the culling test's roundings depend on the order of the axes
        out.append((_turned(o, verts, axes=kind != "cull"), tris, lam))
    return out


# ---- preparation, one pass, its work --------------------------------------------------


def prepare(case, seed):
    meshes = _meshes(case, seed, "cuda")
    kind = case["kind"]
    if kind == "serve":
        # tuning at registration is off: it may settle on other kernels each time
        server = pg.Server(0, tune_meshes=False)
        ids = [server.register(*m) for m in meshes]
        # every request brings its mesh's vertices of that frame from pinned
        # host memory: here the mesh turned to other axes
        o = _Draw(seed + 1, "cuda")
        frames = []
        for k in range(case["requests"]):
            m = k % len(ids)
            frames.append((ids[m], _turned(o, meshes[m][0]).cpu().pin_memory()))
        return {"kind": kind, "server": server, "frames": frames}
    state = {"kind": kind, "ctx": pg.Context(0, cull=kind == "cull"), "meshes": meshes}
    if kind == "host":
        v, t, lam = meshes[0]
        hv, ht = v.cpu().pin_memory(), t.cpu().pin_memory()
        cells, refs, _ = state["ctx"].build_host(hv, ht, lam)
        # output buffers with room for other frames of the mesh, kept by the program
        out = [torch.empty(x.numel() + x.numel() // 8, dtype=torch.int32).pin_memory() for x in (cells, refs)]
        state["meshes"] = [(hv, ht, lam)]
        state["out"] = out
    return state


def _grid(cells, refs, info):
    return {"cells": cells, "refs": refs, "res": list(info.res), "lo": list(info.lo), "hi": list(info.hi),
            "scale": list(info.scale)}


def run(state):
    kind = state["kind"]
    if kind == "serve":
        server = state["server"]
        tickets = [server.submit(m, verts=v) for m, v in state["frames"]]
        grids = [server.wait(t) for t in tickets]
        return [(g.cells, g.refs) for g in grids]
    if kind == "batch":
        b = state["ctx"].build_batched(state["meshes"])
        return {"cells": b.cells, "refs": b.refs, "cells_offsets": np.array(b.cells_offsets),
                "refs_offsets": np.array(b.refs_offsets)}
    verts, tris, lam = state["meshes"][0]
    if kind == "host":
        return _grid(*state["ctx"].build_host(verts, tris, lam, *state["out"]))
    g = state["ctx"].build(verts, tris, lam)
    return _grid(g.cells, g.refs, g.info)


def _plan(verts, tris, lam, n):
    """Scene bounds and the density rule in 64 bits: lo, hi, extent, res."""
    p = verts[tris.reshape(-1).long()].double()
    lo, hi = p.amin(dim=0), p.amax(dim=0)
    e = hi - lo
    flat = e <= 0
    k = (lam * n / torch.where(flat, torch.ones_like(e), e).prod()) ** (1.0 / max(1, int((~flat).sum())))
    res = torch.where(flat, torch.ones_like(e), torch.ceil(e * k).clamp(1, 65535))
    return lo, hi, e, res


def exact(case, seed):
    if case["kind"] in ("serve", "batch"):
        return None   # whole numbers throughout
    verts, tris, lam = _meshes(case, seed, "cuda")[0]
    lo, hi, e, res = _plan(verts, tris, lam, case["n"])
    scale = torch.where(e > 0, res / e, torch.zeros_like(e))
    return {"cells": None, "refs": None, "res": [None] * 3, "lo": lo.tolist(), "hi": hi.tolist(),
            "scale": scale.tolist()}


# Pairs that culling keeps, as a fraction of the box pairs: measured on the
# 1M-triangle soup and on the building; the others are small triangles.
_KEPT = {"nonhomogeneous": 0.056, "architectural": 0.58, "uniform": 0.75, "surface": 0.75}


def _grid_size(scene, n, lam):
    """(vertices, cells, pairs) of a scene of this kind."""
    d = _Draw(SCENE_SEED, "cuda" if torch.cuda.is_available() else "cpu")
    verts, tris = _SCENES[scene](d, d, n)
    lo, _, e, res = _plan(verts, tris, lam, n)
    scale = torch.where(e > 0, res / e, torch.zeros_like(e))
    p = verts[tris.long()].double()
    clo = torch.minimum(torch.floor((p.amin(dim=1) - lo) * scale), res - 1)
    chi = torch.minimum(torch.floor((p.amax(dim=1) - lo) * scale), res - 1)
    return verts.shape[0], int(res.prod()), float((chi - clo + 1).prod(dim=1).sum())


def work(case):
    """Bytes: vertices and triangles read once, cells and refs written once.
    No floating-point operation counts: the path is comparisons and copies."""
    kind = case["kind"]
    if kind == "batch":
        parts = [("nonhomogeneous", n, case["lam"]) for n in _sizes(case)]
    elif kind == "serve":
        sizes = _sizes(case)
        parts = [(("architectural", sizes[k], 8.0) if k % 2 == 0 else ("nonhomogeneous", sizes[k], 4.0))
                 for k in (r % len(sizes) for r in range(case["requests"]))]
    else:
        parts = [(case["scene"], case["n"], case["lam"])]
    total = 0.0
    known = {}
    for scene, n, lam in parts:
        if (scene, n, lam) not in known:
            known[scene, n, lam] = _grid_size(scene, n, lam)
        nverts, ncells, pairs = known[scene, n, lam]
        if kind == "cull":
            pairs *= _KEPT[scene]
        total += 12.0 * nverts + 12.0 * n + 4.0 * (ncells + 1) + 4.0 * pairs
    return {"bytes": total, "flops": 0.0}
