"""Brick builds: radix passes over (brick, object) entries, then per brick the
objects of every cell (split, count, scan, fill).  Each grid equals the
oracle's bit for bit where the bricks can go wrong: grids thinner than a
brick along any axis, grids that end inside a brick, cells and bricks too
crowded for one stage, bricks in many chunks, a cell beyond the 16-bit counts,
and batches of such meshes."""
import numpy as np
import pytest

import oracle
import scenes

from test_gpu_parity import assert_grid_equal, dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _soup(n, box, edge, seed, lam, giants=0, crowd=0):
    """n triangles of edges up to `edge` in `box`, `giants` of which span the
    whole box, and `crowd` tiny ones inside one cell, in random order."""
    g = np.random.Generator(np.random.Philox(seed))
    box = np.asarray(box, np.float64)
    edge = np.minimum(edge, box)
    c = g.random((n, 3)) * (box - edge)
    v = np.stack([c, c + edge * g.random((n, 3)), c + edge * g.random((n, 3))], 1)
    v[:giants] = np.stack([np.zeros(3), box, np.array([box[0], 0.0, box[2]])])
    if crowd:
        v = np.concatenate([v, np.broadcast_to(box * [0.503, 0.507, 0.511], (crowd, 3, 3))])
    v = v[g.permutation(len(v))]
    t = np.arange(3 * len(v), dtype=np.int32).reshape(-1, 3)
    return scenes.Scene("bricks", v.reshape(-1, 3).astype(np.float32), t, lam)


SCENES = {
    # 8 x 8 x 8 bricks, ragged at every face, up to 100 objects per cell
    "cube": lambda: _soup(30_000, (10, 9.3, 11.1), 2.5, 1, 4.0),
    # thin and flat grids: other brick shapes
    "thin_z": lambda: _soup(30_000, (60, 55, 0.9), 8.0, 2, 2.0),
    "flat_z": lambda: _soup(20_000, (60, 55, 0), 9.0, 3, 4.0),
    "flat_x": lambda: _soup(20_000, (0, 60, 55), 9.0, 4, 4.0),
    "flat_y": lambda: _soup(20_000, (60, 0, 55), 9.0, 5, 4.0),
    "line_x": lambda: _soup(20_000, (60, 0, 0), 3.0, 6, 2.0),
    "line_z": lambda: _soup(20_000, (0, 0, 60), 3.0, 7, 2.0),
    # every cell holds thousands: windows of entries, bricks in chunks
    "few_cells": lambda: _soup(40_000, (1, 1.1, 0.9), 0.9, 8, 0.02),
    # one cell of 70,000 objects: 16-bit counts are not enough
    "big_cell": lambda: _soup(20_000, (10, 10, 10), 0.4, 9, 1.0, giants=60, crowd=70_000),
}


@pytest.mark.parametrize("name", sorted(SCENES))
def test_brick_builds_match_oracle(name):
    import paper_2403_10647_gb300 as pg
    s = SCENES[name]()
    o = oracle.build_grid(s.verts, s.tris, s.lam, method="counting")
    c = pg.Context(0)
    try:
        c.profile(True)
        for _ in range(2):   # the second build has the first one's buffers
            g = c.build(dev(s.verts, torch.float32), dev(s.tris, torch.int32), s.lam)
            assert_grid_equal(g, o, name)
        assert "brick_count" in c.kernel_stats(), (o.NO, s.n)
        if name == "big_cell":
            assert np.diff(o.G).max() > 65_535
    finally:
        c.close()


@pytest.mark.parametrize("name", ["cube", "thin_z", "flat_z", "flat_x", "line_z", "few_cells", "soup"])
def test_culled_brick_builds_match_oracle(name):
    """Culled brick builds: the same test decides, whichever pairs reach it
    (boxes of a lane and of the warp, planes that miss most of a box)."""
    import paper_2403_10647_gb300 as pg
    s = scenes.nonhomogeneous_soup(70_000, seed=31, extent=30.0) if name == "soup" else SCENES[name]()
    o = oracle.build_grid(s.verts, s.tris, s.lam, cull=True)
    c = pg.Context(0, cull=True)
    try:
        c.profile(True)
        assert_grid_equal(c.build(dev(s.verts, torch.float32), dev(s.tris, torch.int32), s.lam), o, name)
        assert "cell_scan" in c.kernel_stats()
    finally:
        c.close()


def test_brick_batch_matches_oracle():
    import paper_2403_10647_gb300 as pg
    empty = scenes.Scene("empty", np.zeros((0, 3), np.float32), np.zeros((0, 3), np.int32), 4.0)
    batch = [empty, SCENES["thin_z"](), SCENES["big_cell"](), empty, _soup(3, (1, 2, 3), 0.5, 21, 8.0),
             SCENES["flat_x"](), SCENES["line_z"](), empty]
    c = pg.Context(0)
    try:
        c.profile(True)
        grids = c.build_batched([(dev(s.verts, torch.float32), dev(s.tris, torch.int32), s.lam) for s in batch])
        assert "brick_count" in c.kernel_stats()
        for k, (s, g) in enumerate(zip(batch, grids)):
            assert_grid_equal(g, oracle.build_grid(s.verts, s.tris, s.lam, method="counting"), f"mesh {k}")
    finally:
        c.close()


# cells on both sides of the scan's changes of tile; `crowd`: one cell beyond 16 bits
@pytest.mark.parametrize("lam,crowd", [(50.0, 0), (54.0, 70_000), (414.0, 0), (430.0, 0), (95.0, 70_000)])
def test_cell_scan_sizes_match_oracle(lam, crowd):
    import paper_2403_10647_gb300 as pg
    s = _soup(20_000, (10, 9.3, 11.1), 0.5, 41, lam, giants=2, crowd=crowd)
    o = oracle.build_grid(s.verts, s.tris, s.lam, method="counting")
    c = pg.Context(0)
    try:
        c.profile(True)
        assert_grid_equal(c.build(dev(s.verts, torch.float32), dev(s.tris, torch.int32), s.lam), o, str(lam))
        assert "cell_scan" in c.kernel_stats()
    finally:
        c.close()


@pytest.mark.parametrize("lam", [30.0, 200.0])
def test_cell_scan_of_a_batch_matches_oracle(lam):
    """Slices shorter than a warp's words, between long ones that a warp lies in."""
    import paper_2403_10647_gb300 as pg
    batch = [_soup(k, (1, 2, 3), 0.5, 50 + k, 8.0) for k in (3, 1, 40)] + [_soup(20_000, (10, 9.3, 11.1), 0.7, 42, lam)]
    batch += [_soup(k, (2, 1, 3), 0.5, 60 + k, 5.0) for k in (2, 300)] + [_soup(22_000, (9, 9.3, 8), 0.7, 43, lam)]
    c = pg.Context(0)
    try:
        c.profile(True)
        grids = c.build_batched([(dev(s.verts, torch.float32), dev(s.tris, torch.int32), s.lam) for s in batch])
        assert "cell_scan" in c.kernel_stats()
        for k, (s, g) in enumerate(zip(batch, grids)):
            assert_grid_equal(g, oracle.build_grid(s.verts, s.tris, s.lam, method="counting"), f"mesh {k}")
    finally:
        c.close()
