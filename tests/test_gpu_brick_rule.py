"""Which builds go by bricks: those whose bricks hold enough pairs.  Scenes on
both sides of the rule, single, culled and batched, each grid equal to the
oracle's bit for bit whichever way it is placed."""
import numpy as np
import pytest

import oracle
import scenes

from test_gpu_bricks import _soup
from test_gpu_parity import assert_grid_equal, dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _scene(n, cells, lam, flat=False, seed=81):
    """A soup of n triangles with corners in boxes of `cells` cells a side."""
    e = cells / (lam * n) ** (1 / 2 if flat else 1 / 3)
    return _soup(n, (1, 1, 0 if flat else 1), e, seed, lam)


# name: scene, bricks pay for its box build, for its culled build (None: not built)
CASES = {
    "dense": (lambda: _scene(60_000, 6, 8.0), True, True),                    # 7,650 pairs per brick
    "near": (lambda: _scene(130_000, 3, 64.0), True, False),                  # 200
    "sparse": (lambda: _scene(70_000, 4.5, 512.0), False, False),             # 60
    "flat_dense": (lambda: _scene(60_000, 12, 8.0, flat=True), True, True),   # 1,270
    "flat_sparse": (lambda: _scene(240_000, 4, 64.0, flat=True), False, False),   # 27
    # few cells, sorted in one or two passes: enough pairs beyond so many per entry
    "18_cells": (lambda: _scene(600_000, 1, 8 / 600_000), False, True),
    "64_cells_few": (lambda: _scene(500_000, 1, 62 / 500_000), False, True),
    "64_cells": (lambda: _scene(700_000, 3, 62 / 700_000), True, True),
    "343_cells_few": (lambda: _scene(500_000, 1, 340 / 500_000), False, True),
    "343_cells": (lambda: _scene(500_000, 3, 340 / 500_000), True, True),
    "4096_cells_few": (lambda: _scene(600_000, 1.1, 4_090 / 600_000), False, True),
    "4096_cells": (lambda: _scene(600_000, 3, 4_090 / 600_000), True, True),
    "line_z_few": (lambda: _soup(600_000, (0, 0, 1), 0.012, 82, 1_000 / 600_000), False, False),
    "line_z": (lambda: _soup(200_000, (0, 0, 1), 0.1, 82, 1_000 / 200_000), True, True),
}


@pytest.mark.parametrize("cull", [False, True])
@pytest.mark.parametrize("name", sorted(CASES))
def test_builds_by_bricks_where_they_pay(name, cull):
    import paper_2403_10647_gb300 as pg
    make, box, culled = CASES[name]
    s = make()
    o = oracle.build_grid(s.verts, s.tris, s.lam, method="counting", cull=cull)
    c = pg.Context(0, cull=cull)
    try:
        c.profile(True)
        assert_grid_equal(c.build(dev(s.verts, torch.float32), dev(s.tris, torch.int32), s.lam), o, name)
        assert ("cell_scan" in c.kernel_stats()) == (culled if cull else box), (o.NO, o.plan.res)
    finally:
        c.close()


@pytest.mark.parametrize("name", ["dense", "flat_sparse"])
def test_batches_by_bricks_where_they_pay(name):
    import paper_2403_10647_gb300 as pg
    s, few = CASES[name][0](), _scene(500, 2, 4.0)
    batch = [s, few, s]
    c = pg.Context(0)
    try:
        c.profile(True)
        grids = c.build_batched([(dev(m.verts, torch.float32), dev(m.tris, torch.int32), m.lam) for m in batch])
        assert ("cell_scan" in c.kernel_stats()) == CASES[name][1]
        for k, (m, g) in enumerate(zip(batch, grids)):
            assert_grid_equal(g, oracle.build_grid(m.verts, m.tris, m.lam, method="counting"), f"mesh {k}")
    finally:
        c.close()


@pytest.mark.parametrize("cull", [False, True])
def test_statistics_tell_brick_kernels_apart(cull):
    import paper_2403_10647_gb300 as pg
    pairs, bricks = {"bucket_split", "local_sort"}, {"brick_split", "brick_count", "cell_scan", "brick_fill"}
    if cull:
        pairs, bricks = pairs | {"cull_emit"}, bricks | {"brick_cull"}
    c = pg.Context(0, cull=cull)
    try:
        for name, there, absent in (("dense", bricks, pairs), ("sparse", pairs, bricks)):
            s = CASES[name][0]()
            c.profile(True)
            c.build(dev(s.verts, torch.float32), dev(s.tris, torch.int32), s.lam)
            names = set(c.kernel_stats())
            assert there <= names and not (absent & names), (name, names)
    finally:
        c.close()


@pytest.mark.parametrize("name,launches", [("dense", 1), ("near", 2)])   # 0.5M and 8M cells: one pass, two
def test_scan_launches_are_counted(name, launches):
    import paper_2403_10647_gb300 as pg
    s = CASES[name][0]()
    c = pg.Context(0)
    try:
        c.profile(True)
        c.build(dev(s.verts, torch.float32), dev(s.tris, torch.int32), s.lam)
        assert c.kernel_stats()["cell_scan"]["launches"] == launches
    finally:
        c.close()
