"""Culled brick builds on grids of 20,000 cells along one axis, crossed by oblique
triangles thousands of cells long: there the bound on a cell's distance from a
triangle's plane rests on its rounding terms, not on its constant slack.
Each grid equals the oracle's bit for bit."""
import numpy as np
import pytest

import oracle
import scenes

from test_gpu_parity import assert_grid_equal, dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _long(axis, width, seed):
    """32 triangles with corners anywhere in a box of 20,000 x width x 7 units, half
    of them nearly along a line, and 2,000 small ones, along the given axis."""
    g = np.random.Generator(np.random.Philox(seed))
    box = np.array([20_000.0, width, 7.0])
    big = g.random((32, 3, 3)) * box
    big[:16, 2] = 0.5 * (big[:16, 0] + big[:16, 1]) + g.random((16, 3)) * 0.3
    c = g.random((2_000, 1, 3)) * (box - 2.0)
    v = np.concatenate([big, c + 2.0 * g.random((2_000, 3, 3)), np.stack([np.zeros((3, 3)), np.tile(box, (3, 1))])])
    v = np.roll(v[g.permutation(len(v))], axis, axis=2).reshape(-1, 3).astype(np.float32)
    return scenes.Scene("long", v, np.arange(len(v), dtype=np.int32).reshape(-1, 3), float(box.prod() / (len(v) // 3)))


@pytest.mark.parametrize("axis,width", [(0, 9.0), (1, 9.0), (2, 9.0), (0, 40.0)])
def test_culled_long_grids_match_oracle(axis, width):
    import paper_2403_10647_gb300 as pg
    s = _long(axis, width, 91 + axis)
    o = oracle.build_grid(s.verts, s.tris, s.lam, method="counting", cull=True)
    assert o.plan.res[axis] > 19_000
    c = pg.Context(0, cull=True)
    try:
        c.profile(True)
        assert_grid_equal(c.build(dev(s.verts, torch.float32), dev(s.tris, torch.int32), s.lam), o, str((axis, width)))
        assert "brick_cull" in c.kernel_stats()
    finally:
        c.close()
