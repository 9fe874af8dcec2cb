"""Brick builds of crowded bricks: bricks in many chunks of entries, whose chunk
counts are added up in one or two levels, and cells of more objects than the
16-bit counts hold.  Each grid equals the oracle's bit for bit."""
import numpy as np
import pytest

import oracle

from test_gpu_bricks import _soup
from test_gpu_parity import assert_grid_equal, dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _check(s, cull=False, label=""):
    import paper_2403_10647_gb300 as pg
    o = oracle.build_grid(s.verts, s.tris, s.lam, cull=True) if cull else oracle.build_grid(s.verts, s.tris, s.lam,
                                                                                        method="counting")
    c = pg.Context(0, cull=cull)
    try:
        c.profile(True)
        for _ in range(2):   # the second build has the first one's buffers
            assert_grid_equal(c.build(dev(s.verts, torch.float32), dev(s.tris, torch.int32), s.lam), o, label)
        assert "cell_scan" in c.kernel_stats(), (o.NO, s.n)
    finally:
        c.close()
    return o


# one brick of 8 x 8 x 8 cells: chunk counts on both sides of the change to two
# levels (32 chunks of 1,024 entries), and groups of 32 and 64 with a short last one
@pytest.mark.parametrize("n,edge", [(32_768, 0.95), (32_769, 0.95), (300_001, 0.4), (1_100_000, 0.35)])
@pytest.mark.parametrize("cull", [False, True])
def test_one_crowded_brick_matches_oracle(n, edge, cull):
    s = _soup(n, (1, 1, 1), edge, 71, 500.0 / n)
    o = _check(s, cull, str(n))
    assert list(o.plan.res) == [8, 8, 8]


def test_crowded_bricks_among_others_match_oracle():
    """Some bricks in many chunks, some in a few, some empty, also in a batch."""
    import paper_2403_10647_gb300 as pg
    a = _soup(60_000, (30, 29, 31), 2.0, 72, 4.0)
    v = a.verts.reshape(-1, 3, 3).copy()
    v[5_000:50_000] = v[5_000:50_000] % np.float32(3.0) + np.float32(11.0)   # 45,000 of them in a box of 3 units
    v[50_000:55_000] = v[50_000:55_000] % np.float32(2.0) + np.float32(20.0)
    import scenes
    s = scenes.Scene("crowds", v.reshape(-1, 3), a.tris, 4.0)
    _check(s)
    one = _soup(150_000, (1, 1, 1), 0.5, 73, 500.0 / 150_000)
    c = pg.Context(0)
    try:
        c.profile(True)
        batch = [s, one, _soup(5, (1, 2, 3), 0.5, 74, 8.0), one]
        grids = c.build_batched([(dev(m.verts, torch.float32), dev(m.tris, torch.int32), m.lam) for m in batch])
        assert "cell_scan" in c.kernel_stats()
        for k, (m, g) in enumerate(zip(batch, grids)):
            assert_grid_equal(g, oracle.build_grid(m.verts, m.tris, m.lam, method="counting"), f"mesh {k}")
    finally:
        c.close()


@pytest.mark.parametrize("cells,n,cull", [(60, 700_000, False), (60, 700_000, True), (220, 900_000, False)])
def test_many_cells_beyond_16_bits_match_oracle(cells, n, cull):
    s = _soup(n, (1, 1, 1), 0.7, 75, (cells - 2) / n)
    o = _check(s, cull, str(cells))
    assert (np.diff(o.G) >= 65_535).sum() > 4
