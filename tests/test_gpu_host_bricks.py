"""Builds from and to host memory that go by bricks, whose cells are copied out
while the refs are still being written: into buffers of the exact size, pinned
and pageable, of both placements in turn, and into buffers that are too small."""
import ctypes

import numpy as np
import pytest

import oracle

from test_gpu_brick_rule import _scene

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

MARK = -77


def _call(c, s, cells, refs):
    from paper_2403_10647_gb300 import _lib
    info = _lib.GridInfo()
    v, t = torch.from_numpy(s.verts), torch.from_numpy(s.tris)
    c._bind_stream()
    rc = c._lib.grid_build_host(c._h, v.data_ptr(), v.shape[0], t.data_ptr(), t.shape[0], float(s.lam),
                                cells.data_ptr(), cells.numel(), refs.data_ptr(), refs.numel(), ctypes.byref(info))
    return rc, info


@pytest.mark.parametrize("cull", [False, True])
@pytest.mark.parametrize("pinned", [False, True])
def test_host_builds_by_bricks(cull, pinned):
    import paper_2403_10647_gb300 as pg
    from paper_2403_10647_gb300 import _lib
    s, small = _scene(60_000, 6, 8.0), _scene(3_000, 2, 4.0)
    o = oracle.build_grid(s.verts, s.tris, s.lam, method="counting", cull=cull)
    os = oracle.build_grid(small.verts, small.tris, small.lam, method="counting", cull=cull)

    def buf(n):
        b = torch.full((n,), MARK, dtype=torch.int32)
        return b.pin_memory() if pinned else b

    c = pg.Context(0, cull=cull)
    try:
        c.profile(True)
        for scene, want in ((s, o), (small, os), (s, o)):
            cells, refs = buf(want.G.size), buf(want.refs.size)
            rc, info = _call(c, scene, cells, refs)
            assert rc == _lib.GRID_OK and info.nrefs == want.NO
            assert np.array_equal(cells.numpy(), want.G) and np.array_equal(refs.numpy(), want.refs)
        assert "brick_fill" in c.kernel_stats()
        for scene, want in ((s, o), (small, os)):
            for short_cells, short_refs in ((0, 1), (1, 0), (1, 1)):
                cells, refs = buf(want.G.size - short_cells), buf(want.refs.size - short_refs)
                rc, info = _call(c, scene, cells, refs)
                assert rc == _lib.GRID_ENOSPC
                assert (info.ncells + 1, info.nrefs) == (want.G.size, want.refs.size)
                assert (cells == MARK).all() and (refs == MARK).all(), (short_cells, short_refs)
        cells, refs = buf(o.G.size + 5), buf(o.refs.size + 7)   # more room than the grid takes
        rc, _ = _call(c, s, cells, refs)
        assert rc == _lib.GRID_OK
        assert np.array_equal(cells.numpy()[:-5], o.G) and (cells[-5:] == MARK).all()
        assert np.array_equal(refs.numpy()[:-7], o.refs) and (refs[-7:] == MARK).all()
    finally:
        c.close()
