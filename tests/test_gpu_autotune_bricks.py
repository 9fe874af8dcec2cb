"""The autotuners on scenes that build by bricks: what they are compared with is
the placement that sorted pairs would take at the scene's density."""
import pytest

from test_gpu_brick_rule import _scene
from test_gpu_parity import dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

# pairs per cell: up to 6 sorted pairs end in the hybrid, beyond in radix passes and extraction
SCENES = {"hybrid": (lambda: _scene(130_000, 3, 64.0), True), "chain": (lambda: _scene(60_000, 6, 8.0), False)}


@pytest.mark.parametrize("name", sorted(SCENES))
@pytest.mark.parametrize("batched", [False, True])
def test_other_sort_end_of_brick_builds(name, batched):
    import paper_2403_10647_gb300 as pg
    make, hybrid = SCENES[name]
    s = make()
    mesh = (dev(s.verts, torch.float32), dev(s.tris, torch.int32), s.lam)
    c = pg.Context(0)
    try:
        g = c.build(*mesh)
        assert (g.info.nrefs <= 6 * g.info.ncells) == hybrid
        c.profile(True)
        if batched:   # the batch tuner's other candidates are all brick builds
            r = c.autotune_batched([mesh, mesh], reps=1)
            st = c.kernel_stats()
            assert "brick_fill" in st
            assert ("local_sort" in st) == hybrid and ("extract" in st) == (not hybrid), st.keys()
        else:
            r = c.autotune(*mesh, reps=1)
            st = c.kernel_stats()
            assert "brick_fill" in st
            # pairs written to memory first (EMIT) end the same way
            if r["pair_gen"] == "fused":
                assert ("local_sort" in st) == hybrid and ("extract" in st) == (not hybrid), st.keys()
        assert r["times_ms"]["other_sort_end"] > 0
        if r["local_bits"]:
            assert r["local_bits"] == (-2 if hybrid else -1)
        h = c.build(*mesh)
        assert torch.equal(g.cells, h.cells) and torch.equal(g.refs, h.refs)
    finally:
        c.close()
