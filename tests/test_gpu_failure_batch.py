"""Failure detection inside a batched solve: a wait that runs out in a slot's inner iterations ends that slot and is reported, and
the batch solves correctly afterwards."""
import numpy as np
import pytest

from paper_2009_03762_gb300 import microstructure as M

pytestmark = pytest.mark.gpu


def test_timeout_of_a_batched_solve():
    from paper_2009_03762_gb300 import gfp
    L = gfp.lib()
    sch = gfp.scheme("AFB_R", "PCD", "MIXED")
    grids = []
    for shape in ((16, 12, 64), (12, 8, 16)):  # the first with TMA-fed z-passes, the second without
        g = gfp.Grid(*shape)
        g.set_phases(*M.random_field(*shape, seed=3))
        grids.append(g)
    grids[0].set_tiles(gfp.MIXED, [2, 4, -8])
    assert L.gfp_set_fault_injection(1, 1) == 0
    try:
        bad = gfp.Batch(grids, sch)  # the graph's kernels are captured with the injection
        with pytest.raises(gfp.GfpError) as e:
            bad.solve(1e-8, 320)
        bad.close()
    finally:
        assert L.gfp_set_fault_injection(1, 0) == 0
    assert e.value.code == -6
    good = gfp.Batch(grids, sch)
    C, _, rc = good.solve(1e-8, 5000)
    good.close()
    assert rc == 0
    for g, c in zip(grids, C):
        ref, _, rc = g.effective_stiffness(gfp.scheme("AFB_R", "PCD", "FP64"), 1e-8, 5000)
        assert rc == 0
        assert np.linalg.norm(c - ref) <= 1e-6 * np.linalg.norm(ref)
        g.close()
