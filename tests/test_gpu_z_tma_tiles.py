"""TMA-fed z-tiles of every width, mixed precision, at every length with a register plan, against the FP64 solve (the bar of the
mixed solve, 1e-6 relative): tiles of 8 columns are swizzled at some lengths only."""
import numpy as np
import pytest

from paper_2009_03762_gb300 import microstructure as M

pytestmark = pytest.mark.gpu

E = [0.0, 0.002, 0.0, 0.003, 0.0, -0.001]


@pytest.mark.parametrize("n3", [32, 64, 96, 128, 192, 256])
def test_tma_tiles(n3):
    from paper_2009_03762_gb300 import gfp
    lam, mu = M.random_field(18, 12, n3, seed=1)  # 10 columns: a full and a ragged tile of 8
    g = gfp.Grid(18, 12, n3)
    g.set_phases(lam, mu)
    assert g.solve(gfp.scheme("AFB_R", "PCD", "FP64"), E, 1e-8, 5000).converged
    ref = g.strain()
    for cols in (2, 4, 8):
        g.set_tiles(gfp.MIXED, [2, 4, -cols])
        assert g.solve(gfp.scheme("AFB_R", "PCD", "MIXED"), E, 1e-8, 5000).converged, cols
        assert np.linalg.norm(g.strain() - ref) <= 1e-6 * np.linalg.norm(ref), cols
    g.close()
