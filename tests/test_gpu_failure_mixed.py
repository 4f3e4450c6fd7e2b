"""Failure detection of the TMA-fed z-passes that the mixed solve takes by default at n3 = 256 and 512 (and by choice at 64): a
bounded wait that is made to run out is reported, and the grid solves correctly afterwards."""
import numpy as np
import pytest

from paper_2009_03762_gb300 import microstructure as M

pytestmark = pytest.mark.gpu

E = [0.0, 0.002, 0.0, 0.003, 0.0, -0.001]


@pytest.fixture
def injection():
    from paper_2009_03762_gb300 import gfp
    assert gfp.lib().gfp_set_fault_injection(1, 1) == 0
    yield gfp
    assert gfp.lib().gfp_set_fault_injection(1, 0) == 0


@pytest.mark.parametrize("shape,tiles", [((64, 64, 256), None), ((64, 64, 512), None), ((18, 6, 512), [2, 4, -8]),
                                         ((16, 12, 64), [2, 4, -8])])
def test_timeout_of_a_mixed_solve(injection, shape, tiles):
    gfp = injection
    lam, mu = M.random_field(*shape, seed=8)
    g = gfp.Grid(*shape)
    g.set_phases(lam, mu)
    if tiles:
        g.set_tiles(gfp.MIXED, tiles)
    sch = gfp.scheme("AFB_R", "PCD", "MIXED")
    assert g.solve(sch, E, 1e-8, 5000).status == -6
    assert gfp.lib().gfp_set_fault_injection(1, 0) == 0
    r = g.solve(sch, E, 1e-8, 5000)
    eps = g.strain()
    r64 = g.solve(gfp.scheme("AFB_R", "PCD", "FP64"), E, 1e-8, 5000)
    eps64 = g.strain()
    g.close()
    assert r.converged and r64.converged
    assert np.linalg.norm(eps - eps64) <= 1e-6 * np.linalg.norm(eps64)
