"""The launch shapes that grids take by default, and the z-pass of 512 rows, in mixed precision: against the FP64 GPU solve (the bar of the mixed solve, 1e-6 relative)."""
import numpy as np
import pytest

from paper_2009_03762_gb300 import microstructure as M

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gfp():
    from paper_2009_03762_gb300 import gfp as G
    G.lib()
    return G


def _rel(a, b):
    return np.linalg.norm(np.asarray(a) - np.asarray(b)) / np.linalg.norm(b)


def _check(gfp, shape, tiles=None):
    n1, n2, n3 = shape
    lam, mu = M.random_field(*shape, seed=n1 + n2)
    E = [0.0, 0.002, 0.0, 0.003, 0.0, -0.001]
    g = gfp.Grid(*shape)
    g.set_phases(lam, mu)
    if tiles:
        g.set_tiles(gfp.MIXED, tiles)
    r = g.solve(gfp.scheme("AFB_R", "PCD", "MIXED"), E, 1e-8, 5000)
    assert r.converged
    eps = g.strain()
    r64 = g.solve(gfp.scheme("AFB_R", "PCD", "FP64"), E, 1e-8, 5000)
    assert r64.converged
    assert _rel(eps, g.strain()) <= 1e-6
    assert _rel(r.sigma_mean, r64.sigma_mean) <= 1e-6
    g.close()


@pytest.mark.parametrize("n1", [16, 18, 32, 54])  # 9, 10, 17 and 28 columns of the half spectrum
def test_tall_tiles(gfp, n1):
    _check(gfp, (n1, 6, 512), [2, 4, -8])


@pytest.mark.parametrize("shape", [(64, 64, 256), (64, 64, 512), (32, 512, 8), (512, 8, 8), (192, 12, 8), (8, 8, 512)])
def test_default_shapes(gfp, shape):
    """On both sides of the rules for the z tiles (TMA from 304 tiles on) and the x and y widths."""
    _check(gfp, shape)
