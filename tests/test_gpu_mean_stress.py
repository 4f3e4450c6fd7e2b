"""Mean stress of FP64 solves on layered cells, whose voxels' stresses repeat so that rounding errors would add up instead of
averaging out: against the exactly rounded sum (math.fsum).

With lambda = 0 and a uniform unit shear the stress of a voxel is 2 mu, exactly, and the number of voxels is a power of
two: a compensated sum, off by about 2^-106 of the total, gives the exactly rounded mean."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,seed", [((64, 64, 128), 18), ((64, 64, 128), 45), ((64, 64, 128), 52), ((32, 32, 512), 28),
                                        ((32, 32, 512), 38), ((32, 32, 32), 1)])
@pytest.mark.parametrize("comp", [1, 3])
def test_layers_sum_exactly(shape, seed, comp):
    from paper_2009_03762_gb300 import gfp
    n1, n2, n3 = shape
    rng = np.random.default_rng(seed)
    vals = rng.uniform(1.0, 2.0, n3 // 16)
    layer = vals[rng.integers(0, vals.size, n3)]
    mu = np.repeat(0.5 * layer, n1 * n2).reshape(n3, n2, n1)
    E = [0.0] * 6
    E[comp] = 1.0
    g = gfp.Grid(n1, n2, n3)
    g.set_phases(np.zeros_like(mu), mu)
    r = g.solve(gfp.scheme("AFB_R"), E, 0.0, 1)  # the first iteration leaves the uniform strain
    np.testing.assert_array_equal(g.strain()[comp], 1.0)
    g.close()
    expected = np.zeros(6)
    expected[comp] = math.fsum(np.repeat(layer, n1 * n2)) / mu.size
    np.testing.assert_array_equal(r.sigma_mean, expected)
