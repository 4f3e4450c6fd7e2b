"""FP64 passes on 64-bit block fixed point: every register length on every axis, lengths without a register plan,
fields beyond the comfortable exponent range, infinities, and the Green step's choice of arithmetic, against the FP64
oracle.

Tolerance: an iteration's transforms and Green step each round at a few 2^-53 of the stress, and a handful of
iterations adds them up: 1e-12 relative leaves a factor of about a thousand."""
import numpy as np
import pytest

from oracle import gfp_oracle as O
from paper_2009_03762_gb300 import microstructure as M

pytestmark = pytest.mark.gpu

REL = 1e-12
E = [0.01, -0.004, 0.002, 0.003, -0.001, 0.005]


@pytest.fixture(scope="module")
def gfp():
    from paper_2009_03762_gb300 import gfp as G
    G.lib()
    return G


def _rel(a, b):
    return np.linalg.norm(np.asarray(a) - np.asarray(b)) / np.linalg.norm(b)


def _strain(gfp, lam, mu, op, iters, E=E, tiles=None, **kw):
    n3, n2, n1 = lam.shape
    g = gfp.Grid(n1, n2, n3)
    g.set_phases(lam, mu)
    if tiles:
        g.set_tiles(gfp.FP64, tiles)
    r = g.solve(gfp.scheme(op, "PCD", "FP64", **kw), E, 0.0, iters)
    eps = g.strain()
    g.close()
    return r, eps


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("n", [32, 64, 96, 128, 192, 256, 512, 6, 27, 162])
def test_every_length_on_every_axis(gfp, n, axis):
    shape = [3, 2, 4]
    shape[axis] = n
    lam, mu = M.random_field(*shape, seed=n + axis, lo=0.05, hi=50.0)
    op = ("AFB_R", "ACD", "F")[axis]
    _, eps = _strain(gfp, lam, mu, op, 4)
    assert _rel(eps, O.solve(lam, mu, op, E, max_iters_exact=4, disc="PCD").eps) <= REL


@pytest.mark.parametrize("tiles", [[1, 1, 1], [3, 2, 2], [5, 9, 3], [16, 8, 4], [2, 4, -4]])
def test_tile_widths(gfp, tiles):
    """Widths with and without an instance of their own, on a ragged half spectrum (17 columns)."""
    lam, mu = M.random_field(32, 32, 64, seed=7)
    _, eps = _strain(gfp, lam, mu, "AFB_R", 3, tiles=tiles)
    assert _rel(eps, O.solve(lam, mu, "AFB_R", E, max_iters_exact=3, disc="PCD").eps) <= REL


@pytest.mark.parametrize("shape", [(32, 32, 32), (12, 18, 9)])
@pytest.mark.parametrize("op,k,ke", [("AFB_R", -500, -400), ("ACD", -500, 0), ("DGO", -840, 0), ("DGO", 830, 0)])
def test_power_of_two_scaling_is_exact(gfp, shape, op, k, ke):
    """Moduli times 2^k and a mean strain times 2^ke scale the strain by 2^ke, bit for bit, also where the stress's
    lines leave the range that is converted directly.  (The finite-difference schemes form 1 / (mu (lambda + 2 mu)), so
    their moduli stay above 2^-511.)"""
    lam, mu = M.random_field(*shape, seed=3)
    kw = {"dgo_m": 2} if op == "DGO" else {}
    _, a = _strain(gfp, lam, mu, op, 4, **kw)
    _, b = _strain(gfp, lam * 2.0 ** k, mu * 2.0 ** k, op, 4, E=[v * 2.0 ** ke for v in E], **kw)
    np.testing.assert_array_equal(a * 2.0 ** ke, b)


@pytest.mark.parametrize("shape", [(32, 32, 32), (12, 18, 9)])
def test_overflowing_stress_is_reported(gfp, shape):
    lam, mu = M.random_field(*shape, seed=3)
    r, _ = _strain(gfp, lam * 1e300, mu * 1e300, "AFB_R", 4, E=[v * 1e12 for v in E])
    assert r.status == -5


@pytest.mark.parametrize("shape", [(32, 32, 32), (12, 18, 9)])
def test_reference_media_beyond_the_fixed_point_green_step(gfp, shape):
    """lambda_H < -1.5 mu_H (|(lambda + mu) / (lambda + 2 mu)| > 1) takes the FP64 Green step; lambda_H = 0 and
    lambda_H < 0 the fixed-point one."""
    _, mu = M.random_field(*shape, seed=5)
    for ratio in (-1.6, -0.4, 0.0):
        lam = ratio * mu
        _, eps = _strain(gfp, lam, mu, "AFB_R", 4)
        assert _rel(eps, O.solve(lam, mu, "AFB_R", E, max_iters_exact=4, disc="PCD").eps) <= REL
