"""Real-space FP64 residual of the mixed solve (integer sums for the averaged stencils) against a NumPy FP64
evaluation of the same stencils on the returned strain.

The kernel rounds r to FP32 (relative 2^-24 per value) and adds |r|^2 over at most 16 planes in FP32 (16 x 2^-24 of
the sum), so eta agrees within 0.5 (2 + 16 + 3) 2^-24 = 6.3e-7 relative; the bar is 1e-6.
"""
import numpy as np
import pytest

from paper_2009_03762_gb300 import microstructure as M

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gfp():
    from paper_2009_03762_gb300 import gfp as G
    G.lib()
    return G


def _diff(f, ax, op):
    """Derivative of f [n3][n2][n1] along physical axis ax (array axis 2 - ax)."""
    if op == "CD":
        return 0.5 * (np.roll(f, -1, 2 - ax) - np.roll(f, 1, 2 - ax))
    others = [a for a in range(3) if a != ax]
    if op == "ACD":
        d = np.roll(f, -1, 2 - ax) - np.roll(f, 1, 2 - ax)
        for a in others:
            d = np.roll(d, -1, 2 - a) + np.roll(d, 1, 2 - a)
        return d / 8.0
    d = np.roll(f, -1, 2 - ax) - f
    for a in others:
        d = np.roll(d, -1, 2 - a) + d
    return d / 4.0


def _eta(lam, mu, eps, op, h):
    tr = eps[0] + eps[1] + eps[2]
    s = 2.0 * mu * eps
    s[:3] += lam * tr
    pairs = [(0, 5, 4), (5, 1, 3), (4, 3, 2)]
    r2 = sum(np.sum(sum(_diff(s[c], j, op) for j, c in enumerate(row)) ** 2) for row in pairs)
    t = s.reshape(6, -1).sum(axis=1)
    return np.sqrt(lam.size * r2) / h / np.sqrt((t[:3] ** 2).sum() + 2.0 * (t[3:] ** 2).sum())


@pytest.mark.parametrize("op", ["AFB_R", "AHC", "ACD", "CD"])
@pytest.mark.parametrize("dims", [(6, 3, 2), (32, 8, 16), (36, 9, 18), (72, 12, 36)])
@pytest.mark.parametrize("field", ["mixed", "rising", "falling", "tiny"])
def test_residual_matches_numpy(gfp, op, dims, field):
    n1, n2, n3 = dims
    lam, mu = M.random_field(n1, n2, n3, seed=4)
    lam, mu = np.array(lam, dtype=np.float64), np.array(mu, dtype=np.float64)
    z = np.arange(n3).reshape(n3, 1, 1)
    if field == "rising":  # the largest stress of a tile grows from plane to plane
        w = 2.0 ** (z % 16)
    elif field == "falling":
        w = 2.0 ** (-(z % 16))
    else:
        w = np.ones((n3, 1, 1)) * (2.0 ** -50 if field == "tiny" else 1.0)
    lam, mu = lam * w, mu * w
    E = [0.1, 0.0, -0.2, 0.0, 0.3, 0.05]
    h = 0.3 if n1 == 36 else 0.5  # the outputs' factor 1 / (4h): any number, or a power of two
    g = gfp.Grid(n1, n2, n3, h)
    g.set_phases(lam, mu)
    r = g.solve(gfp.scheme(op, "PCD", "MIXED"), E, 1e-14, 1)
    ref = _eta(lam, mu, g.strain().reshape(6, n3, n2, n1), op, h)
    assert abs(r.residual - ref) <= 1e-6 * ref
