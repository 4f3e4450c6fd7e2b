"""Radix schedules whose neighbouring stages run merged (radices 6, 9, 12 and 18 besides 2, 3, 4, 8 and 16), on lengths
without a register plan, in FP64 and mixed precision, against the FP64 oracle."""
import numpy as np
import pytest

from oracle import gfp_oracle as O
from paper_2009_03762_gb300 import microstructure as M

pytestmark = pytest.mark.gpu

E = [0.01, -0.004, 0.002, 0.003, -0.001, 0.005]


@pytest.fixture(scope="module")
def gfp():
    from paper_2009_03762_gb300 import gfp as G
    G.lib()
    return G


def _rel(a, b):
    return np.linalg.norm(np.asarray(a) - np.asarray(b)) / np.linalg.norm(b)


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("n", [2, 3, 4, 9, 12, 18, 24, 36, 48, 81, 108, 144, 216, 243, 324, 576, 729, 1024])
def test_default_schedules(gfp, n, axis):
    """FP64: 4 iterations to 1e-12 (a few 2^-53 per pass, see test_gpu_fixed_point); mixed: the solve to 1e-6."""
    shape = [4, 3, 2]
    shape[axis] = n
    lam, mu = M.random_field(*shape, seed=n + axis)
    g = gfp.Grid(*shape)
    g.set_phases(lam, mu)
    g.solve(gfp.scheme("AFB_R", "PCD", "FP64"), E, 0.0, 4)
    ref = O.solve(lam, mu, "AFB_R", E, max_iters_exact=4, disc="PCD")
    assert _rel(g.strain(), ref.eps) <= 1e-12
    r = g.solve(gfp.scheme("AFB_R", "PCD", "MIXED"), E, 1e-8, 5000)
    eps = g.strain()
    r64 = g.solve(gfp.scheme("AFB_R", "PCD", "FP64"), E, 1e-8, 5000)
    assert r.converged and r64.converged
    assert _rel(eps, g.strain()) <= 1e-6
    g.close()


@pytest.mark.parametrize("plan", [[2] * 5 + [3], [3, 2, 2, 2, 2, 2], [2, 3, 16], [8, 3, 4], [4, 3, 8], [3, 4, 2, 4]])
def test_explicit_schedules_of_96_times_1(gfp, plan):
    """Every order of merging that a schedule can ask for, on an axis that runs it (the residual's transforms use the
    schedule of every axis in mixed precision)."""
    n = int(np.prod(plan))
    shape = (n, 3, 9) if n != 96 else (96, 3, 9)
    lam, mu = M.random_field(*shape, seed=11)
    g = gfp.Grid(*shape)
    g.set_phases(lam, mu)
    for prec in (gfp.FP64, gfp.MIXED):
        p = g.get_plans(prec) if prec == gfp.FP64 else [plan, [3], [3, 3]]
        p[0] = plan
        g.set_plans(prec, p)
    r = g.solve(gfp.scheme("AFB_R", "PCD", "MIXED"), E, 1e-8, 5000)
    eps = g.strain()
    r64 = g.solve(gfp.scheme("AFB_R", "PCD", "FP64"), E, 1e-8, 5000)
    assert r.converged and r64.converged
    assert _rel(eps, g.strain()) <= 1e-6
    g.close()
