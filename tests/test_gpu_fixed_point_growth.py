"""Lines that grow as far as a line can, in the FP64 passes' fixed-point transforms: modes of equal real and imaginary part
that do not vary along the tested axis, so that every layer adds elements of one phase, on lengths whose schedules scale down by
less than the plain rule.  An overflow would wreck the strain; the bar is that of test_gpu_fixed_point."""
import numpy as np
import pytest

from oracle import gfp_oracle as O

pytestmark = pytest.mark.gpu

E = [0.01, -0.004, 0.002, 0.003, -0.001, 0.005]


@pytest.mark.parametrize("axis", [1, 2])
@pytest.mark.parametrize("n", [243, 432, 486, 729, 864, 972])
def test_lines_of_one_phase(n, axis):
    from paper_2009_03762_gb300 import gfp
    shape = [8, 2, 2]
    shape[axis] = n
    n1, n2, n3 = shape
    x = 2.0 * np.pi * np.arange(n1) / n1
    f = 1.0 + 0.4 * np.cos(x + 0.25 * np.pi) + 0.2 * np.cos(2.0 * x + 0.25 * np.pi)
    m = np.ascontiguousarray(np.broadcast_to(f, (n3, n2, n1)))
    for op in ("AFB_R", "ACD"):
        g = gfp.Grid(n1, n2, n3)
        g.set_phases(0.57 * m, 0.385 * m)
        g.solve(gfp.scheme(op, "PCD", "FP64"), E, 0.0, 4)
        eps = g.strain()
        g.close()
        ref = O.solve(0.57 * m, 0.385 * m, op, E, max_iters_exact=4, disc="PCD").eps
        assert np.linalg.norm(eps - ref) <= 1e-12 * np.linalg.norm(ref)
