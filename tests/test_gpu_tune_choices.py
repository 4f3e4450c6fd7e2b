"""The autotuner decides between launches that differ: FP64 grids keep the sign of the x lines (their x-pass has no cp.async
variant), and schedules that run as the same merged stages are not exchanged for one another (at 16 every candidate runs as
one stage of radix 16)."""
import pytest

from paper_2009_03762_gb300 import microstructure as M

pytestmark = pytest.mark.gpu


def test_choices_that_change_nothing_are_not_made():
    from paper_2009_03762_gb300 import gfp
    g = gfp.Grid(64, 16, 16)
    g.set_phases(*M.random_field(64, 16, 16, seed=1))
    sch = gfp.scheme("AFB_R", "PCD", "FP64")
    before = g.get_plans(gfp.FP64)
    for _ in range(12):  # by noise alone each would hold with odds of one half
        assert g.tune(sch, 1)[0] >= 0
        assert g.get_plans(gfp.FP64) == before
    g.close()
