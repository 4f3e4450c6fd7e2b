"""Shapes next to the scratch limit of the allocation-free solve: those whose spectrum, tables and residual partials fit into
8 MiB with z-tiles of four columns run, also where the default tiles are narrower (more partials)."""
import numpy as np
import pytest

from paper_2009_03762_gb300 import microstructure as M

pytestmark = pytest.mark.gpu

E = [0.01, 0.0, -0.002, 0.0, 0.003, 0.0]


@pytest.mark.parametrize("shape", [(192, 216, 4), (324, 512, 1), (216, 384, 2), (1024, 162, 1), (108, 512, 3)])
def test_shapes_that_just_fit(shape):
    import torch
    from paper_2009_03762_gb300 import gfp
    n1, n2, n3 = shape
    lam, mu = M.random_field(n1, n2, n3, seed=n1)
    lam_t, mu_t = (torch.from_numpy(np.ascontiguousarray(f)).cuda() for f in (lam, mu))
    eps_t = torch.empty((6, n3, n2, n1), dtype=torch.float64, device="cuda")
    rc, r = gfp.solve_noalloc(lam_t, mu_t, eps_t, gfp.scheme("ACD"), E, tol=0.0, maxit=6)
    g = gfp.Grid(n1, n2, n3)
    g.set_phases(lam, mu)
    ref = g.solve(gfp.scheme("ACD"), E, 0.0, 6)
    eps = g.strain()
    g.close()
    assert rc == ref.status == -4 and r.iters == ref.iters == 6
    assert np.linalg.norm(eps_t.cpu().numpy() - eps) <= 1e-12 * np.linalg.norm(eps)


@pytest.mark.parametrize("shape", [(64, 64, 64), (216, 256, 4), (1024, 192, 1)])
def test_shapes_beyond_the_limit(shape):
    import torch
    from paper_2009_03762_gb300 import gfp
    n1, n2, n3 = shape
    one = torch.ones((n3, n2, n1), dtype=torch.float64, device="cuda")
    eps = torch.empty((6, n3, n2, n1), dtype=torch.float64, device="cuda")
    with pytest.raises(gfp.GfpError) as e:
        gfp.solve_noalloc(one, one, eps, gfp.scheme("ACD"), E)
    assert e.value.code == -2
