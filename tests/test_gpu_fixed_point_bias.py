"""Rounding of the FP64 passes has no place of its own: the solve of a translated cell is the translated solve, up to rounding
errors that are as large at the voxels beside the origin as anywhere.

Two solves' errors differ by a random field.  Beside the origin and beside its translate 2 x 27 voxels x 3 shear components are
looked at: for normal errors the largest of them stays below 5 rms (1 in 10^4 runs), and 8 rms leaves room for errors that vary
over the cell.  A shift that truncates adds half a unit of one sign to every mode, and the inverse transforms gather these at
those voxels: sqrt(N) / 2 units against an rms of a few."""
import pytest

pytestmark = pytest.mark.gpu


def _smooth(n3, n2, n1, power, seed):
    import torch
    gen = torch.Generator(device="cuda").manual_seed(seed)
    w = torch.randn(n3, n2, n1, dtype=torch.float64, device="cuda", generator=gen)
    k = [torch.minimum(torch.arange(n, device="cuda"), n - torch.arange(n, device="cuda")).double() for n in (n3, n2, n1)]
    kk = (k[0][:, None, None] ** 2 + k[1][None, :, None] ** 2 + k[2][None, None, :] ** 2).sqrt()
    f = torch.fft.ifftn(torch.fft.fftn(w) / (1.0 + kk) ** power).real
    return torch.exp(0.5 * f / f.std())


@pytest.mark.parametrize("shape", [(128, 128, 128), (64, 64, 512), (54, 54, 243)])
def test_translated_cells(shape):
    import torch
    from paper_2009_03762_gb300 import gfp
    n1, n2, n3 = shape
    m = _smooth(n3, n2, n1, 2, 1)
    shift = (n3 // 3, n2 // 5, n1 // 7)
    out = []
    for s in ((0, 0, 0), shift):
        f = torch.roll(m, s, (0, 1, 2)).contiguous()
        g = gfp.Grid(n1, n2, n3)
        g.set_phases((0.57 * f).contiguous(), (0.385 * f).contiguous())
        g.solve(gfp.scheme("AFB_R", "PCD", "FP64"), [0.01, 0, 0, 0, 0, 0], 0.0, 2)
        eps = g.strain(torch.empty(6, n3, n2, n1, dtype=torch.float64, device="cuda"))
        g.close()
        out.append(torch.roll(eps, tuple(-x for x in s), (1, 2, 3)))
    d = out[0] - out[1]
    for c in (3, 4, 5):  # the shears start from zero: no rounding of a mean strain beside the increment's
        rms = float(d[c].pow(2).mean().sqrt())
        for at in ((0, 0, 0), tuple(-x for x in shift)):
            near = torch.roll(d[c], tuple(1 - x for x in at), (0, 1, 2))[:3, :3, :3]
            assert float(near.abs().max()) <= 8.0 * rms, (c, at)
