"""Listed cells whose own fill lies outside [0, 1] (an overshoot): the plane of such a cell
touches the cube's corner, as that of a full or an empty cell does, whether the number of
its interface neighbours is even or odd."""
import pytest
import torch

from paper_2006_12838_gb300 import plic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flags", [0, plic.FLAG_POINT_CENTROID])
@pytest.mark.parametrize("batched", [False, True])
def test_overshoot(flags, batched):
    dev = torch.device("cuda:0")
    g = torch.Generator(device=dev).manual_seed(2)
    m = 500                                          # one 3^3 stencil per listed cell
    phi = torch.rand((3, 3, m, 3), device=dev, generator=g).mul(2.0).sub(0.5).clamp(0, 1)
    odd = ((phi > 0) & (phi < 1)).sum((0, 1, 3)) - ((phi[1, 1, :, 1] > 0) & (phi[1, 1, :, 1] < 1)).int()
    assert set((odd % 2).tolist()) == {0, 1}
    idx = (9 * m + 3 * m + 3 * torch.arange(m, device=dev) + 1).int()

    def kappa(fill):
        p = phi.clone()
        p[1, 1, :, 1] = fill
        p = p.view(3, 3, 3 * m)
        if not batched:
            return plic.curvature(p, idx, flags=flags)
        out = torch.full((m,), 7.0, device=dev)
        plic.curvature_batched([(p, idx, m, out)], flags=flags)
        return out

    for over, end in ((1.25, 1.0), (1.0 + 1e-6, 1.0), (-0.5, 0.0)):
        a, b = kappa(over), kappa(end)
        assert bool(torch.isfinite(b).all()) and torch.equal(a, b), over
