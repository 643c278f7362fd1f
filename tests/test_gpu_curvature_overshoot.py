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


def test_gradient_of_cells_that_are_not_finite():
    """A listed cell with a NaN or infinite fill adds nothing to the gradient; those beside it
    keep theirs."""
    dev = torch.device("cuda:0")
    g = torch.Generator(device=dev).manual_seed(3)
    m = 60
    phi = torch.rand((3, 3, m, 3), device=dev, generator=g).mul(1.8).sub(0.4).clamp(0, 1)
    phi[1, 1, :, 1].clamp_(0.1, 0.9)
    idx = (9 * m + 3 * m + 3 * torch.arange(m, device=dev) + 1).int()
    w = torch.ones(m, device=dev)
    want = plic.curvature_backward(phi.view(3, 3, 3 * m), idx, w)
    bad = torch.tensor([float("nan"), float("inf"), -float("inf")], device=dev)
    p = phi.clone()
    p[1, 1, ::4, 1] = bad[torch.arange(p[1, 1, ::4, 1].numel(), device=dev) % 3]
    got = plic.curvature_backward(p.view(3, 3, 3 * m), idx, w).view(3, 3, m, 3)
    want = want.view(3, 3, m, 3).clone()
    assert bool((want[:, :, ::4] != 0).any()) and bool(torch.isfinite(want).all())
    want[:, :, ::4] = 0
    assert torch.equal(got, want)
