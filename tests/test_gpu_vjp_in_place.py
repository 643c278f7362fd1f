"""The curvature's adjoint with its result over its inputs: the field itself, a buffer
that overlaps it, the weights; against separate buffers, to the bit."""
import pytest
import torch

from paper_2006_12838_gb300 import plic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(9, 11, 10), (40, 37, 50)])
def test_in_place(shape):
    dev = torch.device("cuda:0")
    z, y, x = (torch.arange(e, device=dev, dtype=torch.float32) for e in shape)
    c = [0.5 * e + 0.2 for e in shape]
    r = 0.35 * min(shape)
    phi = (r - torch.sqrt((x[None, None, :] - c[2]) ** 2 + (y[None, :, None] - c[1]) ** 2
                          + (z[:, None, None] - c[0]) ** 2) + 0.5).clamp(0, 1)
    idx, cnt = plic.interface_compact(phi)
    n = int(cnt.item())
    g = torch.Generator(device=dev).manual_seed(1)
    w = torch.randn(n, device=dev, generator=g)
    want = plic.curvature_backward(phi, idx, w, n_iface=n)
    assert bool((want != 0).any())

    p = phi.clone()
    plic.curvature_backward(p, idx, w, n_iface=n, g_phi=p)
    assert torch.equal(p, want)
    # the result some cells into the field's buffer, and the field some cells into the result's
    m = phi.numel()
    for a, b in ((0, 333), (333, 0)):
        buf = torch.zeros(m + 333, device=dev)
        p, out = buf[a:a + m].view(shape), buf[b:b + m].view(shape)
        p.copy_(phi)
        plic.curvature_backward(p, idx, w, n_iface=n, count=cnt, g_phi=out)
        assert torch.equal(out, want)
    # the weights in the result's buffer
    out = torch.zeros(m, device=dev)
    out[5:5 + n] = w
    plic.curvature_backward(phi, idx, out[5:5 + n], n_iface=n, g_phi=out.view(shape))
    assert torch.equal(out.view(shape), want)
