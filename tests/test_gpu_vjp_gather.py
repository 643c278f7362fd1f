"""The curvature adjoint's gather at the edges of its cuts: fields of a few
cells up to several blocks of runs, a gradient buffer off the 16-byte boundary,
leftovers in the workspace and in the buffer, lists in any order and longer than
their count."""
import numpy as np
import pytest
import torch

from paper_2006_12838_gb300 import plic

pytestmark = pytest.mark.gpu


def _case(shape, seed):
    """A ball's fill, softened over a cell, with noise on its interface."""
    nz, ny, nx = shape
    rng = np.random.default_rng(seed)
    z, y, x = np.meshgrid(*(np.arange(e) - 0.5 * (e - 1) + 0.13 for e in shape), indexing="ij")
    r = 0.33 * min(shape) + 0.7
    p = np.clip(r - np.sqrt((x * min(1, 8 / nx)) ** 2 + y * y + z * z) + 0.5, 0, 1)
    m = (p > 0) & (p < 1)
    p[m] = np.clip(p[m] + 1e-3 * rng.standard_normal(int(m.sum())), 1e-3, 1 - 1e-3)
    if shape == (3, 3, 3):                                # the ball covers it: a tilted plane instead
        p = np.clip(0.5 + 0.45 * z + 0.2 * y + 0.1 * x + 0.01 * rng.standard_normal(shape), 0, 1)
    phi = torch.tensor(p, dtype=torch.float32, device="cuda:0")
    idx, cnt = plic.interface_compact(phi)
    k = int(cnt.item())
    g = torch.tensor(rng.standard_normal(k), dtype=torch.float32, device="cuda:0")
    return phi, idx[:k].contiguous(), g


# 27 cells; one run of 1024 exactly, one cell more, several; more than the 32
# runs of a block, and several blocks
@pytest.mark.parametrize("shape", [(3, 3, 3), (4, 16, 16), (5, 5, 41), (9, 13, 35), (23, 41, 37), (40, 50, 61)])
def test_gather(shape):
    phi, idx, g = _case(shape, sum(shape))
    assert idx.numel() > 0
    ref = plic.curvature_backward(phi, idx, g)
    # outside the stencils exactly 0
    near = torch.zeros(phi.shape, dtype=torch.bool, device=phi.device)
    at = torch.zeros_like(near.view(-1))
    at[idx.long()] = True
    at = at.view(phi.shape)
    for dz in (-1, 0, 1):
        for dy in (-1, 0, 1):
            for dx in (-1, 0, 1):
                near |= torch.roll(at, (dz, dy, dx), (0, 1, 2))
    assert (ref[~near] == 0).all() and torch.isfinite(ref).all()
    # any order, a longer list than its count, leftovers everywhere, any alignment
    perm = torch.randperm(idx.numel(), generator=torch.Generator().manual_seed(1)).to(phi.device)
    n = idx.numel()
    ws = torch.empty(plic.curv_bwd_workspace_bytes(phi.numel(), n + 7), dtype=torch.uint8, device=phi.device)
    tail = torch.full((7,), 5, dtype=torch.int32, device=phi.device)
    count = torch.tensor([n], dtype=torch.int64, device=phi.device)
    for shift, fill in ((0, 0), (1, 255), (2, 1), (3, 127)):
        ws.fill_(fill)
        if fill == 1:                                # entries that point into the list
            ws[:4 * phi.numel()].view(torch.int32).copy_(
                torch.arange(phi.numel(), device=phi.device) % n)
        buf = torch.full((phi.numel() + 8,), float("nan"), device=phi.device)
        out = buf[shift:shift + phi.numel()].view(phi.shape)
        plic.curvature_backward(phi, torch.cat([idx[perm], tail]), torch.cat([g[perm], g.new_full((7,), 9.0)]),
                                n_iface=n + 7, count=count, g_phi=out, workspace=ws)
        assert torch.equal(out, ref)
        assert torch.isnan(buf[:shift]).all() and torch.isnan(buf[shift + phi.numel():]).all()
    # the sum over single-entry lists (each output a sum of at most 27 terms)
    if n <= 600:
        total = torch.zeros(phi.shape, dtype=torch.float64, device=phi.device)
        for k in range(n):
            total += plic.curvature_backward(phi, idx[k:k + 1].contiguous(), g[k:k + 1].contiguous()).double()
        assert torch.allclose(ref.double(), total, rtol=0, atol=27 * 6e-8 * float(total.abs().max()) * 2)
    # an empty list
    assert (plic.curvature_backward(phi, idx, g, n_iface=n, count=count * 0) == 0).all()
