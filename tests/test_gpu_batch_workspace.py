"""The batched call writes nothing outside a workspace of exactly the size asked for:
numbers of fields whose tables end near a multiple of 256 bytes."""
import pytest
import torch

from paper_2006_12838_gb300 import plic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 4, 5, 6, 32, 64, 65, 66])
def test_exact_workspace(n):
    dev = torch.device("cuda:0")
    z, y, x = torch.meshgrid(*(torch.arange(24, device=dev, dtype=torch.float32),) * 3, indexing="ij")
    phi = (7.0 - torch.sqrt((x - 11.3) ** 2 + (y - 12.1) ** 2 + (z - 10.9) ** 2) + 0.5).clamp(0, 1)
    idx, cnt = plic.interface_compact(phi)
    k = int(cnt.item())
    want = plic.curvature(phi, idx, n_iface=k)
    size = plic.workspace_bytes(plic.WS_BATCHED, n)
    room = torch.full((256 + size + 1024,), 0xA5, dtype=torch.uint8, device=dev)
    kappas = torch.zeros((n, k), device=dev)
    batch = plic.BatchedFields([(phi, idx, k, kappas[i]) for i in range(n)], workspace=room[256:256 + size])
    for _ in range(2):
        kappas.fill_(7.0)
        plic.curvature_batched(batch)
        assert torch.equal(kappas, want.expand(n, k))
    assert bool((room[:256] == 0xA5).all()) and bool((room[256 + size:] == 0xA5).all())


@pytest.mark.parametrize("n", [511, 512, 513, 576, 577, 1100])
def test_many_fields(n):
    """Tables of more than one launch: every list comes out, in two captured calls too."""
    dev = torch.device("cuda:0")
    g = torch.Generator(device=dev).manual_seed(n)
    phi = torch.rand((n, 3, 3, 4), device=dev, generator=g).mul(1.6).sub(0.3).clamp(0, 1)     # two inner cells each
    fields, want, kappas = [], [], torch.full((n, 2), 7.0, device=dev)
    for i in range(n):
        idx, cnt = plic.interface_compact(phi[i])
        k = int(cnt.item())
        fields.append((phi[i], idx, k, kappas[i]))
        want.append(torch.cat([plic.curvature(phi[i], idx, n_iface=k), torch.full((2 - k,), 7.0, device=dev)])
                    if k else torch.full((2,), 7.0, device=dev))
    want = torch.stack(want)
    batch = plic.BatchedFields(fields)
    plic.curvature_batched(batch)
    assert torch.equal(kappas, want)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        plic.curvature_batched(batch)
    kappas.fill_(7.0)
    graph.replay()
    assert torch.equal(kappas, want)
