"""The batched call's tables by value: numbers of fields around the table's
size, empty lists among them, and a captured call replayed after the host's
tables are gone."""
import gc

import numpy as np
import pytest
import torch

from paper_2006_12838_gb300 import plic

pytestmark = pytest.mark.gpu


def _fields(n, dev):
    rng = np.random.default_rng(n)
    out = []
    for i in range(n):
        e = int(rng.integers(3, 20))
        z, y, x = np.meshgrid(*(np.arange(e),) * 3, indexing="ij")
        c, r = rng.uniform(0, e, 3), rng.uniform(0.5, 0.6 * e)
        p = np.clip(r - np.sqrt((x - c[0]) ** 2 + (y - c[1]) ** 2 + (z - c[2]) ** 2) + 0.5, 0, 1)
        phi = torch.tensor(p, dtype=torch.float32, device=dev)
        idx, cnt = plic.interface_compact(phi)
        k = int(cnt.item())
        out.append((phi, idx, k, torch.full((max(k, 1),), 7.0, device=dev)))
    return out


@pytest.mark.parametrize("n", [1, 63, 64, 65, 130])
def test_tables_and_capture(n):
    dev = torch.device("cuda:0")
    fields = _fields(n, dev)
    want = [plic.curvature(p, i, n_iface=k) if k else None for p, i, k, _ in fields]
    batch = plic.BatchedFields(fields)

    def check():
        for (_, _, k, kap), w in zip(fields, want):
            if k:
                assert torch.equal(kap[:k], w)
                kap.fill_(7.0)

    plic.curvature_batched(batch)
    check()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        plic.curvature_batched(batch)
        plic.curvature_batched(batch)               # the ticket is cleared in between
    ws = batch.workspace
    del batch
    gc.collect()
    junk = [np.full(1 << 16, 255, np.uint8) for _ in range(8)]      # the host's tables are gone
    for _ in range(2):
        g.replay()
        torch.cuda.synchronize()
        check()
    del junk, ws


@pytest.mark.parametrize("copies", [1, 30, 60, 120])
def test_ticket_sizes(copies):
    """The cells per ticket chosen by the total (32, 64, 128) against fixed ones: the
    same bits, from less than one ticket per warp up to several."""
    dev = torch.device("cuda:0")
    z, y, x = torch.meshgrid(*(torch.arange(96, device=dev, dtype=torch.float32),) * 3, indexing="ij")
    phi = (40.0 - torch.sqrt((x - 47.3) ** 2 + (y - 48.1) ** 2 + (z - 46.9) ** 2) + 0.5).clamp(0, 1)
    idx, cnt = plic.interface_compact(phi)
    k = int(cnt.item())
    want = plic.curvature(phi, idx, n_iface=k)
    for tuning in (None, (128, 32, 0, 1), (128, 128, 0, 1)):
        kappas = torch.full((copies, k), 7.0, device=dev)
        plic.curvature_batched([(phi, idx, k, kappas[i]) for i in range(copies)], tuning=tuning)
        assert torch.equal(kappas, want.expand(copies, k))
