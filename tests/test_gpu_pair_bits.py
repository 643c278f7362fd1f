"""The paired FP32 kernels give a cell the same bits wherever it lies: in aligned and
unaligned arrays, among others or alone, with and without the round trip and the counter."""
import pytest
import torch

from paper_2006_12838_gb300 import plic, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("method", ["analytic", "sz_orig", "sz_opt"])
@pytest.mark.parametrize("prec", ["fp32", "fp32p"])
def test_same_bits(method, prec):
    dev = torch.device("cuda:0")
    n = 4 * 1024 + 1027
    c = synth.plic_cells(n, seed=21, edge_frac=0.05)
    a = [torch.tensor(x, dtype=torch.float32, device=dev) for x in (*c["n"], c["V0"])]

    def shifted(x):
        b = torch.empty(n + 1, device=dev)
        b[1:] = x
        return b[1:]

    def same(x, y):
        return torch.equal(x.contiguous().view(torch.int32), y.clone().view(torch.int32))

    kw = dict(method=method, precision=prec)
    d0 = plic.offset(*a, **kw)
    rt = plic.offset_roundtrip(*a, **kw)
    u = [shifted(x) for x in a]
    rt_u = plic.offset_roundtrip(*u, out=shifted(a[3]), out_rt=shifted(a[3]), **kw)
    bad = torch.zeros(1, dtype=torch.int64, device=dev)
    assert same(d0, plic.offset(*u, out=shifted(a[3]), **kw))
    assert same(d0, plic.offset(*a, invalid=bad, **kw))
    assert same(d0, rt[0]) and same(rt[0], rt_u[0]) and same(rt[1], rt_u[1])
    for i in range(0, n, 97):
        assert same(d0[i:i + 1], plic.offset(*[x[i:i + 1].clone() for x in a], **kw))
