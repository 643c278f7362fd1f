"""The paired FP32 kernels at the sizes and cells where they can go wrong:
arrays off the 16-byte boundary (whole groups of 1024 cells and what is left
over) and cells at the ends of the trigonometric cases, where a component of
the normal is almost zero."""
import numpy as np
import pytest
import torch

from paper_2006_12838_gb300 import plic, synth

pytestmark = pytest.mark.gpu
PAIRED = ["analytic", "sz_orig", "sz_opt"]


@pytest.fixture(scope="module")
def orc():
    import oracle
    oracle.build()
    return oracle


@pytest.mark.parametrize("method", PAIRED)
@pytest.mark.parametrize("n", [1, 2, 255, 1023, 1024, 1025, 2049, 70_001])
def test_unaligned_arrays(method, n):
    dev = torch.device("cuda:0")
    c = synth.plic_cells(n + 3, seed=12, edge_frac=0.02)
    big = [torch.tensor(a, dtype=torch.float32, device=dev) for a in (*c["n"], c["V0"])]
    big[3][::7] = 2.0                                  # invalid cells, counted
    shifted = [x[k:k + n] for k, x in zip((1, 2, 3, 1), big)]
    out = [torch.zeros(n + 2, device=dev)[1:n + 1] for _ in range(2)]
    cnt = torch.zeros(2, dtype=torch.int64, device=dev)
    ref, ref_rt = plic.offset_roundtrip(*[x.clone() for x in shifted], method=method, invalid=cnt[:1])
    for call in (lambda: plic.offset(*shifted, method=method, out=out[0], invalid=cnt[1:]),
                 lambda: plic.offset_roundtrip(*shifted, method=method, out=out[0], out_rt=out[1],
                                               invalid=cnt[1:])):
        cnt[1] = 0
        call()
        assert torch.equal(cnt[:1], cnt[1:])
        # the two loops may contract multiply-adds differently
        assert torch.allclose(out[0], ref, rtol=0, atol=2e-7, equal_nan=True)
    assert torch.allclose(out[1], ref_rt, rtol=0, atol=1e-6, equal_nan=True)


@pytest.mark.parametrize("method", ["analytic", "sz_opt"])
def test_sliver_cases(orc, method):
    """Normals with n1 down to 1e-12 (and 0), volumes at and around every case
    boundary: |d0 error| <= 5e-7, the roundings of a dozen FP32 operations on
    numbers up to 0.87 (3e-8 each) and the cube root of case (1) (2e-7)."""
    rng = np.random.default_rng(5)
    n, V = [], []
    for k in [None] + list(np.linspace(0, 12, 25)):
        for _ in range(40):
            a = np.abs(rng.standard_normal(3))
            a[0] = 0.0 if k is None else a[0] * 10.0 ** -k
            a[1] *= 10.0 ** -(rng.integers(0, 2) * rng.uniform(0, 6))
            a = (a / np.linalg.norm(a)).astype(np.float32).astype(np.float64)
            s = np.sort(a)
            half = 0.5 * s.sum()
            for d in (s[0], s[1], s[2], s[0] + s[1], half):
                for e in (0.0, 1e-7, -1e-7, 1e-5, -1e-5, 0.3 * s[0], -0.3 * s[0]):
                    n.append(rng.permutation(a) * rng.choice([-1.0, 1.0], 3))
                    V.append(min(d + e, half) - half)
    n = np.array(n).T.copy()
    V0 = orc.volume(n[0], n[1], n[2], np.array(V)).astype(np.float32).astype(np.float64)
    V0 = np.clip(np.concatenate([V0, 1 - V0]), 0, 1).astype(np.float32).astype(np.float64)
    n = np.concatenate([n, n], 1)
    ref = orc.offset(n[0], n[1], n[2], V0)
    t = [torch.tensor(a, dtype=torch.float32, device="cuda:0") for a in (*n, V0)]
    for prec in ("fp32", "fp32p"):
        err = np.abs(plic.offset(*t, method=method, precision=prec).cpu().numpy() - ref)
        assert err.max() <= 5e-7, (prec, err.max(), n[:, err.argmax()], V0[err.argmax()])
