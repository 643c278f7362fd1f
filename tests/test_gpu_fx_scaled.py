"""FP64 offsets (optimised SZ and analytic, FP64 and FP64_REFINED) of normals off unit
length, which the fixed-point scheme takes times a power of two."""
import numpy as np
import pytest
import torch

from paper_2006_12838_gb300 import plic

pytestmark = pytest.mark.gpu


def _cells(m):
    rng = np.random.default_rng(m)
    n = rng.standard_normal((3, m))
    n[0, ::5] *= 10.0 ** -rng.uniform(0, 17, n[0, ::5].size)
    n[1, ::7] = n[2, ::7]
    return n / np.sqrt((n * n).sum(0)), rng.random(m), rng


def _solve(n, V, **kw):
    t = [torch.tensor(np.ascontiguousarray(a), device="cuda:0") for a in (*n, V)]
    return plic.offset(*t, **kw).cpu().numpy()


@pytest.mark.parametrize("method", ["sz_opt", "analytic"])
@pytest.mark.parametrize("prec", ["fp64", "fp64r"])
@pytest.mark.parametrize("m", [1, 511, 513, 70_001])
def test_powers_of_two(method, prec, m):
    """2^k n has 2^k d0, to the bit; cells of all lengths side by side."""
    n, V, rng = _cells(m)
    k = rng.integers(-58, 1, m)
    want = _solve(n, V, method=method, precision=prec)
    got = _solve(np.ldexp(n, k), V, method=method, precision=prec)
    assert np.array_equal(got, np.ldexp(want, k))


@pytest.mark.parametrize("method", ["sz_opt", "analytic"])
def test_lengths(method):
    """Unit L1 length and other lengths with L <= 3 against the oracle: 5e-16 of the power of
    two above n3 (the 4e-16 of test_fx_edges_host.py and the oracle's own rounding),
    volumes where the cut polygon's area does not blow that up."""
    import oracle
    oracle.build()
    n, V, rng = _cells(60_000)
    V = 1e-3 + 0.998 * V
    for s in (1 / np.abs(n).sum(0), 0.3, 0.577, 1.2, 2.0 ** rng.uniform(-20, 0.7, V.size)):
        w = n * s
        k = np.abs(w).sum(0) < 2.99
        mid = np.sort(np.abs(n), 0)[1] > 0.1
        want = oracle.offset(*(n * np.ones_like(V)), V) * s
        err = np.abs(_solve(w[:, k], V[k], method=method) - want[k]) / 2.0 ** np.ceil(np.log2(np.abs(w[:, k]).max(0)))
        # n times s is rounded: half an ulp of each component, as much again in d0
        assert err[mid[k]].max() <= 8e-16, err[mid[k]].max()


def test_refused_cells_among_them():
    """L > 3, n = 0, infinite and NaN components, V0 below 2^-96: as before."""
    n, V, _ = _cells(2048)
    n[:, 1::8] = 0.0
    n[:, 2::8] *= 10.0
    n[0, 3::8] = np.nan
    n[2, 4::8] = np.inf
    V[5::8] = 1e-40
    n[:, 6::8] *= 0.3
    V[7::8] = 1.5
    edge = np.array([[3 - 4e-9, 0, 0], [1, 1, 1 - 4e-9], [2, 0.5, 0.5 - 4e-9]])    # L just below 3
    n[:, :24:8] = edge.T
    V[:24:8] = 0.25
    t = [torch.tensor(a, device="cuda:0") for a in (*n, V)]
    bad = torch.zeros(1, dtype=torch.int64, device="cuda:0")
    d0 = plic.offset(*t, invalid=bad).cpu().numpy()
    assert bad.item() == 5 * 256
    assert (np.isnan(d0).reshape(-1, 8) == [False, True, True, True, True, False, False, True]).all()
    half = 0.5 * np.abs(n).sum(0)
    assert np.abs(d0[5::8] + half[5::8]).max() < 1e-12
    import oracle
    oracle.build()
    l = np.sqrt((edge * edge).sum(1))
    assert np.abs(d0[:24:8] - l * oracle.offset(*(edge.T / l), V[:24:8])).max() < 1e-12
