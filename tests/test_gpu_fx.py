"""The fixed-point FP64 offsets (optimised SZ and analytic, PLIC_FP64 and
PLIC_FP64_REFINED) at the edges of the scheme: normals with components down to 0,
pairs and triples of nearly equal components, volumes at every case boundary, down to
the smallest double and at the ends of the range, normals that are not of unit
length (solved by the closed forms), unaligned arrays."""
import numpy as np
import pytest
import torch

from paper_2006_12838_gb300 import plic

pytestmark = pytest.mark.gpu
# d0 is within 2e-16 (tests/test_fx_host.py); the oracle's own bisection
# on doubles is within 3e-16 of the offset (a few ulp of L/2 and of the volume over an
# area of at least 0.1); volumes below are in [1e-3, 1 - 1e-3] for this bound
TIGHT = 5e-16
# the FP64 bound for all volumes: where the cut polygon degenerates the oracle's
# rounding of the volume is divided by its area
WIDE = 1e-12


@pytest.fixture(scope="module")
def orc():
    import oracle
    oracle.build()
    return oracle


def _normals(kind, m, rng):
    n = rng.standard_normal((3, m))
    if kind == "small":
        n[0] *= 10.0 ** -rng.uniform(0, 17, m)
        n[1] *= 10.0 ** -(rng.uniform(0, 17, m) * (rng.random(m) < 0.4))
    if kind == "zero":
        n[0] = 0.0
        n[1, ::2] = 0.0
    if kind == "equal":
        n[1] = n[0] * (1 + rng.choice([0, 1e-16, 1e-9, 1e-6, 1e-5], m))
        n[2, ::2] = n[0, ::2] * (1 + rng.choice([0, 1e-16, 1e-9, 1e-6, 1e-5], n[2, ::2].size))
    n /= np.sqrt((n * n).sum(0))
    n = rng.permuted(n, axis=0)
    return n * rng.choice([-1.0, 1.0], n.shape)


def _volumes(n, rng, orc):
    """Uniform, at and beside the case boundaries, and at the ends."""
    m = n.shape[1]
    s = np.sort(np.abs(n), 0)
    half = 0.5 * s.sum(0)
    which = rng.integers(0, 5, m)
    d = np.choose(which, [s[0], s[1], s[2], s[0] + s[1], half])
    d = d + rng.choice([0, 1e-16, -1e-16, 1e-12, -1e-9, 1e-7, -1e-4], m) * np.where(rng.random(m) < 0.5, s[0], 1)
    V = orc.volume(n[0], n[1], n[2], np.clip(d, 0, half) - half)
    V = np.where(rng.random(m) < 0.4, rng.random(m), np.clip(V, 0, 0.5))
    return np.where(rng.random(m) < 0.5, 1 - V, V)


def _solve(n, V, method, prec):
    t = [torch.tensor(a, device="cuda:0") for a in (*n, V)]
    return plic.offset(*t, method=method, precision=prec).cpu().numpy()


@pytest.mark.parametrize("method", ["sz_opt", "analytic"])
@pytest.mark.parametrize("prec", ["fp64", "fp64r"])
@pytest.mark.parametrize("kind", ["unit", "small", "zero", "equal"])
def test_accuracy(orc, method, prec, kind):
    rng = np.random.default_rng(3)
    n = _normals(kind, 40_000, rng)
    V = _volumes(n, rng, orc)
    d0 = _solve(n, V, method, prec)
    err = np.abs(d0 - orc.offset(n[0], n[1], n[2], V))
    assert err.max() <= WIDE
    s = np.sort(np.abs(n), 0)
    mid = (V > 1e-3) & (V < 1 - 1e-3) & (s[1] > 0.1)
    assert err[mid].max() <= TIGHT


@pytest.mark.parametrize("method", ["sz_opt", "analytic"])
def test_ends(orc, method):
    rng = np.random.default_rng(4)
    n = _normals("unit", 4096, rng)
    V = np.concatenate([[0.0, -0.0, 1.0, 0.5, np.nextafter(0.5, 0), np.nextafter(0.5, 1), 5e-324, 1e-300,
                         np.nextafter(1, 0), 2.0 ** -96, np.nextafter(2.0 ** -96, 0), 1e-29, 1e-28],
                        2.0 ** -rng.uniform(1, 110, 2000), 1 - 2.0 ** -rng.uniform(1, 53, 2083)])
    d0 = _solve(n, V, method, "fp64")
    assert np.abs(d0 - orc.offset(n[0], n[1], n[2], V)).max() <= WIDE
    h = 0.5 * np.abs(n).sum(0)
    assert np.abs(d0[:2] + h[:2]).max() < 1e-15 and abs(d0[2] - h[2]) < 1e-15
    # V0 near 1/2: d0 is A^-1 (V0 - 1/2), of its sign
    assert (np.sign(d0[4:6]) == [-1, 1]).all() or np.abs(d0[4:6]).max() < 1e-16


def test_beyond_the_scheme(orc):
    """Normals of other lengths and invalid input take the closed forms in FP64."""
    rng = np.random.default_rng(5)
    n = _normals("unit", 3000, rng)
    V = _volumes(n, rng, orc)
    for scale in (1e-3, 0.3, 0.99, 1.0 + 1e-7, 1.01, 1.5):
        k = np.abs(n).sum(0) * scale <= 3
        d0 = _solve((n * scale)[:, k], V[k], "sz_opt", "fp64")
        assert np.abs(d0 - scale * orc.offset(*n[:, k], V[k])).max() <= WIDE
    bad = torch.zeros(1, dtype=torch.int64, device="cuda:0")
    one = np.array([1.0, np.nan, np.inf, 0.0, 0.6, 0.6, 0.6, 2.0])
    V = np.array([0.3, 0.3, 0.3, 0.3, -1e-3, 1.0 + 1e-15, np.nan, 0.3])
    t = [torch.tensor(a, device="cuda:0") for a in (one, 0 * V, np.where(one == 2.0, 2.0, 0.0), V)]
    d0 = plic.offset(*t, precision="fp64", invalid=bad).cpu().numpy()
    assert bad.item() == 7 and np.isnan(d0[1:]).all() and abs(d0[0] + 0.2) < 1e-16


@pytest.mark.parametrize("m", [1, 2, 3, 255, 511, 512, 513, 1023, 1025, 4099])
def test_unaligned(m):
    rng = np.random.default_rng(m)
    n = _normals("unit", m + 1, rng)
    V = rng.random(m + 1)
    big = [torch.tensor(a, device="cuda:0") for a in (*n, V)]
    a = plic.offset(*[x[1:] for x in big])
    b = plic.offset(*[x[1:].clone() for x in big])
    assert torch.equal(a, b)
