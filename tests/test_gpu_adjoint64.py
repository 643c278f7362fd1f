"""The FP64 adjoints at the edges of their scheme, against the derivatives of Eq. 10's
case volumes in long double: components down to 0 and pairs of equal ones, planes near
a corner and at every case boundary, normals off unit length (the general formula),
planes that miss the cube, invalid cells, unaligned arrays."""
import numpy as np
import pytest
import torch

from paper_2006_12838_gb300 import plic

pytestmark = pytest.mark.gpu
LD = np.longdouble


def _reference(n, d0):
    """A, c of the cut polygons (rows: cells) in long double."""
    n, d0 = n.astype(LD), d0.astype(LD)
    a = np.abs(n)
    order = np.argsort(a, axis=0, kind="stable")
    n1, n2, n3 = np.take_along_axis(a, order, 0)
    d = (n1 + n2 + n3) / 2 - np.abs(d0)
    r1, r2 = [np.where(x > 0, 1 / np.where(x > 0, x, 1), 0) for x in (n1, n2)]
    e2, e3 = np.maximum(d - n2, 0), np.maximum(d - n3, 0)
    cub, sq = (e2 ** 3 + e3 ** 3) * r1, (e2 ** 2 + e3 ** 2) * r1
    N, G = 3 * d * (d - n1) + n1 ** 2 - cub, 6 * d - 3 * n1 - 3 * sq
    five, one = d >= n1 + n2, d < n1
    G = np.where(five | one, 1, G)
    pick = lambda c5, c1, c: np.where(five, c5, np.where(one, c1, c))
    A = pick(1 / n3, d * d * r1 * r2 / (2 * n3), G * r2 / (6 * n3)) * np.sqrt(n1 ** 2 + n2 ** 2 + n3 ** 2)
    c = [pick(LD(0.5), d * r1 / 3, (3 * d - 2 * n1 - cub * r1) / G),
         pick(LD(0.5), d * r2 / 3, (N * r2 - 3 * e2 ** 2 * r1) / G),
         pick((d - (n1 + n2) / 2) / n3, d / (3 * n3), (N / n3 - 3 * e3 ** 2 * r1) / G)]
    c = np.take_along_axis(np.stack(c), np.argsort(order, axis=0), 0) - LD(0.5)
    c = np.where(d0 > 0, -c, c) * np.where(n < 0, -1, 1)
    least = np.where(n1 > 0, n1, np.where(n2 > 0, n2, n3))
    return A, c, d, least


def _cells(kind, m):
    rng = np.random.default_rng(len(kind) + m)
    n = rng.standard_normal((3, m))
    if kind == "small":
        n[0] *= 2.0 ** -rng.uniform(0, 40, m)
        n[1] *= 2.0 ** -(rng.uniform(0, 40, m) * (rng.random(m) < 0.5))
    if kind == "zero":
        n[0] = 0.0
        n[1, ::3] = -0.0
    if kind == "equal":
        n[1] = n[0] * rng.choice([1, 1 + 1e-15, 1 - 1e-12], m)
        n[2, ::2] = -n[0, ::2]
    n = np.stack([n[(np.arange(m) + k) % 3, np.arange(m)] for k in range(3)])
    n /= np.sqrt((n * n).sum(0))
    if kind == "length":
        n *= 2.0 ** rng.uniform(-6, 6, m) * np.where(rng.random(m) < 0.3, 0, 1) + (rng.random(m) < 0.3) * 1e-6 + 1e-3
    a = np.sort(np.abs(n), axis=0)
    L = a.sum(0)
    d = L / 2 * rng.random(m)
    if kind == "edges":
        d = np.choose(rng.integers(0, 5, m), [a[0], a[1], a[2], a[0] + a[1], L / 2])
        d = np.clip(d * (1 + rng.choice([-1e-15, 0, 1e-15], m)), 0, L / 2)
    if kind == "corner":
        d = L / 2 * 2.0 ** -rng.uniform(0, 34, m)
    return n, (L / 2 - d) * rng.choice([-1, 1], m)


# Tolerances: d carries a rounding of 1e-16 (twice that with the sums in another order)
# that moves c by at most 1/n1 (n2 where n1 = 0) and 1/d times as much, A by
# 1/(n2 n3) and 1/A, relatively, by 2/d; each formula adds at most a dozen roundings of its terms.
@pytest.mark.parametrize("kind", ["random", "small", "zero", "equal", "length", "edges", "corner"])
@pytest.mark.parametrize("m,shift", [(1, 0), (4097, 0), (50_001, 1)])
def test_against_long_double(kind, m, shift):
    dev = torch.device("cuda:0")
    n, d0 = _cells(kind, m)
    g = np.random.default_rng(m).standard_normal(m)
    buf = torch.zeros(5, m + 4, dtype=torch.float64, device=dev)
    buf[:, shift:shift + m] = torch.from_numpy(np.stack([*n, d0, g]))
    nx, ny, nz, td, tg = [r[shift:shift + m] for r in buf]
    A, c, d, least = _reference(n, d0)
    ok = d > 1e-13
    size = np.sqrt((n * n).sum(0))                   # everything but |n| scales with it
    cond = 3e-15 * (1 + size / least + size / np.where(ok, d, 1))

    def close(got, want, tol):
        err = np.abs(got.cpu().numpy().astype(LD) - want)[ok]
        assert (err <= tol[ok]).all(), (err / tol[ok]).max()

    gv, gx, gy, gz = plic.offset_backward(nx, ny, nz, td, tg)
    with np.errstate(divide="ignore"):
        close(gv, g / A, cond * np.abs(g / A))
    for k, r in enumerate((gx, gy, gz)):
        close(r, g * c[k], cond * np.abs(g))
    gd, gx, gy, gz = plic.volume_backward(nx, ny, nz, td, tg)
    close(gd, g * A, cond * np.abs(g))
    for k, r in enumerate((gx, gy, gz)):
        close(r, -g * A * c[k], 2 * cond * np.abs(g))


def test_cells_without_a_polygon():
    """Planes that miss the cube, zero and NaN cells: what the general formula answers,
    also between cells of the scheme."""
    dev = torch.device("cuda:0")
    inf, nan = float("inf"), float("nan")
    cells = np.array([[0.6, 0.0, 0.8, 0.1, 1.0], [0.6, 0.0, 0.8, 0.7, 2.0], [0.6, 0.0, 0.8, -0.9, -2.0],
                      [0.6, 0.0, 0.8, 0.9, 0.0], [0.0, 0.0, 0.0, 0.0, 1.0], [0.6, 0.0, 0.8, nan, 1.0],
                      [1.0, 0.0, 0.0, 0.5, 1.0], [1.0, 0.0, -0.0, -0.25, 1.0]]).T
    t = [torch.tensor(r, dtype=torch.float64, device=dev) for r in cells]
    gv, gx, gy, gz = [r.cpu().numpy() for r in plic.offset_backward(*t)]
    np.testing.assert_allclose(gv, [0.8, inf, -inf, 0, nan, inf, inf, 1.0], rtol=1e-14)
    np.testing.assert_array_equal(np.isnan(gx), [0, 0, 0, 0, 1, 0, 0, 0])
    np.testing.assert_allclose(gx[[1, 2, 3, 5, 6]], 0.0)
    np.testing.assert_allclose([gx[7], gy[7], gz[7]], [-0.25, 0, 0], atol=1e-15)
    gd, *_ = [r.cpu().numpy() for r in plic.volume_backward(*t)]
    np.testing.assert_allclose(gd, [1.25, 0, 0, 0, 0, 0, 0, 1.0], rtol=1e-14)
