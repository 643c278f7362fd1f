"""The curvature step's own PLIC solves (one normal, many volumes): normals with one
component almost zero and volumes at the boundary of cases (2), (3) and (5), where the
thresholds' roundings meet the large constants of case (3)."""
import ctypes
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

from paper_2006_12838_gb300 import build as B
from paper_2006_12838_gb300 import plic

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, HERE)
from kappa_gate import gate_kappa  # noqa: E402


@pytest.fixture(scope="module")
def orc():
    import oracle
    oracle.build()
    return oracle


@pytest.fixture(scope="module")
def solve(tmp_path_factory):
    """(paired, single) offsets of float32 normals (3, n) and volumes."""
    lib = str(tmp_path_factory.mktemp("curv") / "curv_offset.so")
    subprocess.run([B._nvcc()] + B.ARCH + B.NVCC_FLAGS +
                   ["-shared", "-o", lib, os.path.join(HERE, "curv_offset.cu")], check=True)
    f = ctypes.CDLL(lib).curv_offsets
    f.argtypes = [ctypes.c_void_p] * 6 + [ctypes.c_int64]

    def run(n, V0):
        t = [torch.tensor(np.ascontiguousarray(a), dtype=torch.float32, device="cuda:0") for a in (*n, V0)]
        out = [torch.zeros_like(t[3]) for _ in range(2)]
        torch.cuda.synchronize()
        assert f(*(x.data_ptr() for x in t + out), t[3].numel()) == 0
        return [o.double().cpu().numpy() for o in out]

    return run


def _ulps(v, k):
    """v moved by k (an array) units in the last place."""
    return (np.asarray(v, np.float32).view(np.int32) + k.astype(np.int32)).view(np.float32)


def test_degenerate_normals(orc, solve):
    """Smallest component 1e-12 to 1e-34 of the others, V within a few ulp of the
    boundary n2/(2 n3): |d0 error| <= 5e-7, the roundings of a dozen FP32 operations on
    numbers up to 0.87 (3e-8 each) and the cube root of case (1) (2e-7)."""
    rng = np.random.default_rng(3)
    N = 400_000
    th = rng.uniform(0.0, np.pi / 4, N)
    n = np.stack([np.cos(th), np.sin(th), 10.0 ** -rng.uniform(12, 34, N)]).astype(np.float32)
    V = np.minimum(_ulps(0.5 * np.tan(th), rng.integers(-3, 4, N)), np.float32(0.5))
    V = np.where(rng.random(N) < 0.5, V, np.float32(1) - V).astype(np.float32)
    want = orc.offset(*n.astype(np.float64), V.astype(np.float64))
    for got in solve(n, V):
        assert np.isfinite(got).all(), np.sum(~np.isfinite(got))
        assert np.abs(got - want).max() <= 5e-7


def test_extruded_planes_with_a_residue(orc):
    """Stencils of planes along x, fills in steps of 1/1024 (their sums in x cancel
    exactly) and 1e-14 to 1e-30 left in the empty neighbour that is summed last (the
    normal's smallest component is of that size), the middle row's fill within a few
    ulp of n2/(2 n3) of the stencil's normal: kappa against the oracle."""
    rng = np.random.default_rng(1)
    N = 40_000
    e = np.arange(-1, 2)
    th = rng.uniform(0.05, 0.78, N)
    ny, nz = np.sin(th), np.cos(th)
    c = rng.uniform(-0.45, 0.45, N) * (ny + nz) / 2
    d = c[:, None, None] + nz[:, None, None] * e[None, :, None] + ny[:, None, None] * e[None, None, :]
    full = np.broadcast_to
    plane = orc.volume(np.zeros(9 * N), full(ny[:, None], (N, 9)).ravel().copy(),
                       full(nz[:, None], (N, 9)).ravel().copy(), d.ravel()).reshape(N, 3, 3)   # (z, y)
    plane = np.round(1024 * plane) / 1024
    phi = np.repeat(plane[:, :, :, None], 3, axis=3).astype(np.float32)                       # (z, y, x)
    phi = phi[phi[:, 0, 0, 2] == 0]
    N = len(phi)
    phi[:, 0, 0, 2] = (10.0 ** -rng.uniform(14, 30, N)).astype(np.float32)
    # the normal's y and z sums (Eq. 38); the middle row has no weight in them
    w1 = np.array([1.0, 2.0, 1.0])
    p = phi.astype(np.float64)
    gy = np.einsum("nzyx,z,y,x->n", p, w1, e.astype(float), w1)
    gz = np.einsum("nzyx,z,y,x->n", p, e.astype(float), w1, w1)
    n2, n3 = np.minimum(abs(gy), abs(gz)), np.maximum(abs(gy), abs(gz))
    V = np.clip(_ulps(0.5 * n2 / n3, rng.integers(-3, 4, N)), np.float32(1e-3), np.float32(0.5))
    phi[:, 1, 1, :] = V[:, None]
    field = np.ascontiguousarray(phi.transpose(1, 2, 0, 3).reshape(3, 3, 3 * N))
    idx = (9 * N + 3 * N + 3 * np.arange(N) + 1).astype(np.int32)
    ref, dim, _, cond = orc.curvature(field, idx, with_cond=True)
    t, i = torch.tensor(field, device="cuda:0"), torch.tensor(idx, device="cuda:0")
    kappa = plic.curvature(t, i)
    assert bool(torch.isfinite(kappa).all())
    gate_kappa(kappa.cpu().numpy(), ref, dim, "extruded planes", cond=cond)
    g = plic.curvature_backward(t, i, torch.ones_like(kappa))
    assert bool(torch.isfinite(g).all())


@pytest.mark.parametrize("equal", [False, True])
def test_error_by_case(orc, solve, equal):
    """Random normals, and normals of nearly equal components (spread 1e-1 to 1e-6): the
    offsets of cases (3) and (4) as accurate as a solve that ends with a Newton step on
    Eq. 10: rms 2.6e-8 and 2.9e-8, at most 1.3e-7 (half an ulp each of L and L s, 3e-8
    or 6e-8, and of the three or four numbers below 1/2 that s is formed from, 1.5e-8
    each)."""
    rng = np.random.default_rng(7)
    N = 600_000
    n = rng.standard_normal((3, N))
    if equal:
        n = rng.standard_normal(N) * (1 + 10.0 ** -rng.uniform(1, 6, N) * n)
    n = (n / np.linalg.norm(n, axis=0)).astype(np.float32)
    V = rng.random(N).astype(np.float32)
    want = orc.offset(*n.astype(np.float64), V.astype(np.float64))
    s = np.sort(np.abs(n.astype(np.float64)), axis=0)
    d = 0.5 * s.sum(0) - np.abs(want)
    hard = (d >= s[1]) & (d < s[0] + s[1])
    for got in solve(n, V):
        err = np.abs(got - want)
        for case, rms in ((hard & (d < s[2]), 2.6e-8), (hard & (d >= s[2]), 2.9e-8)):
            assert np.sqrt(np.mean(err[case] ** 2)) <= rms, np.sqrt(np.mean(err[case] ** 2))
            assert err[case].max() <= 1.3e-7, err[case].max()
