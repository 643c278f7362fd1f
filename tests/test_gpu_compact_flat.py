"""The flat compaction passes at the edges of their cuts: fields that start off
the 16-byte boundary, every tile size and the block sums of large fields, last
tiles of a few cells, values at the ends of (0, 1), lists shorter than the count;
the entry without bits against the entry with them."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2006_12838_gb300 import plic

pytestmark = pytest.mark.gpu
SPECIAL = np.array([0.0, -0.0, 1.0, np.nextafter(np.float32(1), np.float32(0)), 1e-45, -1e-45, 1.17e-38,
                    np.nan, np.inf, -np.inf, -0.5, 1.5, np.nextafter(np.float32(1), np.float32(2)), 0.5],
                   np.float32)


def _field(shape, seed, density):
    rng = np.random.default_rng(seed)
    p = (rng.random(shape) < 0.5).astype(np.float32)
    pick = rng.random(shape) < density
    p[pick] = SPECIAL[rng.integers(0, SPECIAL.size, int(pick.sum()))]
    return p


def _expect(p):
    m = (p > 0) & (p < 1)
    inner = np.zeros_like(m)
    inner[1:-1, 1:-1, 1:-1] = m[1:-1, 1:-1, 1:-1]
    return np.flatnonzero(inner.reshape(-1)).astype(np.int32)


# (nz, ny, nx): tiles of 1024, 4096 and 8192 cells with last tiles of a few
# cells, rows of every remainder, and (the last) two tiles per block
@pytest.mark.parametrize("shape,density", [((3, 3, 3), 0.9), ((5, 4, 7), 0.5), ((4, 3, 1025), 0.3),
                                           ((7, 31, 33), 1.0), ((40, 41, 43), 0.02), ((70, 131, 130), 0.1),
                                           ((102, 101, 104), 0.001), ((190, 173, 171), 0.05),
                                           ((130, 211, 206), 1.0), ((266, 281, 283), 0.01),
                                           ((260, 513, 519), 0.003)])
@pytest.mark.parametrize("shift", [0, 1, 2, 3])
def test_shapes_and_alignment(shape, density, shift):
    if shape[0] >= 260 and shift > 1:
        pytest.skip("one shift of the large fields is enough")
    dev = torch.device("cuda:0")
    p = _field(shape, shape[2] + shift, density)
    want = _expect(p)
    buf = torch.full((p.size + 8,), 0.5, device=dev)          # interface values around the field
    phi = buf[shift:shift + p.size].view(shape)
    phi.copy_(torch.from_numpy(p))
    idx, cnt = plic.interface_compact(phi)
    assert int(cnt.item()) == want.size
    np.testing.assert_array_equal(idx[:want.size].cpu().numpy(), want)
    # without bits, and a list shorter than the count
    cap = max(1, want.size // 2)
    short = torch.full((cap + 4,), -7, dtype=torch.int32, device=dev)
    cnt2 = torch.zeros(1, dtype=torch.int64, device=dev)
    st = plic.load().vof_interface_compact_noalloc(
        ctypes.c_void_p(phi.data_ptr()), shape[2], shape[1], shape[0], ctypes.c_void_p(short.data_ptr()), cap,
        ctypes.c_void_p(cnt2.data_ptr()), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == 0 and int(cnt2.item()) == want.size
    k = min(cap, want.size)
    np.testing.assert_array_equal(short[:k].cpu().numpy(), want[:k])
    assert (short[cap:].cpu().numpy() == -7).all()
    idx2, cnt3 = plic.interface_compact(phi, idx=torch.full((cap + 4,), -7, dtype=torch.int32, device=dev)[:cap])
    assert int(cnt3.item()) == want.size
    np.testing.assert_array_equal(idx2[:k].cpu().numpy(), want[:k])
