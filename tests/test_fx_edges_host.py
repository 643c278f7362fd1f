"""The fixed-point FP64 offset on the host (the same source as on the GPU) against
quadruple precision, where fx_host.cpp's draws are thin."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("no g++")
    out = str(tmp_path_factory.mktemp("fx") / "fx_edges_host")
    subprocess.run(["g++", "-O2", "-o", out, os.path.join(HERE, "fx_edges_host.cpp")], check=True)
    return out


def _run(exe, kind):
    r = subprocess.run([exe, "40000", str(kind)], check=True, capture_output=True, text=True)
    refused, worst, shifts = r.stdout.split()
    return int(refused), float(worst), int(shifts)


def test_sliver_beside_one_half(exe):
    """A component of 1e-12 to 1e-18 beside two nearly equal ones of 0.5 to 0.95, V0 within
    1e-12 of 1/2 (case (4) and its neighbours): d0 is below 1e-12 here, and what is left
    of the 2e-16 of test_fx_host.py is half the rounding of n1 + n2 and of y/2."""
    refused, worst, shifts = _run(exe, 0)
    assert (refused, shifts) == (0, 0) and worst <= 2e-16, (refused, worst, shifts)


@pytest.mark.parametrize("kind", [1, 2, 3, 4])
def test_normals_off_unit_length(exe, kind):
    """Lengths 1/2 to 2, unit L1 length, lengths down to 2^-58, components around 3/4: no
    cell with L < 2.999 is refused, and of the power of two above n3 |d0 error| <= 4e-16:
    half an ulp of s and of y/2 (below 1.5 and 1: 1.1e-16, 5.6e-17), half the rounding of
    n1 + n2 (5.6e-17, all doubled where three components of 3/4 and more are halved once
    more) and the root's own."""
    refused, worst, shifts = _run(exe, kind)
    assert (refused, shifts) == (0, 0) and worst <= 4e-16, (refused, worst, shifts)
