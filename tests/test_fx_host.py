"""The fixed-point FP64 offset on the host (the same source as on the GPU),
against quadruple precision: |d0 error| <= 2e-16, the sum of half an ulp of numbers
up to 0.87 (5.6e-17), of y/2 with y up to 1.74 (5.6e-17) and of half the rounding of
n1 + n2 up to 1.41 (5.6e-17), and the root's own error (a few units of 2^-58 over a
derivative of at least 3); no cell inside the scheme's range is refused, no shift
count is negative."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("no g++")
    out = str(tmp_path_factory.mktemp("fx") / "fx_host")
    subprocess.run(["g++", "-O2", "-o", out, os.path.join(HERE, "fx_host.cpp")], check=True)
    return out


@pytest.mark.parametrize("kind", range(6))
def test_against_quadruple_precision(exe, kind):
    r = subprocess.run([exe, "40000", str(kind)], check=True, capture_output=True, text=True)
    refused, worst, shifts = r.stdout.split()
    assert (int(refused), int(shifts)) == (0, 0) and float(worst) <= 2e-16, r.stdout
