"""The FP64 adjoints' area and centroid on the host (the same source as on the GPU),
normals of unit length and others: no cell is refused, and the errors against quadruple
precision are no larger than those of the general formula in doubles (which has the
same number of roundings or more; a fifth more allowed for the draw)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("no g++")
    out = str(tmp_path_factory.mktemp("adj") / "adjoint64_host")
    subprocess.run(["g++", "-O2", "-o", out, os.path.join(HERE, "adjoint64_host.cpp")], check=True)
    return out


# unit length; lengths 1/2 to 2; unit L1 length; lengths 2^-8 to 1
@pytest.mark.parametrize("kind", range(4))
def test_lengths(exe, kind):
    r = subprocess.run([exe, "100000", str(kind)], check=True, capture_output=True, text=True)
    v = r.stdout.split()
    assert int(v[0]) == 0, r.stdout
    e = [float(x) for x in v[1:]]
    for k in range(3):
        worst, rms, worst_general, rms_general = e[4 * k:4 * k + 4]
        assert rms <= 1.2 * rms_general and worst <= 1.2 * worst_general, (k, r.stdout)
