"""The workspaces' layouts on the host (the same source as in the library): every part
ends inside the size that plic_workspace_bytes answers."""
import os
import shutil
import subprocess

import pytest

from paper_2006_12838_gb300 import build as B
from paper_2006_12838_gb300 import plic

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lines(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("no g++")
    out = str(tmp_path_factory.mktemp("ws") / "workspace_host")
    subprocess.run(["g++", "-O1", "-o", out, os.path.join(HERE, "workspace_host.cpp")], check=True)
    return [int(v) for v in subprocess.run([out], check=True, capture_output=True, text=True).stdout.split()]


def test_batch_layout_inside_the_workspace(lines):
    assert lines[0] == 0, "%d counts of fields end beyond the workspace" % lines[0]


def test_compaction_layout_inside_the_workspace(lines):
    assert lines[1] == 0, "%d shapes" % lines[1]


def test_batch_size_query(lines):
    B.build()
    sizes = lines[2:]
    assert [plic.workspace_bytes(plic.WS_BATCHED, n) for n in range(len(sizes))] == sizes
    # sizes that callers hold from before stay enough
    assert sizes == [(56 * n + 16 + 255) // 256 * 256 + 256 for n in range(len(sizes))]
