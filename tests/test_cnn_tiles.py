"""The network's work items (csrc/cnn_tiles.h), without a GPU: over many shapes
and dilations every image pixel lies in one tile at its place, every product of
the weight gradients is formed once, reads stay in the guarded arrays, and small
networks take no more rounds of tiles than parts of four tiles, one tile an item
or tiles over the flattened rows would (a fixed four and no flat form had been
slower than the kernels before them: 64 x 64 with dilations 1 84 us against 63)."""
import os
import shutil
import subprocess

import pytest

from test_host_geometry import CSRC, ROOT


def test_items(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("g++ is missing")
    exe = str(tmp_path / "cnn_tiles_check")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, os.path.join(ROOT, "tests", "cnn_tiles_check.cpp"), "-o", exe],
                   check=True)
    out = subprocess.run([exe], capture_output=True, text=True, timeout=600)
    rows = {ln.split()[0]: [int(v) for v in ln.split()[1:]] for ln in out.stdout.splitlines()}
    assert out.returncode == 0 and rows, out.stdout + out.stderr
    assert all(v[0] == 0 and v[1] > 20 for v in rows.values()), rows
