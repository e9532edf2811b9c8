"""The 3D cluster programs (csrc/cluster3d.cpp), without a GPU: the host code
is compiled with g++ together with cluster3_check.cpp, which runs the phases
of every level's program rank by rank -- a whole sweep each, own values sent into
the other ranks' inboxes, two values a ghost -- and compares them bitwise with
the same sweeps over the level's lists; a phase reads nothing that it writes,
every copy is sent in the sweep that changes it, and every index stays in its
section.  Levels from 9^3 (a few nodes
a rank) up, with and without a junction zone, sizes off powers of two."""
import os
import shutil
import subprocess

import pytest

from test_host_geometry import CSRC, ROOT, _cuda_include


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    inc = _cuda_include()
    if shutil.which("g++") is None or inc is None:
        pytest.skip("g++ or the CUDA headers are missing")
    exe = str(tmp_path_factory.mktemp("c3") / "cluster3_check")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
                    "-I", inc, os.path.join(ROOT, "tests", "cluster3_check.cpp"), os.path.join(CSRC, "cluster3d.cpp"),
                    os.path.join(CSRC, "setup.cpp"), "-o", exe], check=True)
    return exe


@pytest.mark.parametrize("n,nc", [(65, 9), (85, 22), (97, 25)])
def test_cluster_programs_equal_the_list_sweeps(checker, n, nc):
    out = subprocess.run([checker, str(n), str(nc)], capture_output=True, text=True, timeout=600)
    rows = [ln.split() for ln in out.stdout.splitlines()]
    assert rows and out.returncode == 0, out.stdout + out.stderr
    assert all(int(r[1]) == 0 for r in rows), rows
    assert {r[0] for r in rows} >= {"band_and_zone", "zone", "stale", "race", "bounds"}
    assert all(int(r[2]) > 0 for r in rows), rows
