"""The band-sweep blocks of the larger 3D levels (csrc/cluster3d.cpp), without
a GPU: the host code is compiled with g++ together with sweep3_check.cpp, which
runs the sweeps block by block -- values between sweeps through the compact
arrays -- and compares them bitwise with the same sweeps over the level's
lists; every node belongs to one block, a phase reads nothing that it writes,
every index stays in its section.  One block, more blocks than some levels have
nodes to share, sizes off powers of two."""
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
    exe = str(tmp_path_factory.mktemp("s3") / "sweep3_check")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-pthread", "-I", os.path.join(ROOT, "include"),
                    "-I", CSRC, "-I", inc, os.path.join(ROOT, "tests", "sweep3_check.cpp"),
                    os.path.join(CSRC, "cluster3d.cpp"), os.path.join(CSRC, "setup.cpp"), "-o", exe], check=True)
    return exe


@pytest.mark.parametrize("n,nc,blocks", [(65, 9, 1), (65, 9, 304), (85, 22, 40), (97, 25, 61)])
def test_sweep_blocks_equal_the_list_sweeps(checker, n, nc, blocks):
    out = subprocess.run([checker, str(n), str(nc), str(blocks)], capture_output=True, text=True, timeout=600)
    rows = [ln.split() for ln in out.stdout.splitlines()]
    assert rows and out.returncode == 0, out.stdout + out.stderr
    assert all(int(r[1]) == 0 for r in rows), rows
    assert {r[0] for r in rows} == {"values", "coverage", "race", "bounds"}
