"""The 2D boundary blocks as per-thread records (build_blocks2), without a GPU:
the setup code is compiled with g++ together with blocks2_check.cpp, which runs
every block's phases and compares the nodes it stores bitwise with a
relaxation's sweeps over the whole grid; a phase reads nothing that it writes,
and every source lies in the block's values.  Cases reach one and two records a
thread, no extra sweeps, and a halo too large for the records (the two-launch
form then runs)."""
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
    exe = str(tmp_path_factory.mktemp("b2") / "blocks2_check")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
                    "-I", inc, os.path.join(ROOT, "tests", "blocks2_check.cpp"), os.path.join(CSRC, "setup.cpp"),
                    "-o", exe], check=True)
    return exe


@pytest.mark.parametrize("n,nc,lam,delta,forms", [(257, 33, 5, 3.0, {(1, 256), (2, 256)}), (305, 39, 5, 3.0, None),
                                                  (129, 33, 0, 3.0, {(1, 256)}), (257, 129, 5, 8.0, {(2, 512)}),
                                                  (513, 257, 12, 12.0, {(0, 0)})])
def test_blocks_equal_the_grid_sweeps(checker, n, nc, lam, delta, forms):
    """forms: the (records a thread, threads) that the finer levels' blocks take."""
    out = subprocess.run([checker, str(n), str(nc), str(lam), str(delta)], capture_output=True, text=True, timeout=600)
    rows = [ln.split() for ln in out.stdout.splitlines()]
    assert rows and out.returncode == 0, out.stdout + out.stderr
    checks = [r for r in rows if r[0] != "records"]
    assert all(int(r[1]) == 0 and int(r[2]) > 0 for r in checks), checks
    got = {(int(r[2]), int(r[3])) for r in rows if r[0] == "records" and int(r[1]) > nc}
    assert forms is None or forms <= got, got
