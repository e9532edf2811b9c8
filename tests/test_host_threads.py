"""The setup's loops over the host's threads (csrc/host_threads.h), without a
GPU: an exception inside one thread -- an allocation that fails while a batch's
domains, coarsest inverses or junction solves are built -- reaches the entry
point, which returns a status; it used to end the process."""
import os
import shutil
import subprocess

import pytest

from test_host_geometry import CSRC, ROOT


def test_exceptions_reach_the_caller(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("g++ is missing")
    exe = str(tmp_path / "host_threads_check")
    subprocess.run(["g++", "-O2", "-std=c++17", "-pthread", "-I", CSRC,
                    os.path.join(ROOT, "tests", "host_threads_check.cpp"), "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0 and out.stdout.strip() == "0", out.stdout + out.stderr


def test_no_other_threads_in_the_setup():
    """Threads started in any other way are the two that hold their own exception."""
    found = {}
    for f in sorted(os.listdir(CSRC)):
        src = open(os.path.join(CSRC, f)).read()
        n = src.count("emplace_back(work)") + src.count("pool.emplace_back([") + src.count("= std::thread(")
        if n:
            found[f] = n
    assert found == {"api.cu": 1, "cluster3d.cpp": 1, "host_threads.h": 1}, found
