"""The ring decomposition (csrc/rings.h) where memory runs out: an exception that a caller can catch, never the
end of the process."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def limits_check(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("g++ not found")
    exe = str(tmp_path_factory.mktemp("limits") / "ring_limits_check")
    src = os.path.join(HERE, "ring_limits_check.cpp")
    subprocess.run([cxx, "-O1", "-std=c++17", "-fopenmp", src, "-o", exe], check=True)
    return exe


def test_every_failed_allocation_reaches_the_caller(limits_check):
    r = subprocess.run([limits_check, "alloc", "7"], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, (r.returncode, r.stderr)
