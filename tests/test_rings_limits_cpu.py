"""The ring decomposition (csrc/rings.h) where memory or 32-bit tables run out: an exception that a caller
can catch, or a decline, never the end of the process."""
import os
import resource
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


@pytest.mark.parametrize("far,taken", [(1e3, 1), (1e6, 1), (3e8, 0), (3e9, 0), (1e18, 0), (1e300, 0)])
def test_far_nodes(limits_check, far, taken):
    """Balls far past the spectral box (its periods fold them back), in bounded memory."""
    r = subprocess.run([limits_check, "far", repr(far)], capture_output=True, text=True, timeout=300,
                       preexec_fn=lambda: resource.setrlimit(resource.RLIMIT_AS, (4 << 30, 4 << 30)))
    assert r.returncode == 0, (r.returncode, r.stderr)
    assert r.stdout.split() == [str(taken)] * 2
