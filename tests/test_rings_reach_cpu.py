"""The pruned FFT passes write the forward spectrum as far as ring_reach (csrc/rings.h) says: every cell
that a node's footprint covers, those of zero weight among them, has to lie within it."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def reach_check(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("g++ not found")
    exe = str(tmp_path_factory.mktemp("reach") / "ring_reach_check")
    src = os.path.join(HERE, "ring_reach_check.cpp")
    subprocess.run([cxx, "-O2", "-std=c++17", "-fopenmp", src, "-o", exe], check=True)
    return exe


@pytest.mark.parametrize("w,pad", [(w, 1) for w in range(4, 11)] + [(8, 0), (13, 0)])
@pytest.mark.parametrize("grid,rings", [((128, 96, 80), (24, 6, 48)), ((1, 96, 128), (24, 0, 48))])
def test_footprints_lie_within_the_reach(reach_check, grid, rings, w, pad):
    ends = 0
    for k in range(36):   # balls from 0.3 of Nyquist on, in steps that move the last first tap over even and odd
        f = 0.3 + 0.0131 * k
        args = [str(v) for v in (*grid, *rings, f, 0.9 * f, f, w, pad)]
        r = subprocess.run([reach_check, *args], capture_output=True, text=True)
        assert r.returncode == 0, (f, r.returncode, r.stdout)
        ends += int(r.stdout)
    assert ends > 0   # the reach is met, not merely an upper bound
