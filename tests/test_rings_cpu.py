"""The ring decomposition of the 3D and 2D nodes (csrc/rings.h) on the CPU: its tables, followed as the
kernels follow them, against the direct sums over every node's taps on the periodic grid."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def ring_check(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("g++ not found")
    exe = str(tmp_path_factory.mktemp("rings") / "ring_check")
    subprocess.run([cxx, "-O2", "-std=c++17", "-fopenmp", os.path.join(HERE, "ring_check.cpp"), "-o", exe], check=True)
    return exe


# fine grid, rings (radii x angles) and nodes a ring, ball radius over the Nyquist radius per axis, w,
# padded footprints, most cells of a strip
@pytest.mark.parametrize("grid,rings,radius,w,pad,cells", [
    ((36, 40, 30), (8, 5, 24), (1, 1, 1), 7, 1, 768),             # taps past Nyquist wrap and mirror
    ((36, 40, 30), (8, 5, 24), (1, 1, 1), 7, 1, 100),             # many short arcs
    ((36, 40, 30), (8, 5, 24), (.6, .9, .7), 13, 0, 1600),        # an ellipsoid inside the box
    ((18, 20, 24), (6, 4, 10), (1.7, 2.3, 1.9), 7, 1, 768),       # a ball larger than the box
    ((18, 20, 24), (6, 4, 10), (1.7, 2.3, 3.9), 8, 0, 1600),      # ... whose last-axis images repeat
    ((64, 64, 64), (16, 16, 64), (1, 1, 1), 10, 1, 768),
    ((16, 16, 16), (6, 3, 4098), (1, 1, 1), 4, 1, 768),           # dense rings, arcs at the node limit
    ((16, 16, 16), (2, 1, 2), (.3, .3, .3), 15, 0, 1600),         # two nodes a ring, windows wider than the ball
    ((64, 48, 40), (16, 16, 2), (40, 37, 1), 13, 0, 1600),        # far nodes: one node an arc
    ((1, 64, 48), (20, 0, 36), (1, 1, 1), 7, 1, 768),             # 2D (no angle theta), to Nyquist
    ((1, 50, 36), (12, 0, 20), (1, .4, .6), 13, 0, 1600),
    ((1, 20, 24), (9, 0, 14), (1, 1.7, 2.3), 13, 0, 1600),        # 2D, a ball larger than the box
    ((1, 36, 20), (6, 0, 600), (1, .9, .9), 7, 1, 100),
])
def test_ring_tables_reproduce_the_direct_sums(ring_check, grid, rings, radius, w, pad, cells):
    args = [str(v) for v in (*grid, *rings, *radius, w, pad, cells)]
    r = subprocess.run([ring_check, *args], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    interp, spread = (float(v) for v in r.stdout.split())
    # sums of at most a few thousand FP64 terms of the size of the largest value
    assert interp < 1e-12 and spread < 1e-12, r.stdout
