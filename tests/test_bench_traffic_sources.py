"""The digest that marks captured DRAM traffic as stale covers every source that decides it: the ring
kernels and their tables' builder, with what these include."""
import os
import re
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import bench  # noqa: E402

CSRC = "paper_1410_3584_gb300/csrc/"


def _closure(start):
    seen, todo = set(), list(start)
    while todo:
        f = todo.pop()
        if f in seen:
            continue
        seen.add(f)
        with open(os.path.join(ROOT, CSRC, f), encoding="utf-8") as fh:
            todo += [i for i in re.findall(r'#include "([^"]+)"', fh.read()) if "/" not in i]
    return {CSRC + f for f in seen}


def test_digest_covers_the_ring_kernels_sources():
    assert _closure(["ring_dev.cuh", "rings.h"]) <= set(bench.TRAFFIC_SOURCES)
    assert {CSRC + "plan.cu", CSRC + "ring_launch.cuh"} <= set(bench.TRAFFIC_SOURCES)
