"""Potentials on grids of every common FFT length, few lines and many, against the FP64 oracle on the same
quadrature (the bars of the parity tests).  The other lengths are in test_gpu_rings.py."""
import math
import os
import sys

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import workloads as W  # noqa: E402
from oracle import potential  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nl():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_1410_3584_gb300 as mod
    return mod


@pytest.mark.parametrize("n", [32, 48, 64, 80, 96, 128, 160, 192])
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("shape", [(16, 18, 0), (0, 10, 16), (8, 0, 30), (0, 12), (20, 0)])
def test_common_lengths_vs_oracle(nl, prec, n, shape):
    import torch
    g = W.Grid(tuple(m or n for m in shape), tuple(0.25 * (m or n) for m in shape))
    kernel, counts = ("coulomb3d", (8, 8, 16)) if g.dim == 3 else ("coulomb2d", (12, 32))
    rho = W.random_density(g, 3)
    P = 0.9 * math.pi / max(g.h)
    for method in (0, 1):
        plan = nl.Plan(g.n, g.L, kernel, prec, kmax=P, counts=counts, tol=1e-6 if prec == "fp32" else 1e-12,
                       method=method)
        out = plan.eval(torch.from_numpy(rho).to("cuda", torch.float64 if prec == "fp64" else torch.float32))
        plan.close()
        ref = potential.eval_nufft(rho, g, kernel, P, counts, tol=1e-13)
        err = np.max(np.abs(out.double().cpu().numpy() - ref)) / np.max(np.abs(ref))
        assert err < (1e-5 if prec == "fp32" else 1e-10), (method, err)
