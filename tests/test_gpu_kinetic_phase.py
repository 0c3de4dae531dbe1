"""FP32 time splitting: the kinetic flow's phase is formed in FP64 and rounded once.

The transform of a delta function is exactly one everywhere, so a step from it without a potential leaves
the square of the phase factors in the modes, with the random error of three FP32 transforms on top.
The error of a factor rounded once is known; the modes' errors, projected on it, give 1 if that is the error
the factors have.  Factors rounded per axis and multiplied in FP32 have another one (projection near 0).
"""
import math
import os
import sys

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nl():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_1410_3584_gb300 as mod
    return mod


@pytest.mark.parametrize("n", [(64, 16, 20), (24, 32, 20)])   # an outer axis whose passes carry the phase, and one whose don't
def test_factors_are_rounded_once(nl, n):
    import torch
    g = W.Grid(n, (8.0, 2.3, 2.9))
    N, tau = float(np.prod(n)), 0.05
    mu2 = sum(k * k for k in np.meshgrid(*(np.fft.fftfreq(m) * m * math.pi / L for m, L in zip(g.n, g.L)), indexing="ij"))
    f = np.exp(-0.25j * tau * mu2)
    rounded = (f / N).astype(np.complex64).astype(np.complex128) * N - f
    plan = nl.Plan(g.n, g.L, "coulomb3d", "fp32", kmax=2.0, counts=(4, 4, 8))
    psi = torch.zeros(n, dtype=torch.complex64, device="cuda")
    psi[0, 0, 0] = 1.0
    nl.nlp_ts_step(plan.handle, psi, torch.zeros(n, dtype=torch.float32, device="cuda"), 0.0, 0.0, tau, 2)
    plan.close()
    err = np.fft.fftn(psi.cpu().numpy().astype(np.complex128)) - f * f
    want = 2.0 * f * rounded
    slope = float(np.sum((err * want.conj()).real) / np.sum(np.abs(want) ** 2))
    # the transforms' error is about 1.5e-7 rms a mode and independent of `rounded` (4e-8 in the square): the
    # projection is uncertain by 4 / sqrt(2 N) = 0.03 at the most, the bar is five times that
    assert abs(slope - 1.0) < 0.15, slope
