"""The ring kernels on the GPU against the generic one-warp-per-node kernel (spread_variant=1):
the same w-tap NUFFT in another order of summation, so the two differ by rounding alone (FP64:
sums of ~1e4 terms; FP32: both evaluate kernel values to ~1e-6)."""
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
BOUND = {"fp64": 1e-12, "fp32": 1e-5}


@pytest.fixture(scope="module")
def nl():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_1410_3584_gb300 as mod
    return mod


def _both(nl, g, kernel, prec, **kw):
    import torch
    rho = torch.from_numpy(W.random_density(g, 5)).to("cuda", torch.float64 if prec == "fp64" else torch.float32)
    out = []
    for variant in (0, 1):
        plan = nl.Plan(g.n, g.L, kernel, prec, spread_variant=variant, **kw)
        assert (plan.info["sub_tile"] > 0) == (variant == 0)
        out.append(plan.eval(rho).double().cpu().numpy())
        plan.close()
    return np.max(np.abs(out[0] - out[1])) / np.max(np.abs(out[1]))


@pytest.mark.parametrize("prec,tol", [("fp32", t) for t in (1e-3, 1e-4, 1e-5, 1e-6, 1e-7, 1e-8, 1e-9)] +
                         [("fp64", t) for t in (1e-7, 1e-8, 1e-9, 1e-10, 1e-11, 1e-12, 1e-13, 1e-14)])
def test_every_width(nl, prec, tol):
    """w = 4 ... 10 (FP32) and 8 ... 15 (FP64), an uneven box, taps that wrap past Nyquist."""
    g = W.Grid((30, 24, 20), (7.0, 6.0, 5.0))
    assert _both(nl, g, "coulomb3d", prec, kmax=math.pi / max(g.h), counts=(24, 16, 40), tol=tol) < BOUND[prec]


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("n,L,frac,counts", [
    ((8, 8, 8), (3.0, 3.0, 3.0), 1.0, (4, 2, 2)),            # two nodes a ring, the window wider than the grid's half
    ((18, 10, 50), (4.0, 3.0, 9.0), 1.0, (16, 8, 30)),       # fine grid not a multiple of the patches
    ((36, 36, 36), (8.0, 8.0, 8.0), 0.2, (12, 12, 34)),      # a small ball: most of the spectrum left out
    ((32, 32, 32), (8.0, 8.0, 8.0), 1.4, (16, 16, 24)),      # a ball past the spectral box
    ((24, 24, 24), (6.0, 6.0, 6.0), 1.0, (8, 2, 2050)),      # dense rings: arcs at the node limit
    ((64, 48, 40), (8.0, 6.0, 5.0), 1.0, (32, 32, 2)),       # far nodes
])
def test_shapes(nl, prec, n, L, frac, counts):
    g = W.Grid(n, L)
    tol = 1e-6 if prec == "fp32" else 1e-12
    err = _both(nl, g, "dipole3d", prec, kmax=frac * math.pi / max(g.h), counts=counts, tol=tol,
                dipole_axis=(1.0, 0.5, 2.0))
    assert err < BOUND[prec]


@pytest.mark.parametrize("kernel,kw", [("coulomb2d", {}), ("poisson2d", {}), ("confined2d", {"eps": 0.5})])
@pytest.mark.parametrize("prec,tol", [("fp32", 1e-6), ("fp64", 1e-7), ("fp64", 1e-12), ("fp64", 1e-14)])
@pytest.mark.parametrize("n,L,frac,counts", [
    ((64, 48), (8.0, 6.0), 1.0, (32, 96)),
    ((8, 10), (3.0, 3.0), 1.0, (4, 4)),                # windows as wide as the grid
    ((90, 36), (9.0, 5.0), 0.3, (16, 702)),            # a small disc, dense rings
    ((24, 24), (6.0, 6.0), 1.5, (10, 16)),             # a disc past the spectral box
])
def test_2d(nl, kernel, kw, prec, tol, n, L, frac, counts):
    g = W.Grid(n, L)
    # Poisson: W(k) divides differences of rho-hat by |k|, about 1/(r_1 P) = n_r^2 times the rounding of rho-hat
    amp = 10.0 if kernel == "poisson2d" else 1.0
    err = _both(nl, g, kernel, prec, kmax=frac * math.pi / max(g.h), counts=counts, tol=tol, **kw)
    assert err < amp * BOUND[prec]


@pytest.mark.parametrize("prec,method", [("fp32", 0), ("fp64", 0), ("fp64", 2)])
def test_an_evaluation_leaves_nothing_behind(nl, prec, method):
    """A density of NaNs and infinities does not reach the next evaluation of the plan."""
    import torch
    g = W.cube(24, 6.0)
    plan = nl.Plan(g.n, g.L, "coulomb3d", prec, kmax=2.0, counts=(16, 16, 32), method=method)
    dt = torch.float64 if prec == "fp64" else torch.float32
    rho = torch.from_numpy(W.random_density(g, 3)).to("cuda", dt)
    first = plan.eval(rho).clone()
    bad = rho.clone()
    bad[3, 4, 5] = float("nan")
    bad[7, 8, 9] = float("inf")
    plan.eval(bad)
    assert torch.equal(plan.eval(rho), first)
    plan.close()


@pytest.mark.parametrize("n", [24, 30, 36, 40, 50, 54, 60, 72, 90, 100, 108, 120, 144, 150, 162, 180])
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_fft_lengths_vs_oracle(nl, prec, n):
    """Every fine-grid length 2 n with kernels of its own radices, on each axis, against the FP64
    oracle on the same quadrature (the bars of the parity tests)."""
    import torch
    from oracle import potential
    for shape in ((n, n, 16), (16, 18, n)):
        g = W.Grid(shape, tuple(0.25 * m for m in shape))
        rho = W.random_density(g, 3)
        P, counts = 0.9 * math.pi / max(g.h), (8, 8, 16)
        plan = nl.Plan(g.n, g.L, "coulomb3d", prec, kmax=P, counts=counts, tol=1e-6 if prec == "fp32" else 1e-12)
        out = plan.eval(torch.from_numpy(rho).to("cuda", torch.float64 if prec == "fp64" else torch.float32))
        plan.close()
        ref = potential.eval_nufft(rho, g, "coulomb3d", P, counts, tol=1e-13)
        err = np.max(np.abs(out.double().cpu().numpy() - ref)) / np.max(np.abs(ref))
        assert err < (1e-5 if prec == "fp32" else 1e-11), (shape, err)


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("nx", [720, 800, 864, 960, 1000])
def test_2d_long_first_axis(nl, prec, nx):
    """Fine axes of 2 nx points that run as two passes of 45 ... 125 points (in FP64 the blocks of 60
    and 125 points hold fewer lines), against the FP64 oracle."""
    import torch
    from oracle import potential
    g = W.Grid((nx, 48), (0.02 * nx, 4.0))
    rho = W.random_density(g, 4)
    P, counts = 0.5 * math.pi / max(g.h), (12, 32)
    plan = nl.Plan(g.n, g.L, "coulomb2d", prec, kmax=P, counts=counts, tol=1e-6 if prec == "fp32" else 1e-12)
    out = plan.eval(torch.from_numpy(rho).to("cuda", torch.float64 if prec == "fp64" else torch.float32))
    plan.close()
    ref = potential.eval_nufft(rho, g, "coulomb2d", P, counts, tol=1e-13)
    err = np.max(np.abs(out.double().cpu().numpy() - ref)) / np.max(np.abs(ref))
    assert err < (1e-5 if prec == "fp32" else 1e-11), err
