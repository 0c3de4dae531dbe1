"""FP32 ring plans of even width on balls that leave part of the spectrum out: their padded footprints
cover cells of zero weight past the last tap, which must have been written by this evaluation (zero times
what an allocation or an earlier call left there is NaN if that was NaN or infinite)."""
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
EVEN = (1e-3, 1e-5, 1e-7, 1e-9)   # w = 4, 6, 8, 10


@pytest.fixture(scope="module")
def nl():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_1410_3584_gb300 as mod
    return mod


def _fill_free_memory_with_nan(nl):
    """What a program leaves behind that freed other data: NaN patterns, and a plan of the other precision."""
    import torch
    plan = nl.Plan((48, 48, 48), (6.0, 6.0, 6.0), "coulomb3d", "fp64", kmax=6.0, counts=(8, 8, 16))
    plan.eval(torch.full((48, 48, 48), float("nan"), dtype=torch.float64, device="cuda"))
    plan.close()
    bufs = [torch.full((n,), float("nan"), device="cuda") for n in (1 << 19, 1 << 22, 1 << 22, 1 << 24, 1 << 26)]
    torch.cuda.synchronize()
    del bufs
    torch.cuda.empty_cache()


@pytest.mark.parametrize("tol", EVEN)
def test_even_widths_on_restricted_balls(nl, tol):
    import torch
    g = W.cube(64, 6.0)
    rho = torch.from_numpy(W.random_density(g, 5)).to("cuda", torch.float32)
    for frac in (0.5, 0.512, 0.524, 0.54, 0.56, 0.59, 0.62, 0.66, 0.7, 0.75):
        kw = dict(kmax=frac * math.pi / g.h[0], counts=(24, 12, 48), tol=tol)
        _fill_free_memory_with_nan(nl)
        out = []
        for variant in (0, 1):
            plan = nl.Plan(g.n, g.L, "coulomb3d", "fp32", spread_variant=variant, **kw)
            assert (plan.info["sub_tile"] > 0) == (variant == 0)
            out.append(plan.eval(rho).double().cpu().numpy())
            plan.close()
        err = np.max(np.abs(out[0] - out[1])) / np.max(np.abs(out[1]))
        assert err < 1e-5, (frac, err)


@pytest.mark.parametrize("tol", EVEN)
def test_improved_algorithm_after_a_density_of_nans(nl, tol):
    """Method 2 leaves the spectrum of I_1, on the whole frequency box, in the memory that I_2 reads next."""
    import torch
    for L in (6.0, 6.3, 6.6, 7.0, 7.4):
        g = W.cube(24, L)
        rho = torch.from_numpy(W.random_density(g, 3)).to("cuda", torch.float32)
        plan = nl.Plan(g.n, g.L, "coulomb3d", "fp32", counts=(16, 16, 32), method=2, tol=tol)
        first = plan.eval(rho).clone()
        assert bool(torch.isfinite(first).all())
        plan.eval(torch.full_like(rho, float("nan")))
        assert torch.equal(plan.eval(rho), first), L
        plan.close()


@pytest.mark.parametrize("kernel,prec", [("coulomb3d", "fp32"), ("coulomb3d", "fp64"), ("coulomb2d", "fp64")])
@pytest.mark.parametrize("kmax", [1e9, 1e18, 1e307])
def test_a_ball_past_every_table_is_refused(nl, kernel, prec, kmax):
    g = W.cube(16, 4.0, dim=int(kernel[-2]))
    with pytest.raises(nl.NlpError):
        nl.Plan(g.n, g.L, kernel, prec, kmax=kmax, counts=(8, 4, 16) if g.dim == 3 else (8, 16))
