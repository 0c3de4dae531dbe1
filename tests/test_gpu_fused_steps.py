"""Gradient-flow and time steps on grids whose axes take different routes, against the FP64 oracle: the
pointwise work rides in the FFT passes where the last axis (gradient flow) and the outer axis have
compile-time lengths, whatever axis 1 is.  Every axis has its own length, box and trap, so that tables of two axes
cannot be swapped unnoticed.  Bars of the one-step parity tests: 1e-10 (FP64) and 1e-5 (FP32)."""
import math

import numpy as np
import pytest

import workloads as W
from oracle import gf, potential, ts

pytestmark = pytest.mark.gpu

GRIDS = [
    ((64, 48, 96), (5.0, 4.2, 6.5)),     # fused, axis 1 on a length of the other kind
    ((96, 64, 128), (6.0, 4.6, 8.5)),    # fused on every axis
    ((96, 64, 54), (6.5, 5.0, 4.4)),     # the outer axis fused (time steps), the last one not
    ((60, 64, 64), (4.6, 5.2, 5.8)),     # the last axis alone
    ((64, 96), (6.0, 8.0)),              # 2D, fused
    ((96, 60), (8.0, 5.0)),
    ((160, 128), (10.0, 7.0)),           # 2D, the other fused lengths of few lines
    ((320, 160), (13.0, 9.0)),
    ((64, 24, 160), (5.0, 3.0, 8.0)),
]
BAR = {"fp64": 1e-10, "fp32": 1e-5}


@pytest.fixture(scope="module")
def nl():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_1410_3584_gb300 as m
    return m


@pytest.fixture(scope="module", params=GRIDS, ids=lambda p: "x".join(map(str, p[0])))
def setup(request):
    n, L = request.param
    g = W.Grid(n, L)
    kernel, counts = ("coulomb3d", (24, 16, 48)) if g.dim == 3 else ("coulomb2d", (32, 64))
    P = 0.6 * math.pi / max(g.h)
    V = W.harmonic_trap(g, (1.0, 1.4, 0.8)[:g.dim])
    return g, kernel, counts, P, V, potential.ConvolutionOperator(g, kernel, P, counts)


@pytest.mark.parametrize("max_inner", [200, 5])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_gf_step(nl, setup, prec, max_inner):
    import torch
    g, kernel, counts, P, V, op = setup
    beta, gc, tau, tol = 5.0, 0.7, 1e-2, 1e-12 if prec == "fp64" else 1e-6
    phi0 = W.normalized_gaussian_start(g, (1.3, 0.8, 1.5)[:g.dim])
    # 200 are never needed, five are used up
    G = gf.GradientFlow(g, V, beta, op, tau=tau, g=gc, inner_tol=tol, max_inner=max_inner)
    ref, ch_ref = G.step(phi0)
    assert (G.last_inner == max_inner) == (max_inner == 5)
    plan = nl.Plan(g.n, g.L, kernel, prec, kmax=P, counts=counts)
    dt = plan.torch_dtype
    phi = torch.from_numpy(phi0).to("cuda", dt)
    ch, it, _, _ = nl.nlp_gf_step(plan.handle, phi, torch.from_numpy(V).to("cuda", dt), beta, gc, tau, tol, max_inner,
                                  raise_on_nonconv=False)
    plan.close()
    err = np.max(np.abs(phi.double().cpu().numpy() - ref)) / np.max(np.abs(ref))
    assert err < BAR[prec], err
    assert abs(ch - ch_ref) < BAR[prec] * 50 * max(1.0, ch_ref)
    if prec == "fp64":
        assert abs(it - G.last_inner) <= 1


@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_ts_step(nl, setup, prec, order):
    import torch
    g, kernel, counts, P, V, op = setup
    psi0 = W.gaussian(g, [math.sqrt(2.0)] * g.dim, center=(0.5, -0.3, 0.2)[:g.dim]).astype(np.complex128)
    S = ts.TimeSplitting(g, V, 5.0, op, g=0.3)
    ref = psi0
    for _ in range(2):
        ref = S.step(ref, 0.02, order)
    plan = nl.Plan(g.n, g.L, kernel, prec, kmax=P, counts=counts)
    psi = torch.from_numpy(psi0).to("cuda", torch.complex128 if prec == "fp64" else torch.complex64)
    tV = torch.from_numpy(V).to("cuda", plan.torch_dtype)
    for _ in range(2):
        nl.nlp_ts_step(plan.handle, psi, tV, 5.0, 0.3, 0.02, order)
    plan.close()
    err = np.max(np.abs(psi.cpu().numpy().astype(np.complex128) - ref)) / np.max(np.abs(ref))
    assert err < BAR[prec], err
