"""Plans made on a non-blocking stream while the legacy stream is busy give the same results, bit for bit,
as those made on the legacy stream: their tables are copied and filled on their own stream."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu

KINDS = [
    ("coulomb3d", "fp32", {}), ("coulomb3d", "fp64", {}), ("coulomb3d", "fp32", {"spread_variant": 1}),
    ("dipole3d", "fp64", {"method": 1}), ("coulomb3d", "fp32", {"method": 2}),
    ("coulomb2d", "fp32", {}), ("poisson2d", "fp64", {}), ("coulomb2d", "fp64", {"spread_variant": 1}),
    ("coulomb2d", "fp64", {"method": 1}), ("poisson1d", "fp64", {}),
]


@pytest.fixture(scope="module")
def nl():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_1410_3584_gb300 as mod
    return mod


def _grid(kernel):
    if kernel.endswith("3d"):
        return W.Grid((24, 20, 30), (5.0, 4.5, 6.0)), {"kmax": 3.0, "counts": (16, 8, 32)}
    if kernel.endswith("2d"):
        return W.Grid((48, 60), (6.0, 8.0)), {"kmax": 3.0, "counts": (24, 48)}
    return W.Grid((128,), (8.0,)), {}


@pytest.mark.parametrize("kernel,prec,opt", KINDS)
def test_plans(nl, kernel, prec, opt):
    import torch
    g, kw = _grid(kernel)
    dt = torch.float64 if prec == "fp64" else torch.float32
    rho = torch.from_numpy(W.random_density(g, 5)).to("cuda", dt)
    plan = nl.Plan(g.n, g.L, kernel, prec, **kw, **opt)
    want = plan.eval(rho).clone()
    plan.close()
    st = torch.cuda.Stream()   # non-blocking
    busy = torch.randn(4096, 4096, device="cuda")
    torch.cuda.synchronize()
    for _ in range(40):
        busy = busy @ busy * 1e-2   # (tens of ms of the legacy stream)
    plan = nl.Plan(g.n, g.L, kernel, prec, stream=st, **kw, **opt)
    with torch.cuda.stream(st):
        out = plan.eval(rho)
        st.synchronize()
    assert torch.equal(out, want)
    plan.close()
