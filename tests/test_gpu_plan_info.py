"""Plan info tells which node kernels a plan runs: those it has tables for."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nl():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_1410_3584_gb300 as mod
    return mod


@pytest.mark.parametrize("kernel,prec,opt,ring", [
    ("coulomb3d", "fp32", {}, True), ("coulomb3d", "fp64", {}, True), ("coulomb2d", "fp32", {}, True),
    ("poisson2d", "fp64", {}, True), ("coulomb3d", "fp64", {"method": 2}, True),
    ("coulomb3d", "fp32", {"spread_variant": 1}, False), ("coulomb3d", "fp32", {"tol": 1e-2}, False),
    ("coulomb2d", "fp32", {"tol": 1e-5}, False),
    ("coulomb3d", "fp64", {"method": 1}, False), ("coulomb2d", "fp32", {"method": 1}, False),
])
def test_sub_tile(nl, kernel, prec, opt, ring):
    n, L = ((16, 18, 20), (4.0, 4.5, 5.0)) if kernel.endswith("3d") else ((32, 36), (8.0, 9.0))
    plan = nl.Plan(n, L, kernel, prec, kmax=3.0, counts=(8, 8, 16) if len(n) == 3 else (16, 32), **opt)
    info = plan.info
    plan.close()
    assert (info["sub_tile"] > 0) == ring
    assert (info["segments"] > 0) == ring
