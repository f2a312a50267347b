"""Solves whose vectors lie where a factorisation keeps its update matrices: factors of changing
type in one context, and factors with little or no room there."""
import numpy as np
import pytest

import gen
import paper_2508_16094_gb300 as gb

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.fixture(scope="module", autouse=True)
def _built():
    gb.build()


def test_factors_of_changing_type_in_one_context():
    lp = gen.grid_lp(9, 8, 7, seed=8)
    ctx = gb.IpmContext(lp.n, lp.m, lp.rowptr, lp.col, lp.l, lp.u, options=gb.default_options(storage_fp64=1))
    ctx.kkt_analyze(gen.nd_order_grid3d(9, 8, 7))
    ctx.ipm_set_workspace()
    B = dev(gen.normal(4, 8 * lp.n).reshape(8, lp.n))
    for step, prec in enumerate([gb.IPM_FP64, gb.IPM_TF32X3, gb.IPM_FP64, gb.IPM_FP32, gb.IPM_TF32, gb.IPM_FP64]):
        ctx.kkt_assemble(dev(lp.val), dev(10.0 ** gen.uniform(step, lp.m + 2 * lp.n, -1, 1)), 1e-8)
        ctx.kkt_factor(prec)
        for nrhs in (1, 8, 3, 1):
            X = torch.full((nrhs, lp.n), np.nan, dtype=torch.float64, device="cuda")
            assert ctx.kkt_solve(B[:nrhs], X, gb.IPM_REFINE_IR).rel_residual <= 1e-10


@pytest.mark.parametrize("prec", [gb.IPM_FP64, gb.IPM_TF32X3])
@pytest.mark.parametrize("n", [1, 500, 3000, 40000])
def test_factors_without_update_matrices(n, prec):
    # bounds only: K is diagonal
    ctx = gb.IpmContext(n, 0, np.zeros(1, np.int64), np.zeros(0, np.int32), np.zeros(n), np.ones(n),
                        options=gb.default_options(precision=prec, storage_fp64=int(prec == gb.IPM_FP64)))
    ctx.kkt_analyze(None)
    ctx.ipm_set_workspace()
    D = 10.0 ** gen.uniform(3, 2 * n, -1, 1)
    ctx.kkt_assemble(dev(np.zeros(1)), dev(D), 0.0)
    ctx.kkt_factor(prec)
    B = gen.normal(4, 11 * n).reshape(11, n)
    X = torch.empty((11, n), dtype=torch.float64, device="cuda")
    ctx.kkt_solve(dev(B), X, gb.IPM_REFINE_IR)
    ref = B / (D[:n] + D[n:])
    assert np.all(np.abs(X.cpu().numpy() - ref) <= 2e-10 * np.abs(B).max() / (D[:n] + D[n:]).min())
