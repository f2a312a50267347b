"""The persistent FP64 triangular solve at the edges of its 64-wide blocks and
across fronts, the signed factor included, and its bounded waits."""
import numpy as np
import pytest

import gen
import paper_2508_16094_gb300 as gb
from tests.test_gpu_dense_front import dense_front

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
U = 2.0 ** -53


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.fixture(scope="module", autouse=True)
def _built():
    gb.build()


@pytest.mark.parametrize("n", [1, 2, 7, 8, 9, 63, 64, 65, 127, 128, 129, 200, 321])
def test_dense_front_solve(n):
    ctx, K = dense_front(n, gb.default_options(storage_fp64=1), seed=5)
    ctx.kkt_factor(gb.IPM_FP64)
    b = np.random.default_rng(n).standard_normal(n)
    x = torch.empty(n, dtype=torch.float64, device="cuda")
    ctx.kkt_solve(dev(b), x, gb.IPM_REFINE_NONE)
    # forward error of a backward-stable solve: at most a small multiple of n u cond(K)
    xr = np.linalg.solve(K, b)
    err = np.linalg.norm(x.cpu().numpy() - xr) / np.linalg.norm(xr)
    assert err <= 8 * (n + 2) * U * np.linalg.cond(K)


@pytest.mark.parametrize("shape,prec_tc", [((9, 8, 7), 0), ((5, 17, 11), 0), ((14, 14, 14), 1)])
def test_fronts_agree_with_the_level_schedule(shape, prec_tc):
    """kkt_solve (persistent) against kkt_solve_noalloc (level kernels) on one factor."""
    lp = gen.grid_lp(*shape, seed=8)
    o = gb.default_options(storage_fp64=1, fp64_tc=prec_tc)
    ctx = gb.IpmContext(lp.n, lp.m, lp.rowptr, lp.col, lp.l, lp.u, options=o)
    ctx.kkt_analyze(gen.nd_order_grid3d(*shape))
    ctx.ipm_set_workspace()
    ctx.kkt_assemble(dev(lp.val), dev(10.0 ** gen.uniform(9, lp.m + 2 * lp.n, -1, 1)), 1e-8)
    ctx.kkt_factor(gb.IPM_FP64)
    b = dev(gen.normal(4, lp.n))
    x, y = torch.empty_like(b), torch.empty_like(b)
    info = ctx.kkt_solve(b, x, gb.IPM_REFINE_NONE)
    ctx.kkt_solve_noalloc(b, y)
    assert info.rel_residual <= 1e-13  # of a matrix with cond < 1e5
    assert float((x - y).norm() / y.norm()) <= 1e-12


def test_signed_factor_solves_the_augmented_system():
    lp = gen.grid_lp(6, 5, 7, seed=12)
    o = gb.default_options(storage_fp64=1, formulation=gb.IPM_FORM_AUGMENTED)
    ctx = gb.IpmContext(lp.n, lp.m, lp.rowptr, lp.col, lp.l, lp.u, options=o)
    ctx.kkt_analyze(None)
    ctx.ipm_set_workspace()
    D = 10.0 ** gen.uniform(3, lp.m + 2 * lp.n, -1, 1)
    ctx.kkt_assemble(dev(lp.val), dev(D), 1e-8)
    ctx.kkt_factor(gb.IPM_FP64)
    A = lp.dense_A()
    H = np.diag(1e-8 + D[lp.m:lp.m + lp.n] + D[lp.m + lp.n:])
    M = np.block([[H, A.T], [A, -np.diag(1.0 / D[:lp.m])]])
    b = gen.normal(4, lp.n + lp.m)
    x = torch.empty(lp.n + lp.m, dtype=torch.float64, device="cuda")
    ctx.kkt_solve(dev(b), x, gb.IPM_REFINE_NONE)
    xr = np.linalg.solve(M, b)
    assert np.linalg.norm(x.cpu().numpy() - xr) <= 8 * len(b) * U * np.linalg.cond(M) * np.linalg.norm(xr)


@pytest.mark.parametrize("withheld", [0, 1])
def test_a_wait_that_runs_out_is_reported(withheld):
    lp = gen.grid_lp(8, seed=3)
    ctx = gb.IpmContext(lp.n, lp.m, lp.rowptr, lp.col, lp.l, lp.u, options=gb.default_options(storage_fp64=1))
    ctx.kkt_analyze(gen.nd_order_grid3d(8))
    ctx.ipm_set_workspace()
    ctx.kkt_assemble(dev(lp.val), dev(10.0 ** gen.uniform(9, lp.m + 2 * lp.n, -1, 1)), 1e-8)
    ctx.kkt_factor(gb.IPM_FP64)
    b = dev(gen.normal(4, lp.n))
    x = torch.empty_like(b)
    ctx.kkt_test_solve_timeout(2000, withheld)
    with pytest.raises(gb.IpmError) as e:
        ctx.kkt_solve(b, x, gb.IPM_REFINE_NONE)
    assert e.value.status == 8
    info = ctx.kkt_solve(b, x, gb.IPM_REFINE_NONE)
    assert info.rel_residual <= 1e-13
