"""Right-hand sides that share a persistent solve: every group size and remainder
agrees with solving them one by one, in each storage type and for a signed factor."""
import numpy as np
import pytest

import gen
import paper_2508_16094_gb300 as gb

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
SHAPE = (7, 9, 8)


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.fixture(scope="module", autouse=True)
def _built():
    gb.build()


def factored(prec, form=gb.IPM_FORM_PRIMAL):
    lp = gen.grid_lp(*SHAPE, seed=8)
    o = gb.default_options(storage_fp64=int(prec == gb.IPM_FP64), formulation=form)
    ctx = gb.IpmContext(lp.n, lp.m, lp.rowptr, lp.col, lp.l, lp.u, options=o)
    ctx.kkt_analyze(gen.nd_order_grid3d(*SHAPE) if form == gb.IPM_FORM_PRIMAL else None)
    ctx.ipm_set_workspace()
    ctx.kkt_assemble(dev(lp.val), dev(10.0 ** gen.uniform(9, lp.m + 2 * lp.n, -1, 1)), 1e-8)
    ctx.kkt_factor(prec)
    return ctx


@pytest.mark.parametrize("nrhs", [2, 3, 4, 5, 9])
@pytest.mark.parametrize("prec,form,refine", [
    (gb.IPM_FP64, gb.IPM_FORM_PRIMAL, gb.IPM_REFINE_NONE),
    (gb.IPM_FP64, gb.IPM_FORM_AUGMENTED, gb.IPM_REFINE_IR),
    (gb.IPM_TF32X3, gb.IPM_FORM_PRIMAL, gb.IPM_REFINE_IR),
    (gb.IPM_BF16, gb.IPM_FORM_PRIMAL, gb.IPM_REFINE_IR),
    (gb.IPM_TF32, gb.IPM_FORM_PRIMAL, gb.IPM_REFINE_PCG),
    (gb.IPM_FP32, gb.IPM_FORM_PRIMAL, gb.IPM_REFINE_IR)])
def test_groups_agree_with_single_solves(prec, form, refine, nrhs):
    ctx = factored(prec, form)
    n = ctx.kkt_order()
    B = gen.normal(4, n * nrhs).reshape(nrhs, n) * 10.0 ** np.arange(nrhs)[:, None]
    B[1] = 0.0  # needs no steps: leaves the group at once
    B = dev(B)
    X = torch.full_like(B, np.nan)
    info = ctx.kkt_solve(B, X, refine)
    Y = torch.full_like(B, np.nan)
    ones = [ctx.kkt_solve(B[k], Y[k], refine) for k in range(nrhs)]
    # both sides end at a residual of at most 1e-10 of a system with cond < 1e5 (FP64, unrefined:
    # of a few u), so they differ by less than the sum of the two errors
    scale = 1e-10 if prec == gb.IPM_FP64 and refine == gb.IPM_REFINE_NONE else 2e-5
    assert torch.isfinite(X).all() and not X[1].any()
    for k in range(nrhs):
        assert float((X[k] - Y[k]).norm()) <= scale * float(Y[k].norm())
    assert info.iterations == sum(o.iterations for o in ones)
    assert info.used_pcg == max(o.used_pcg for o in ones)
    Z = B.clone()  # in place
    ctx.kkt_solve(Z, Z, refine)
    assert float((Z - Y).abs().max()) <= scale * float(Y.abs().max())


@pytest.mark.parametrize("prec", [gb.IPM_FP64, gb.IPM_TF32X3])
def test_a_wait_that_runs_out_drains_every_right_hand_side(prec):
    ctx = factored(prec)
    B = dev(gen.normal(4, 3 * ctx.kkt_order()).reshape(3, -1))
    X = torch.empty_like(B)
    ctx.kkt_test_solve_timeout(2000, 1)
    with pytest.raises(gb.IpmError) as e:
        ctx.kkt_solve(B, X, gb.IPM_REFINE_NONE)
    assert e.value.status == 8
    assert ctx.kkt_solve(B, X, gb.IPM_REFINE_IR).rel_residual <= 1e-10
