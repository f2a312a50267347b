"""NaN in a right-hand side, a matrix or a problem: no call may report success, and the
other right-hand sides of the same call keep their results."""
import numpy as np
import pytest

import gen
import paper_2508_16094_gb300 as gb

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
SHAPE = (6, 5, 7)
OK = 0


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.fixture(scope="module", autouse=True)
def _built():
    gb.build()


def context(prec, **kw):
    lp = gen.grid_lp(*SHAPE, seed=8)
    o = gb.default_options(precision=prec, storage_fp64=int(prec == gb.IPM_FP64), **kw)
    ctx = gb.IpmContext(lp.n, lp.m, lp.rowptr, lp.col, lp.l, lp.u, options=o)
    ctx.kkt_analyze(gen.nd_order_grid3d(*SHAPE))
    ctx.ipm_set_workspace()
    return ctx, lp


def solve_status(ctx, b, x, refine):
    try:
        ctx.kkt_solve(b, x, refine)
    except gb.IpmError as e:
        return e.status
    return OK


@pytest.mark.parametrize("prec", [gb.IPM_FP64, gb.IPM_TF32X3, gb.IPM_FP32])
@pytest.mark.parametrize("refine", [gb.IPM_REFINE_NONE, gb.IPM_REFINE_IR, gb.IPM_REFINE_PCG])
@pytest.mark.parametrize("whole", [False, True])
def test_nan_in_a_right_hand_side(prec, refine, whole):
    ctx, lp = context(prec, accept_tol=1e-2)
    ctx.kkt_assemble(dev(lp.val), dev(10.0 ** gen.uniform(9, lp.m + 2 * lp.n, -1, 1)), 1e-8)
    ctx.kkt_factor(prec)
    B = dev(gen.normal(4, 3 * lp.n).reshape(3, lp.n))
    X, Y = torch.empty_like(B), torch.empty_like(B)
    assert solve_status(ctx, B, X, refine) == OK
    bad = B.clone()
    if whole:
        bad[1] = float("nan")
    else:
        bad[1, lp.n // 3] = float("nan")
    assert solve_status(ctx, bad[1], Y[1], refine) != OK
    assert solve_status(ctx, bad, Y, refine) != OK
    assert torch.equal(X[0], Y[0]) and torch.equal(X[2], Y[2])


@pytest.mark.parametrize("prec", [gb.IPM_TF32X3, gb.IPM_FP32])
@pytest.mark.parametrize("refine", [gb.IPM_REFINE_NONE, gb.IPM_REFINE_IR, gb.IPM_REFINE_PCG])
def test_nan_in_the_matrix(prec, refine):
    # (these factors replace a pivot that is not a number and go on)
    ctx, lp = context(prec)
    D = 10.0 ** gen.uniform(9, lp.m + 2 * lp.n, -1, 1)
    D[lp.m // 2] = np.nan
    ctx.kkt_assemble(dev(lp.val), dev(D), 1e-8)
    ctx.kkt_factor(prec, raise_on_error=False)
    b = dev(gen.normal(4, lp.n))
    assert solve_status(ctx, b, torch.empty_like(b), refine) != OK


@pytest.mark.parametrize("n,at", [(4, 0), (4, 3), (700, 300)])
@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("refine", [gb.IPM_REFINE_NONE, gb.IPM_REFINE_IR, gb.IPM_REFINE_PCG])
def test_a_solution_past_the_largest_number(n, at, sign, refine):
    # bounds only: K is diagonal, and one entry of the solution, 5 / 1e-308, overflows
    ctx = gb.IpmContext(n, 0, np.zeros(1, np.int64), np.zeros(0, np.int32), np.zeros(n), np.ones(n),
                        options=gb.default_options(storage_fp64=1))
    ctx.kkt_analyze(None)
    ctx.ipm_set_workspace()
    D, b = np.ones(2 * n), np.ones((2, n))
    D[at], D[n + at], b[1, at] = 1e-308, 0.0, 5.0 * sign
    ctx.kkt_assemble(dev(np.zeros(1)), dev(D), 0.0)
    ctx.kkt_factor(gb.IPM_FP64)
    x, X = torch.empty(n, dtype=torch.float64, device="cuda"), torch.empty((2, n), dtype=torch.float64, device="cuda")
    assert solve_status(ctx, dev(b[0]), x, refine) == OK
    assert solve_status(ctx, dev(b[1]), x, refine) != OK
    assert solve_status(ctx, dev(b), X, refine) != OK


@pytest.mark.parametrize("prec", [gb.IPM_FP64, gb.IPM_TF32X3])
@pytest.mark.parametrize("what", ["val", "b", "c"])
def test_nan_in_a_problem(prec, what):
    ctx, lp = context(prec)
    data = {"val": lp.val.copy(), "b": lp.b.copy(), "c": lp.c.copy()}
    data[what][len(data[what]) // 2] = np.nan
    x, s, lam = (torch.empty(k, dtype=torch.float64, device="cuda") for k in (lp.n, ctx.m_tot, ctx.m_tot))
    assert ctx.ipm_solve(dev(data["val"]), dev(data["b"]), dev(data["c"]), x, s, lam).status != OK
