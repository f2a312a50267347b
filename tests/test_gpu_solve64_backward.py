"""Backward error of one unrefined FP64 solve beside that of substitution.

kkt_solve works with inverses of the factor's 64-wide diagonal blocks, kkt_solve_noalloc
substitutes; both on one factor. A product with an inverse alone leaves a residual of
|L| |L^-1| |v| u where substitution leaves |L| |y| u, which differ by the condition of the
block: tried on a block where that is large, and on fronts with D over many decades.
"""
import numpy as np
import pytest

import gen
import paper_2508_16094_gb300 as gb

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
U = 2.0 ** -53


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.fixture(scope="module", autouse=True)
def _built():
    gb.build()


def backward_errors(ctx, K, B):
    """Normwise (largest row sum), kkt_solve's and kkt_solve_noalloc's, per right-hand side."""
    out = []
    Kl = K.astype(np.longdouble)
    norm = float(np.abs(K).sum(axis=1).max())
    for b in B:
        bd = dev(b)
        for f in (lambda x: ctx.kkt_solve(bd, x, gb.IPM_REFINE_NONE, raise_on_error=False),
                  lambda x: ctx.kkt_solve_noalloc(bd, x)):
            x = torch.empty_like(bd)
            f(x)
            x = x.cpu().numpy()
            r = np.abs(Kl @ x - b).max()
            out.append(float(r) / (norm * np.abs(x).max() + np.abs(b).max()))
    e = np.array(out).reshape(-1, 2)
    return e[:, 0], e[:, 1]


def check(new, ref):
    # the same bound, gamma_k |L| |y| a block, holds for both and the sums differ in their order
    # only; medians over many right-hand sides: within a factor of two, and the rounding of x
    assert np.median(new) <= 2.0 * np.median(ref) + U


@pytest.mark.parametrize("n,c", [(20, 0.5), (32, 0.35), (63, 0.2), (64, 0.2), (65, 0.2), (100, 0.1), (130, 0.1)])
def test_ill_conditioned_diagonal_block(n, c):
    # L: ones, -c below the diagonal; its inverse grows as (1 + c)^k
    L = np.eye(n) - c * np.tril(np.ones((n, n)), -1)
    W = L @ L.T
    i, j = np.tril_indices(n)
    order = np.lexsort((i, j))  # lower CSC
    i, j = i[order], j[order]
    wp = np.concatenate([[0], np.cumsum(np.arange(n, 0, -1))]).astype(np.int64)
    ctx = gb.IpmContext(n, 1, np.array([0, 1]), np.zeros(1, np.int32), None, None, wp, i.astype(np.int32),
                        options=gb.default_options(storage_fp64=1))
    ctx.kkt_analyze(np.arange(n, dtype=np.int32))
    ctx.ipm_set_workspace()
    ctx.kkt_assemble(dev(np.zeros(1)), dev(np.ones(1)), 0.0, dev(W[i, j]))
    ctx.kkt_factor(gb.IPM_FP64)
    rng = np.random.default_rng(n)
    K = np.tril(W) + np.tril(W, -1).T
    B = np.concatenate([rng.standard_normal((20, n)), rng.standard_normal((20, n)) @ K])
    check(*backward_errors(ctx, K, B))


@pytest.mark.parametrize("decades", [1, 4, 8])
@pytest.mark.parametrize("form", [gb.IPM_FORM_PRIMAL, gb.IPM_FORM_AUGMENTED])
def test_fronts(form, decades):
    shape = (7, 8, 6)
    lp = gen.grid_lp(*shape, seed=8)
    ctx = gb.IpmContext(lp.n, lp.m, lp.rowptr, lp.col, lp.l, lp.u,
                        options=gb.default_options(storage_fp64=1, formulation=form))
    ctx.kkt_analyze(gen.nd_order_grid3d(*shape) if form == gb.IPM_FORM_PRIMAL else None)
    ctx.ipm_set_workspace()
    D = 10.0 ** gen.uniform(9, lp.m + 2 * lp.n, -decades, decades)
    ctx.kkt_assemble(dev(lp.val), dev(D), 1e-8)
    ctx.kkt_factor(gb.IPM_FP64)
    A = lp.dense_A()
    H = np.diag(1e-8 + D[lp.m:lp.m + lp.n] + D[lp.m + lp.n:])
    if form == gb.IPM_FORM_PRIMAL:
        K = A.T @ (D[:lp.m, None] * A) + H
    else:
        K = np.block([[H, A.T], [A, -np.diag(1.0 / D[:lp.m])]])
    B = np.random.default_rng(3).standard_normal((20, len(K)))
    check(*backward_errors(ctx, K, B))
