"""FMA-pipe factor of one dense front at the edges of its tiles (panels of 16
columns, blocks of 64, update tiles of 32 and 64, FP32 super-steps of 256).

One dense row of J makes K a full n x n matrix, so the analysis has a single
front of n columns; K and L come back through the library's exports.
"""
import numpy as np
import pytest

import gen
import paper_2508_16094_gb300 as gb

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    gb.build()


def dense_front(n, options, seed=3, decades=1.0):
    """Context of the dense problem, assembled; K from the library's export."""
    rng = np.random.default_rng(seed)
    m = 3
    rowptr = np.arange(m + 1, dtype=np.int64) * n
    col = np.tile(np.arange(n, dtype=np.int32), m)
    ctx = gb.IpmContext(n, m, rowptr, col, np.zeros(n), np.ones(n), options=options)
    info = ctx.kkt_analyze(None)
    assert info.max_ncol == n
    ctx.ipm_set_workspace()
    dev = lambda a: torch.as_tensor(a, dtype=torch.float64, device="cuda")
    ctx.kkt_assemble(dev(rng.standard_normal(m * n)), dev(10.0 ** rng.uniform(-decades, decades, m + 2 * n)), 1e-8)
    K = np.zeros((n, n))
    i, j = np.tril_indices(n)
    order = np.lexsort((i, j))  # lower CSC
    K[i[order], j[order]] = ctx.kkt_export_assembled()
    return ctx, np.tril(K) + np.tril(K, -1).T


def factor_of(ctx, n):
    i, j = np.tril_indices(n)
    L = np.zeros((n, n))
    L[i, j] = ctx.kkt_factor_entries(i, j)
    return L


@pytest.mark.parametrize("prec", [gb.IPM_FP64, gb.IPM_FP32])
@pytest.mark.parametrize("n", [1, 2, 15, 16, 17, 33, 48, 63, 64, 65, 80, 96, 97, 128, 129, 191, 255, 256, 257, 320, 513])
def test_factor_backward_error_at_tile_edges(n, prec):
    ctx, K = dense_front(n, gb.default_options(precision=prec, storage_fp64=1))
    P = ctx.kkt_symbolic_export()["perm"]
    K = K[np.ix_(P, P)]
    ctx.kkt_factor(prec)
    L = factor_of(ctx, n)
    # |L L^T - K|_ij <= (n + 1) u sqrt(k_ii k_jj) for any order of the sums; a few
    # more u for the reciprocal of the pivot and for K rounded to FP32
    u = 2.0 ** -53 if prec == gb.IPM_FP64 else 2.0 ** -24
    d = np.sqrt(np.diag(K))
    assert np.all(np.abs(L @ L.T - K) <= (n + 10) * u * 1.01 * np.outer(d, d))


@pytest.mark.parametrize("n,bad", [(40, 0), (64, 63), (100, 70), (130, 129)])
def test_first_non_positive_pivot_is_reported(n, bad):
    # W = -2 on one variable makes exactly that leading minor the first indefinite one:
    # its diagonal becomes -1 plus small terms, the ones before it stay positive
    m = 1
    wp, wi = np.arange(n + 1), np.arange(n)
    ctx = gb.IpmContext(n, m, np.array([0, n]), np.arange(n, dtype=np.int32), None, None, wp, wi,
                        options=gb.default_options(storage_fp64=1))
    ctx.kkt_analyze(None)
    ctx.ipm_set_workspace()
    P = ctx.kkt_symbolic_export()["perm"]
    w = np.ones(n)
    w[P[bad]] = -2.0
    dev = lambda a: torch.as_tensor(a, dtype=torch.float64, device="cuda")
    ctx.kkt_assemble(dev(np.full(n, 1e-3)), dev(np.ones(m)), 1e-8, dev(w))
    st, col = ctx.kkt_factor(gb.IPM_FP64, raise_on_error=False)
    assert st == 5 and col == bad
