"""Triangular solves through a narrow front (solved by one task a sweep) at the edges of
its range: k columns over r rows, beside a root that takes both."""
import numpy as np
import pytest

import paper_2508_16094_gb300 as gb

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
U = 2.0 ** -53


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.fixture(scope="module", autouse=True)
def _built():
    gb.build()


@pytest.mark.parametrize("prec", [gb.IPM_FP64, gb.IPM_TF32X3, gb.IPM_FP32])
@pytest.mark.parametrize("k,r", [(1, 1), (2, 3), (3, 130), (4, 31), (5, 300), (8, 257), (15, 16), (16, 255), (17, 256),
                                 (31, 257), (32, 511), (32, 512), (32, 513), (33, 64)])
def test_one_narrow_front(k, r, prec):
    # variables a (k), b (k) and s (r); one dense row over a and s, one over b and s: a's front
    # has k columns and the r rows of s, and b joins s in the root
    n = 2 * k + r
    rng = np.random.default_rng(100 * k + r)
    cols = [np.r_[0:k, 2 * k:n], np.arange(k, n)]
    rowptr = np.cumsum([0] + [len(c) for c in cols]).astype(np.int64)
    col, val = np.concatenate(cols).astype(np.int32), rng.standard_normal(rowptr[-1])
    ctx = gb.IpmContext(n, 2, rowptr, col, np.zeros(n), np.ones(n),
                        options=gb.default_options(precision=prec, storage_fp64=int(prec == gb.IPM_FP64)))
    ctx.kkt_analyze(np.arange(n, dtype=np.int32))
    S = ctx.kkt_symbolic_export()
    widths, rows = np.diff(S["super"]), np.diff(S["srp"])
    assert (k, r) in set(zip(widths.tolist(), rows.tolist()))
    ctx.ipm_set_workspace()
    D = 10.0 ** rng.uniform(-1, 1, 2 + 2 * n)
    ctx.kkt_assemble(dev(val), dev(D), 1e-8)
    ctx.kkt_factor(prec)
    J = np.zeros((2, n))
    for i, c in enumerate(cols):
        J[i, c] = val[rowptr[i]:rowptr[i + 1]]
    K = J.T @ (D[:2, None] * J) + np.diag(D[2:2 + n] + D[2 + n:] + 1e-8)
    B = rng.standard_normal((3, n))
    X = torch.empty((3, n), dtype=torch.float64, device="cuda")
    refine = gb.IPM_REFINE_NONE if prec == gb.IPM_FP64 else gb.IPM_REFINE_IR
    one = torch.empty(n, dtype=torch.float64, device="cuda")
    ctx.kkt_solve(dev(B[0]), one, refine)
    ctx.kkt_solve(dev(B), X, refine)
    # forward error of a backward-stable solve (FP64), or of a residual of at most 1e-10
    # (largest entries; sqrt(n) for the norms)
    c = np.linalg.cond(K)
    tol = 8 * (n + 2) * U * c if prec == gb.IPM_FP64 else 1e-10 * np.sqrt(n) * c
    ref = np.linalg.solve(K, B.T).T
    for x, y in [(one.cpu().numpy(), ref[0])] + list(zip(X.cpu().numpy(), ref)):
        assert np.linalg.norm(x - y) <= tol * np.linalg.norm(y)
