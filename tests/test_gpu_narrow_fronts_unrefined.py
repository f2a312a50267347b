"""Narrow fronts of FP32-storage factors, unrefined: refinement would hide a row or a column
that a sweep drops."""
import numpy as np
import pytest

import paper_2508_16094_gb300 as gb

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
U32 = 2.0 ** -24


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.fixture(scope="module", autouse=True)
def _built():
    gb.build()


@pytest.mark.parametrize("prec", [gb.IPM_TF32X3, gb.IPM_FP32])
@pytest.mark.parametrize("k,r", [(1, 1), (2, 3), (3, 130), (4, 31), (5, 300), (8, 257), (15, 16), (16, 255), (17, 256),
                                 (31, 257), (32, 511), (32, 512), (32, 513), (33, 64)])
def test_backward_error(k, r, prec):
    # the pattern of test_gpu_narrow_fronts.py: a's front has k columns and the r rows of s
    n = 2 * k + r
    rng = np.random.default_rng(100 * k + r)
    cols = [np.r_[0:k, 2 * k:n], np.arange(k, n)]
    rowptr = np.cumsum([0] + [len(c) for c in cols]).astype(np.int64)
    col, val = np.concatenate(cols).astype(np.int32), rng.standard_normal(rowptr[-1])
    ctx = gb.IpmContext(n, 2, rowptr, col, np.zeros(n), np.ones(n),
                        options=gb.default_options(precision=prec, storage_fp64=0, accept_tol=1.0))
    ctx.kkt_analyze(np.arange(n, dtype=np.int32))
    ctx.ipm_set_workspace()
    D = 10.0 ** rng.uniform(-1, 1, 2 + 2 * n)
    ctx.kkt_assemble(dev(val), dev(D), 1e-8)
    ctx.kkt_factor(prec)
    J = np.zeros((2, n))
    for i, c in enumerate(cols):
        J[i, c] = val[rowptr[i]:rowptr[i + 1]]
    K = J.T @ (D[:2, None] * J) + np.diag(D[2:2 + n] + D[2 + n:] + 1e-8)
    B = rng.standard_normal((3, n))
    X, one = torch.empty((3, n), dtype=torch.float64, device="cuda"), torch.empty(n, dtype=torch.float64, device="cuda")
    ctx.kkt_solve(dev(B[0]), one, gb.IPM_REFINE_NONE)
    ctx.kkt_solve(dev(B), X, gb.IPM_REFINE_NONE)
    # factor and two sweeps of n-term sums in FP32 (the split products keep 2^-22): a small
    # multiple of n u of |K| |x|; a row left out is an error of the order of |K| |x| / n
    norm = np.linalg.norm(K, np.inf)
    for x, b in [(one.cpu().numpy(), B[0])] + list(zip(X.cpu().numpy(), B)):
        eta = np.abs(K @ x - b).max() / (norm * np.abs(x).max() + np.abs(b).max())
        assert eta <= 16 * U32 * np.sqrt(n)
