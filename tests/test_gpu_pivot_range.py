"""FP64 diagonal blocks whose pivots leave the range of the branch-free panel (FP32's normal
range), in every panel or in one of them."""
import numpy as np
import pytest

import paper_2508_16094_gb300 as gb
from tests.test_gpu_dense_front import factor_of

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
U = 2.0 ** -53


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.fixture(scope="module", autouse=True)
def _built():
    gb.build()


@pytest.mark.parametrize("n", [5, 16, 17, 64, 100])
@pytest.mark.parametrize("scale", ["small", "large", "one"])
def test_pivots_outside_fp32(n, scale):
    rng = np.random.default_rng(n)
    m = 2
    rowptr, col = np.arange(m + 1, dtype=np.int64) * n, np.tile(np.arange(n, dtype=np.int32), m)
    ctx = gb.IpmContext(n, m, rowptr, col, np.zeros(n), np.ones(n), options=gb.default_options(storage_fp64=1))
    ctx.kkt_analyze(np.arange(n, dtype=np.int32))
    ctx.ipm_set_workspace()
    s = {"small": 2.0 ** -300, "large": 2.0 ** 300, "one": 1.0}[scale]
    D = 10.0 ** rng.uniform(-1, 1, m + 2 * n) * s
    if scale == "one":
        D[m + n // 2] *= 2.0 ** 300  # a single diagonal entry far past the others
    ctx.kkt_assemble(dev(rng.standard_normal(m * n)), dev(D), 1e-8 * s)
    K = np.zeros((n, n))
    i, j = np.tril_indices(n)
    order = np.lexsort((i, j))  # lower CSC
    K[i[order], j[order]] = ctx.kkt_export_assembled()
    K = np.tril(K) + np.tril(K, -1).T
    P = ctx.kkt_symbolic_export()["perm"]
    K = K[np.ix_(P, P)]
    ctx.kkt_factor(gb.IPM_FP64)
    L = factor_of(ctx, n)
    # |L L^T - K|_ij <= (n + 10) u sqrt(k_ii k_jj), as for pivots of ordinary size, and the
    # products formed here round n times more
    d = np.sqrt(np.diag(K))
    assert np.all(np.isfinite(L))
    assert np.all(np.abs(L / d[:, None] @ (L / d[:, None]).T - K / np.outer(d, d)) <= (n + 10) * U * 1.01 + 4 * U * n)
