"""The first column of a front's factor, which nothing but its pivot's root and one quotient
per entry makes: correctly rounded in the signed FP64 and the FP32 factors of the FMA pipe, in the
diagonal block and in the rows below it."""
import numpy as np
import pytest

import paper_2508_16094_gb300 as gb
from tests.test_gpu_dense_front import dense_front, factor_of

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    gb.build()


@pytest.mark.parametrize("seed", [3, 4, 5])
@pytest.mark.parametrize("n", [17, 64, 200])
def test_fp32(n, seed):
    ctx, K = dense_front(n, gb.default_options(precision=gb.IPM_FP32), seed=seed)
    P = ctx.kkt_symbolic_export()["perm"]
    col = K[np.ix_(P, P)][:, 0].astype(np.float32)
    ctx.kkt_factor(gb.IPM_FP32)
    L = factor_of(ctx, n)[:, 0]
    l0 = np.sqrt(col[0])
    assert L[0] == l0
    assert np.array_equal(L[1:], (col[1:] / l0).astype(np.float64))


@pytest.mark.parametrize("seed", [3, 4, 5])
@pytest.mark.parametrize("n,m", [(9, 3), (50, 14), (150, 50)])
def test_signed_fp64(n, m, seed):
    # every row of J dense: one front of n + m columns
    rng = np.random.default_rng(seed)
    rowptr = np.arange(m + 1, dtype=np.int64) * n
    ctx = gb.IpmContext(n, m, rowptr, np.tile(np.arange(n, dtype=np.int32), m), np.zeros(n), np.ones(n),
                        options=gb.default_options(storage_fp64=1, formulation=gb.IPM_FORM_AUGMENTED))
    N = n + m
    ctx.kkt_analyze(np.r_[n:N, 0:n].astype(np.int32))  # the negative pivots first
    dev = lambda a: torch.as_tensor(a, dtype=torch.float64, device="cuda")
    ctx.ipm_set_workspace()
    J, D = rng.standard_normal((m, n)), 10.0 ** rng.uniform(-1, 1, m + 2 * n)
    ctx.kkt_assemble(dev(J.ravel()), dev(D), 1e-8)
    ctx.kkt_factor(gb.IPM_FP64)
    S = ctx.kkt_symbolic_export()
    P = S["perm"]
    H = 1e-8 + D[m:m + n] + D[m + n:]
    K = np.block([[np.diag(H), J.T], [J, -np.diag(1.0 / D[:m])]])[np.ix_(P, P)]
    first = 0 if P[0] >= n else None
    assert first == 0
    rows = np.flatnonzero(K[:, 0])
    L = ctx.kkt_factor_entries(rows, np.zeros(len(rows), np.int32))
    l0 = np.sqrt(-K[0, 0])
    assert L[0] == l0
    assert np.array_equal(L[1:], K[rows[1:], 0] / -l0)
