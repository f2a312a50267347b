"""FP32-storage factors of a matrix whose entries are FP32 subnormals: its factor is of
ordinary size and stays finite, and no pivot counts as perturbed."""
import numpy as np
import pytest

import paper_2508_16094_gb300 as gb
from tests.test_gpu_dense_front import factor_of

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    gb.build()


@pytest.mark.parametrize("prec", [gb.IPM_FP32, gb.IPM_TF32, gb.IPM_TF32X3])
@pytest.mark.parametrize("n", [1, 5, 16, 17, 40, 64, 100, 128])
def test_factor_is_finite(n, prec):
    # diagonal 8 s, the rest +-s / 4 or 0 with at most 16 entries a row: positive definite, and
    # s K0 exact in FP32 (s = 2^-137: units of 2^-149 are 2^-12 s)
    rng = np.random.default_rng(n)
    K0 = 8.0 * np.eye(n)
    for k in range(n):
        for q in rng.permutation(n)[:8]:
            if q != k:
                K0[k, q] = K0[q, k] = 0.25 * rng.choice([-1.0, 1.0])
    s = 2.0 ** -137
    i, j = np.tril_indices(n)
    order = np.lexsort((i, j))  # lower CSC
    i, j = i[order], j[order]
    wp = np.concatenate([[0], np.cumsum(np.arange(n, 0, -1))]).astype(np.int64)
    dev = lambda a: torch.as_tensor(a, dtype=torch.float64, device="cuda")
    ctx = gb.IpmContext(n, 1, np.array([0, 1]), np.zeros(1, np.int32), None, None, wp, i.astype(np.int32),
                        options=gb.default_options(precision=prec, storage_fp64=0))
    ctx.kkt_analyze(np.arange(n, dtype=np.int32))
    ctx.ipm_set_workspace()
    ctx.kkt_assemble(dev(np.zeros(1)), dev(np.ones(1)), 0.0, dev(s * K0[i, j]))
    ctx.kkt_factor(prec)
    assert ctx.ipm_last_perturbed() == 0
    L = factor_of(ctx, n)
    assert np.all(np.isfinite(L))
    # every term of an entry's sum is rounded to a multiple of 2^-149 at worst
    assert np.all(np.abs(L @ L.T - s * K0) <= (n + 10) * (2.0 ** -149 + 2.0 ** -24 * 8 * s))
