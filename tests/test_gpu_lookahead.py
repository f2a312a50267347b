"""FP64 factors whose updates run beside the next diagonal blocks: one front just below
and above the size from which the FMA-pipe factor looks ahead, and the tensor-core one
over odd and even numbers of 64-column blocks."""
import numpy as np
import pytest

import paper_2508_16094_gb300 as gb
from tests.test_gpu_dense_front import dense_front, factor_of

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
U = 2.0 ** -53


@pytest.fixture(scope="module", autouse=True)
def _built():
    gb.build()


@pytest.mark.parametrize("tc", [0, 1])
@pytest.mark.parametrize("n", [193, 256, 320, 385, 639, 672, 673, 833, 960])
def test_backward_error_and_repeats(n, tc):
    ctx, K = dense_front(n, gb.default_options(storage_fp64=1, fp64_tc=tc))
    P = ctx.kkt_symbolic_export()["perm"]
    K = K[np.ix_(P, P)]
    d = np.sqrt(np.diag(K))
    # |l_ik| <= sqrt(k_ii), so a sum of n products errs by at most (n + 10) u sqrt(k_ii k_jj) in
    # FP64; a slice window of 128 columns drops at most 2^-53 times 128 such products more,
    # twice that with the rounding of the slices themselves
    bound = (4 if tc else 1.01) * (n + 10) * U * np.outer(d, d)
    first = None
    for _ in range(3):
        ctx.kkt_factor(gb.IPM_FP64)
        L = factor_of(ctx, n)
        assert np.all(np.abs(L @ L.T - K) <= bound)
        if first is None:
            first = L
        if not tc:  # (the tensor-core factor adds the parts of long sums in any order)
            assert np.array_equal(L, first)
