"""Two FP64 factors of one matrix on the tensor cores agree to the last bit where no sum is long
enough to be split over CTAs, whatever runs beside what: work on another stream delays now the
one, now the other of the factor's own streams."""
import contextlib
import threading

import numpy as np
import pytest

import gen
import paper_2508_16094_gb300 as gb
from tests.test_gpu_dense_front import dense_front, factor_of

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.fixture(scope="module", autouse=True)
def _built():
    gb.build()


@contextlib.contextmanager
def busy_gpu():
    """Matrix products on a stream of their own for as long as the block runs."""
    stop = threading.Event()

    def run():
        st = torch.cuda.Stream()
        rng = np.random.default_rng(1)
        with torch.cuda.stream(st):
            a = torch.ones((2048, 2048), device="cuda")
            while not stop.is_set():
                for _ in range(int(rng.integers(1, 8))):
                    a @ a
                st.synchronize()

    t = threading.Thread(target=run)
    t.start()
    try:
        yield
    finally:
        stop.set()
        t.join()


@pytest.mark.parametrize("n", [449, 896])
def test_one_front(n):
    ctx, _ = dense_front(n, gb.default_options(storage_fp64=1, fp64_tc=1))
    ctx.kkt_factor(gb.IPM_FP64)
    first = factor_of(ctx, n)
    with busy_gpu():
        for _ in range(20):
            ctx.kkt_factor(gb.IPM_FP64)
            assert np.array_equal(factor_of(ctx, n), first)


@pytest.mark.parametrize("shape", [(16, 16, 64), (24, 24, 24)])
def test_many_fronts(shape):
    lp = gen.grid_lp(*shape, seed=2)
    ctx = gb.IpmContext(lp.n, lp.m, lp.rowptr, lp.col, lp.l, lp.u,
                        options=gb.default_options(storage_fp64=1, fp64_tc=1))
    info = ctx.kkt_analyze(gen.nd_order_grid3d(*shape))
    ctx.ipm_set_workspace()
    ctx.kkt_assemble(dev(lp.val), dev(10.0 ** gen.uniform(9, lp.m + 2 * lp.n, -1, 1)), 1e-8)
    S = ctx.kkt_symbolic_export()
    width = np.diff(S["super"])
    # sums of 15 blocks of 64 columns and more may be split; a front's entries also hold its descendants' sums
    split = width > 896
    for f in range(info.nsuper):  # children come before their parent
        p = S["sparent"][f]
        if p >= 0 and split[f]:
            split[p] = True
    rng = np.random.default_rng(0)
    rows, cols = [], []
    for f in np.flatnonzero(~split & (width >= 193)):
        a, b = S["super"][f], S["super"][f + 1]
        r = np.r_[a:b, S["sri"][S["srp"][f]:S["srp"][f + 1]]]
        i, j = rng.choice(r, 20000), rng.integers(a, b, 20000)
        rows.append(i[i >= j])
        cols.append(j[i >= j])
    assert rows
    rows, cols = np.concatenate(rows), np.concatenate(cols)
    ctx.kkt_factor(gb.IPM_FP64)
    first = ctx.kkt_factor_entries(rows, cols)
    with busy_gpu():
        for _ in range(10):
            ctx.kkt_factor(gb.IPM_FP64)
            assert np.array_equal(ctx.kkt_factor_entries(rows, cols), first)
