"""Batched MPC in FP64 with bounds far from the other data: infinite ones are no problem the
method can solve and must not come back as solved; wide and narrow ones solve."""
import numpy as np
import pytest

import gen
import paper_2508_16094_gb300 as gb

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    gb.build()


def solve(u_max, x_max, **kw):
    mb = gen.mpc_batch(8, seed=3, t_min=1, t_max=40)
    mb.u_max, mb.x_max = u_max, x_max
    m = gb.BatchedMPC(mb)
    m.ipm_solve_batched(**kw)
    return m.status.cpu().numpy(), m.kkt.cpu().numpy(), m.z.cpu().numpy()


@pytest.mark.parametrize("u_max,x_max", [(1.0, np.inf), (np.inf, np.inf), (np.inf, 5.0)])
def test_infinite_bounds_are_not_reported_as_solved(u_max, x_max):
    status, _, _ = solve(u_max, x_max)
    assert (status != 0).all()


@pytest.mark.parametrize("x_max", [1e160, 1e200, 1e300])
def test_bounds_whose_products_overflow(x_max):
    # s = x_max and lambda = 1: s lambda over max(1, |f|) is what is left of the optimum
    status, kkt, _ = solve(1.0, x_max, max_iter=0)
    assert (status == 7).all() and np.allclose(kkt, x_max, rtol=1e-12)
    status, kkt, _ = solve(1.0, x_max)
    assert (status != 0).all() and (kkt > 1e3).all()


@pytest.mark.parametrize("x_max", [5.0, 1e3, 1e6, 1e8])
def test_wide_bounds(x_max):
    status, kkt, _ = solve(1.0, x_max)
    assert (status == 0).all() and (kkt <= 1e-6).all()
