"""The FP64 batched MPC kernel at the edges of its stage loops (one to a few more
stages than it keeps in flight) and with fewer CTAs than instances, against the
CPU oracle and against itself."""
import numpy as np
import pytest

import gen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2508_16094_gb300 as gb  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    gb.build()
    oracle.build()


@pytest.mark.parametrize("t", [1, 2, 3, 4, 5, 8, 9, 17])
def test_short_horizons_match_oracle(t):
    mb = gen.mpc_batch(3, seed=40 + t, t_min=t, t_max=t)
    b = gb.BatchedMPC(mb)
    b.ipm_solve_batched(precision=gb.IPM_FP64, tol=1e-8)
    torch.cuda.synchronize()
    assert np.all(b.status.cpu().numpy() == 0)
    assert np.all(b.kkt.cpu().numpy() <= 1e-8)
    obj = b.obj.cpu().numpy()
    for i in range(mb.count):
        lp, W = gen.mpc_instance_qp(*mb.instance(i), u_max=mb.u_max, x_max=mb.x_max)
        r = oracle.ipm_lp(oracle.analyze(lp.n, lp.m, lp.rowptr, lp.col, None, W[0], W[1]), lp, tol=1e-8, W=W)
        assert r["status"] == 0
        # both are within 1e-8 (scaled KKT) of the same optimum
        assert abs(obj[i] - r["objective"]) <= 1e-6 * max(1.0, abs(r["objective"]))


def test_queue_order_does_not_matter():
    mb = gen.mpc_batch(13, seed=5, t_min=2, t_max=30)
    b = gb.BatchedMPC(mb)
    out = []
    for ipc, ctas in ((2, 1), (16, 1), (8, 0)):
        b.z.zero_()
        b.ipm_solve_batched(precision=gb.IPM_FP64, instances_per_cta=ipc, ctas=ctas)
        out.append((b.z.clone(), b.obj.clone(), b.iters.clone()))
    torch.cuda.synchronize()
    for z, obj, it in out[1:]:
        assert torch.equal(z, out[0][0]) and torch.equal(obj, out[0][1]) and torch.equal(it, out[0][2])
