"""Workspace of a context (host only): what solves use beside the factor lies in the place of the
update matrices, so it costs nothing beyond what one right-hand side needs."""
import pytest

import gen
import paper_2508_16094_gb300 as gb

# bytes with substitution for the FP64 solves and one right-hand side at a time, before there were block
# inverses, published entries or groups of right-hand sides
BEFORE = {(10, "fp64"): 6756096, (10, "fp64_tc"): 9418752, (10, "tf32x3"): 5941248,
          (20, "fp64"): 93794560, (20, "fp64_tc"): 155309824, (20, "tf32x3"): 74199552,
          (32, "fp64"): 656058624, (32, "fp64_tc"): 1147002368, (32, "tf32x3"): 506479872}
OPTIONS = {"fp64": dict(storage_fp64=1), "fp64_tc": dict(storage_fp64=1, fp64_tc=1),
           "tf32x3": dict(precision=gb.IPM_TF32X3, storage_fp64=0)}


@pytest.mark.parametrize("g,name", sorted(BEFORE))
def test_workspace_is_no_larger(g, name):
    lp = gen.grid_lp(g, seed=1)
    ctx = gb.IpmContext(lp.n, lp.m, lp.rowptr, lp.col, lp.l, lp.u, options=gb.default_options(**OPTIONS[name]))
    info = ctx.kkt_analyze(gen.nd_order_grid3d(g))
    assert info.workspace_bytes <= 1.01 * BEFORE[g, name]
