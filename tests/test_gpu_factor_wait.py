"""IC(0) of warp units waits, in the kernel, for rows of the same block: a wait that
outlasts the limit (1 ns here: any wait at all) ends the factorization with the
timeout status, not with a pivot's; the context factors again with the default
limit, to the same bits, and a matrix that does break down still says so."""
import numpy as np
import pytest
import scipy.sparse as sp

import gen
import oracle
from paper_2609_00561_gb300 import build as libbuild
from paper_2609_00561_gb300 import iccg

pytestmark = pytest.mark.gpu

pytest.importorskip("torch")

BREAKDOWN, TIMEOUT = 3, 6


@pytest.mark.parametrize("no_graph", [0, 1])
def test_factor_wait_runs_out_then_context_factors(no_graph):
    libbuild.build()
    a = gen.diffusion3d_27pt(24)
    bl = oracle.blocking(a, "abmc", 32)
    S = iccg.Solver(a, bl, no_graph=no_graph)
    ref = iccg.iccg_get_factor(S.ctx)
    iccg.iccg_set_wait_limit(S.ctx, 1)
    with pytest.raises(iccg.IccgError) as ei:
        iccg.iccg_factor(S.ctx)
    assert ei.value.status == TIMEOUT
    assert "gave up" in iccg.iccg_last_error(S.ctx)[1]
    with pytest.raises(iccg.IccgError):   # no factor: no solve
        iccg.iccg_solve(S.ctx, np.ones(a.n), np.zeros(a.n), 1e-8, 10)
    iccg.iccg_set_wait_limit(S.ctx, 0)
    iccg.iccg_factor(S.ctx)
    assert np.array_equal(iccg.iccg_get_factor(S.ctx), ref)
    S.close()


def test_breakdown_is_still_a_breakdown():
    libbuild.build()
    a = gen.diffusion3d_27pt(12)
    m = a.to_scipy().tolil()
    m[700, 700] = -1.0
    a = gen.from_scipy(sp.csr_matrix(m))
    with pytest.raises(iccg.IccgError) as ei:
        iccg.Solver(a, oracle.blocking(a, "abmc", 32))
    assert ei.value.status == BREAKDOWN
