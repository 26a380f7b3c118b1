"""The batched solve's <r, z>: r in 64 bits times the z that enters the search
direction, also with the FP32 preconditioner.

Line search.  With x0 = 0 and one iteration, x = alpha z and
alpha = <b, z> / <z, A z>, so <b, x> / <x, A x> = 1 whatever the
preconditioner's rounding.  Bar 1e-10: sums of n <= 3000 FP64 products are off
by at most n 2^-53 cond = 3e-13 cond, cond = sum |b_i z_i| / <b, z> below 100
here; another product in alpha (y^T y, y = L^-1 r in FP32) is off by 1e-8.

Overflow.  A x 1e-45: y = L^-1 r of about 1e22 fits FP32, z = L^-T y of about
1e45 does not, so <r, z> is not finite at the start: that status at once,
whatever maxit, and x0 back."""
import numpy as np
import pytest

import gen
import oracle
from paper_2609_00561_gb300 import build as libbuild
from paper_2609_00561_gb300 import iccg

pytestmark = pytest.mark.gpu

pytest.importorskip("torch")

NONFINITE = 7
MATRICES = {"graph": lambda: gen.rgg_laplacian(2500, 12.0, 3), "diffusion": lambda: gen.diffusion3d_27pt(13)}


def _first(m):
    return m[0] if isinstance(m, tuple) else m


@pytest.mark.parametrize("fp32", [False, True])
@pytest.mark.parametrize("block", [1, 8, 32])
@pytest.mark.parametrize("name", sorted(MATRICES))
def test_first_step_is_a_line_search(name, block, fp32):
    libbuild.build()
    a = _first(MATRICES[name]())
    bl = oracle.blocking(a, "abmc", block)
    B = np.random.default_rng(5).uniform(-1.0, 1.0, (5, a.n))
    S = iccg.Solver(a, bl, lane_block_max=-1, precond_fp32=fp32)
    batch = iccg.BatchSolver([S], 5)
    X = [np.zeros_like(B)]
    st, it, _, _ = batch.solve([B], X, 0.0, 1)
    assert st == iccg.ICCG_NOT_CONVERGED and np.all(it == 1)
    m = a.to_scipy()
    for b, x in zip(B, X[0]):
        assert abs((b @ x) / (x @ (m @ x)) - 1.0) <= 1e-10
    batch.close()
    S.close()


@pytest.mark.parametrize("maxit", [0, 1, 5])
@pytest.mark.parametrize("block", [1, 8, 32])
def test_overflow_of_the_backward_sweep_ends_the_solve(block, maxit):
    libbuild.build()
    a = _first(gen.poisson3d_7pt(8, shift=0.1))
    bl = oracle.blocking(a, "abmc", block)
    s = gen.from_scipy(a.to_scipy() * 1e-45)
    S = iccg.Solver(s, bl, lane_block_max=-1, precond_fp32=True)
    batch = iccg.BatchSolver([S], 3)
    rng = np.random.default_rng(6)
    B, x0 = rng.uniform(0.5, 1.0, (3, a.n)), rng.uniform(-1.0, 1.0, (3, a.n))
    X = [x0.copy()]
    st, it, stv, _ = batch.solve([B], X, 1e-8, maxit)
    assert st == NONFINITE and np.all(stv == NONFINITE) and np.all(it == 0)
    assert np.array_equal(X[0], x0)
    batch.close()
    S.close()
