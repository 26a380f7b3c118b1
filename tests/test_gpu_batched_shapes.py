"""Launch shapes of the batched solve at the limit of an SM's shared memory: the
warps of a CTA with the largest blocks and a full warp of right-hand sides, each
as many as fit with one row scratch per right-hand side alone; against the
oracle (bars of test_gpu_batched.py).  One warp more than that is refused.
Then the block sizes and right-hand-side counts between which the kernel's form
changes."""
import numpy as np
import pytest

import gen
import oracle
from paper_2609_00561_gb300 import build as libbuild
from paper_2609_00561_gb300 import iccg

pytestmark = pytest.mark.gpu

pytest.importorskip("torch")


def _systems(fp32, block, wide):
    a = gen.random_spd_small(400, 0.1, 3) if wide else gen.poisson3d_7pt(9, shift=1e-2)
    bl = oracle.blocking(a, "abmc", block)
    return a, bl, iccg.Solver(a, bl, lane_block_max=-1, precond_fp32=fp32)


@pytest.mark.parametrize("rows_per_thread", [1, 2, 4])
@pytest.mark.parametrize("wide", [False, True])
@pytest.mark.parametrize("fp32,block,warps", [(False, 64, 13), (False, 32, 16), (True, 64, 16), (True, 32, 16)])
def test_largest_shapes_match_oracle(fp32, block, warps, wide, rows_per_thread):
    libbuild.build()
    a, bl, S = _systems(fp32, block, wide)
    B = np.random.default_rng(7).uniform(-1.0, 1.0, (32, a.n))
    batch = iccg.BatchSolver([S, S], 32, warps_per_cta=warps, rows_per_thread=rows_per_thread)
    assert batch.info()["warps_per_cta"] == warps
    X = [np.zeros_like(B), np.zeros_like(B)]
    st, it, _, _ = batch.solve([B, B], X, 1e-8, 3000)
    assert st == iccg.ICCG_OK
    m = a.to_scipy()
    for j in range(0, 32, 7):
        ref = oracle.iccg(a, B[j], bl["perm"], tol=1e-8, maxit=3000)
        if fp32:
            assert np.linalg.norm(B[j] - m @ X[0][j]) <= 1e-7 * np.linalg.norm(B[j])
            assert abs(int(it[0, j]) - ref["iterations"]) <= 3 + ref["iterations"] // 10
        else:
            assert np.linalg.norm(X[0][j] - ref["x"]) <= 1e-10 * np.linalg.norm(ref["x"])
            assert abs(int(it[0, j]) - ref["iterations"]) <= 1
    batch.close()
    S.close()


def test_one_warp_more_is_refused():
    libbuild.build()
    _, _, S = _systems(False, 64, False)
    with pytest.raises(iccg.IccgError) as ei:
        iccg.BatchSolver([S], 32, warps_per_cta=14)
    assert ei.value.status == iccg.ICCG_ERR_ARG
    S.close()


@pytest.mark.parametrize("nrhs", [1, 8, 9, 16, 17])
@pytest.mark.parametrize("block", [2, 3, 5, 6])
@pytest.mark.parametrize("wide", [False, True])
def test_small_blocks_match_oracle(wide, block, nrhs):
    libbuild.build()
    a, bl, S = _systems(False, block, wide)
    B = np.random.default_rng(8).uniform(-1.0, 1.0, (nrhs, a.n))
    batch = iccg.BatchSolver([S, S], nrhs)
    X = [np.zeros_like(B), np.zeros_like(B)]
    st, it, _, _ = batch.solve([B, B], X, 1e-8, 3000)
    assert st == iccg.ICCG_OK
    for j in range(0, nrhs, 8):
        ref = oracle.iccg(a, B[j], bl["perm"], tol=1e-8, maxit=3000)
        for x in X:
            assert np.linalg.norm(x[j] - ref["x"]) <= 1e-10 * np.linalg.norm(ref["x"])
        assert abs(int(it[0, j]) - ref["iterations"]) <= 1
    batch.close()
    S.close()
