"""The batched kernel's block handling at its edges: one-row blocks, blocks of
the largest size (64 rows), blocks and product tiles with more entries than a
warp stages in shared memory, and right-hand-side counts from one lane to a
full warp, against the oracle (bars of test_gpu_batched.py)."""
import numpy as np
import pytest

import gen
import oracle
from paper_2609_00561_gb300 import build as libbuild
from paper_2609_00561_gb300 import iccg

pytestmark = pytest.mark.gpu

pytest.importorskip("torch")

MATRICES = {
    "grid7": lambda: gen.poisson3d_7pt(9, shift=1e-2),
    # 27-point rows: blocks of 64 rows hold more than 512 entries
    "aniso27": lambda: gen.stencil_aniso("27pt", 1000, 4.0),
    # rows of up to 60 entries: a product tile of 16 rows holds more than 512
    "dense": lambda: gen.random_spd_small(300, 0.1, 3),
}


@pytest.mark.parametrize("nrhs", [1, 5, 32])
@pytest.mark.parametrize("block", [1, 13, 64])
@pytest.mark.parametrize("name", sorted(MATRICES))
def test_block_edges_match_oracle(name, block, nrhs):
    libbuild.build()
    a = MATRICES[name]()
    bl = oracle.blocking(a, "abmc", block)
    B = np.random.default_rng(7).uniform(-1.0, 1.0, (nrhs, a.n))
    S = iccg.Solver(a, bl, lane_block_max=-1)
    batch = iccg.BatchSolver([S, S], nrhs, rows_per_thread=1 if nrhs > 1 else 4)
    X = [np.zeros_like(B), np.zeros_like(B)]
    st, it, _, _ = batch.solve([B, B], X, 1e-8, 3000)
    assert st == iccg.ICCG_OK
    assert np.array_equal(X[0], X[1]) or np.allclose(X[0], X[1], rtol=1e-9, atol=1e-12)
    for j in range(0, nrhs, 7):
        ref = oracle.iccg(a, B[j], bl["perm"], tol=1e-8, maxit=3000)
        assert np.linalg.norm(X[0][j] - ref["x"]) <= 1e-10 * np.linalg.norm(ref["x"])
        assert abs(int(it[0, j]) - ref["iterations"]) <= 1
    batch.close()
    S.close()
