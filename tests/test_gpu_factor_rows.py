"""IC(0) kernels at the edges of their row widths: banded matrices (every row
from 0 to w strictly-lower entries, full fill inside the band) with one block
per color, so that every color is one level (one-row blocks), one warp unit of
several levels, or many; the factor against the oracle's.

Bar: a banded factor is a chain of at most w products per entry; 1e-12 of the
largest entry is the bar of the other factor tests."""
import numpy as np
import pytest
import scipy.sparse as sp

import gen
import oracle
from paper_2609_00561_gb300 import build as libbuild
from paper_2609_00561_gb300 import iccg

pytestmark = pytest.mark.gpu

pytest.importorskip("torch")


def _band(n, w, seed):
    rng = np.random.default_rng(seed)
    offs = [-rng.uniform(0.1, 1.0, n - k) for k in range(1, w + 1)]
    off = sp.diags(offs + offs, list(range(1, w + 1)) + [-k for k in range(1, w + 1)], shape=(n, n), format="csr")
    d = -np.asarray(off.sum(axis=1)).ravel() + rng.uniform(0.1, 1.0, n)
    return gen.from_scipy(off + sp.diags(d, 0))


@pytest.mark.parametrize("no_graph", [0, 1])
@pytest.mark.parametrize("block", [1, 5, 8, 31, 32])
@pytest.mark.parametrize("w", [1, 8, 9, 31, 32, 33, 63, 64, 65])
def test_banded_factor_matches_oracle(w, block, no_graph):
    libbuild.build()
    n = 161
    a = _band(n, w, 100 * w + block)
    bptr = np.append(np.arange(0, n, block), n).astype(np.int32)
    nb = bptr.size - 1
    bl = {"perm": np.arange(n, dtype=np.int32), "block_ptr": bptr, "color_ptr": np.arange(nb + 1, dtype=np.int32),
          "n_b": nb, "n_c": nb}
    S = iccg.Solver(a, bl, no_graph=no_graph)
    lptr, lcol, aval = oracle.tril_csr(a.to_scipy())
    lref, brow = oracle.ic0(lptr, lcol, aval)
    assert brow == -1
    for _ in range(2):   # a second factorization overwrites the first's scratch
        iccg.iccg_factor(S.ctx)
        lgpu = iccg.iccg_get_factor(S.ctx)
        assert np.max(np.abs(lgpu - lref)) <= 1e-12 * np.max(np.abs(lref))
    r = np.random.default_rng(3).uniform(-1, 1, n)
    z = np.zeros(n)
    iccg.iccg_precond(S.ctx, r, z)
    zref = oracle.backward(lptr, lcol, lref, oracle.forward(lptr, lcol, lref, r))
    assert np.max(np.abs(z - zref)) <= 1e-12 * np.max(np.abs(zref))
    S.close()
