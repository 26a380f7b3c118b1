"""The allocation-free product at the edges of its two forms and of its slices: as
many rows as one CTA each of the persistent grid holds, one fewer and more, one
slice and many; rows whose 32 together have up to, exactly and more than the
entries that a warp stages, wide and narrow slices in turn, empty rows, a full row.

Bar: a row's sum of w products in order is within w 2^-53 of the sum of their
magnitudes; <p, q> within n 2^-53 of the sum of its terms' (compared at four
times that, the reference's own rounding included)."""
import numpy as np
import pytest
import scipy.sparse as sp

from paper_2609_00561_gb300 import build as libbuild
from paper_2609_00561_gb300 import iccg

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

GRID = 608 * 256   # rows of the persistent grid


def _lengths(n, kind, rng):
    if kind == "narrow":
        return rng.integers(0, 9, n)
    if kind == "eight":      # 256 entries a slice, then 257 in every third
        w = np.full(n, 8)
        w[::96] += 1
        return w
    if kind == "wide":
        return rng.integers(9, 40, n)
    w = rng.integers(0, 8, n)   # slices in turn
    for s in range(0, n, 96):
        w[s:s + 32] = rng.integers(0, 60, min(32, n - s))
    return w


@pytest.mark.parametrize("kind", ["narrow", "eight", "wide", "mixed"])
@pytest.mark.parametrize("n", [1, 31, 257, GRID - 1, GRID, GRID + 1, GRID + 33, 2 * GRID + 300])
def test_product_matches_scipy(n, kind):
    libbuild.build()
    rng = np.random.default_rng(n + len(kind))
    w = np.minimum(_lengths(n, kind, rng), n)
    if kind == "mixed" and n <= 257:
        w[n // 2] = n
    ptr = np.zeros(n + 1, dtype=np.int64)
    ptr[1:] = np.cumsum(w)
    col = rng.integers(0, n, ptr[-1]).astype(np.int32)
    val, p = rng.uniform(-1, 1, ptr[-1]), rng.uniform(-1, 1, n)
    a = sp.csr_matrix((val, col, ptr), shape=(n, n))
    q, pq = torch.full((n,), 7.0, dtype=torch.float64, device="cuda"), torch.zeros(1, dtype=torch.float64, device="cuda")
    dev = [torch.as_tensor(x).cuda() for x in (ptr, col, val, p)]
    for _ in range(2):
        assert iccg.iccg_spmv_dot_noalloc(n, *dev, q, pq) == iccg.ICCG_OK
    torch.cuda.synchronize()
    ref, mag = a @ p, abs(a) @ abs(p)
    eps = 2.0 ** -53
    assert np.all(np.abs(q.cpu().numpy() - ref) <= 4 * eps * np.maximum(w, 1) * mag)
    assert abs(pq.item() - p @ ref) <= 4 * eps * (n + w.max()) * (np.abs(p) @ mag) + 1e-300
