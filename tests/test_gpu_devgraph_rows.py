"""Device graph and coloring at the edges of the row lengths: rows whose pairs
(both directions of every stored entry) number up to, exactly and above what a
warp sorts in registers, unsorted and repeated columns, one-sided entries, empty
rows; equal to the host's graph, coloring and ordering integer for integer."""
import numpy as np
import pytest

from paper_2609_00561_gb300 import build as libbuild
from paper_2609_00561_gb300 import iccg

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _pattern(n, per_row, seed):
    """per_row off-diagonal columns a row (with repeats, unsorted, one-sided) and
    the diagonal; row 0 is linked to `per_row` rows more than once."""
    rng = np.random.default_rng(seed)
    rows = [np.append(rng.integers(0, n, per_row), i) for i in range(n)]
    rows[0] = np.concatenate([np.repeat(np.arange(1, 1 + per_row // 2), 2), [0]])
    rows[n // 2] = np.array([n // 2])
    ptr = np.zeros(n + 1, dtype=np.int64)
    ptr[1:] = np.cumsum([r.size for r in rows])
    return ptr, np.concatenate(rows).astype(np.int32)


@pytest.mark.parametrize("n,per_row", [(40, 1), (300, 8), (300, 15), (300, 16), (200, 24), (150, 31), (150, 32), (150, 40)])
def test_graph_and_coloring_equal_host(n, per_row):
    libbuild.build()
    ptr, col = _pattern(n, per_row, 10 * n + per_row)
    gptr, gadj = iccg.iccg_graph(n, ptr, col)
    dp, da = iccg.iccg_dev_graph(torch.as_tensor(ptr).cuda(), torch.as_tensor(col).cuda())
    assert np.array_equal(dp.cpu().numpy(), gptr) and np.array_equal(da.cpu().numpy(), gadj)
    for size in (1, 3):
        block_of, nb = iccg.iccg_block_abmc(n, gptr, gadj, size)
        ref = iccg.iccg_color_order(n, gptr, gadj, nb, block_of)
        out = iccg.iccg_dev_color_order(dp, da, nb, torch.as_tensor(block_of).cuda())
        assert out[1] == ref[1]
        for k in (0, 2, 3, 4):
            assert np.array_equal(out[k].cpu().numpy(), ref[k])
