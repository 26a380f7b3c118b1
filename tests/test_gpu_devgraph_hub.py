"""Device graph and coloring of patterns with one very long row among short ones (a
hub linked with every row, at the start, the end and in between): equal to the
host's."""
import numpy as np
import pytest

from paper_2609_00561_gb300 import build as libbuild
from paper_2609_00561_gb300 import iccg

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,hub", [(66, 0), (5000, 0), (5000, 4999), (200000, 77)])
def test_hub_graph_equals_host(n, hub):
    libbuild.build()
    ptr = 2 * np.arange(n + 1, dtype=np.int64)
    col = np.empty(2 * n, dtype=np.int32)
    col[0::2] = hub
    col[1::2] = (np.arange(n) + 1) % n
    gptr, gadj = iccg.iccg_graph(n, ptr, col)
    dp, da = iccg.iccg_dev_graph(torch.as_tensor(ptr).cuda(), torch.as_tensor(col).cuda())
    assert np.array_equal(dp.cpu().numpy(), gptr) and np.array_equal(da.cpu().numpy(), gadj)
    for size in (1, 40):
        bo, nb = iccg.iccg_block_abmc(n, gptr, gadj, size)
        ref = iccg.iccg_color_order(n, gptr, gadj, nb, bo)
        out = iccg.iccg_dev_color_order(dp, da, nb, torch.as_tensor(bo).cuda())
        assert out[1] == ref[1]
        for k in (0, 2, 3, 4):
            assert np.array_equal(out[k].cpu().numpy(), ref[k])
