"""The solve's graph runs its first iterations one a pass and the later ones several
a pass: solves that end at every place of a pass (iteration limits around the
change and behind it, tolerance reached early) equal the host-driven loop bit for
bit (the same kernels in the same order), for every kind of color kernel, one
after another on one context."""
import numpy as np
import pytest

import gen
import oracle
from paper_2609_00561_gb300 import build as libbuild
from paper_2609_00561_gb300 import iccg

pytestmark = pytest.mark.gpu

pytest.importorskip("torch")

LAYOUTS = {
    "pair": dict(bl=("leiden_cpm", dict(gamma=0.5)), opts=dict()),
    "units": dict(bl=("abmc", 16), opts=dict()),
    "warp": dict(bl=("abmc", 1), opts=dict()),
    "lane": dict(bl=("abmc", 4), opts=dict(tile_mapping="cta")),
    "groups": dict(bl=("abmc", 8), opts=dict(lane_block_max=-1)),
    "tail": dict(bl=("leiden_cpm", dict(gamma=0.5)), opts=dict(fuse_sweep=2)),
    "coop": dict(bl=("leiden_cpm", dict(gamma=0.5)), opts=dict(fuse_sweep=1)),
}


def _blocking(a, spec):
    if spec[0] == "abmc":
        return oracle.blocking(a, "abmc", spec[1])
    return oracle.blocking(a, spec[0], **spec[1])


@pytest.mark.parametrize("fp32", [False, True])
@pytest.mark.parametrize("name", sorted(LAYOUTS))
def test_every_end_of_a_pass_equals_the_host_loop(name, fp32):
    libbuild.build()
    a = gen.poisson3d_7pt(14)
    bl = _blocking(a, LAYOUTS[name]["bl"])
    b = gen.rhs_uniform(a.n, 4)
    G = iccg.Solver(a, bl, precond_fp32=fp32, **LAYOUTS[name]["opts"])
    H = iccg.Solver(a, bl, precond_fp32=fp32, no_graph=1, **LAYOUTS[name]["opts"])
    z0 = np.zeros(a.n)
    iccg.iccg_precond(G.ctx, b, z0)
    ends = [(0.0, m) for m in (0, 1, 2, 15, 16, 17, 18, 19, 20, 21, 24, 3)] + [(t, 500) for t in (0.5, 1e-2, 1e-8, 1e-1)]
    for tol, maxit in ends:
        xg, xh = np.full(a.n, 0.25), np.full(a.n, 0.25)
        sg, ig, hg = iccg.iccg_solve(G.ctx, b, xg, tol, maxit)
        sh, ih, hh = iccg.iccg_solve(H.ctx, b, xh, tol, maxit)
        assert (sg, ig) == (sh, ih)
        assert np.array_equal(xg, xh) and np.array_equal(hg, hh)
    z1 = np.zeros(a.n)
    iccg.iccg_precond(G.ctx, b, z1)   # after a solve that ended
    assert np.array_equal(z0, z1)
    G.close()
    H.close()
