"""The network kernels' forms: networks whose weights do not fit a CTA's shared
memory (a launch per layer), and batches at which the forward pass changes from
one launch to a launch per layer; against the oracle (bars of test_gpu_mlp.py),
and the two forms of the forward pass bit for bit."""
import numpy as np
import pytest

from oracle import learn as ol
from paper_2609_00561_gb300 import build as libbuild
from paper_2609_00561_gb300 import iccg

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _net(nf, h, c, B, seed):
    rng = np.random.default_rng(seed)
    p = rng.normal(0.0, 0.4 * min(1.0, 8.0 / np.sqrt(h)), ol.mlp_offsets(nf, h, c)["total"]).astype(np.float32)
    return (p, rng.normal(size=(B, nf)).astype(np.float32), rng.integers(0, c, B).astype(np.int32),
            rng.normal(size=B).astype(np.float32))


@pytest.mark.parametrize("shape", [(20, 96, 6, 40), (20, 130, 5, 33), (300, 70, 9, 17), (20, 64, 5, 1300),
                                   (20, 8, 2, 5001)])
def test_forward_loss_and_gradient_match_oracle(shape):
    libbuild.build()
    nf, h, c, B = shape
    p, X, y, yr = _net(nf, h, c, B, 5)
    P, Xd = torch.tensor(p).cuda(), torch.tensor(X).cuda()
    out = torch.zeros((B, c + 1), device="cuda")
    act = torch.zeros(2 * B * h, device="cuda")
    iccg.mlp_forward(P, nf, h, c, Xd, out, act)
    zr, h1, h2 = ol.mlp_forward(p, nf, h, c, X)
    assert np.allclose(out.cpu().numpy(), zr, rtol=1e-5, atol=1e-5 * np.abs(zr).max())
    assert np.allclose(act.cpu().numpy()[:B * h].reshape(B, h), h1, rtol=1e-5, atol=1e-5 * np.abs(h1).max())
    G, loss = torch.zeros_like(P), torch.zeros(1, device="cuda")
    work = torch.zeros(B * (4 * h + 2 * (c + 1) + 1), device="cuda")
    iccg.mlp_grad(P, nf, h, c, Xd, torch.tensor(y).cuda(), torch.tensor(yr).cuda(), 0.5, G, loss, work)
    gr = ol.mlp_grad(p, nf, h, c, X, y, yr, 0.5)
    assert np.max(np.abs(G.cpu().numpy() - gr)) <= 1e-4 * np.max(np.abs(gr)) + 1e-7
    assert float(loss.item()) == pytest.approx(ol.mlp_loss(p, nf, h, c, X, y, yr, 0.5), rel=1e-5)


@pytest.mark.parametrize("shape", [(20, 64, 5), (3, 5, 2), (20, 95, 5)])
def test_forward_forms_are_the_same_bits(shape):
    libbuild.build()
    nf, h, c = shape
    B = 6000
    p, X, _, _ = _net(nf, h, c, B, 6)
    P, Xd = torch.tensor(p).cuda(), torch.tensor(X).cuda()
    whole, part = torch.zeros((B, c + 1), device="cuda"), torch.zeros((B, c + 1), device="cuda")
    iccg.mlp_forward(P, nf, h, c, Xd, whole)
    for k in range(0, B, 300):
        iccg.mlp_forward(P, nf, h, c, Xd[k:k + 300], part[k:k + 300])
    assert torch.equal(whole, part)
