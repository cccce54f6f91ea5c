"""The proposer's tiled kernels at the edges of their tiles (64 samples per gradient tile, 128 per inference tile):
logits do not depend on the tile a sample falls into, and the gradient of a batch is the mean of its parts'."""
import numpy as np
import pytest
import torch

from oracle import proposer as P

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__ as g
    g.build()
    import paper_2402_13861_gb300 as p
    torch.cuda.set_device(0)
    return p


@pytest.mark.parametrize("n", [1, 63, 64, 65, 129, 64 * 152 + 1])
def test_tile_edges(pkg, n):
    layers = P.init_params(5)
    packed = np.concatenate([np.concatenate([W.reshape(-1), b.reshape(-1)]) for W, b in layers]).astype(np.float32)
    prop = pkg.Proposer(packed, np.zeros(8), np.ones(8))
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    x = torch.randn((n, 8), generator=g, device="cuda")
    y = (torch.rand(n, generator=g, device="cuda") < 0.4).float()
    z = prop.predict(x)
    i = n // 2
    assert torch.equal(z[i:], prop.predict(x[i:].contiguous()))
    grad, loss = prop.grad(x, y)
    parts = [(0, i), (i, n)] if i else [(0, n)]
    want = sum(prop.grad(x[a:b].contiguous(), y[a:b].contiguous())[0].double() * (b - a) for a, b in parts) / n
    # float32 sums of the same terms in another order: 2 n u of their absolute sum, bounded by n times the largest
    # of one sample's entries; sqrt(n) u of the norm in practice
    assert (grad.double() - want).norm() <= 1e-5 * want.norm() + 1e-9
    one = torch.nn.functional.binary_cross_entropy_with_logits(z.double(), y.double())
    assert abs(loss.item() - one.item()) <= 1e-5 * abs(one.item()) + 1e-7
    prop.close()
