"""The proposer's gradient of a long batch: the float32 sums over its samples do not grow less accurate with it."""
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


@pytest.mark.parametrize("seed,label", [(0, 1.0), (1, 0.0), (2, 1.0)])
def test_equal_samples(pkg, seed, label):
    """2^20 equal samples: the mean's scale is a power of two, so that every term is the single sample's, scaled
    exactly, and the gradient has to be that sample's.  Roundings of an entry: 64 samples of a tile, the tiles of a
    block, the blocks' additions, and the single sample's own."""
    n = 1 << 20
    layers = P.init_params(5 + seed)
    packed = np.concatenate([np.concatenate([W.reshape(-1), b.reshape(-1)]) for W, b in layers]).astype(np.float32)
    prop = pkg.Proposer(packed, np.zeros(8), np.ones(8))
    x1 = torch.tensor(np.random.default_rng(seed).normal(size=(1, 8)).astype(np.float32), device="cuda")
    y1 = torch.full((1,), label, device="cuda")
    g1, l1 = (t.clone().double() for t in prop.grad(x1, y1))
    g, l = (t.double() for t in prop.grad(x1.expand(n, 8).contiguous(), y1.expand(n).contiguous()))
    blocks = torch.cuda.get_device_properties(0).multi_processor_count
    roundings = 64 + -(-n // (64 * blocks)) + blocks + 4
    tol = 1.01 * roundings * 2.0 ** -24
    assert torch.all((g - g1).abs() <= tol * g1.abs())
    assert abs(l.item() - l1.item()) <= tol * abs(l1.item())
    assert (g1 != 0).sum() > 500
    prop.close()
