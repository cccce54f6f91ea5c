"""Float32 evaluation of networks with one hidden layer (no matrix tile; the points per CTA follow the list's length):
a point's value does not depend on the list and lies in the float32 band of the oracle."""
import numpy as np
import pytest
import torch

from oracle import mlp
from synth import inr

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__ as g
    g.build()
    import paper_2402_13861_gb300 as p
    torch.cuda.set_device(0)
    return p


@pytest.mark.parametrize("w,act", [(16, "relu"), (48, "elu"), (80, "relu"), (128, "sine"), (400, "relu"), (512, "relu")])
def test_lists_either_side_of_each_tile(pkg, w, act):
    """As in the deeper networks' test: 2 H (w + 8) 2^-24 of the absolute-value propagation, whose hidden layer is
    bounded by |z| + 1 for every activation and errs by what its argument does and four roundings of its own."""
    layers = inr.random_inr([3, w, 1], 150 + w, act=act)
    net = pkg.Inr(layers, act=act)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    top = max(8, 16384 // w // 8 * 8)
    n = sms * top + 5
    rng = np.random.default_rng(151)
    x = rng.uniform(-1, 1, size=(n, 3)).astype(np.float32)
    dx = torch.tensor(x, device="cuda")
    v = net.eval_points(dx)
    lengths, p = [1, 7, 8, 9], 8
    while p <= top:
        lengths += [p * sms - 1, p * sms, p * sms + 1]
        p *= 2
    for m in (m for m in lengths if m <= n):
        assert torch.equal(net.eval_points(dx[:m]), v[:m]), m
    pick = np.unique(np.r_[0:64, n - 64:n, rng.integers(0, n, 500)])
    ref = mlp.mlp_forward(layers, x[pick]) if act == "relu" else mlp.mlp_forward(layers, x[pick], act=act)
    (W0, b0), (W1, b1) = [(np.abs(W.astype(np.float64)), np.abs(b.astype(np.float64))) for W, b in layers]
    a = (np.abs(x[pick].astype(np.float64)) @ W0.T + b0 + 1.0) @ W1.T + b1
    assert np.all(np.abs(v.cpu().numpy()[pick] - ref) <= 4 * (w + 8) * 2.0 ** -24 * a[:, 0])
    net.close()
