"""The float32 matrix tile of sgemm.cuh at the edges of its launch shapes (ragged widths, partial tiles,
both tile forms of the point evaluation) against the float64 oracle."""
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


@pytest.mark.parametrize("w,H", [(16, 1), (16, 3), (48, 2), (64, 2), (112, 3), (256, 2), (400, 2), (512, 2)])
def test_eval_fp32_tile_edges(pkg, w, H):
    """1 point to just above one tile per SM: a chain of w + 1 multiply-adds per layer, so every value is
    within H (w + 8) 2^-24 of the absolute-value propagation (doubled for the sums' own roundings)."""
    layers = inr.random_inr([3] + [w] * H + [1], 40 + w)
    rng = np.random.default_rng(41)
    layers = [(W, rng.normal(0, 0.1, size=b.shape).astype(np.float32)) for W, b in layers]
    net = pkg.Inr(layers)
    big = 152 * 8192 // w
    x = rng.uniform(-1, 1, size=(2 * big + 129, 3)).astype(np.float32)
    ref = mlp.mlp_forward(layers, x)
    a = np.abs(x.astype(np.float64))
    for W, b in layers:
        a = a @ np.abs(W.astype(np.float64)).T + np.abs(b.astype(np.float64))
    tol = 2 * (H + 1) * (w + 8) * 2.0 ** -24 * a[:, 0]
    first = None
    for n in (1, 7, 8, 9, 4096 // w + 1, big - 1, big, big + 1, 2 * big + 129):
        v = net.eval_points(torch.tensor(x[:n], device="cuda")).cpu().numpy()
        assert np.all(np.abs(v - ref[:n]) <= tol[:n]), n
        if first is None:
            first = v[0]
        assert v[0] == first                       # the chain of one point does not depend on the shape
    net.close()
