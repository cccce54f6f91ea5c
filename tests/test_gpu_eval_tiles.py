"""The pipelined tensor-core evaluation (eval_tc.cu) at the edges of its tiles and rings: one point to one more
tile than CTAs, one hidden GEMM (the output layer of a tile overlaps the next tile's only GEMM) to the most layers
(fewer weight stages), both widths and every activation."""
import numpy as np
import pytest
import torch

from oracle import activations
from synth import inr

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__ as g
    g.build()
    import paper_2402_13861_gb300 as p
    torch.cuda.set_device(0)
    return p


@pytest.mark.parametrize("w,H,act", [(128, 2, "relu"), (128, 3, "sine"), (128, 12, "elu"), (256, 2, "elu"),
                                     (256, 3, "relu"), (256, 12, "relu")])
def test_eval_tc_tile_edges(pkg, w, H, act):
    """Two-term products err by less than 2^-15 of the absolute-value propagation per layer (3 2^-18 per
    product and the float32 accumulation of 3 K of them); the activations are 1-Lipschitz."""
    layers = inr.random_inr([3] + [w] * H + [1], 90 + H, act="relu" if act == "sine" else act)
    rng = np.random.default_rng(91)
    layers = [(W, rng.normal(0, 0.1, size=b.shape).astype(np.float32)) for W, b in layers]
    net = pkg.Inr(layers, act=act)
    x = rng.uniform(-1, 1, size=(2 * 152 * 128 + 130, 3)).astype(np.float32)
    first = None
    for n in (1, 127, 128, 129, 152 * 128 + 1, 2 * 152 * 128 + 130):
        v = net.eval_points(torch.tensor(x[:n], device="cuda"), prec="bf16").cpu().numpy()
        idx = np.unique(np.r_[0, n // 3, max(0, n - 129), n - 1])
        ref, a = x[idx].astype(np.float64), np.abs(x[idx].astype(np.float64))
        for l, (W, b) in enumerate(layers):
            ref = ref @ W.astype(np.float64).T + b.astype(np.float64)
            ref = activations.forward(act, ref) if l < H else ref
            a = a @ np.abs(W.astype(np.float64)).T + np.abs(b.astype(np.float64))
        assert np.all(np.abs(v[idx] - np.ravel(ref)) <= (H + 1) * 2.0 ** -15 * a[:, 0]), n
        if first is None:
            first = v[0]
        assert v[0] == first                       # a point's value does not depend on its tile
    net.close()
