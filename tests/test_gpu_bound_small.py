"""The one-launch float32 bound of small networks against the row path, over the rule that chooses it (up to
8192 cells with one or two hidden layers, up to one cell per SM with more; widths up to 64)."""
import numpy as np
import pytest
import torch

from synth import boxes, inr

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__ as g
    g.build()
    import paper_2402_13861_gb300 as p
    torch.cuda.set_device(0)
    return p


@pytest.mark.parametrize("w,H,act", [(16, 1, "relu"), (32, 2, "relu"), (48, 2, "elu"), (64, 1, "sine"), (64, 2, "relu"),
                                     (16, 8, "relu"), (48, 4, "relu"), (64, 5, "relu"), (64, 7, "relu"), (80, 2, "relu")])
def test_small_network_bounds_equal_the_row_path(pkg, w, H, act):
    layers = inr.random_inr([3] + [w] * H + [1], 80 + w + H, act=act)
    rng = np.random.default_rng(81)
    layers = [(W, rng.normal(0, 0.1, size=b.shape).astype(np.float32)) for W, b in layers]
    net = pkg.Inr(layers, act=act)
    edge = 8192 if H <= 2 else torch.cuda.get_device_properties(0).multi_processor_count
    lo, hi = (torch.tensor(x, device="cuda") for x in boxes.random_boxes(edge + 1, 82, -9, 0))
    modes = [("clt", False), ("sound", False), ("sound", True), ("raua", False)] if act == "relu" else [("clt", False)]
    for mode, inflate in modes:
        c, s = net.bound_cells(lo, hi, mode=mode, prec="fp32", inflate=inflate)
        for n in (1, 7, edge - 1, edge):
            a, b = net.bound_cells(lo[:n], hi[:n], mode=mode, prec="fp32", inflate=inflate)
            assert torch.equal(a, c[:n]) and torch.equal(b, s[:n]), (mode, inflate, n)
        assert torch.isfinite(c).all() and torch.isfinite(s).all()
    net.close()
