"""Float32 bounds of few cells against those of many: the one-launch form of small networks (up to 8192 cells
with one or two hidden layers, up to 64 neurons per SM with more; widths up to 64), the row path's kernels with
several blocks per cell (up to one cell per SM), and the reduced form with two cells per thread."""
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
    edge = 8192 if H <= 2 else 64 * torch.cuda.get_device_properties(0).multi_processor_count // w
    lo, hi = (torch.tensor(x, device="cuda") for x in boxes.random_boxes(edge + 1, 82, -9, 0))
    modes = [("clt", False), ("sound", False), ("sound", True), ("raua", False)] if act == "relu" else [("clt", False)]
    for mode, inflate in modes:
        c, s = net.bound_cells(lo, hi, mode=mode, prec="fp32", inflate=inflate)
        for n in (1, 7, edge - 1, edge):
            a, b = net.bound_cells(lo[:n], hi[:n], mode=mode, prec="fp32", inflate=inflate)
            assert torch.equal(a, c[:n]) and torch.equal(b, s[:n]), (mode, inflate, n)
        assert torch.isfinite(c).all() and torch.isfinite(s).all()
    net.close()


@pytest.mark.parametrize("w,H,act", [(80, 5, "sine"), (112, 3, "relu"), (256, 4, "elu"), (400, 3, "relu"), (512, 4, "relu")])
def test_few_cells_equal_many(pkg, w, H, act):
    """From every symbol dead or alive to more rows than one hand-over of the output layer takes, either side of
    the cell counts where the kernels change."""
    net = pkg.Inr(inr.random_inr([3] + [w] * H + [1], 85 + w, act=act), act=act)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    lo, hi = (torch.tensor(x, device="cuda") for x in boxes.random_boxes(sms + 1, 86, -9, 0))
    modes = [("clt", False), ("sound", False), ("sound", True), ("raua", False)] if act == "relu" else [("clt", False)]
    for mode, inflate in modes:
        c, s = net.bound_cells(lo, hi, mode=mode, prec="fp32", inflate=inflate)
        for n in (1, sms // 4, sms // 4 + 1, sms):
            a, b = net.bound_cells(lo[:n], hi[:n], mode=mode, prec="fp32", inflate=inflate)
            assert torch.equal(a, c[:n]) and torch.equal(b, s[:n]), (mode, inflate, n)
        assert torch.isfinite(c).all() and torch.isfinite(s).all()
    net.close()


@pytest.mark.parametrize("w,H,inflate", [(64, 2, True), (128, 3, False), (272, 2, True), (400, 2, False), (512, 3, True)])
def test_few_cells_equal_many_rafixed(pkg, w, H, inflate):
    net = pkg.Inr(inr.random_inr([3] + [w] * H + [1], 95 + w))
    edge = torch.cuda.get_device_properties(0).multi_processor_count * 2 * (1024 // w)
    lo, hi = (torch.tensor(x, device="cuda") for x in boxes.random_boxes(edge + 1, 87, -9, 0))
    c, s = net.bound_cells(lo, hi, mode="rafixed", prec="fp32", inflate=inflate)
    for n in (1, 2, 5, edge - 1, edge):
        a, b = net.bound_cells(lo[:n], hi[:n], mode="rafixed", prec="fp32", inflate=inflate)
        assert torch.equal(a, c[:n]) and torch.equal(b, s[:n]), n
    net.close()
