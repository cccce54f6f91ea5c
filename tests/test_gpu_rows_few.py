"""BF16 bounds of few cells (several warps per cell and column for the new rows up to four cells per SM, a
cluster of blocks per cell for the output layer up to one) against those of many: the same bits."""
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


@pytest.mark.parametrize("w,H,act", [(64, 5, "relu"), (128, 4, "elu"), (256, 4, "relu"), (512, 3, "relu"), (512, 4, "sine")])
def test_few_cells_equal_many(pkg, w, H, act):
    """Fine to coarse boxes: from no new row to all of them, in one hand-over of the output layer and in several."""
    net = pkg.Inr(inr.random_inr([3] + [w] * H + [1], 30 + w, act=act), act=act)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    lo, hi = (torch.tensor(x, device="cuda") for x in boxes.random_boxes(4 * sms + 1, 31, -9, 0))
    modes = [("clt", False), ("sound", False), ("sound", True), ("raua", False)] if act == "relu" else [("clt", False)]
    for mode, inflate in modes:
        c, s = net.bound_cells(lo, hi, mode=mode, prec="bf16", inflate=inflate)
        for n in (1, 2, sms, sms + 1, 4 * sms):
            a, b = net.bound_cells(lo[:n], hi[:n], mode=mode, prec="bf16", inflate=inflate)
            assert torch.equal(a, c[:n]) and torch.equal(b, s[:n]), (mode, inflate, n)
        assert torch.isfinite(c).all() and torch.isfinite(s).all()
    net.close()


@pytest.mark.parametrize("w,H", [(64, 4), (128, 3), (256, 3), (512, 3)])
def test_one_cell_per_warp_equals_several(pkg, w, H):
    """Lists either side of the length from which a warp takes several cells (48 or 64 cells per SM), with every
    remainder of a batch of rows among the cells."""
    net = pkg.Inr(inr.random_inr([3] + [w] * H + [1], 50 + w))
    edge = torch.cuda.get_device_properties(0).multi_processor_count * (48 if w == 256 else 64)
    lo, hi = (torch.tensor(x, device="cuda") for x in boxes.random_boxes(edge + 3, 51, -9, -2))
    for mode, inflate in (("clt", False), ("sound", True)):
        c, s = net.bound_cells(lo, hi, mode=mode, prec="bf16", inflate=inflate)
        a, b = net.bound_cells(lo[:edge - 1], hi[:edge - 1], mode=mode, prec="bf16", inflate=inflate)
        assert torch.equal(a, c[:edge - 1]) and torch.equal(b, s[:edge - 1]), (mode, inflate)
    net.close()
