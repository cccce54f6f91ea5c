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
