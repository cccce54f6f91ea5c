"""BF16 bounds either side of the list lengths where the row path takes another kernel: 16 cells per SM (the first
activation, UP with ReLU) and 32 (the output layer at width 128).  The same bits, cell by cell."""
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


@pytest.mark.parametrize("w,H,per_sm", [(64, 1, 16), (64, 3, 16), (128, 3, 16), (256, 3, 16), (512, 2, 16), (128, 1, 16),
                                        (128, 2, 32), (128, 4, 32)])
def test_either_side_of_a_switch(pkg, w, H, per_sm):
    net = pkg.Inr(inr.random_inr([3] + [w] * H + [1], 160 + w + H))
    edge = torch.cuda.get_device_properties(0).multi_processor_count * per_sm
    lo, hi = (torch.tensor(x, device="cuda") for x in boxes.random_boxes(edge, 161, -9, 0))
    for mode, inflate in (("clt", False), ("sound", False), ("sound", True), ("raua", False)):
        c, s = net.bound_cells(lo, hi, mode=mode, prec="bf16", inflate=inflate)
        a, b = net.bound_cells(lo[:edge - 1], hi[:edge - 1], mode=mode, prec="bf16", inflate=inflate)
        assert torch.equal(a, c[:edge - 1]) and torch.equal(b, s[:edge - 1]), (mode, inflate)
        assert torch.isfinite(c).all() and torch.isfinite(s).all()
    net.close()
