"""Float32 bounds of a long list where the device has room for the smaller row buffers only."""
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


def test_less_memory_gives_the_same_bounds(pkg):
    """8000 cells of a 256 x 5 network ask for 12 GB of rows, and 6 GB are enough for chunks of half their length."""
    layers = inr.random_inr([3] + [256] * 5 + [1], 170)
    lo, hi = (torch.tensor(x, device="cuda") for x in boxes.random_boxes(8000, 171, -10, -4))
    net = pkg.Inr(layers)
    want = net.bound_cells(lo, hi, mode="clt", prec="fp32")
    torch.cuda.synchronize()
    net.close()
    net = pkg.Inr(layers)
    torch.cuda.empty_cache()
    free, total = torch.cuda.mem_get_info()
    room = 9 << 30                               # the smaller buffers and their eighth in reserve: 6.8 GB
    taken = torch.empty(max(0, free - room), dtype=torch.uint8, device="cuda")
    assert torch.cuda.mem_get_info()[0] < 12 << 30
    try:
        for _ in range(2):                       # the second call finds its workspace in place
            before = torch.cuda.mem_get_info()[0]
            c, s = net.bound_cells(lo, hi, mode="clt", prec="fp32")
            torch.cuda.synchronize()
        assert torch.cuda.mem_get_info()[0] == before
    finally:
        del taken
        torch.cuda.empty_cache()
    assert torch.equal(c, want[0]) and torch.equal(s, want[1])
    net.close()
