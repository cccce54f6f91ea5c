"""Entry points that read nothing back only enqueue: they return while earlier work of their stream still runs."""
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


@pytest.mark.parametrize("w,H,n,mode,inflate", [(16, 2, 70001, "clt", False), (48, 3, 70001, "sound", True),
                                                (256, 5, 4001, "clt", False), (512, 2, 200, "sound", False),
                                                (64, 2, 50001, "rafixed", True)])
def test_fp32_bounds_only_enqueue(pkg, w, H, n, mode, inflate):
    """From a few cells to more than one chunk of the row buffers.  The first call sizes the workspace and times the
    tile shapes; about a second of other work is ahead of the second one, which must be back before that ends."""
    net = pkg.Inr(inr.random_inr([3] + [w] * H + [1], 140 + w))
    lo, hi = (torch.tensor(x, device="cuda") for x in boxes.random_boxes(n, 141, -10, -4))
    c, s = torch.empty(n, device="cuda"), torch.empty(n, device="cuda")
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        c0, s0 = net.bound_cells(lo, hi, mode=mode, prec="fp32", inflate=inflate)
        stream.synchronize()
        torch.cuda._sleep(2_000_000_000)
        net.bound_cells(lo, hi, mode=mode, prec="fp32", inflate=inflate, center=c, spread=s)
        assert not stream.query()
        stream.synchronize()
        assert torch.equal(c, c0) and torch.equal(s, s0)
    net.close()


@pytest.mark.parametrize("w,H,long,short", [(16, 2, 70001, 65536), (256, 5, 4001, 3000)])
def test_a_shorter_list_needs_no_more_workspace(pkg, w, H, long, short):
    """A capture may not allocate: after a list of several chunks any shorter one, also of one larger chunk, can be
    captured."""
    net = pkg.Inr(inr.random_inr([3] + [w] * H + [1], 145 + w))
    lo, hi = (torch.tensor(x, device="cuda") for x in boxes.random_boxes(long, 146, -10, -4))
    c0, s0 = net.bound_cells(lo, hi, mode="clt", prec="fp32")
    c, s = torch.zeros(short, device="cuda"), torch.zeros(short, device="cuda")
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        net.bound_cells(lo[:short], hi[:short], mode="clt", prec="fp32", center=c, spread=s)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(c, c0[:short]) and torch.equal(s, s0[:short])
    net.close()
