"""Reduced bounds of long lists on narrow networks, where a CTA takes the most cells and its weight ring is smallest:
the output layer's sums, which go over the ring, must leave the cells' largest magnitudes behind it alone."""
import numpy as np
import pytest
import torch

from oracle import affine
from synth import boxes, inr

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__ as g
    g.build()
    import paper_2402_13861_gb300 as p
    torch.cuda.set_device(0)
    return p


@pytest.mark.parametrize("w,H,inflate", [(16, 1, True), (16, 2, True), (16, 3, True), (16, 2, False), (32, 3, True),
                                         (48, 2, True), (64, 2, True), (64, 3, False)])
def test_long_lists_equal_short_ones(pkg, w, H, inflate):
    """132, 200 and 256 cells per CTA at w = 16 against at most 128 (both parities of H: the magnitudes are
    double-buffered across layers): the same bits, and the oracle's bound enclosed or met as in short lists."""
    layers = inr.random_inr([3] + [w] * H + [1], 110 + w + H)
    net = pkg.Inr(layers)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 100003
    lo, hi = boxes.random_boxes(n, 111, -10, -2)
    dlo, dhi = torch.tensor(lo, device="cuda"), torch.tensor(hi, device="cuda")
    step = 2 * (1024 // w) * sms                   # up to one CTA per SM of 128 threads
    short = [net.bound_cells(dlo[a:a + step].contiguous(), dhi[a:a + step].contiguous(), mode="rafixed", inflate=inflate)
             for a in range(0, n, step)]
    c, s = (torch.cat(x) for x in zip(*short))
    for m in (132 * sms - 3, 200 * sms - 3, 20003, 30001, n):
        a, b = net.bound_cells(dlo[:m], dhi[:m], mode="rafixed", inflate=inflate)
        assert torch.equal(a, c[:m]) and torch.equal(b, s[:m]), m
    idx = np.r_[0:40, n - 40:n]
    oc, os_ = affine.bound(layers, lo[idx], hi[idx], "rafixed", batch=40)
    c, s = c.cpu().numpy().astype(np.float64)[idx], s.cpu().numpy().astype(np.float64)[idx]
    if inflate:
        assert np.all(c - s <= oc - os_ + 1e-7) and np.all(c + s >= oc + os_ - 1e-7)
    else:
        tol = 8 * H * w * 2.0 ** -24 * (np.abs(oc) + os_) + 1e-7
        assert np.all(np.abs(c - oc) <= tol) and np.all(np.abs(s - os_) <= tol)
    net.close()
