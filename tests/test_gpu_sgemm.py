"""The float32 matrix tile of sgemm.cuh at the edges of its launch shapes (ragged widths, partial tiles,
both tile forms of the point evaluation) against the float64 oracle."""
import numpy as np
import pytest
import torch

from oracle import affine, mlp
from synth import boxes, inr

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


@pytest.mark.parametrize("w,H,act,mode,inflate", [(16, 1, "relu", "sound", True), (16, 3, "relu", "clt", False),
                                                  (48, 4, "sine", "clt", False), (64, 2, "relu", "raua", False),
                                                  (112, 3, "relu", "sound", False), (128, 3, "elu", "clt", False),
                                                  (272, 2, "relu", "sound", True), (512, 2, "relu", "clt", False)])
def test_fp32_bounds_row_edges(pkg, w, H, act, mode, inflate):
    """Coarse to fine boxes, from one cell to more than fit with every symbol alive (where the host reads the
    row counts and a chunk is shrunk and restarted): a cell's bound does not depend on its neighbours or
    the chunking, and stays within the float32 band 8 H w 2^-24 (|x0| + s) of the oracle."""
    layers = inr.random_inr([3] + [w] * H + [1], 60 + w, act=act)
    net = pkg.Inr(layers, act=act)
    full = min(1 << 16, (6 << 30) // (2 * (3 + w * (H - 1)) * w * 4))
    n = min(70001, full + 513)
    lo, hi = boxes.random_boxes(n, 61, -10, -1)
    order = np.argsort(hi[:, 0] - lo[:, 0], kind="stable")          # fine boxes first, coarse ones last
    dlo, dhi = (torch.tensor(x[order], device="cuda") for x in (lo, hi))
    c, s = net.bound_cells(dlo, dhi, mode=mode, prec="fp32", inflate=inflate)
    pick = np.unique(np.r_[0, 1, n // 2, n - 2, n - 1, np.random.default_rng(62).integers(0, n, 24)])
    for i in pick[[0, 3, len(pick) // 2, -1]]:
        ci, si = net.bound_cells(dlo[i:i + 1], dhi[i:i + 1], mode=mode, prec="fp32", inflate=inflate)
        assert ci[0] == c[i] and si[0] == s[i]
    a, b = net.bound_cells(dlo[pick].contiguous(), dhi[pick].contiguous(), mode=mode, prec="fp32", inflate=inflate)
    assert torch.equal(a, c[pick]) and torch.equal(b, s[pick])
    c, s = c.cpu().numpy().astype(np.float64)[pick], s.cpu().numpy().astype(np.float64)[pick]
    if act == "relu":
        oc, os_ = affine.bound(layers, lo[order][pick], hi[order][pick], mode, batch=8)
    else:
        oc, os_ = affine.bound(layers, lo[order][pick], hi[order][pick], mode, batch=8, act=act)
    tol = 8 * H * w * 2.0 ** -24 * (np.abs(oc) + os_) + 1e-7
    if inflate:
        assert np.all(c - s <= oc - os_ + 1e-7) and np.all(c + s >= oc + os_ - 1e-7)
    else:
        assert np.all(np.abs(c - oc) <= tol) and np.all(np.abs(s - os_) <= tol)
    net.close()


def test_fp32_bounds_under_capture(pkg):
    """A stream capture takes the float32 bound (no host reads), after a plain call sized the workspace."""
    net = pkg.Inr(inr.random_inr([3, 64, 64, 64, 1], 70))
    lo, hi = (torch.tensor(x, device="cuda") for x in boxes.random_boxes(200, 71, -8, -1))
    c0, s0 = [x.clone() for x in net.bound_cells(lo, hi, mode="clt", prec="fp32")]
    c, s = torch.zeros_like(c0), torch.zeros_like(s0)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        net.bound_cells(lo, hi, mode="clt", prec="fp32", center=c, spread=s)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(c, c0) and torch.equal(s, s0)
    net.close()


@pytest.mark.parametrize("w,H,inflate", [(16, 2, False), (48, 3, True), (64, 2, False), (80, 2, True), (256, 2, False),
                                         (400, 2, False), (512, 2, True)])
def test_rafixed_tile_edges(pkg, w, H, inflate):
    """Both tile forms (two cells per thread up to w = 64, four above), ragged last tiles and few cells: a cell's
    bound is the same whatever its tile, and within the float32 band of the oracle (an enclosure with inflation)."""
    layers = inr.random_inr([3] + [w] * H + [1], 100 + w)
    net = pkg.Inr(layers)
    lo, hi = boxes.random_boxes(20003, 101, -10, -2)
    dlo, dhi = torch.tensor(lo, device="cuda"), torch.tensor(hi, device="cuda")
    c, s = net.bound_cells(dlo, dhi, mode="rafixed", inflate=inflate)
    for n in (1, 3, 63, 305, 4001):
        a, b = net.bound_cells(dlo[:n].contiguous(), dhi[:n].contiguous(), mode="rafixed", inflate=inflate)
        assert torch.equal(a, c[:n]) and torch.equal(b, s[:n]), n
    idx = np.r_[0:40, 20003 - 40:20003]
    oc, os_ = affine.bound(layers, lo[idx], hi[idx], "rafixed", batch=40)
    c, s = c.cpu().numpy().astype(np.float64)[idx], s.cpu().numpy().astype(np.float64)[idx]
    if inflate:
        assert np.all(c - s <= oc - os_ + 1e-7) and np.all(c + s >= oc + os_ - 1e-7)
    else:
        tol = 8 * H * w * 2.0 ** -24 * (np.abs(oc) + os_) + 1e-7
        assert np.all(np.abs(c - oc) <= tol) and np.all(np.abs(s - os_) <= tol)
    net.close()
