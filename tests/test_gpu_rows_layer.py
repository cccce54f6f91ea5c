"""The fused layer kernel of the row-batched BF16 path (rows_layer.cu) at the edges of its tiles: partial tiles of
32 cells, the two forms at width 64, cells with no, one and many 64-row blocks of symbol rows, against the
oracle with per-result bands (tests/_rounding_model.py)."""
import numpy as np
import pytest
import torch

from synth import boxes, inr

import _rounding_model as rm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__ as g
    g.build()
    import paper_2402_13861_gb300 as p
    torch.cuda.set_device(0)
    return p


@pytest.mark.parametrize("w,H,act,mode", [(64, 2, "relu", "clt"), (64, 4, "relu", "sound"), (64, 3, "elu", "clt"),
                                          (128, 2, "relu", "raua"), (128, 3, "elu", "clt"), (256, 2, "relu", "clt"),
                                          (256, 4, "relu", "sound"), (256, 2, "sine", "clt"), (512, 3, "relu", "clt"),
                                          (512, 2, "relu", "sound")])
def test_rows_layer_tile_edges(pkg, w, H, act, mode):
    layers = inr.random_inr([3] + [w] * H + [1], 80 + w + H, act=act)
    rng = np.random.default_rng(81)
    layers = [(W, rng.normal(0, 0.1, size=b.shape).astype(np.float32)) for W, b in layers]
    net = pkg.Inr(layers, act=act)
    top = 32 * 152 + 33 if w == 64 else 97
    lo, hi = boxes.random_boxes(top, 82, -10, -2)
    for n in (1, 31, 32, 33, top):
        c, s = net.bound_cells(torch.tensor(lo[:n], device="cuda"), torch.tensor(hi[:n], device="cuda"), mode=mode,
                               prec="bf16")
        idx = np.unique(np.r_[0, n // 2, max(0, n - 2), n - 1])
        b = rm.bound_bands(layers, lo[idx], hi[idx], mode, batch=4, act=act)
        c, s = c.cpu().numpy().astype(np.float64)[idx], s.cpu().numpy().astype(np.float64)[idx]
        assert np.all(np.abs(c - b["centre"]) <= b["band_c"]) and np.all(np.abs(s - b["spread"]) <= b["band_s"]), n
    net.close()
