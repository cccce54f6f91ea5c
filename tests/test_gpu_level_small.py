"""Short level lists (culled, ranked and scattered by one block) against the general passes, either side of
the length where the choice changes (2048 cells)."""
import numpy as np
import pytest
import torch

from synth import inr

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__ as g
    g.build()
    import paper_2402_13861_gb300 as p
    torch.cuda.set_device(0)
    return p


@pytest.mark.parametrize("kd", [False, True])
def test_full_lists_either_side_of_the_limit(pkg, kd):
    """A network that no cell excludes: with the k-d split the lists are 1, 2, 4, ..., 2048, 4096 cells, with
    the octree 1, 8, 64, 512, 4096; every cell survives with both iso bits, once."""
    rng = np.random.default_rng(90)
    layers = [(W, rng.normal(0, 0.1, size=b.shape).astype(np.float32)) for W, b in inr.random_inr([3, 16, 16, 1], 91)]
    net = pkg.Inr(layers)
    r = net.extract(4, [0.0, 1e-3], mode="sound", prec="fp32", kd_tree=kd, bound_stop_level=0)
    codes, masks = r["codes"][:r["n_active"]].cpu().numpy(), r["masks"][:r["n_active"]].cpu().numpy()
    i = np.arange(16, dtype=np.int64)
    want = np.sort((i[:, None, None] | (i[None, :, None] << 10) | (i[None, None, :] << 20)).ravel())
    assert np.array_equal(np.sort(codes.astype(np.int64)), want)
    assert np.all(masks == 3)
    net.close()


def test_pruned_lists_nest(pkg):
    """Lists that grow past the limit while cells are culled: the survivors of a level are the children of
    survivors above it, and a finer extraction repeats them."""
    net = pkg.Inr(inr.random_inr([3, 32, 32, 1], 92))
    runs = [net.extract(L, [0.0], mode="sound", prec="fp32", kd_tree=kd) for kd in (False, True) for L in (3, 4, 5, 6)]
    for a, b in ((0, 1), (1, 2), (2, 3)):
        up = runs[a]["codes"][:runs[a]["n_active"]].cpu().numpy().astype(np.int64)
        dn = runs[b]["codes"][:runs[b]["n_active"]].cpu().numpy().astype(np.int64)
        assert dn.size > 0 and np.unique(dn).size == dn.size
        par = (dn >> 1) & ~((1 << 9) | (1 << 19))
        assert np.all(np.isin(par, up))
    assert runs[3]["n_active"] > 2048
    net.close()
