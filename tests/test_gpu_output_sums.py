"""The float32 output layer's sum over the last activation's symbols keeps small terms beside a large one."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__ as g
    g.build()
    import paper_2402_13861_gb300 as p
    torch.cuda.set_device(0)
    return p


@pytest.mark.parametrize("n", [1, 2000])
def test_small_symbols_beside_a_large_one(pkg, n):
    """512 neurons alike but for signs that cancel in every input row, so that the spread is sum gamma |w_m|: one
    weight 1 per column of 32 and fifteen of just below half an ulp of gamma, which a plain running sum drops
    (14.25 ulp in all).  Three of them may be lost beside the large term, and the three sums of four, the tree
    over the lanes and the last additions round: at most (3 + 3 + 1) / 2 ulp for each of the two columns."""
    w = 512
    sign = np.where(np.arange(w) % 2 == 0, 1.0, -1.0)
    W0 = (sign[:, None] * np.array([[1.0, 0.5, 0.25]])).astype(np.float32)
    b0, b1 = np.zeros(w, np.float32), np.zeros(1, np.float32)
    lo = torch.full((n, 3), -0.3, device="cuda")
    hi = torch.full((n, 3), 0.3, device="cuda")

    def spread(small):
        w1 = np.zeros((1, w), np.float32)
        w1[0, 0:2] = 1.0
        for k in range(1, 16):
            w1[0, 32 * k:32 * k + 2] = small
        net = pkg.Inr([(W0, b0), (w1, b1)])
        c, s = net.bound_cells(lo, hi, mode="sound", prec="fp32")
        c, s = c.cpu().numpy().astype(np.float64), s.cpu().numpy().astype(np.float64)
        net.close()
        assert np.all(s == s[0])
        return s[0]

    gamma = spread(0.0) / 2
    ulp = 2.0 ** (np.floor(np.log2(gamma)) - 23)
    small = np.float32(0.475 * ulp / gamma)
    grown = spread(small) - 2 * gamma
    assert abs(grown - 30 * gamma * float(small)) <= 7 * ulp
