"""FP64 products and sums that the adaptive kernels issue as fused multiply-adds
round as plain ones, zero signs, subnormals and infinities included."""
import numpy as np
import pytest

import paper_2011_01740_gb300 as ens

pytestmark = pytest.mark.gpu


def test_products_and_sums_round_as_plain_ones():
    """Valve right-hand side with kappa = 0 and q = 0, so that the evaluation's own
    multiply-adds round as a product (whose sum with +0 differs only if it is an
    exact zero) or a sum: no tolerance."""
    import torch
    v = np.array([0.0, -0.0, 1.0, -1.0, 1 / 3, 5e-324, -5e-324, 1e-310, 3e-308, -1e-200, 1e200, 1.7e308, -1.7e308,
                  np.inf, -np.inf])
    sq = np.array([0.0, 1.0, 4.0, 2.0 ** -1060, 2.0 ** 1020, np.inf])       # their roots are exact
    y1, d, y3, b = (a.ravel() for a in np.meshgrid(v, v, sq, v, indexing="ij"))
    n = y1.size
    P = np.stack([np.zeros(n), np.zeros(n), d, b, np.ones(n)])
    y = np.stack([y1, np.full(n, 0.75), y3])
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    dy = torch.empty(y.shape, dtype=torch.float64, device="cuda")
    ens.ens_eval_rhs(ens.ENS_SYS_RELIEF_VALVE, n, dev(P), dev(np.zeros(n)), dev(y), dy)
    got = dy.cpu().numpy()
    with np.errstate(all="ignore"):
        p = -y1 * np.sqrt(y3)
        p = np.where((y1 == 0) | (y3 == 0), p + 0.0, p)      # one that underflows keeps its sign
        want = np.stack([y[1], -0.0 * y[1] + (y3 - (y1 + d)), b * p])
    nan = np.isnan(want)
    assert np.array_equal(np.isnan(got), nan)
    assert np.array_equal(got.view(np.int64)[~nan], want.view(np.int64)[~nan])
