"""Held-out densities where their FP64 arithmetic can go wrong: z from 0 to
beyond the table's end at 9.5, coincident points, y zero or subnormal,
negative coordinates, sigma very small and very large, one draw (scaled sums
of 1) and several, and pair counts from 1 to more than one pass of the grid."""
import numpy as np
import pytest

import oracle
from paper_1905_04582_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32c", "fp64"])
@pytest.mark.parametrize("n,d,sigma,draws", [(3, 1, 0.5, 1), (129, 1, 0.3, 2), (130, 2, 1e-4, 1), (200, 3, 1e5, 3),
                                             (97, 8, 0.3, 2), (640, 2, 0.4, 1)])
def test_lpd_matches_oracle(prec, n, d, sigma, draws):
    from paper_1905_04582_gb300.mds import MDS
    rng = np.random.default_rng(11 * n + d)
    x = 1e-3 * sigma * rng.standard_normal((n, d))
    x[:, 0] = 0.0973 * sigma * (np.arange(n) - n // 2)
    if n > 8:
        x[5] = x[2]
    x = x.astype(np.float32).astype(np.float64)
    iu, ju = np.triu_indices(n, 1)
    dist = np.sqrt(((x[iu] - x[ju]) ** 2).sum(-1))
    yp = np.abs(dist + 0.7 * sigma * rng.standard_normal(len(iu))).astype(np.float32)
    yp[0] = 0.0
    yp[1] = 1e-42  # subnormal
    fold = np.stack([iu, ju], axis=1)[:-1]  # all pairs but the last
    xs = [(x + 0.05 * sigma * k).astype(np.float32) * (1 if k % 2 == 0 else -1) for k in range(draws)]
    sg = [sigma * (1 + 0.25 * k) for k in range(draws)]
    with MDS(n, d, prec) as m:
        m.set_data(yp)
        m.set_sigma(sigma)
        m.set_locations(xs[0])
        m.set_heldout([tuple(p) for p in fold.tolist()])
        for xk, sk in zip(xs, sg):
            m.set_locations(xk)
            m.set_sigma(sk)
            m.lpd_accumulate()
        got, count = m.lpd()
    assert count == draws
    ref = oracle.lpd(yp, fold, [xk.astype(np.float64) for xk in xs], sg)
    # a pair's terms are u^2 / 2 of order 1, log Phi of order 1 and log sigma, each to a few ulps of FP64
    assert abs(got - ref) <= 1e-13 * len(fold) * (4 + abs(np.log(sigma)))
