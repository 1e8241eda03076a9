"""Batches whose chunked pass takes several launches (more chains than one
launch's arguments hold) and whose reduction takes whole column blocks (more
quarter blocks than resident CTAs), against the oracle: likelihood, gradient
and one HMC iteration of the first, a middle and the last chain."""
import numpy as np
import pytest

import oracle
from paper_1905_04582_gb300 import workloads as W
from gpu_util import TOL, grad_check, scalar_check
from test_batch_gpu import build

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes,chains,d,strip", [((130, 65), (66, 3), 2, -2), ((257,), (64,), 1, -30),
                                                  ((700, 90), (30, 35), 3, -9), ((130,), (5,), 6, -4)])
def test_batch_launches_match_oracle(sizes, chains, d, strip):
    datasets = [W.custom(n, d, sigma=0.5, seed=60 + n) for n in sizes]
    b, xs = build(datasets, list(chains), strip=strip)
    eps, steps, seed = 8e-4, 3, 77
    where = [(k, j) for k, c in enumerate(chains) for j in range(c)]
    pick = sorted({0, len(where) // 2, len(where) - 1})
    tol = TOL["fp32c"]
    with b:
        ll, _ = b.evaluate()
        for g in pick:
            k, j = where[g]
            w, x64 = datasets[k], xs[k][j].astype(np.float64)
            g_ref, s_abs, s_sq = oracle.gradient(w.y_packed, x64, w.sigma, with_abs=True, with_sq=True)
            scalar_check(ll[g], oracle.loglik(w.y_packed, x64, w.sigma)[0], tol["ll"], what=f"L chain {g}")
            grad_check(b.get_gradient(k, j), g_ref, s_abs, tol["g"], s_sq=s_sq, u=tol["u"], what=f"grad {g}")
        acc, dh = b.hmc(1, steps, [eps] * len(sizes), seed=seed)
        for g in pick:
            k, j = where[g]
            w, x64 = datasets[k], xs[k][j].astype(np.float64)
            p0 = oracle.draw_momentum(seed, g, 0, w.n * d)[0].reshape(w.n, d)
            xr, pr, h0, h1 = oracle.leapfrog(w.y_packed, x64, p0, w.sigma, eps, steps)
            assert abs(dh[0, g] - (h1 - h0)) <= 2e-6 * abs(ll[g]) + 1e-6 * w.n * d, (g, dh[0, g], h1 - h0)
            ref = xr if acc[0, g] else x64
            np.testing.assert_allclose(b.get_locations(k, j), ref, rtol=0, atol=2e-5 * (1 + np.abs(xr).max()))
