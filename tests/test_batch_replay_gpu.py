"""Batched HMC calls one after another with something changed between them:
a dataset's sigma, its Y (also after mds_batch_reorder, where new data moves
Y to a new buffer), its step size.  Each call is compared with the oracle's
trajectory from the locations the call started at, with the tolerances of
test_batch_gpu; the draws are those of global chain g and iteration t."""
import numpy as np
import pytest

import oracle
from paper_1905_04582_gb300 import workloads as W
from test_batch_gpu import build

pytestmark = pytest.mark.gpu

SEED, STEPS = 99, 6


def one_iteration(b, datasets, sigmas, eps, t):
    """b.hmc(1, ...), its iteration t, against the oracle from the present locations."""
    where = [(k, j) for k, c in enumerate(b.chains) for j in range(c)]
    start = [b.get_locations(k, j) for k, j in where]
    acc, dh = b.hmc(1, STEPS, eps, seed=SEED)
    for g, (k, j) in enumerate(where):
        w = datasets[k]
        p0 = oracle.draw_momentum(SEED, g, t, w.n * w.d)[0].reshape(w.n, w.d)
        xr, _, h0, h1 = oracle.leapfrog(w.y_packed, start[g], p0, sigmas[k], eps[k], STEPS)
        ll = oracle.loglik(w.y_packed, xr, sigmas[k])[0]
        assert abs(dh[0, g] - (h1 - h0)) <= 2e-6 * abs(ll) + 1e-6 * w.n * w.d, (g, dh[0, g], h1 - h0)
        ref = xr if acc[0, g] else start[g]
        np.testing.assert_allclose(b.get_locations(k, j), ref, rtol=0, atol=5e-5 * (1 + np.abs(xr).max()))


@pytest.mark.parametrize("strip", [2, -6])
@pytest.mark.parametrize("d", [2, 5])
def test_hmc_after_new_sigma(strip, d):
    datasets = [W.custom(220, d, sigma=0.5, seed=51), W.custom(130, d, sigma=0.4, seed=52)]
    sigmas, eps = [0.5, 0.4], [4e-3, 5e-3]
    b, _ = build(datasets, [2, 1], strip=strip)
    with b:
        one_iteration(b, datasets, sigmas, eps, 0)
        for t, (k, s) in enumerate([(1, 0.9), (0, 0.35), (0, 0.5)], start=1):
            b.set_sigma(k, s)
            sigmas[k] = s
            one_iteration(b, datasets, sigmas, eps, t)
        eps = [2e-3, 5e-3]
        one_iteration(b, datasets, sigmas, eps, 4)


@pytest.mark.parametrize("strip", [2, -6])
@pytest.mark.parametrize("order", [False, True])
def test_hmc_after_new_data(strip, order):
    datasets = [W.custom(220, 2, sigma=0.5, seed=51), W.custom(130, 2, sigma=0.4, seed=52)]
    sigmas, eps = [0.5, 0.4], [4e-3, 5e-3]
    b, _ = build(datasets, [2, 2], strip=strip)
    with b:
        if order:
            b.reorder()
        one_iteration(b, datasets, sigmas, eps, 0)
        for t, (k, seed) in enumerate([(0, 61), (1, 62)], start=1):
            w = W.custom(datasets[k].n, 2, sigma=sigmas[k], seed=seed)
            b.set_data(k, w.y_packed)
            datasets[k] = w
            one_iteration(b, datasets, sigmas, eps, t)
