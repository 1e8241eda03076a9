"""Batched reductions on both sides of the line between quarter blocks and
whole column blocks (more quarters than CTAs that are resident at once: four
per SM up to D = 4, three at D = 5, two beyond), against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1905_04582_gb300 import workloads as W
from gpu_util import TOL, grad_check, scalar_check
from test_batch_gpu import build

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,per_sm", [(4, 4), (5, 3), (6, 2), (8, 2)])
@pytest.mark.parametrize("past", [False, True])
def test_batch_reduction_at_the_line(d, per_sm, past):
    torch = pytest.importorskip("torch")
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 130  # 3 column blocks: 12 quarters a chain
    chains = per_sm * sms // 12 + (1 if past else 0)
    wl = W.custom(n, d, sigma=0.5, seed=60 + d)
    b, xs = build([wl], [chains], strip=-2)
    with b:
        ll, ds = b.evaluate()
        for g in (0, chains // 2, chains - 1):
            x64 = xs[0][g].astype(np.float64)
            g_ref, s_abs, s_sq = oracle.gradient(wl.y_packed, x64, wl.sigma, with_abs=True, with_sq=True)
            tol = TOL["fp32c"]
            scalar_check(ll[g], oracle.loglik(wl.y_packed, x64, wl.sigma)[0], tol["ll"], what=f"L chain {g}")
            grad_check(b.get_gradient(0, g), g_ref, s_abs, tol["g"], s_sq=s_sq, u=tol["u"], what=f"grad {g}")
        x0 = [b.get_locations(0, g) for g in (0, chains - 1)]
        acc, dh = b.hmc(1, 3, [8e-4], seed=5)
        for g, x64 in zip((0, chains - 1), x0):
            p0 = oracle.draw_momentum(5, g, 0, n * d)[0].reshape(n, d)
            xr, _, h0, h1 = oracle.leapfrog(wl.y_packed, x64, p0, wl.sigma, 8e-4, 3)
            assert abs(dh[0, g] - (h1 - h0)) <= 2e-6 * abs(ll[g]) + 1e-6 * n * d
            ref = xr if acc[0, g] else x64
            np.testing.assert_allclose(b.get_locations(0, g), ref, rtol=0, atol=2e-5 * (1 + np.abs(xr).max()))
