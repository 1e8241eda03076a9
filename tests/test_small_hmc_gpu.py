"""HMC of small problems as a user runs it: no shape of the pass forced, the
momenta and uniforms drawn on the device, so the iterations run whole in the
cluster's launch (csrc/small_traj.cu), up to 16 of them in one.  Every
iteration is compared with the oracle's from the locations it started at
(tolerances of test_hmc_gpu and test_small_traj_gpu); many iterations in one
call, in several calls, queued, and resumed from a snapshot are bitwise the
same chain; rejections and a growing split of the locations among them."""
import math

import numpy as np
import pytest

import oracle
from paper_1905_04582_gb300 import workloads as W
from gpu_util import TOL, grad_check

pytestmark = pytest.mark.gpu

SEED, ITERS = 7, 21  # two launches: 16 iterations and 5


def model(wl, scale=1.0, reorder=False, lam=0.0, fold=None):
    from paper_1905_04582_gb300.mds import MDS
    m = MDS(wl.n, wl.d, "fp32c")
    m.set_data(wl.y_packed)
    m.set_locations((wl.x_eval * scale).astype(np.float32))
    m.set_sigma(wl.sigma)
    m.set_prior(lam)
    if reorder:
        m.reorder()
    if fold is not None:
        m.set_heldout(fold)
    return m


def check_iteration(m, wl, t, steps, eps, lam=0.0, keep=None):
    """hmc(1), the chain's iteration t, against the oracle; (accepted, dH)."""
    x0 = m.get_locations()
    acc, dh, _ = m.hmc(1, steps, eps, seed=SEED)
    p, u = oracle.draw_momentum(SEED, 0, t, wl.n * wl.d)
    xr, pr, h0, h1 = oracle.leapfrog(wl.y_packed, x0, p.reshape(wl.n, wl.d), wl.sigma, eps, steps, keep=keep, lam=lam)
    ll = max(abs(oracle.loglik(wl.y_packed, v, wl.sigma, keep=keep)[0]) for v in (x0, xr))
    tol = 2e-6 * ll + 1e-6 * max(1.0, abs(h0), abs(h1))
    assert abs(dh[0] - (h1 - h0)) <= tol, (t, dh[0], h1 - h0)
    if abs(math.log(u) + h1 - h0) > 2 * tol:
        assert bool(acc[0]) == (math.log(u) < h0 - h1), (t, dh[0], u)
    x = m.get_locations()
    if acc[0]:
        np.testing.assert_allclose(x, xr, rtol=0, atol=2e-5 * (1 + np.abs(xr).max()))
        np.testing.assert_allclose(m.get_momentum(), pr, rtol=0, atol=1e-4 * (1 + np.abs(pr).max()))
    else:
        np.testing.assert_array_equal(x, x0)
    return bool(acc[0]), dh[0]


def check_gradient(m, wl, keep=None):
    x = m.get_locations()
    _, g, _ = m.gradient()
    g_ref, s_abs, s_sq = oracle.gradient(wl.y_packed, x, wl.sigma, keep=keep, with_abs=True, with_sq=True)
    grad_check(g, g_ref, s_abs, TOL["fp32c"]["g"], s_sq=s_sq, u=TOL["fp32c"]["u"])


@pytest.mark.parametrize("n,d,eps,scale,reorder,lam", [
    (200, 2, 0.02, 1.0, False, 0.0),   # rejections
    (300, 1, 0.012, 1.0, True, 0.0),
    (130, 4, 0.04, 1.0, False, 0.8),
    (65, 7, 0.09, 1.0, True, 0.0),
    (200, 2, 0.005, 0.05, False, 0.0),  # locations that spread 15 times: the split grows between iterations
    (130, 6, 0.01, 0.02, True, 0.0),
])
def test_iterations_match_oracle_and_one_another(n, d, eps, scale, reorder, lam):
    wl = W.custom(n, d, sigma=0.5, seed=900 + n + d)
    steps = 4
    with model(wl, scale, reorder, lam) as m:
        single = [check_iteration(m, wl, t, steps, eps, lam=lam) for t in range(ITERS)]
        x, p, ll = m.get_locations(), m.get_momentum(), m.log_likelihood()
        check_gradient(m, wl)
    acc, dh = np.array([s[0] for s in single]), np.array([s[1] for s in single])
    if scale == 1.0:
        assert acc.any() and not acc.all()
    else:
        assert np.abs(x).max() > 8 * np.abs(wl.x_eval * scale).max()  # beyond the first split's bound

    def same(m, a, h):
        np.testing.assert_array_equal(a, acc)
        np.testing.assert_array_equal(h, dh)
        np.testing.assert_array_equal(m.get_locations(), x)
        np.testing.assert_array_equal(m.get_momentum(), p)
        assert m.log_likelihood() == ll

    with model(wl, scale, reorder, lam) as m:
        a, h, stats = m.hmc(ITERS, steps, eps, seed=SEED)
        same(m, a, h)
        assert stats["accepted"] == acc.sum() and stats["iterations"] == ITERS
    with model(wl, scale, reorder, lam) as m:
        m.hmc_enqueue(7, steps, eps, seed=SEED)
        m.hmc_enqueue(ITERS - 7, steps, eps, seed=SEED)
        a, h, stats = m.hmc_collect()
        same(m, a, h)
        assert stats["accepted"] == acc.sum()
    # a snapshot resumes as the chain whose locations are set anew (the split then follows from them)
    with model(wl, scale, reorder, lam) as m:
        m.hmc(4, steps, eps, seed=SEED)
        state = m.get_state()
        m.set_locations(m.get_locations())
        a1, h1, _ = m.hmc(ITERS - 4, steps, eps, seed=SEED)
        np.testing.assert_array_equal(a1, acc[4:])
        x1, p1, ll1 = m.get_locations(), m.get_momentum(), m.log_likelihood()
    with model(wl, scale, False, lam) as m:
        m.set_state(state)
        a2, h2, _ = m.hmc(ITERS - 4, steps, eps, seed=SEED)
        np.testing.assert_array_equal(a2, a1)
        np.testing.assert_array_equal(h2, h1)
        np.testing.assert_array_equal(m.get_locations(), x1)
        np.testing.assert_array_equal(m.get_momentum(), p1)
        assert m.log_likelihood() == ll1


def test_rejections_of_a_fold_with_injected_draws():
    wl = W.custom(330, 2, sigma=0.4, seed=77)
    rng = np.random.default_rng(5)
    iu, ju = np.triu_indices(wl.n, 1)
    fold = [(int(iu[q]), int(ju[q])) for q in rng.choice(len(iu), size=900, replace=False)]
    keep = oracle.keep_mask(wl.n, fold)
    p_all, u_all = W.momenta(35, ITERS, wl.n, wl.d)
    u_all[::3] = 1.0 - 1e-9  # these accept only where the energy falls
    steps, eps = 4, 0.012
    with model(wl, fold=fold) as m:
        acc, dh, _ = m.hmc(ITERS, steps, eps, p_all=p_all, u_all=u_all)
        x = m.get_locations()
        check_gradient(m, wl, keep)
    with model(wl, fold=fold) as m:
        for t in range(ITERS):
            x0 = m.get_locations()
            a, h, _ = m.hmc(1, steps, eps, p_all=p_all[t:t + 1], u_all=u_all[t:t + 1])
            assert a[0] == acc[t] and h[0] == dh[t]
            xr, _, h0, h1 = oracle.leapfrog(wl.y_packed, x0, p_all[t], wl.sigma, eps, steps, keep=keep)
            ll = max(abs(oracle.loglik(wl.y_packed, v, wl.sigma, keep=keep)[0]) for v in (x0, xr))
            assert abs(h[0] - (h1 - h0)) <= 2e-6 * ll + 1e-6 * max(1.0, abs(h0), abs(h1)), (t, h[0], h1 - h0)
            if not a[0]:
                np.testing.assert_array_equal(m.get_locations(), x0)
        np.testing.assert_array_equal(m.get_locations(), x)
    assert acc.any() and not acc.all()
