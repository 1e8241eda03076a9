"""Evaluations and trajectories of small problems, each in one launch: the
edges of its tiles, its units and its items per CTA, every dimension, a
locality order, a fold and the isotropic prior, against the oracle with the
tolerances of test_parity_gpu and test_hmc_gpu; the same with a forced shape
of the pass (a launch per pass and reduction) agrees to the same tolerance."""
import math

import numpy as np
import pytest

import oracle
from paper_1905_04582_gb300 import workloads as W
from gpu_util import TOL, grad_check, scalar_check

pytestmark = pytest.mark.gpu


def check(m, wl, p0, steps, eps, keep=None, lam=0.0):
    x64 = wl.x_eval.astype(np.float32).astype(np.float64)
    xr, pr, h0, h1 = oracle.leapfrog(wl.y_packed, x64, p0, wl.sigma, eps, steps, keep=keep, lam=lam)
    dh = m.leapfrog(steps, eps, p0=p0)
    x, p = m.get_locations(), m.get_momentum()
    ll, _ = m.log_likelihood()
    np.testing.assert_allclose(x, xr, rtol=0, atol=2e-6 * (1 + np.abs(xr).max()))
    np.testing.assert_allclose(p, pr, rtol=0, atol=1e-4 * (1 + np.abs(pr).max()))
    assert abs(dh - (h1 - h0)) <= 2e-6 * abs(ll) + 1e-6, (dh, h1 - h0)
    ll_ref, _ = oracle.loglik(wl.y_packed, xr, wl.sigma, keep=keep)
    assert math.isclose(ll, ll_ref, rel_tol=1e-6, abs_tol=3e-6)


def model(wl, **kw):
    from paper_1905_04582_gb300.mds import MDS
    m = MDS(wl.n, wl.d, "fp32c", **kw)
    m.set_data(wl.y_packed)
    m.set_locations(wl.x_eval)
    m.set_sigma(wl.sigma)
    return m


@pytest.mark.parametrize("n,d,steps", [(2, 1, 3), (17, 2, 2), (63, 2, 5), (64, 3, 5), (65, 2, 5), (128, 1, 4),
                                       (200, 2, 10), (200, 7, 3), (257, 4, 4), (321, 8, 3), (449, 5, 3), (385, 6, 3),
                                       (577, 2, 4), (640, 3, 3), (704, 2, 3), (832, 1, 2)])
def test_small_trajectory_matches_oracle(n, d, steps):
    wl = W.custom(n, d, sigma=0.5, seed=900 + n + d)
    p_all, _ = W.momenta(31, 1, n, d)
    eps = 0.014 / math.sqrt(n)
    with model(wl) as m:
        check(m, wl, p_all[0], steps, eps)
        check_again = m.get_locations()
        m.set_locations(wl.x_eval)
        m.leapfrog(steps, eps, p0=p_all[0])
        np.testing.assert_array_equal(m.get_locations(), check_again)  # bitwise reproducible
    with model(wl, chunks=1) as m:
        check(m, wl, p_all[0], steps, eps)


@pytest.mark.parametrize("reorder,fold,lam", [(True, False, 0.0), (False, True, 0.7), (True, True, 0.0)])
def test_small_trajectory_order_fold_prior(reorder, fold, lam):
    wl = W.custom(330, 2, sigma=0.4, seed=77)
    p_all, _ = W.momenta(32, 1, wl.n, wl.d)
    rng = np.random.default_rng(5)
    keep = None
    with model(wl) as m:
        m.set_prior(lam)
        if reorder:
            m.reorder()
        if fold:
            iu, ju = np.triu_indices(wl.n, 1)
            pick = rng.choice(len(iu), size=900, replace=False)
            pairs = [(int(iu[q]), int(ju[q])) for q in pick] + [(1, 2), (wl.n - 1, 0), (5, wl.n - 2)]
            m.set_heldout(pairs)
            keep = oracle.keep_mask(wl.n, pairs)
        check(m, wl, p_all[0], 4, 8e-4, keep=keep, lam=lam)


def test_small_hmc_device_draws_match_single_steps():
    # several iterations in the captured graph: the state of each start is the end of the one before
    wl = W.custom(200, 2, sigma=0.5, seed=12)
    x64 = wl.x_eval.astype(np.float32).astype(np.float64)
    p_all, u_all = W.momenta(33, 4, wl.n, wl.d)
    xr, acc_r, dh_r = oracle.hmc(wl.y_packed, x64, wl.sigma, 1e-3, 6, p_all, u_all)
    with model(wl) as m:
        ll0, _ = m.log_likelihood()
        acc, dh, _ = m.hmc(4, 6, 1e-3, p_all=p_all, u_all=u_all)
        x = m.get_locations()
    np.testing.assert_array_equal(np.asarray(acc), acc_r)
    assert np.all(np.abs(np.asarray(dh) - dh_r) <= 2e-6 * abs(ll0) + 1e-6)
    np.testing.assert_allclose(x, xr, rtol=0, atol=2e-5 * (1 + np.abs(xr).max()))


@pytest.mark.parametrize("n,d,mixture", [(2, 1, None), (17, 2, None), (63, 2, None), (64, 3, None), (65, 4, None),
                                         (128, 1, (6, 0.3)), (200, 2, None), (257, 2, (6, 0.3)), (321, 8, None),
                                         (385, 5, (3, 0.3)), (449, 6, None), (513, 2, (6, 0.3)), (641, 7, None),
                                         (832, 1, None)])
def test_small_evaluation_matches_oracle(n, d, mixture):
    torch = pytest.importorskip("torch")
    wl = W.custom(n, d, sigma=0.3 if mixture else 0.5, seed=700 + n + d, mixture=mixture)
    x64 = wl.x_eval.astype(np.float32).astype(np.float64)
    iu, ju = np.triu_indices(n, 1)
    rng = np.random.default_rng(n)
    pick = rng.choice(len(iu), size=max(1, len(iu) // 20), replace=False)
    folds = [None] if n < 17 else [None, [(int(iu[q]), int(ju[q])) for q in pick]]
    for reorder in (False, True):
        for fold in folds:
            keep = None if fold is None else oracle.keep_mask(n, fold)
            ll_ref, _ = oracle.loglik(wl.y_packed, x64, wl.sigma, keep=keep)
            ds_ref = oracle.dsigma(wl.y_packed, x64, wl.sigma, keep=keep)
            g_ref, s_abs, s_sq = oracle.gradient(wl.y_packed, x64, wl.sigma, keep=keep, with_abs=True, with_sq=True)
            m_pairs = n * (n - 1) // 2 if keep is None else int(keep.sum())
            tol = TOL["fp32c"]
            with model(wl) as m:
                if reorder:
                    m.reorder()
                if fold is not None:
                    m.set_heldout(fold)
                out = torch.empty(n, d, device="cuda")
                for how in ("host", "device f32", "device f64"):
                    if how == "host":
                        ll, g, ds = m.gradient()
                    else:
                        buf = out if how == "device f32" else out.double()
                        ll, _, ds = m.gradient(out=buf)
                        g = buf.double().cpu().numpy()
                    scalar_check(ll, ll_ref, tol["ll"], scale=max(abs(ll_ref), m_pairs), what=f"L {how}")
                    scalar_check(ds, ds_ref, tol["g"], scale=abs(ds_ref) + 2 * m_pairs / wl.sigma, what=f"ds {how}")
                    grad_check(g, g_ref, s_abs, tol["g"], s_sq=s_sq, u=tol["u"], what=f"gradient {how}")
