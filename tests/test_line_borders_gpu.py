"""Items on a line (D = 1) that lie close together on the two sides of a border
between multiples of the split's quantum q, from a rounding apart to a
hundredth of q: L and the gradient by every FP32C pass against the oracle
(there d^2 as Dh^2 plus a correction is a difference of equal numbers).  The
tolerances are those of the parity tests."""
import math

import numpy as np
import pytest

import oracle
from paper_1905_04582_gb300 import workloads as W
from gpu_util import TOL, grad_check, scalar_check

pytestmark = pytest.mark.gpu


def problem(n, sigma, seed):
    """(y, x): a cloud, and pairs about the borders (k + 1/2) q, a few and many quanta from 0."""
    rng = np.random.default_rng(seed)
    x = rng.standard_normal(n).astype(np.float32)
    x[0] = 3.75  # the largest: q = 2^ceil(log2(4 * 3.75 / 2047))
    q = 2.0 ** math.ceil(math.log2(4 * 3.75 / 2047))
    x = np.clip(x, -3.7, 3.75).astype(np.float32)
    gaps = [0.0, 2.0 ** -24, 1e-7, 3e-7, 1e-6, 3e-6, 1e-5, 1e-4]
    spots = [0, 1, -1, 37, -90, 200, 301]
    m = 1
    for i, k in enumerate(spots):
        for g in gaps:
            if m + 2 > n:
                break
            border = (k + 0.5) * q
            x[m], x[m + 1] = np.float32(border - g * (1 + i) / 4), np.float32(border + g * 0.6)
            m += 2
    perm = rng.permutation(n)
    x = x[perm][:, None].copy()
    assert np.abs(x).max() == np.float32(3.75)
    iu, ju = np.triu_indices(n, 1)
    d = np.abs(x[iu, 0].astype(np.float64) - x[ju, 0])
    return np.abs(d + sigma * rng.standard_normal(len(iu))).astype(np.float32), x


def check(ll, g, y, x, sigma, what):
    n = len(x)
    x64 = x.astype(np.float64)
    ll_ref, _ = oracle.loglik(y, x64, sigma)
    g_ref, s_abs, s_sq = oracle.gradient(y, x64, sigma, with_abs=True, with_sq=True)
    tol = TOL["fp32c"]
    m_pairs = n * (n - 1) / 2
    scalar_check(ll, ll_ref, tol["ll"], scale=max(abs(ll_ref), m_pairs), what=f"L {what}")
    grad_check(g, g_ref, s_abs, tol["g"], s_sq=s_sq, u=tol["u"], what=f"gradient {what}")


@pytest.mark.parametrize("n,sigma", [(150, 0.5), (700, 0.3), (60, 0.05)])
@pytest.mark.parametrize("kw", [{}, {"strip": 2}, {"chunks": 1}, {"reorder": True}, {"fold": True}])
def test_pairs_about_a_border(n, sigma, kw):
    from paper_1905_04582_gb300.mds import MDS
    y, x = problem(n, sigma, n)
    shape = {k: v for k, v in kw.items() if k in ("strip", "chunks")}
    with MDS(n, 1, "fp32c", **shape) as m:
        m.set_data(y)
        m.set_locations(x)
        m.set_sigma(sigma)
        if kw.get("reorder"):
            m.reorder()
        if kw.get("fold"):
            m.set_heldout([(0, n - 1)])
            _, g, _ = m.gradient()
            keep = oracle.keep_mask(n, [(0, n - 1)])
            g_ref, s_abs, s_sq = oracle.gradient(y, x.astype(np.float64), sigma, keep=keep, with_abs=True, with_sq=True)
            grad_check(g, g_ref, s_abs, TOL["fp32c"]["g"], s_sq=s_sq, u=TOL["fp32c"]["u"])
            return
        ll, g, _ = m.gradient()
        check(ll, g, y, x, sigma, str(kw))


@pytest.mark.parametrize("strip", [2, -6])
def test_batched_pairs_about_a_border(strip):
    from paper_1905_04582_gb300.mds import Batch
    n, sigma = 300, 0.4
    y, x = problem(n, sigma, 5)
    with Batch([n], 1, [2], strip=strip) as b:
        b.set_data(0, y)
        b.set_sigma(0, sigma)
        b.set_locations(0, 0, x)
        b.set_locations(0, 1, -x)
        ll, _ = b.evaluate()
        for c, xc in enumerate((x, -x)):
            check(ll[c], b.get_gradient(0, c), y, xc, sigma, f"chain {c}")
