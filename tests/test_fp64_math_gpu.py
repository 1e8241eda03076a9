"""FP64 pair arithmetic (root and its inverse, phi/Phi and log Phi from the
table) where it can go wrong: z from 0 to beyond the table's end at 9.5 in
steps finer than its nodes, coincident points, y that is zero or subnormal,
sigma from very small to very large, and tile edges; both FP64 entry points
against the oracle with the FP64 tolerances of the parity tests."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_1905_04582_gb300 import capi
from paper_1905_04582_gb300 import workloads as W
from gpu_util import TOL, grad_check, scalar_check

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _points(n, d, sigma, seed):
    """A line of points 0.0973 sigma apart (z up to 12 and beyond) with a
    little noise across it, one coincident pair, one pair 1e-9 sigma apart."""
    rng = np.random.default_rng(seed)
    x = 1e-3 * sigma * rng.standard_normal((n, d))
    x[:, 0] = 0.0973 * sigma * np.arange(n)
    if n > 8:
        x[5] = x[2]
        x[7] = x[6]
        x[7, 0] += 1e-9 * sigma
    dist = np.sqrt(((x[:, None, :] - x[None, :, :]) ** 2).sum(-1))
    y = np.abs(dist + 0.7 * sigma * rng.standard_normal((n, n))).astype(np.float32)
    yp = y[np.triu_indices(n, 1)]
    yp[0] = 0.0
    if yp.size > 2:
        yp[1] = 1e-42  # subnormal
    return x, yp


@pytest.mark.parametrize("n,d,sigma", [(2, 1, 0.5), (33, 1, 0.3), (64, 2, 1e-4), (129, 2, 0.3), (200, 3, 1e6),
                                       (191, 4, 0.05), (130, 5, 2.0), (97, 8, 0.3), (160, 2, 1e-30)])
def test_fp64_pair_arithmetic(n, d, sigma):
    from paper_1905_04582_gb300.mds import MDS
    x, yp = _points(n, d, sigma, 7 * n + d)
    ll_ref, _ = oracle.loglik(yp, x, sigma)
    g_ref, s_abs, s_sq = oracle.gradient(yp, x, sigma, with_abs=True, with_sq=True)
    ds_ref = oracle.dsigma(yp, x, sigma)
    m_pairs = n * (n - 1) / 2
    tol = TOL["fp64"]
    got = []
    with MDS(n, d, "fp64") as m:
        m.set_data(yp)
        m.set_locations(x)
        m.set_sigma(sigma)
        got.append(("mds_gradient", *m.gradient()))
    y_dev = torch.from_numpy(W.packed_to_full(yp, n)).cuda()
    x_dev = torch.from_numpy(x).cuda()
    g_dev = torch.full((n, d), float("nan"), dtype=torch.float64, device="cuda")
    ll, ds = ctypes.c_double(), ctypes.c_double()
    capi.check(capi.lib().mds_loglik_grad_noalloc(n, d, y_dev.data_ptr(), n, x_dev.data_ptr(), sigma,
                                                  g_dev.data_ptr(), ctypes.byref(ll), ctypes.byref(ds), None))
    got.append(("noalloc", ll.value, g_dev.cpu().numpy(), ds.value))
    for who, ll_v, g, ds_v in got:
        scalar_check(ll_v, ll_ref, tol["ll"], scale=m_pairs * (1 + abs(np.log(sigma))), what=f"L {who}")
        scalar_check(ds_v, ds_ref, tol["g"], scale=abs(ds_ref) + 2 * m_pairs / sigma, what=f"dL/dsigma {who}")
        grad_check(g, g_ref, s_abs, tol["g"], what=f"gradient {who}", s_sq=s_sq, u=tol["u"])
