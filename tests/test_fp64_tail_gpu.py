"""phi/Phi and log Phi of the FP64 path by themselves: with y equal to delta a
pair's residual is zero, so that dL/dX is phi/Phi and sum r is log Phi alone.
z from the table's first nodes over its end at 10 to where both underflow,
single pairs through both FP64 entry points and sums of pairs of one z (two
clusters, the pairs within them held out), and residuals from 0 to where the
two terms vanish beside them.

Bounds: the oracle takes erfc and exp of rounded arguments, z^2 u each for the
argument's rounding and as much again for its square, the table's side z^2 u
for z; 4 (z^2 + 4) u holds both sides, u = 2^-53, and the FP64 tolerance of the
parity tests, 1e-12, is above it.  dL/dsigma and L are sums with M / sigma and
M log sigma: the scalar tolerances of the parity tests."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_1905_04582_gb300 import capi
from paper_1905_04582_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
U = 2.0 ** -53


def bound(z):
    return 4 * (z * z + 4) * U


def noalloc(y, x, sigma):
    n, d = x.shape
    y_dev = torch.from_numpy(W.packed_to_full(y, n)).cuda()
    x_dev = torch.from_numpy(x).cuda()
    g = torch.full((n, d), float("nan"), dtype=torch.float64, device="cuda")
    ll, ds = ctypes.c_double(), ctypes.c_double()
    capi.check(capi.lib().mds_loglik_grad_noalloc(n, d, y_dev.data_ptr(), n, x_dev.data_ptr(), sigma, g.data_ptr(),
                                                  ctypes.byref(ll), ctypes.byref(ds), None))
    return ll.value, g.cpu().numpy(), ds.value


@pytest.mark.parametrize("sigma", [1.0, 0.25])
def test_single_pairs_without_residual(sigma):
    from paper_1905_04582_gb300.mds import MDS
    rng = np.random.default_rng(3)
    zs = np.concatenate([rng.uniform(a, a + 0.5, 6) for a in np.arange(0.5, 12, 0.5)] +
                        [[1 / 128, 0.25, 3 - 1 / 128, 7 + 1 / 128, 9.5, 10 - 2 ** -20, 10, 10 + 2 ** -20, 20, 30, 37]])
    with MDS(2, 1, "fp64") as m:
        m.set_sigma(sigma)
        for z in zs:
            dist = np.float32(z * sigma)  # sigma a power of two: z' = dist / sigma exactly
            zz = float(dist) / sigma
            x = np.array([[0.0], [float(dist)]])
            y = np.array([dist], dtype=np.float32)
            _, r_ref = oracle.loglik(y, x, sigma)
            g_ref = oracle.gradient(y, x, sigma)
            m.set_data(y)
            m.set_locations(x)
            _, g, _ = m.gradient()
            _, r = m.log_likelihood()
            assert abs(r - r_ref) <= bound(zz) * abs(r_ref), (zz, r, r_ref)
            ll_na, g_na, _ = noalloc(y, x, sigma)
            if sigma == 1.0:
                assert abs(ll_na + r_ref) <= bound(zz) * abs(r_ref), (zz, ll_na, r_ref)
            for who in (g, g_na):
                assert np.all(np.abs(who - g_ref) <= bound(zz) * np.abs(g_ref)), (zz, who, g_ref)


@pytest.mark.parametrize("z", [4.5, 8.25, 9.75, 10.5, 11.5, 20.0, 36.0])
@pytest.mark.parametrize("d", [1, 3, 6])
def test_sums_of_pairs_without_residual(z, d):
    from paper_1905_04582_gb300.mds import MDS
    # two clusters on a line: every distance between them is exact
    sigma, half = 0.5, 37
    n = 2 * half
    x = np.zeros((n, d))
    x[half:, 0] = z * sigma
    x[:, 0] += np.tile(np.arange(half) / 1024.0, 2)
    iu, ju = np.triu_indices(n, 1)
    y = np.abs(x[iu, 0] - x[ju, 0]).astype(np.float32)
    within = [(int(i), int(j)) for i, j in zip(iu, ju) if (i < half) == (j < half)]
    keep = oracle.keep_mask(n, within)
    _, r_ref = oracle.loglik(y, x, sigma, keep=keep)
    g_ref = oracle.gradient(y, x, sigma, keep=keep)
    tol = bound(z + 0.1)
    with MDS(n, d, "fp64") as m:
        m.set_data(y)
        m.set_locations(x)
        m.set_sigma(sigma)
        m.set_heldout(within)
        _, g, _ = m.gradient()
        _, r = m.log_likelihood()
    assert abs(r - r_ref) <= (tol + n * U) * abs(r_ref)
    assert np.all(np.abs(g - g_ref) <= (tol + n * U) * np.abs(g_ref))


@pytest.mark.parametrize("z", [9.99, 10.01, 10.7, 11.3, 12.5, 25.0])
def test_small_residuals(z):
    from paper_1905_04582_gb300.mds import MDS
    # y = dist (1 + k 2^-23): residuals from none to far above the vanishing terms
    sigma = 1.0
    dist = np.float32(z)
    with MDS(2, 1, "fp64") as m:
        m.set_sigma(sigma)
        for k in [0, 1, -1, 3, 64, -1000, 20000, 300000]:
            y = np.array([dist * np.float32(1 + k * 2.0 ** -23)], dtype=np.float32)
            x = np.array([[0.0], [float(dist)]])
            _, r_ref = oracle.loglik(y, x, sigma)
            g_ref = oracle.gradient(y, x, sigma)
            m.set_data(y)
            m.set_locations(x)
            _, g, _ = m.gradient()
            _, r = m.log_likelihood()
            _, g_na, _ = noalloc(y, x, sigma)
            assert abs(r - r_ref) <= bound(z) * abs(r_ref), (k, r, r_ref)
            for who in (g, g_na):
                assert np.all(np.abs(who - g_ref) <= bound(z) * np.abs(g_ref)), (k, who, g_ref)
