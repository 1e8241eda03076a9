"""The trajectory-start kernel's energy partials at a size where they take
more than one allocation unit (512 bytes): H(end) - H(start) of a trajectory
against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1905_04582_gb300 import workloads as W
from test_hmc_gpu import dh_tol

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d", [(2300, 8), (5000, 4)])
def test_energy_partials_of_many_start_ctas(n, d):
    from paper_1905_04582_gb300.mds import MDS
    wl = W.custom(n, d, sigma=0.5, seed=19)
    x0 = wl.x_eval.astype(np.float64)
    p0 = np.random.default_rng(4).standard_normal((n, d))
    _, _, h0, h1 = oracle.leapfrog(wl.y_packed, x0, p0, wl.sigma, 1e-3, 2, nthreads=8)
    with MDS(n, d, "fp64") as m:
        m.set_data(wl.y_packed)
        m.set_locations(x0)
        m.set_sigma(wl.sigma)
        ll, _ = m.log_likelihood()
        dh = m.leapfrog(2, 1e-3, p0=p0)
    assert abs(dh - (h1 - h0)) <= dh_tol("fp64", ll), (dh, h1 - h0)
