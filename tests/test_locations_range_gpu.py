"""Locations beyond the range of the FP32C split: FP64 entries that are finite
but no FP32 numbers are refused like other locations out of range, before
anything is written; infinite entries like NaN entries; and a trajectory that
diverges to infinity is reported and leaves the split of the locations it
restores as it was."""
import numpy as np
import pytest

from paper_1905_04582_gb300 import workloads as W
from paper_1905_04582_gb300.capi import MDS_ERR_INVALID_ARG, MDS_ERR_NONFINITE, MDSError

pytestmark = pytest.mark.gpu


def model(wl, **kw):
    from paper_1905_04582_gb300.mds import MDS
    m = MDS(wl.n, wl.d, "fp32c", **kw)
    m.set_data(wl.y_packed)
    m.set_sigma(wl.sigma)
    m.set_locations(wl.x_eval)
    return m


@pytest.mark.parametrize("n,d", [(120, 2), (4500, 8)])  # max |x| found by each CTA, by a kernel of its own
@pytest.mark.parametrize("where", ["host", "device"])
@pytest.mark.parametrize("bad", [1e36, 1e39, -3.5e38, -1e300])
def test_locations_beyond_fp32_are_refused(n, d, where, bad):
    torch = pytest.importorskip("torch")
    wl = W.custom(n, d, seed=12)
    with model(wl) as m:
        ll0, g0, _ = m.gradient()
        far = wl.x_eval.astype(np.float64)
        far[n - 3, d - 1] = bad
        with pytest.raises(MDSError) as e:
            m.set_locations(torch.from_numpy(far).cuda() if where == "device" else far)
        assert e.value.status == MDS_ERR_INVALID_ARG and "FP32C range" in str(e.value)
        np.testing.assert_array_equal(m.get_locations(dtype=np.float32), wl.x_eval)
        ll1, g1, _ = m.gradient()
        assert ll1 == ll0
        np.testing.assert_array_equal(g1, g0)


@pytest.mark.parametrize("n,d", [(120, 2), (4500, 8)])
@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("also", [0.5, 1e39])
def test_infinite_locations_are_refused(n, d, bad, also):
    wl = W.custom(n, d, seed=12)
    with model(wl) as m:
        x = wl.x_eval.astype(np.float64)
        x[5, 0] = bad
        x[6, 0] = also
        with pytest.raises(MDSError) as e:
            m.set_locations(x)
        assert e.value.status == MDS_ERR_INVALID_ARG
        if not (np.isnan(bad) and also == 1e39):
            assert "NaN or Inf" in str(e.value)


@pytest.mark.parametrize("kw", [{}, {"strip": 2}, {"chunks": 1}])
def test_diverged_trajectory_keeps_the_split(kw):
    wl = W.custom(200, 2, sigma=0.5, seed=14)
    with model(wl, **kw) as m:
        before = m.gradient()
        with pytest.raises(MDSError) as e:
            m.hmc(2, 3, 3e38, seed=5)
        assert e.value.status == MDS_ERR_NONFINITE
        np.testing.assert_array_equal(m.get_locations(dtype=np.float32), wl.x_eval)
        after = m.gradient()
        assert before[0] == after[0] and before[2] == after[2]
        np.testing.assert_array_equal(before[1], after[1])
        m.hmc(2, 3, 1e-3, seed=5)  # and the sampler goes on
