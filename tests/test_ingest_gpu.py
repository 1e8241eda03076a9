"""Every form in which Y is taken stores the same values: full matrices with
rows on and off 16-byte boundaries (leading dimension and base), FP32 and FP64,
host and device, the packed upper triangle; results are bitwise those of the
packed host form.  The diagonal and the lower triangle hold NaN throughout.
A negative, NaN or Inf entry is refused and named wherever it lies."""
import numpy as np
import pytest

from paper_1905_04582_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def results(wl, y, **kw):
    from paper_1905_04582_gb300.mds import MDS
    with MDS(wl.n, wl.d, "fp64", strip=2) as m:
        m.set_data(y, **kw)
        m.set_sigma(wl.sigma)
        m.set_locations(wl.x_eval)
        ll, g, ds = m.gradient()
    return ll, g, ds


def full(wl, ld, shift, dtype):
    """An N x N view with leading dimension ld, its first entry `shift` entries into the buffer."""
    n = wl.n
    buf = np.full(shift + n * ld, np.nan, dtype=dtype)
    iu, ju = np.triu_indices(n, 1)
    buf[shift + iu * ld + ju] = wl.y_packed
    return buf


@pytest.mark.parametrize("n", [2, 5, 63, 64, 65, 130, 192, 260, 301])
def test_all_forms_store_the_same(n):
    wl = W.custom(n, 2, sigma=0.5, seed=80 + n)
    ref = results(wl, wl.y_packed)
    forms = []
    for ld in sorted({n, n + 1, (n + 3) // 4 * 4, (n + 3) // 4 * 4 + 8}):
        for shift in (0, 1, 4):
            for dtype in (np.float32, np.float64):
                buf = full(wl, ld, shift, dtype)
                forms.append((torch.from_numpy(buf).cuda()[shift:], dict(layout="full", ld=ld)))
                if shift == 0:
                    forms.append((buf, dict(layout="full", ld=ld)))
    forms.append((torch.from_numpy(wl.y_packed).cuda(), {}))
    forms.append((wl.y_packed.astype(np.float64), {}))
    for y, kw in forms:
        got = results(wl, y, **kw)
        assert got[0] == ref[0] and got[2] == ref[2], (kw, y.dtype)
        np.testing.assert_array_equal(got[1], ref[1])


@pytest.mark.parametrize("n,i,j", [(130, 0, 1), (130, 3, 64), (130, 62, 127), (130, 127, 129), (192, 64, 191),
                                   (260, 17, 200), (260, 255, 259)])
@pytest.mark.parametrize("bad", [-1.0, -1e-30, float("nan"), float("inf")])
def test_bad_entries_are_refused_and_named(n, i, j, bad):
    from paper_1905_04582_gb300.capi import MDSError
    from paper_1905_04582_gb300.mds import MDS
    wl = W.custom(n, 2, sigma=0.5, seed=7)
    for ld in (n, n + 1, (n + 3) // 4 * 4):
        buf = full(wl, ld, 0, np.float32)
        buf[i * ld + j] = bad
        with MDS(n, 2) as m:
            with pytest.raises(MDSError, match=rf"Y\({i}, {j}\)"):
                m.set_data(torch.from_numpy(buf).cuda(), layout="full", ld=ld)
