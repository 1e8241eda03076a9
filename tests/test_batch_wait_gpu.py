"""Every batched call that synchronises does so on all of its ways out: with
work queued before it on the batch's stream, mds_batch_hmc returns only when
that work is done, also with no iteration to run, whether the device tables
are as they were or change with the call (another step size)."""
import pytest

from paper_1905_04582_gb300 import workloads as W
from test_batch_gpu import build

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("strip", [2, -6])
@pytest.mark.parametrize("eps", [1e-3, 2e-3])
def test_hmc_without_iterations_waits(strip, eps):
    torch = pytest.importorskip("torch")
    stream = torch.cuda.Stream()
    b, _ = build([W.custom(130, 2, sigma=0.5, seed=51)], [2], strip=strip)
    with b:
        b._check(b._lib.mds_batch_set_stream(b._h, stream.cuda_stream))
        b.evaluate()
        b.hmc(1, 2, [1e-3], seed=1)
        with torch.cuda.stream(stream):
            torch.cuda._sleep(40_000_000)  # about 20 ms
        b.hmc(0, 2, [eps], seed=1)
        assert stream.query()
