"""A batch's tuned shape is one of its own candidates: the strip kernel,
chunks of 2-16 tiles, or chunks that make one to three full waves of the chunk
slots, which depends on the number of chains.  A batch of one chain, tuned
first, leaves its shape to no batch of more chains over the same datasets."""
import pytest

from paper_1905_04582_gb300 import workloads as W
from test_batch_gpu import build

pytestmark = pytest.mark.gpu


def candidates(ns, chains, slots):
    tiles = [((n + 63) // 64) * ((n + 63) // 64 + 1) // 2 for n in ns]
    out = {1, 2, 3, 4, -2, -4, -8, -16}
    for m in (1, 2, 3):
        per = 1
        while per < 256 and sum(c * max(1, t // per) for t, c in zip(tiles, chains)) > slots * m:
            per += 1
        out.add(-per)
    return out


@pytest.mark.parametrize("ns", [(1330,), (700, 90), (1000,), (1600,), (900, 900, 900)])
def test_tuned_shape_is_of_the_batch(ns):
    torch = pytest.importorskip("torch")
    slots = 3 * torch.cuda.get_device_properties(0).multi_processor_count  # D = 2: three chunk CTAs per SM
    datasets = [W.custom(n, 2, sigma=0.5, seed=80 + n) for n in ns]
    for count in (1, 24):
        chains = [count] * len(ns)
        b, _ = build(datasets, chains)
        with b:
            b.evaluate()
            assert b.get_strip() in candidates(ns, chains, slots), (count, b.get_strip())
