"""Launches of similar numbers of ranges share a captured graph: what goes in
is laid out for a power of two of ranges."""
import pytest

from paper_2411_01964_gb300 import inputs
from test_gpu_parity import assert_same_range

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("counts", [(1,), (2,), (3, 4), (5, 6, 7, 8), (9, 13, 16), (17, 25, 32), (33, 50, 64)])
def test_one_layout_per_power_of_two(gpu, orc, counts):
    sent = set()
    for n in counts + counts:
        reqs = [(lo, lo + 20001 + lo % 100) for lo, _ in inputs.batch_requests(n, n)]
        res = gpu.verify_batch([a for a, _ in reqs], [b for _, b in reqs])
        for g, o in zip(res, orc.verify_ranges(reqs)):
            assert_same_range(g, o, per_n=False)
        sent.add(gpu.last_transfer()[0])
    assert len(sent) == 1
