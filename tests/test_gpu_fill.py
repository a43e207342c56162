"""The bucket fill against the CPU oracle where its quick tests and its split
into items can go wrong: batches of 1 to 600 ranges (one range per multiplier
item, then chunks of up to 16), empty and tiny ranges among long ones, hits at
either end of a range, and every threshold between the two kinds of items."""
import pytest

from paper_2411_01964_gb300 import Verifier, inputs
from test_gpu_parity import assert_same_range

pytestmark = pytest.mark.gpu


def check(v, orc, reqs):
    res = v.verify_batch([a for a, _ in reqs], [b for _, b in reqs])
    for g, o in zip(res, orc.verify_ranges(reqs)):
        assert_same_range(g, o, per_n=False)


@pytest.mark.parametrize("count", [1, 31, 33, 63, 65, 200, 600])
def test_batch_sizes(gpu, orc, count):
    reqs = [(lo, lo + min(hi - lo, 1 << 18)) for lo, hi in inputs.batch_requests(count, count)]
    reqs[::7] = [(lo, lo + 1 + lo % 5) for lo, _ in reqs[::7]]
    check(gpu, orc, reqs)


@pytest.mark.parametrize("knobs", [dict(mult_prime_log2=m) for m in (10, 15, 18, 20, 31)],
                         ids=lambda k: str(k["mult_prime_log2"]))
def test_hits_at_the_ends(orc, knobs):
    # ranges around odd multiples j p^2 of primes of every size: the multiple
    # is the value 2 below the first or the last n
    reqs = []
    for p in (2053, 4099, 65537, 262147, 1048583, 8388617, 16777259):
        for j in (1, 3, 65, 101, 4097):
            m = j * p * p
            if (1 << 12) < m < (1 << 50) - (1 << 14):
                reqs += [(m + 2, m + 2 + 500), (m + 2 - 998, m + 3), (m - 5000, m + 5000)]
    with Verifier(max_hi=1 << 50, **knobs) as v:
        check(v, orc, reqs)
        check(v, orc, reqs[:3])
