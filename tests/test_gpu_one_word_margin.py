"""A margin of one word (margin_log2 = 6) under the lean scan of the linear
layout, in ranges long enough that most tiles search no first occurrence any
more and take the scan's unmasked loop where its alignment allows.  Integers:
equality with the CPU oracle."""
import pytest

from paper_2411_01964_gb300 import Verifier
from test_gpu_parity import assert_same_range

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("knobs,log2_len", [(dict(tile_log2=14, threads=128), 26), (dict(stamp_primes=2), 31),
                                            (dict(tile_log2=16, threads=256), 29)],
                         ids=["tile14", "stamp2", "tile16"])
@pytest.mark.parametrize("margin_log2", [6, 7])
def test_long_ranges(orc, knobs, log2_len, margin_log2):
    lo = (1 << 45) + 1
    hi = lo + (1 << log2_len)
    o = orc.verify_range(lo, hi)
    with Verifier(max_hi=1 << 46, margin_log2=margin_log2, **knobs) as v:
        assert_same_range(v.verify_range(lo, hi), o, per_n=False)
        assert_same_range(v.verify_range_plain(lo, hi), o, per_n=False)
