"""Block sizes whose half is not a whole number of warps, for launches whose
tiles are halved: such a launch must still scan every n once.  Histograms,
lists, per-n values and bitmaps against the CPU oracle; integers: equality."""
import numpy as np
import pytest

from paper_2411_01964_gb300 import Verifier
from test_gpu_parity import assert_same_range, unpack_bitmap

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("threads", [544, 608, 864, 992])
def test_halved_blocks_are_whole_warps(orc, threads):
    # 2^24 odd n in tiles of 2^16 are 257 tiles, fewer than two per SM: halved once
    lo = (1 << 44) + 12345
    hi = lo + (1 << 25)
    o = orc.verify_range(lo, hi, per_n=True)
    with Verifier(max_hi=1 << 45, tile_log2=16, threads=threads) as v:
        assert_same_range(v.verify_range(lo, hi), o, per_n=False)
        assert_same_range(v.verify_range(lo, hi, per_n=True), o)
        bits, f0, cnt = unpack_bitmap(v.sieve_bitmap(lo, hi).cpu().numpy().view(np.uint32), lo, hi)
        assert np.array_equal(bits[f0:f0 + cnt], orc.sieve_odd(lo, hi))


def test_halved_default_tiles(orc):
    lo = (1 << 47) + 1
    hi = lo + (1 << 28)
    with Verifier(max_hi=1 << 48, threads=544) as v:
        assert_same_range(v.verify_range(lo, hi), orc.verify_range(lo, hi), per_n=False)
