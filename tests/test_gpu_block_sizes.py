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
    # 160 tiles of 2^16 odd n, fewer than three for two SMs: halved once
    lo = (1 << 44) + 12345
    hi = lo + 160 * (1 << 17)
    o = orc.verify_range(lo, hi, per_n=True)
    with Verifier(max_hi=1 << 45, tile_log2=16, threads=threads) as v:
        assert_same_range(v.verify_range(lo, hi), o, per_n=False)
        assert_same_range(v.verify_range(lo, hi, per_n=True), o)
        bits, f0, cnt = unpack_bitmap(v.sieve_bitmap(lo, hi).cpu().numpy().view(np.uint32), lo, hi)
        assert np.array_equal(bits[f0:f0 + cnt], orc.sieve_odd(lo, hi))


def test_halved_default_tiles(orc):
    lo = (1 << 47) + 1
    hi = lo + 160 * (1 << 20)
    with Verifier(max_hi=1 << 48, threads=544) as v:
        assert_same_range(v.verify_range(lo, hi), orc.verify_range(lo, hi), per_n=False)


@pytest.mark.parametrize("T", [2, 3, 4, 6])
@pytest.mark.parametrize("tiles", [1, 15, 16, 226, 227, 228])
def test_around_the_halving(orc, T, tiles):
    # tiles of 2^16 odd n where the halving starts and stops
    lo = (1 << 44) + 12345
    hi = lo + tiles * (1 << 17) - 1000
    with Verifier(max_hi=1 << 45, tile_log2=16, record_k_threshold=T) as v:
        o = orc.verify_range(lo, hi, per_n=True, list_cap=1 << 22, list_k_threshold=T)
        assert_same_range(v.verify_range(lo, hi, list_cap=1 << 22), o, per_n=False)
        assert_same_range(v.verify_range(lo, hi, list_cap=1 << 22, per_n=True), o)


@pytest.mark.parametrize("large_prime_min", [3500, 8192, 1 << 14, 1 << 20])
@pytest.mark.parametrize("log2_len", [18, 20, 24, 26])
def test_many_sparse_primes(orc, large_prime_min, log2_len):
    # the stream layout's block stops shrinking at eight sparse primes per thread
    lo = (1 << 44) + 12345
    hi = lo + (1 << log2_len) + 999
    with Verifier(max_hi=1 << 45, large_prime_min=large_prime_min) as v:
        assert_same_range(v.verify_range(lo, hi), orc.verify_range(lo, hi), per_n=False)
