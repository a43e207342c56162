"""The stream layout of the fused range path (streams.cu) against the CPU
oracle, at the sizes where it can go wrong: windows of every size, ranges that
end on and around a tile's last bit, ranges near 0, and first occurrences
outside a range's first tile.  All integers: equality."""
import pytest

from paper_2411_01964_gb300 import Verifier, inputs
from test_gpu_parity import assert_same_range

pytestmark = pytest.mark.gpu

MARGIN = 4320                                            # bits below a tile at the default margin


def core(threads):
    return 32 * 36 * threads - MARGIN                    # odd n per tile


@pytest.mark.parametrize("threads", [32, 64, 128, 256, 512])
@pytest.mark.parametrize("extra", [-1, 0, 1, 37])
def test_ranges_around_a_window(gpu, orc, threads, extra):
    for lo in (3, (1 << 30) + 1, (1 << 49) + 12345):
        hi = lo + 2 * (core(threads) + extra)
        assert_same_range(gpu.verify_range(lo, hi), orc.verify_range(lo, hi), per_n=False)


@pytest.mark.parametrize("lo,n_odd", [(0, 1), (3, 35), (3, 36), (5, 37), (4001, 4500), ((1 << 44) + 63, 1152),
                                      ((1 << 44) + 1, 3 * core(512) + 11)])
def test_odd_starts_and_lengths(gpu, orc, lo, n_odd):
    for d in (0, 1, 64, 2 * 1151):
        assert_same_range(gpu.verify_range(lo + d, lo + d + 2 * n_odd), orc.verify_range(lo + d, lo + d + 2 * n_odd),
                          per_n=False)


@pytest.mark.parametrize("knobs", [dict(tile_log2=17, threads=128, ctas_per_sm=4, margin_log2=6),
                                   dict(tile_log2=18, threads=256, margin_log2=14),
                                   dict(large_prime_min=40), dict(large_prime_min=16384, margin_log2=9)],
                         ids=lambda k: "-".join(f"{a}{b}" for a, b in k.items()))
def test_shapes_of_the_stream_layout(orc, knobs):
    with Verifier(max_hi=(1 << 50) + (1 << 24), **knobs) as v:
        for lo, hi in [(3, 1 << 22), ((1 << 40) + 7, (1 << 40) + 7 + (1 << 23) + 99), ((1 << 50) - 70001, 1 << 50)]:
            assert_same_range(v.verify_range(lo, hi), orc.verify_range(lo, hi), per_n=False)


def test_first_occurrence_outside_the_first_tile(gpu, orc):
    # the first n with mink = 5 lies 85605 odd n above lo: the range's first
    # tile (69408 odd n at this length) has none
    lo, hi = 1099749996181, 1099749996181 + (1 << 24)
    o = orc.verify_range(lo, hi)
    assert o.first_n[5] == 1099750167391
    assert_same_range(gpu.verify_range(lo, hi), o, per_n=False)
    gpu.launch_range(lo, hi)
    assert_same_range(gpu.fetch_range(), o, per_n=False)


def test_batches_of_short_ranges(gpu, orc):
    reqs = [(lo, lo + 2 * n) for lo, n in zip((a for a, _ in inputs.batch_requests(5, 400)),
                                              (1 + 97 * i for i in range(400)))]
    res = gpu.verify_batch([a for a, _ in reqs], [b for _, b in reqs])
    for g, o in zip(res, orc.verify_ranges(reqs)):
        assert_same_range(g, o, per_n=False)


@pytest.mark.parametrize("n,k,margin", [(60690478781437, 13, 12), (9579717479644589, 14, 13)])
def test_an_n_beyond_the_look_back(orc, n, k, margin):
    # a look-back of 2^12 or more: the exact test of the n beyond it is
    # launched only after the results have counted one
    rng = (n - 40000, n + 60000)
    o = orc.verify_range(*rng)
    assert o.hist[k] == 1 and o.first_n[k] == n
    with Verifier(max_hi=1 << (n.bit_length() + 1), margin_log2=margin) as v:
        assert_same_range(v.verify_range(*rng), o, per_n=False)
        v.launch_range(*rng)
        assert_same_range(v.fetch_range(), o, per_n=False)
        for count in (3, 40):
            for g in v.verify_batch([rng[0]] * count, [rng[1]] * count):
                assert_same_range(g, o, per_n=False)
