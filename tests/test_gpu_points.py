"""Point queries at the counts where the kernel changes (a block per point with
four or two exponents at a time, then a warp per four points), against the
oracle's trial division: all sizes of n, small, even and CRT-forced ones among
them.  All integers: equality."""
import numpy as np
import pytest

from paper_2411_01964_gb300 import Verifier, inputs

pytestmark = pytest.mark.gpu


def mixed_points(count):
    pts = list(range(0, 40)) + [9, 25, 49, 3 ** 5 + 2, 5 ** 8 + 4, (1 << 50) - 1, (1 << 50) - 3]
    pts += inputs.crt_forced(6, 20, max_bits=50)
    pts += [p * p + 2 for p in (104723, 1000003, 33554393)]           # n - 2 the square of a prime
    pts += [p * p * 3 + 4 for p in (104729, 1000003, 19369999)]       # n - 4 three times one
    for bits, seed in ((50, 1), (40, 2), (30, 3), (20, 4), (10, 5)):
        pts += inputs.random_points(seed, max(count // 5, 1), 2, 1 << bits)
    return (pts[-count:] if count < len(pts) // 2 else pts * (count // len(pts) + 1))[:count]


@pytest.mark.parametrize("count", [1, 2, 33, 304, 305, 3648, 7296, 7297, 7400, 12345])
def test_point_counts(gpu, orc, count):
    pts = mixed_points(count)
    assert len(pts) == count
    assert np.array_equal(gpu.min_k(pts), orc.min_k(pts))


@pytest.mark.parametrize("count", [40, 400, 8000])
def test_points_around_the_32_bit_test(orc, count):
    # below 2^52 primes are ruled out in 32 bits, from there on in 64
    pts = [(1 << 52) + d for d in range(-39, 41, 2)] + inputs.random_points(6, count, 1 << 51, 1 << 53)
    pts = pts[:count]
    with Verifier(max_hi=(1 << 53) + 1) as v:
        assert np.array_equal(v.min_k(pts), orc.min_k(pts))


def test_small_tables(orc):
    # tables with fewer primes than one step takes
    for max_hi in (30, 4000, 1 << 20):
        with Verifier(max_hi=max_hi) as v:
            for count in (5, 400, 8000):
                pts = [i % max_hi for i in range(count)]
                assert np.array_equal(v.min_k(pts), orc.min_k(pts))
