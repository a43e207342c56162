"""A prime table that grows (sv_init_primes with a larger bound) while a launch
is waiting to be fetched, or between launches that replay one captured graph:
the results are the oracle's.  The ranges hold an n beyond the look-back, whose
exact test is launched only when the results are fetched."""
import numpy as np
import pytest

from paper_2411_01964_gb300 import B, Verifier
from test_gpu_parity import assert_same_range

pytestmark = pytest.mark.gpu

N, K = 60690478781437, 13
RANGE = (N - 40000, N + 60000)


@pytest.fixture(scope="module")
def want(orc):
    o = orc.verify_range(*RANGE)
    assert o.hist[K] == 1 and o.first_n[K] == N
    return o


def test_between_launch_and_fetch(want):
    with Verifier(max_hi=1 << 46, margin_log2=12) as v:
        for bits in (48, 50, 51):
            v.launch_range(*RANGE)
            B.sv_init_primes(v.ctx, 1 << bits)
            assert_same_range(v.fetch_range(), want, per_n=False)


@pytest.mark.parametrize("count", [3, 40])
def test_between_launch_and_fetch_of_a_batch(want, count):
    with Verifier(max_hi=1 << 46, margin_log2=12) as v:
        v.launch_batch([RANGE[0]] * count, [RANGE[1]] * count)
        B.sv_init_primes(v.ctx, 1 << 49)
        for g in v.fetch_batch():
            assert_same_range(g, want, per_n=False)


def test_between_calls(orc, want):
    # 1 << 46 and the next bounds end in the same prime gap: tables of equal size
    big = (1 << 46) + (1 << 20)
    with Verifier(max_hi=1 << 46, margin_log2=12) as v:
        for hi in (1 << 46, (1 << 46) + 1000, (1 << 46) + 2000, big, 1 << 49):
            B.sv_init_primes(v.ctx, hi)
            for _ in range(2):
                assert_same_range(v.verify_range(*RANGE), want, per_n=False)
            lo = hi - (1 << 17)
            assert_same_range(v.verify_range(lo, hi), orc.verify_range(lo, hi), per_n=False)


def test_while_the_server_has_launches_in_flight(want):
    with Verifier(max_hi=1 << 46, margin_log2=12) as v:
        for bits in (47, 48, 49, 50):
            ts = [v.submit_range(*RANGE) for _ in range(24)]
            B.sv_init_primes(v.ctx, 1 << bits)
            for t in ts:
                assert v.poll(t, -1) == B.SV_OK
                got = t.result()
                assert got.hist == want.hist and got.first_n == want.first_n
                assert np.array_equal(got.list_n, want.list_n)
