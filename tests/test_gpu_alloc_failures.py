"""Allocations that fail after others of the same call have succeeded (made on
the host): the call returns SV_ENOMEM, and the next calls on the same context
are exact.  Integers: equality with the CPU oracle."""
import numpy as np
import pytest

from paper_2411_01964_gb300 import B, Verifier, inputs
from test_gpu_parity import unpack_bitmap

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def no_failures_left():
    yield
    from paper_2411_01964_gb300 import binding
    binding.load().sv_inject_alloc_failures(binding._CTX(1), 0)


def enomem(call):
    with pytest.raises(B.SvError) as e:
        call()
    assert e.value.status == B.SV_ENOMEM


def test_bucket_counts_grown_before_the_buckets_fail(orc):
    # stale counts would fill the buckets up: wrong strikes, or a launch repeated with deeper buckets
    lo = (1 << 40) + 64
    short, long = lo + (1 << 21), lo + (1 << 24)
    want = orc.sieve_odd(lo, short)
    with Verifier(max_hi=1 << 41, tile_log2=14, margin_log2=6) as v:
        def bitmap_is_exact():
            before = v.kernel_launches()
            bits, f0, cnt = unpack_bitmap(v.sieve_bitmap(lo, short).cpu().numpy().view(np.uint32), lo, short)
            assert np.array_equal(bits[f0:f0 + cnt], want)
            return v.kernel_launches() - before

        launches = bitmap_is_exact()
        B.sv_inject_alloc_failures_after(v.ctx, 1, 1)  # the counts grow, the buckets do not
        enomem(lambda: v.sieve_bitmap(lo, long))
        B.sv_inject_alloc_failures(v.ctx, 0)
        assert bitmap_is_exact() == launches


@pytest.mark.parametrize("skip", range(10))
def test_any_allocation_of_a_growing_call(orc, skip):
    # whichever buffer fails, a call that fits the buffers of before is exact
    lo = (1 << 44) + 12345
    small, large = lo + (1 << 22), lo + (1 << 30)
    o = orc.verify_range(lo, small)
    with Verifier(max_hi=1 << 45) as v:
        assert v.verify_range(lo, small).hist == o.hist
        B.sv_inject_alloc_failures_after(v.ctx, skip, 1)
        try:
            v.verify_range(lo, large)
        except B.SvError as e:
            assert e.status == B.SV_ENOMEM
        B.sv_inject_alloc_failures(v.ctx, 0)
        for hi in (small, lo + (1 << 24)):
            o = orc.verify_range(lo, hi)
            g = v.verify_range(lo, hi)
            assert g.hist == o.hist and g.first_n == o.first_n and np.array_equal(g.list_n, o.list_n)


def test_points_of_a_launch_whose_ranges_fail(orc):
    # the points of a slot are launched first; when its ranges then fail for
    # want of memory, the slot's next points are answered from their own staging
    lo = (1 << 44) + 12345
    with Verifier(max_hi=1 << 46, serve_slots=1) as v:
        t = v.submit_points([3])
        assert v.poll(t, -1) == B.SV_OK
        for i, count in enumerate((2048, 1024, 40000, 2048)):
            B.sv_inject_alloc_failures(v.ctx, 1 << 20)
            burst = [v.prepare_points(inputs.random_points(10 + i, count, 2, 1 << 44)),
                     v.prepare_range(lo, lo + (1 << 24))]
            v.submit_many(burst)
            assert v.poll(burst[1], -1) == B.SV_ENOMEM
            B.sv_inject_alloc_failures(v.ctx, 0)
            pts = inputs.random_points(20 + i, 1500, 2, 1 << 44)
            after = v.submit_points(pts)
            v.poll(burst[0], -1)
            assert v.poll(after, -1) == B.SV_OK
            assert np.array_equal(after.result(), orc.min_k(pts))
