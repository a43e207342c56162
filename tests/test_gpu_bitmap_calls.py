"""sv_sieve_bitmap beside its captured graph: the timing of other kernels than
the tile kernel, and a context on the legacy default stream, which cannot be
captured."""
import numpy as np
import pytest

from paper_2411_01964_gb300 import B, Verifier
from test_gpu_parity import unpack_bitmap

pytestmark = pytest.mark.gpu

LO, HI = (1 << 40) + 12345, (1 << 40) + 12345 + (1 << 22) + 77


def assert_bitmap(v, orc):
    bits, f0, cnt = unpack_bitmap(v.sieve_bitmap(LO, HI).cpu().numpy().view(np.uint32), LO, HI)
    assert np.array_equal(bits[f0:f0 + cnt], orc.sieve_odd(LO, HI))


@pytest.mark.parametrize("kernels", [["init"], ["bucket_fill"], ["tile"], ["init", "bucket_fill", "tile"]],
                         ids="-".join)
def test_timed_kernels(orc, kernels):
    with Verifier(max_hi=1 << 41) as v:
        assert_bitmap(v, orc)
        B.sv_kernel_timing(v.ctx, kernels)
        assert_bitmap(v, orc)
        for name, i in B.KERNEL_IDS.items():
            ms, n = B.sv_kernel_time(v.ctx, i)
            assert n == (name in kernels) and (ms > 0) == (name in kernels)


def test_legacy_stream(orc):
    with Verifier(max_hi=1 << 41, stream=1) as v:
        assert_bitmap(v, orc)
        assert_bitmap(v, orc)


def test_a_refused_capture_leaves_no_error(orc):
    # a range on the legacy stream is refused; the next calls are unaffected
    with Verifier(max_hi=1 << 41, stream=1) as v:
        with pytest.raises(B.SvError) as e:
            v.verify_range(LO, HI)
        assert e.value.status == B.SV_ECUDA
        assert_bitmap(v, orc)
    with Verifier(max_hi=1 << 41) as v:
        assert v.verify_range(LO, HI).hist == orc.verify_range(LO, HI).hist
