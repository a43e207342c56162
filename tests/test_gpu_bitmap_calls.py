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
