"""The per-n output (one byte per n) where its 32-byte groups can go wrong:
output addresses of every alignment, ranges that start and end anywhere in a
group, tiles of several sizes, list thresholds from 1 on, and n that go to the
exact test.  Integers: equality with the CPU oracle, and no byte outside the
output is written."""
import numpy as np
import pytest
import torch

from paper_2411_01964_gb300 import Verifier
from test_gpu_parity import assert_same_range

pytestmark = pytest.mark.gpu


def device_per_n(v, lo, hi, shift):
    n = (hi - (max(lo, 3) | 1) + 1) // 2
    room = torch.full((n + 256,), 77, dtype=torch.uint8, device="cuda")
    d = room[64 + shift: 64 + shift + n]
    v.launch_range(lo, hi, d)
    g = v.fetch_range(list_cap=1 << 20)
    r = room.cpu().numpy()
    assert (r[:64 + shift] == 77).all() and (r[64 + shift + n:] == 77).all()
    g.per_n_k = r[64 + shift: 64 + shift + n]
    return g


@pytest.mark.parametrize("shift", [0, 1, 15, 16, 31])
@pytest.mark.parametrize("n_odd", [1, 31, 32, 33, 100, 5000, (1 << 15) + 1, 3 * (1 << 19) + 7])
def test_alignments(gpu, orc, shift, n_odd):
    for lo in (3, (1 << 40) + 7, (1 << 49) + 64 * 12345 + 63):
        hi = lo + 2 * n_odd
        o = orc.verify_range(lo, hi, per_n=True)
        assert_same_range(device_per_n(gpu, lo, hi, shift), o)


@pytest.mark.parametrize("knobs", [dict(record_k_threshold=t) for t in (1, 2, 3, 4, 5)] +
                         [dict(margin_log2=6, tile_log2=14), dict(margin_log2=7), dict(tile_log2=20, margin_log2=18),
                          dict(threads=128, tile_log2=16)],
                         ids=lambda k: "-".join(f"{a}{b}" for a, b in k.items()))
def test_options(orc, knobs):
    with Verifier(max_hi=1 << 45, **knobs) as v:
        T = v.config.record_k_threshold
        for lo, n_odd in ((3, 70001), ((1 << 44) + 1, 100003)):
            if T < 3:
                n_odd //= 8
            o = orc.verify_range(lo, lo + 2 * n_odd, per_n=True, list_k_threshold=T)
            assert_same_range(device_per_n(v, lo, lo + 2 * n_odd, 5), o)
