"""Point queries whose points are small, large and mixed, at the counts where
the line between the two moves (it lies at 2^20, 2^34 or 2^38), against the
oracle's trial division; host and device arrays.  Integers: equality."""
import random

import numpy as np
import pytest
import torch

from paper_2411_01964_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count", [1, 31, 33, 304, 305, 1216, 1217, 3040, 3041, 7296, 7297, 9000])
def test_small_and_large_points(gpu, orc, count):
    pts = list(range(12)) + [x + d for x in (1 << 20, 1 << 34, 1 << 38) for d in range(-4, 5)]
    pts += [p * p + 2 for p in (101, 103, 131, 137, 139, 4099, 8191)] + inputs.crt_forced(5, 8, max_bits=40)
    for seed, bits in enumerate((8, 14, 20, 22, 34, 35, 38, 40)):
        pts += inputs.random_points(seed, count // 8 + 1, 2, 1 << bits)
    random.Random(count).shuffle(pts)
    pts = np.array(pts[:count], dtype=np.uint64)
    want = orc.min_k([int(x) for x in pts])
    assert np.array_equal(gpu.min_k(pts), want)
    out = torch.full((count + 2,), 77, dtype=torch.uint8, device="cuda")
    gpu.min_k_device(torch.from_numpy(pts.view(np.int64)).cuda(), out[1:count + 1])
    gpu.synchronize()
    got = out.cpu().numpy()
    assert np.array_equal(got[1:-1], want) and got[0] == got[-1] == 77
    for below in (1 << 20, 1 << 36):                       # all small
        low = pts % np.uint64(below)
        assert np.array_equal(gpu.min_k(low), orc.min_k([int(x) for x in low]))
