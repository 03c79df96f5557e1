"""GPU: averaging blobs that crowd into one binning cell, on a grid where the blobs are taken in cell
order (256^3 and at least 1,024 blobs).

A blob's cost is its own box of grid points, wherever the others are, so crowded blobs may take
no more than ten times as long as the same number spread out (the rest is contention on one
cell's counter: 8,190 atomic adds, about 10 us); sorting that cell's entries serially took 3,500
times as long.  The values are compared bit for bit with averaging in index order, which fewer
than 1,024 blobs take.
"""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIGMA = 1.0 / np.sqrt(np.pi)


def _seconds(f):
    import torch
    f()
    t = []
    for _ in range(3):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        f()
        torch.cuda.synchronize()
        t.append(time.perf_counter() - t0)
    return min(t)


def test_crowded_average(lib):
    import torch
    N, L, n = 256, 70.0, 8190
    rng = np.random.default_rng(3)
    spread = torch.as_tensor(rng.uniform(0.0, L, size=(n, 3)), device="cuda")
    crowded = 0.3 * L + 1e-3 * spread
    F = lib.Fcm(N, L, SIGMA, 3.0, max_blobs=n)
    F.brownian(spread, 5, 0, 2, 1.0, 0.01)
    v = F.average(crowded)
    few = torch.cat([F.average(crowded[i:i + 1000]) for i in range(0, n, 1000)])
    assert torch.equal(v, few)
    t_spread, t_crowded = _seconds(lambda: F.average(spread)), _seconds(lambda: F.average(crowded))
    assert t_crowded < 10.0 * t_spread, (t_crowded, t_spread)
    b_spread, b_crowded = (_seconds(lambda: F.brownian(r, 5, 0, 2, 1.0, 0.01)) for r in (spread, crowded))
    assert b_crowded < 10.0 * b_spread, (b_crowded, b_spread)
