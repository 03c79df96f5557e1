"""GPU: reference points of many suspensions of which one is larger: eight blocks for every
suspension, which one suspension of more than 256 bodies used to bring, cost more than the sums.

Loading a configuration with one suspension of 300 bodies beside 2,000 single ones is the work of
one of 250 and 2,050 to 2%; the times may differ by half (eight blocks each: 2.8 times).
"""
import time

import numpy as np
import pytest

from synthetic import shapes

pytestmark = pytest.mark.gpu


def _load_time(lib, first, rest):
    import torch
    n = first + rest
    rng = np.random.default_rng(1)
    Y = rng.uniform(0.0, 1e3, size=(n, 3))
    off = np.concatenate([[0], first + np.arange(rest + 1)])
    ctx = lib.Context(lib.Params(autotune=0, gmres_restart=4, lanczos_max_iter=4), [shapes.icosahedron()],
                      np.zeros(n, dtype=np.int32), off, Y, np.tile([1.0, 0.0, 0.0, 0.0], (n, 1)))
    r = ctx.blob_positions().cpu().numpy().reshape(n, 12, 3)
    assert np.abs(r.mean(axis=1) - Y).max() < 1e-9
    t = []
    for _ in range(20):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        ctx.blob_positions()
        t.append(time.perf_counter() - t0)
    return min(t)


def test_one_larger_suspension_among_many(lib):
    small, large = _load_time(lib, 250, 2050), _load_time(lib, 300, 2000)
    assert large < 1.5 * small, (large, small)
