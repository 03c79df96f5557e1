"""GPU: the symmetric FP32 and double-float pair kernels with source ranges shorter than a tile (the
work lists of small and mid-size suspensions), at the edges of tiles and sweeps, against the
oracle.  Tolerances as in the parity tests of these products: 2e-6 and 1e-11 (relative 2-norm).
"""
import numpy as np
import pytest

from oracle import rpy

from gpu_common import rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("counts", [[1], [31], [33], [511], [512], [513], [545], [1030], [1537],
                                    [1, 16, 0, 17, 200, 511, 513, 1029], [60] * 40])
def test_products_at_range_edges(lib, counts):
    """Single-blob bodies, uniform in a cube: every pair, overlapping ones included."""
    rng = np.random.default_rng(counts[0] + len(counts))
    n = int(sum(counts))
    Y = rng.uniform(0.0, 2.0 + 2.6 * max(counts) ** (1.0 / 3.0), size=(n, 3))
    off = np.concatenate([[0], np.cumsum(counts)])
    ctx = lib.Context(lib.Params(), [np.zeros((1, 3))], np.zeros(n, dtype=np.int32), off, Y,
                      np.tile([1.0, 0.0, 0.0, 0.0], (n, 1)))
    lam = rng.standard_normal((n, 3))
    u32 = ctx.rpy_apply(lam, lib.FP32_MIXED).cpu().numpy().reshape(-1, 3)
    udf = ctx.rpy_apply(lam, 2).cpu().numpy().reshape(-1, 3)
    for s in range(len(counts)):
        a, b = off[s], off[s + 1]
        if b > a:
            ref = rpy.rpy_matrix(Y[a:b], 1.0, 1.0) @ lam[a:b].reshape(-1)
            assert rel(u32[a:b], ref) < 2e-6, (counts[s], rel(u32[a:b], ref))
            assert rel(udf[a:b], ref) < 1e-11, (counts[s], rel(udf[a:b], ref))
