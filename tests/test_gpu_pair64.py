"""GPU: the symmetric FP64 pair kernel where its work split can go wrong -- tile and sweep edges,
uneven and empty suspensions, overlapping pairs -- against the oracle.

Tolerance: a pair term carries fewer than 12 roundings (about 12 x 1.1e-16) and the sums are
short chains joined in FP64, so products agree with the dense oracle to below 1e-14 in the
relative 2-norm.
"""
import numpy as np
import pytest

from oracle import rpy

from gpu_common import rel

pytestmark = pytest.mark.gpu


def _free_blobs(lib, counts, seed, box):
    """A context of single-blob bodies: counts[s] blobs in suspension s, uniform in a cube."""
    rng = np.random.default_rng(seed)
    n = int(sum(counts))
    Y = rng.uniform(0.0, box, size=(n, 3))
    q = np.tile([1.0, 0.0, 0.0, 0.0], (n, 1))
    off = np.concatenate([[0], np.cumsum(counts)])
    ctx = lib.Context(lib.Params(autotune=0), [np.zeros((1, 3))], np.zeros(n, dtype=np.int32), off, Y, q)
    return ctx, Y, off, rng.standard_normal((n, 3))


@pytest.mark.parametrize("counts", [[1], [5], [33], [128], [129], [257], [640], [1000],
                                    [1, 2, 0, 7, 31, 127, 128, 129, 300], [15] * 36])
def test_fp64_product_at_tile_edges(lib, counts):
    ctx, Y, off, lam = _free_blobs(lib, counts, len(counts) + counts[0], 2.0 + 3.0 * max(counts) ** (1.0 / 3.0))
    u = ctx.rpy_apply(lam, lib.FP64).cpu().numpy().reshape(-1, 3)
    for s in range(len(counts)):
        a, b = off[s], off[s + 1]
        if b > a:
            ref = rpy.rpy_matrix(Y[a:b], 1.0, 1.0) @ lam[a:b].reshape(-1)
            assert rel(u[a:b], ref) < 1e-14, (counts[s], rel(u[a:b], ref))


def test_fp64_product_over_distances(lib):
    """Pairs from far overlap to a million radii, and across r = 2a: every suspension is one pair."""
    d = np.concatenate([np.logspace(-6, 6, 97), 2.0 + np.array([-1, 1]) * 1e-9, [2.0, np.nextafter(2.0, 0.0)]])
    n = len(d)
    Y = np.zeros((2 * n, 3))
    Y[1::2] = d[:, None] * np.array([0.6, 0.0, 0.8])
    lam = np.random.default_rng(4).standard_normal((2 * n, 3))
    ctx = lib.Context(lib.Params(autotune=0), [np.zeros((1, 3))], np.zeros(2 * n, dtype=np.int32),
                      np.arange(0, 2 * n + 1, 2), Y, np.tile([1.0, 0, 0, 0], (2 * n, 1)))
    u = ctx.rpy_apply(lam, lib.FP64).cpu().numpy().reshape(-1, 3)
    for k in range(n):
        ref = rpy.rpy_matrix(Y[2 * k:2 * k + 2], 1.0, 1.0) @ lam[2 * k:2 * k + 2].reshape(-1)
        assert rel(u[2 * k:2 * k + 2], ref) < 1e-14, (d[k], rel(u[2 * k:2 * k + 2], ref))
