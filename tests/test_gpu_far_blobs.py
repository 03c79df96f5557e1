"""GPU: FP64 products of blobs so far apart that the square of their distance overflows.

Such a pair's mobility (about 1/r) is below 1e-150 of a blob's own, so the product is each blob's
self-mobility times its lambda, to FP64 rounding (1e-13, the tolerance of the FP64 products).
Blobs lie on a line at multiples of 2e157 (the reference point, their mean, keeps them apart);
128 blobs share a tile of the pair kernel, further ones lie in later tiles.
"""
import numpy as np
import pytest

from oracle import rpy, wall

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("walled", [0, 1])
@pytest.mark.parametrize("n", [2, 128, 300])
def test_fp64_product_of_blobs_out_of_range(lib, n, walled):
    rng = np.random.default_rng(n)
    Y = np.zeros((n, 3))
    Y[:, 0] = 2e157 * np.arange(n)
    Y[:, 2] = 3.0
    lam = rng.standard_normal((n, 3))
    ctx = lib.Context(lib.Params(autotune=0, wall=walled), [np.zeros((1, 3))], np.zeros(n, dtype=np.int32), [0, n], Y,
                      np.tile([1.0, 0.0, 0.0, 0.0], (n, 1)))
    u = ctx.rpy_apply(lam, lib.FP64).cpu().numpy().reshape(n, 3)
    one = np.array([[0.0, 0.0, 3.0]])
    M = wall.wall_matrix(one, 1.0, 1.0) if walled else rpy.rpy_matrix(one, 1.0, 1.0)
    assert np.abs(u - lam @ M.T).max() <= 1e-13 * np.abs(lam @ M.T).max()
