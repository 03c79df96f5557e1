"""GPU: FCM spreading and averaging where their kernels change -- cells of fewer than 8 points per
side and of two layer chunks, more staged blobs than one round takes, and grids on which
averaging takes the blobs in cell order -- against the oracle (2e-5, the FP32 grid's tolerance
in test_gpu_fcm.py) and, for the order, bit for bit against another order of the same blobs.
"""
import numpy as np
import pytest

from oracle import fcm

from gpu_common import rel

pytestmark = pytest.mark.gpu

SIGMA = 1.0 / np.sqrt(np.pi)


# cells per side, points per cell side: (6, 6), (4, 8), (4, 16), (18, 8)
@pytest.mark.parametrize("N,L,R_t,n", [(32, 20.0, 3.0, 500), (32, 16.0, 3.9, 1500), (64, 20.0, 4.6, 900),
                                       (128, 40.0, 2.2, 700)])
def test_spread_cell_shapes(lib, N, L, R_t, n):
    rng = np.random.default_rng(N + n)
    r = rng.uniform(-L, 2.0 * L, size=(n, 3))
    lam = rng.standard_normal((n, 3))
    u = lib.Fcm(N, L, SIGMA, R_t, max_blobs=n).apply(r, lam).cpu().numpy()
    ref = fcm.mobility_apply(fcm.Grid(N, L, SIGMA, R_t), r, lam)
    assert rel(u, ref) < 2e-5, rel(u, ref)


def test_average_in_cell_order(lib):
    N, L, n = 256, 70.0, 1200
    rng = np.random.default_rng(7)
    r = rng.uniform(0.0, L, size=(n, 3))
    F = lib.Fcm(N, L, SIGMA, 3.0, max_blobs=n)
    v = F.brownian(r, 5, 0, 2, 1.0, 0.01).cpu().numpy()
    np.testing.assert_array_equal(F.average(r).cpu().numpy(), v)
    perm = rng.permutation(n)
    np.testing.assert_array_equal(F.average(r[perm]).cpu().numpy(), v[perm])
    np.testing.assert_array_equal(F.average(r[:100]).cpu().numpy(), v[:100])   # few blobs: index order
