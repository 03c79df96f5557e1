"""GPU: the FP32 pair kernel's work list for batches of suspensions: with work enough to fill the
chip many times over, ranges grow to whole tiles and beyond (32-source items made such products
up to 18% slower), whatever the size of a suspension; tiny suspensions in great number are not
such work, and a larger one beside them keeps short ranges.  Products agree with the FP64 path.

Tolerance: that of the FP32 products in the parity tests, 2e-6.
"""
import numpy as np
import pytest

from synthetic import shapes, workloads as WL

from gpu_common import rel

pytestmark = pytest.mark.gpu


def _context(lib, off, Y, rng):
    n = len(Y)
    return lib.Context(lib.Params(precision=lib.FP32_MIXED, autotune=0, gmres_restart=4, lanczos_max_iter=4),
                       [shapes.icosahedron()], np.zeros(n, dtype=np.int32), off, Y, WL.random_unit_quaternions(rng, n))


# bodies of 12 blobs per suspension, suspensions, source tiles per item by the rule on 152 SMs
@pytest.mark.parametrize("bodies,susp,tiles", [(225, 310, 2), (750, 24, 1), (125, 310, 1), (42, 100, 1)])
def test_batches_take_long_ranges(lib, bodies, susp, tiles):
    rng = np.random.default_rng(bodies)
    n = bodies * susp
    side = int(np.ceil(bodies ** (1.0 / 3.0)))
    g = np.stack(np.meshgrid(*[np.arange(side)] * 3, indexing="ij"), -1).reshape(-1, 3)[:bodies]
    Y = np.tile(6.4 * g, (susp, 1)) + rng.uniform(-0.2, 0.2, size=(n, 3))
    ctx = _context(lib, bodies * np.arange(susp + 1), Y, rng)
    assert ctx.profile_read()["sym_width"] >= tiles
    lam = rng.standard_normal(3 * ctx.n_blobs)
    u = ctx.rpy_apply(lam, lib.FP32_MIXED).cpu().numpy()
    assert rel(u, ctx.rpy_apply(lam, lib.FP64).cpu().numpy()) < 2e-6


def test_tiny_suspensions_do_not_lengthen_ranges(lib):
    rng = np.random.default_rng(5)
    counts = [170] + [1] * 4000
    g = np.stack(np.meshgrid(*[np.arange(6)] * 3, indexing="ij"), -1).reshape(-1, 3)
    Y = np.concatenate([6.4 * g[:170], np.zeros((4000, 3))]) + rng.uniform(-0.2, 0.2, size=(4170, 3))
    ctx = _context(lib, np.concatenate([[0], np.cumsum(counts)]), Y, rng)
    assert ctx.profile_read()["sym_width"] == 1
    lam = rng.standard_normal(3 * ctx.n_blobs)
    u = ctx.rpy_apply(lam, lib.FP32_MIXED).cpu().numpy()
    assert rel(u, ctx.rpy_apply(lam, lib.FP64).cpu().numpy()) < 2e-6
