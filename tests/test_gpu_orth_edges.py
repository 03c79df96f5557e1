"""GPU: the fused orthogonalisation where its cluster doubles -- from 512 elements per block on for
few suspensions (512, 1,024, 2,048, 4,096 and 8,192 elements: 1, 2, 4, 8 and 16 blocks), from
4,096 on for many -- by two identities of the square root that Lanczos converges to.

Bodies are single blobs (3 elements each), so the root is M^(1/2).  Applied twice it is the FP64
product, and a batch equals its suspensions one by one, which take other clusters.  Roots stop at
a change of 1e-11; an error of a few times that is carried through a second root of condition
number below 1e2: 1e-8.
"""
import numpy as np
import pytest

from gpu_common import rel

pytestmark = pytest.mark.gpu


def _context(lib, counts, seed):
    rng = np.random.default_rng(seed)
    n = int(sum(counts))
    side = int(np.ceil(max(counts) ** (1.0 / 3.0)))
    g = np.stack(np.meshgrid(*[np.arange(side)] * 3, indexing="ij"), -1).reshape(-1, 3).astype(float)
    Y = np.concatenate([3.1 * g[:c] + rng.uniform(-0.5, 0.5, size=(c, 3)) for c in counts])
    return _of(lib, counts, Y), Y, rng.standard_normal((n, 3))


def _of(lib, counts, Y):
    n = len(Y)
    p = lib.Params(autotune=0, kT=1.0, dt=2.0, lanczos_tol=1e-11, lanczos_max_iter=100, gmres_restart=4)
    return lib.Context(p, [np.zeros((1, 3))], np.zeros(n, dtype=np.int32), np.concatenate([[0], np.cumsum(counts)]), Y,
                       np.tile([1.0, 0.0, 0.0, 0.0], (n, 1)))


@pytest.mark.parametrize("n", [170, 171, 341, 342, 682, 683, 1365, 1366, 2730, 2731])
def test_root_twice_is_the_product(lib, n):
    ctx, _, W = _context(lib, [n], n)
    v = ctx.brownian_slip(ctx.brownian_slip(W.reshape(-1))[0])[0].cpu().numpy()
    assert rel(v, ctx.rpy_apply(W, lib.FP64).cpu().numpy()) < 1e-8


def test_batch_with_parts_of_513_to_4096_elements(lib):
    """310 suspensions: two blocks each, of which the shorter suspensions fill one and a part."""
    counts = np.random.default_rng(2).integers(30, 900, size=310).tolist()
    counts[:6] = [1400, 171, 682, 683, 1365, 1366]
    ctx, Y, W = _context(lib, counts, 5)
    off = np.concatenate([[0], np.cumsum(counts)])
    v = ctx.brownian_slip(W.reshape(-1))[0].cpu().numpy().reshape(-1, 3)
    for s in (0, 1, 2, 3, 4, 5, 100, 309):
        a, b = off[s], off[s + 1]
        one = _of(lib, [counts[s]], Y[a:b]).brownian_slip(W[a:b].reshape(-1))[0].cpu().numpy()
        assert rel(v[a:b], one) < 1e-8, (s, rel(v[a:b], one))
