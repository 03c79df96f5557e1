"""GPU: one Krylov iteration's orthogonalisation in one launch, where its split changes -- 1, 2, 4
and 8 blocks per suspension (1,024 elements each), uneven and empty suspensions, and both
sides of the length at which the separate kernels take over (32,768 elements).

Bodies are single blobs, so the block factor of M is a multiple of I and the square root that
Lanczos converges to is M^(1/2).  Converged roots agree to 1e-9 (stopping change 1e-11 times the
Krylov bound of a few, FP64 rounding far below); solves are checked by their own residual.
"""
import numpy as np
import pytest

from oracle import rigid, rpy

from gpu_common import rel

pytestmark = pytest.mark.gpu


def _free(lib, counts, seed, **kw):
    rng = np.random.default_rng(seed)
    n = int(sum(counts))
    side = int(np.ceil(max(counts) ** (1.0 / 3.0)))
    g = np.stack(np.meshgrid(*[np.arange(side)] * 3, indexing="ij"), -1).reshape(-1, 3).astype(float)
    Y = np.concatenate([3.1 * g[:c] + rng.uniform(-0.5, 0.5, size=(c, 3)) for c in counts if c])
    q = np.tile([1.0, 0.0, 0.0, 0.0], (n, 1))
    off = np.concatenate([[0], np.cumsum(counts)])
    p = dict(autotune=0, kT=1.0, dt=2.0, lanczos_max_iter=100)
    p.update(kw)
    return lib.Context(lib.Params(**p), [np.zeros((1, 3))], np.zeros(n, dtype=np.int32), off, Y, q), Y, off, rng


@pytest.mark.parametrize("counts", [[1], [2], [40], [341], [342], [683], [1366], [300, 0, 7, 1, 700, 64]])
def test_root_at_cluster_edges(lib, counts):
    ctx, Y, off, rng = _free(lib, counts, counts[0], lanczos_tol=1e-11)
    W = rng.standard_normal((len(Y), 3))
    vb = ctx.brownian_slip(W)[0].cpu().numpy().reshape(-1, 3)
    for s in range(len(counts)):
        a, b = off[s], off[s + 1]
        if b > a:
            ref = rigid.sqrtm_sym(rpy.rpy_matrix(Y[a:b], 1.0, 1.0)) @ W[a:b].reshape(-1)
            assert rel(vb[a:b], ref) < 1e-9, (counts[s], rel(vb[a:b], ref))


@pytest.mark.parametrize("n", [3640, 3641])
def test_solve_on_both_sides_of_the_fused_length(lib, n):
    """9 saddle entries per single-blob body: 32,760 and 32,769."""
    ctx, Y, off, rng = _free(lib, [n], n, gmres_tol=1e-9, gmres_restart=20)
    FT = np.zeros((n, 6))
    FT[:, :3] = rng.standard_normal((n, 3))
    V, lam, info = ctx.mobility_solve(FT.reshape(-1), None, want_lambda=True)
    assert info["converged"] and info["residual"] <= 1e-9
    x = np.concatenate([lam.cpu().numpy(), V.cpu().numpy()])
    y = ctx.saddle_apply(x, lib.FP64).cpu().numpy()
    b = np.concatenate([np.zeros(3 * n), -FT.reshape(-1)])
    assert rel(y, b) < 2e-9, rel(y, b)
