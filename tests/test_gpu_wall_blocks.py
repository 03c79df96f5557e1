"""GPU: the per-body blocks above a wall (factor, inverse, 6 x 6 solve) at the sizes where their
set-up changes -- one blob, a collinear body (pseudo-inverse), 128- and 256-thread blocks (64
rows), and bodies whose triangle no longer fits shared memory (56 blobs) -- against the oracle.

Tolerances as for the boomerangs of test_gpu_wall.py: 1e-10 for the block solve and 1e-9 for the
converged square root, which carry the condition number of a body's block (below 1e4 at blob
spacing 2a) times FP64 rounding.
"""
import numpy as np
import pytest

from oracle import geometry as G, rigid, wall
from synthetic import shapes, workloads as WL

from gpu_common import rel

pytestmark = pytest.mark.gpu


def _cluster(n):
    """n blobs of a cubic lattice of spacing 2a, nearest the origin first."""
    g = np.stack(np.meshgrid(*[np.arange(-3, 4)] * 3, indexing="ij"), -1).reshape(-1, 3)
    order = np.lexsort((g[:, 2], g[:, 1], g[:, 0], (g * g).sum(1)))
    return 2.0 * g[order[:n]].astype(float)


TEMPLATES = {"single": np.zeros((1, 3)), "rod": shapes.rod(9, 2.0), "c21": _cluster(21), "c22": _cluster(22),
             "c55": _cluster(55), "c56": _cluster(56)}


@pytest.mark.parametrize("name", list(TEMPLATES))
def test_wall_block_sizes(lib, name):
    T = TEMPLATES[name]
    rng = np.random.default_rng(len(T))
    reach = np.linalg.norm(T - T.mean(axis=0), axis=1).max()
    Y = np.array([[0.0, 0.0, reach + 2.0], [40.0, 1.0, reach + 2.7], [-3.0, 45.0, reach + 1.6]])
    q = WL.random_unit_quaternions(rng, 3)
    off = np.array([0, 2, 3])
    ctx = lib.Context(lib.Params(wall=1, autotune=0, kT=1.0, dt=0.02, lanczos_tol=1e-11, lanczos_max_iter=128), [T],
                      np.zeros(3, dtype=np.int32), off, Y, q)
    rvec = rng.standard_normal(int(ctx.saddle_off[-1]))
    z = ctx.precond_apply(rvec).cpu().numpy()
    W = rng.standard_normal((3 * len(T), 3))
    vb = ctx.brownian_slip(W.reshape(-1))[0].cpu().numpy()
    n = len(T)
    for s in range(2):
        a, b = off[s], off[s + 1]
        lay = G.Layout([T], np.zeros(b - a, dtype=np.int32))
        r = G.blob_positions(lay, Y[a:b], q[a:b])
        M, K = wall.wall_matrix(r, 1.0, 1.0), rigid.k_matrix(r, Y[a:b], lay.blob_body)
        o, nl = int(ctx.saddle_off[s]), 3 * n * (b - a)
        for p in range(b - a):
            rows, cols = slice(3 * n * p, 3 * n * (p + 1)), slice(6 * p, 6 * p + 6)
            Kp = K[rows, cols]
            lp, vp = rigid.saddle_solve(M[rows, rows], Kp, rigid.rigid_basis(Kp, 1), -rvec[o:o + nl][rows],
                                        -rvec[o + nl:][cols])
            assert rel(z[o:o + nl][rows], lp) < 1e-10, rel(z[o:o + nl][rows], lp)
            assert rel(z[o + nl:][cols], vp) < 1e-10, rel(z[o + nl:][cols], vp)
        ref = np.sqrt(2.0 / 0.02) * rigid.sqrtm_block(M, rigid.block_factor_lab(lay, M)) @ W[n * a:n * b].reshape(-1)
        assert rel(vb[3 * n * a:3 * n * b], ref) < 1e-9, rel(vb[3 * n * a:3 * n * b], ref)
