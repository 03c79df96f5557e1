"""GPU: the per-body products with several bodies of one template per block (FP32, from 512 bodies
on), with templates of 1 to 22 blobs whose body counts leave partly filled groups, against the
FP64 path of the library, which takes one body per block and forms the body rows separately.

Tolerances: those of the FP32 products (2e-6) and of the FP32 square root at tight stopping
(2e-5) in the parity tests; the solve is checked by its reported and recomputed residual.
"""
import numpy as np
import pytest

from synthetic import shapes, workloads as WL

from gpu_common import rel

pytestmark = pytest.mark.gpu

TEMPLATES = [np.zeros((1, 3)), shapes.dumbbell(2.0), shapes.rod(5, 2.0), shapes.icosahedron(),
             np.concatenate([shapes.rod(11, 2.0), shapes.rod(11, 2.0) + [2.5, 0.0, 0.0]])]


@pytest.mark.parametrize("n", [511, 515, 6083])
def test_grouped_body_products(lib, n):
    rng = np.random.default_rng(n)
    tmpl = rng.choice(len(TEMPLATES), size=n, p=[0.3, 0.3, 0.2, 0.15, 0.05]).astype(np.int32)
    side = int(np.ceil(n ** (1.0 / 3.0)))
    g = np.stack(np.meshgrid(*[np.arange(side)] * 3, indexing="ij"), -1).reshape(-1, 3)[:n]
    Y = 26.0 * g + rng.uniform(-0.5, 0.5, size=(n, 3))
    q = WL.random_unit_quaternions(rng, n)
    off = np.array([0, n // 3, n // 3, n])
    ctx = {}
    for prec in (0, 1):
        ctx[prec] = lib.Context(lib.Params(precision=prec, autotune=0, kT=1.0, dt=2.0, lanczos_tol=1e-7,
                                           lanczos_max_iter=100), TEMPLATES, tmpl, off, Y, q)
    x = rng.standard_normal(int(ctx[0].saddle_off[-1]))
    y0, y1 = (ctx[0].saddle_apply(x, p).cpu().numpy() for p in (0, 1))
    assert rel(y1, y0) < 2e-6, rel(y1, y0)
    for s in range(3):   # the body rows alone: FP64 sums on both sides
        lo, hi = int(ctx[0].saddle_off[s + 1]) - 6 * (off[s + 1] - off[s]), int(ctx[0].saddle_off[s + 1])
        if hi > lo:
            assert rel(y1[lo:hi], y0[lo:hi]) < 1e-12
    W = rng.standard_normal(3 * ctx[0].n_blobs)
    v0, v1 = (ctx[p].brownian_slip(W)[0].cpu().numpy() for p in (0, 1))
    assert rel(v1, v0) < 2e-5, rel(v1, v0)
    FT = np.zeros((n, 6))
    FT[:, :3] = rng.standard_normal((n, 3))
    V, lam, info = ctx[1].mobility_solve(FT.reshape(-1), W, want_lambda=True)
    V0 = ctx[0].mobility_solve(FT.reshape(-1), W)[0].cpu().numpy()
    assert info["converged"] and info["residual"] <= 1e-6
    assert rel(V.cpu().numpy(), V0) < 1e-5, rel(V.cpu().numpy(), V0)
