"""GPU: GMRES cycles whose back substitution has the fewest columns a restart allows (2), a few, and
more than one lane row of 32 (the FP32-mixed cycle aims a decade below its tolerance).

Forces without torques (a torque along a rod's axis has no solution).  Each solve is judged by its
own residual through the FP64 saddle product: at most the solver's tolerance, plus the product's
rounding (1e-13), whatever the restart length."""
import numpy as np
import pytest

from synthetic import workloads as WL

from gpu_common import rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("restart,prec,tol", [(2, 0, 1e-10), (5, 0, 1e-10), (100, 0, 1e-10), (100, 1, 2e-13)])
def test_residual(lib, restart, prec, tol):
    wl = WL.mixed_small(90, seed=2)
    ctx = lib.context_from_workload(wl, precision=prec, gmres_tol=tol, gmres_restart=restart, gmres_max_iter=4000)
    rng = np.random.default_rng(restart)
    FT = np.zeros((ctx.n_bodies, 6))
    FT[:, :3] = rng.standard_normal((ctx.n_bodies, 3))
    FT = FT.reshape(-1)
    V, lam, info = ctx.mobility_solve(FT, None, want_lambda=True)
    assert info["converged"]
    x = np.concatenate([lam.cpu().numpy(), V.cpu().numpy()])
    y = ctx.saddle_apply(x, lib.FP64).cpu().numpy()
    assert rel(y, np.concatenate([np.zeros(3 * ctx.n_blobs), -FT])) < tol + 1e-13, info
