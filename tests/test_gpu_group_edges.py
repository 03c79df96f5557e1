"""GPU: the FP32 per-body products with groups of four and eight bodies of the largest templates that
are grouped (43 to 85 blobs: one thread per row), every suspension one body, the last groups
partly filled, against the FP64 path.

Tolerances: 2e-6, that of the FP32 products in the parity tests; the solve by its reported
residual, and 1e-5 for its velocities.
"""
import numpy as np
import pytest

from synthetic import workloads as WL

from gpu_common import rel
from test_gpu_row_sums import _shell

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [515, 6083])
def test_large_templates_in_groups(lib, n):
    rng = np.random.default_rng(n)
    T = [_shell(43), _shell(85), np.zeros((1, 3))]
    tmpl = rng.choice(3, size=n, p=[0.5, 0.3, 0.2]).astype(np.int32)
    Y, q = rng.uniform(-5.0, 5.0, size=(n, 3)), WL.random_unit_quaternions(rng, n)
    ctx = [lib.Context(lib.Params(precision=p, autotune=0, gmres_restart=10, lanczos_max_iter=8), T, tmpl,
                       np.arange(n + 1), Y, q) for p in (0, 1)]
    x = rng.standard_normal(int(ctx[0].saddle_off[-1]))
    y0, y1 = (ctx[0].saddle_apply(x, p).cpu().numpy() for p in (0, 1))
    assert rel(y1, y0) < 2e-6, rel(y1, y0)
    FT = rng.standard_normal(6 * n)
    FT[np.repeat(tmpl == 2, 6) & np.tile([False] * 3 + [True] * 3, n)] = 0.0   # a single blob takes no torque
    V, _, info = ctx[1].mobility_solve(FT)
    assert info["converged"] and info["residual"] <= 1e-6
    V0 = ctx[0].mobility_solve(FT)[0].cpu().numpy()
    assert rel(V.cpu().numpy(), V0) < 1e-5, rel(V.cpu().numpy(), V0)
