"""GPU: the symmetric FP64 pair kernel with four targets per lane (a suspension above 16,384 blobs),
beside smaller suspensions in the same tiles of 512, at sampled blobs against the oracle's pairs.

Tolerance: as for the one-target form, below 1e-14 in the relative 2-norm over the sampled rows.
"""
import numpy as np
import pytest

from gpu_common import rel

pytestmark = pytest.mark.gpu


def _rows(Y, lam, rows):
    """Rows of M lam (a = eta = 1): unbounded RPY with the overlapping form below r = 2."""
    out = []
    for i in rows:
        d = Y[i] - Y
        r = np.linalg.norm(d, axis=1)
        s = np.where(r > 0.0, r, 1.0)
        dl = np.einsum("ij,ij->i", d, lam) / (s * s)
        far = r >= 2.0
        A = np.where(far, (1.0 + 2.0 / (3.0 * s * s)) / (8.0 * np.pi * s), (1.0 - 9.0 * r / 32.0) / (6.0 * np.pi))
        B = np.where(far, (1.0 - 2.0 / (s * s)) / (8.0 * np.pi * s), 3.0 * r / 32.0 / (6.0 * np.pi))
        out.append((A[:, None] * lam + (B * dl)[:, None] * d).sum(axis=0))
    return np.array(out)


@pytest.mark.parametrize("counts", [[16385], [16896], [17000, 1, 513, 40]])
def test_four_targets_per_lane(lib, counts):
    rng = np.random.default_rng(counts[0])
    n = sum(counts)
    Y = rng.uniform(0.0, 70.0, size=(n, 3))
    lam = rng.standard_normal((n, 3))
    off = np.concatenate([[0], np.cumsum(counts)])
    ctx = lib.Context(lib.Params(autotune=0, gmres_restart=4, lanczos_max_iter=4), [np.zeros((1, 3))],
                      np.zeros(n, dtype=np.int32), off, Y, np.tile([1.0, 0.0, 0.0, 0.0], (n, 1)))
    u = ctx.rpy_apply(lam, lib.FP64).cpu().numpy().reshape(-1, 3)
    for s, c in enumerate(counts):
        a, b = off[s], off[s + 1]
        rows = np.unique(np.clip(np.concatenate([[0, 1, 127, 128, 511, 512, 513, c - 2, c - 1],
                                                 rng.integers(0, c, 40)]), 0, c - 1))
        assert rel(u[a:b][rows], _rows(Y[a:b], lam[a:b], rows)) < 1e-14, (c, rel(u[a:b][rows], _rows(Y[a:b], lam[a:b], rows)))
