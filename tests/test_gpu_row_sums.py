"""GPU: accuracy of the same-body block of the FP32 products, whose row sums run in FP32.

Every suspension holds one body, so an FP32 product is the body's own block: the template's
matrix in FP32, a row in four FP32 chains or more joined in FP64, plus what is left of the pair
kernel's terms for those blobs (chains of 32 sources) after the same terms are taken out again.
Both are emulated here operation by operation, and the product's error against FP64 may exceed
the emulated one by a tenth: the terms' order within a chain and the reciprocal root's last bit
differ, which moves a root mean square over 1e3 to 1e5 rows by a few percent.  Two chains a row
give 1.19 (43 blobs) to 1.35 (340 blobs) times the emulated error.

Template sizes: rows split over two threads (42 blobs) and not (43 and more), one body per block
(few bodies, or templates above 85 blobs) and four (from 512 bodies on, the last group partly
filled).
"""
import numpy as np
import pytest

from oracle import rpy

from gpu_common import rel

pytestmark = pytest.mark.gpu

F = np.float32


def _shell(n):
    """n blobs on a golden spiral over a sphere, closest spacing 2a."""
    i = np.arange(n) + 0.5
    z, t = 1.0 - 2.0 * i / n, np.pi * (1.0 + 5.0 ** 0.5) * i
    s = np.sqrt(1.0 - z * z)
    p = np.stack([s * np.cos(t), s * np.sin(t), z], 1)
    d = np.linalg.norm(p[:, None] - p[None], axis=-1) + 9.0 * np.eye(n)
    p = p * 2.0 / d.min()
    return p - p.mean(axis=0)


def _fma(a, b, c):
    return (a.astype(np.float64) * b + c).astype(F)


def _row_error(M, lam, chains):
    """Error of M lam (units 1/(8 pi eta)) as FP32 chains joined in FP64; lam (3n, bodies)."""
    M32, l32 = M.astype(F), lam.astype(F)
    acc = [np.zeros(lam.shape, F) for _ in range(chains)]
    for k in range(len(M)):
        acc[k % chains] = _fma(M32[:, k:k + 1], l32[k][None], acc[k % chains])
    return sum(a.astype(np.float64) for a in acc) - M @ lam


def _pair_error(p, lam):
    """Rounding of the pair kernel's 32-source chains against the same terms added exactly."""
    x, l, n = p.astype(F), lam.astype(F), len(p)
    q, total, terms = np.zeros(lam.shape, F), np.zeros(lam.shape), np.zeros(lam.shape)
    for j in range(n):
        d = x[j] - x
        r2 = _fma(d[:, 0], d[:, 0], _fma(d[:, 1], d[:, 1], d[:, 2] * d[:, 2]))
        ri = (1.0 / np.sqrt(np.maximum(r2, F(4)).astype(np.float64))).astype(F)
        ri2 = ri * ri
        ri3 = ri2 * ri
        A = _fma(np.full(n, F(2.0 / 3.0)), ri3, ri)[:, None]
        B = (ri3 * _fma(np.full(n, F(-2)), ri2, np.ones(n, F)))[:, None]
        s = B * _fma(d[:, 0:1], l[j, 0][None], _fma(d[:, 1:2], l[j, 1][None], d[:, 2:3] * l[j, 2][None]))
        for c in range(3):
            lc, dc = np.broadcast_to(l[j, c], s.shape), np.broadcast_to(d[:, c:c + 1], s.shape)
            terms[:, c] += _fma(np.broadcast_to(A, s.shape), lc, s * dc)
            q[:, c] = _fma(np.broadcast_to(A, s.shape), lc, _fma(s, dc, q[:, c]))
        if j % 32 == 31 or j == n - 1:
            total += q
            q[:] = 0
    return total - terms


@pytest.mark.parametrize("n,bodies", [(42, 513), (43, 513), (85, 514), (162, 24), (340, 12)])
def test_same_body_row_sums(lib, n, bodies):
    rng = np.random.default_rng(n)
    p = _shell(n)
    Y = np.zeros((bodies, 3))
    q = np.tile([1.0, 0.0, 0.0, 0.0], (bodies, 1))
    ctx = lib.Context(lib.Params(autotune=0, precision=lib.FP32_MIXED, gmres_restart=4, lanczos_max_iter=4), [p],
                      np.zeros(bodies, dtype=np.int32), np.arange(bodies + 1), Y, q)
    lam = rng.standard_normal((bodies, n, 3))
    M = rpy.rpy_matrix(p, 1.0, 1.0)
    ref = np.einsum("ij,bj->bi", M, lam.reshape(bodies, -1))
    u64 = ctx.rpy_apply(lam, lib.FP64).cpu().numpy().reshape(bodies, -1)
    assert rel(u64, ref) < 1e-13
    err = rel(ctx.rpy_apply(lam, lib.FP32_MIXED).cpu().numpy(), u64)
    cols = lam.reshape(bodies, 3 * n).T
    scaled = 8.0 * np.pi * M
    pair = _pair_error(p, np.moveaxis(lam, 0, -1)).reshape(3 * n, bodies)
    expected = np.linalg.norm(_row_error(scaled, cols, 4) + pair) / np.linalg.norm(scaled @ cols)
    assert err < 1.1 * expected, (err, expected)
