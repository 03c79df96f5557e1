"""GPU: the allocation-free product where its preparation's split changes -- fewer blobs than the
cluster has blocks, parts one past a block's 1,024 threads, the last sizes below the largest -- on
clouds far from the origin, whose centroid has to be right for FP32 coordinates to keep digits.

Bound: 2e-6 of the FP64 product, the FP32 product's own (sums of 1e-7 terms); coordinates within 64
of the centroid round to 4e-6 of a radius, and shift a term by less than that."""
import numpy as np
import pytest

from test_zz_no_alloc import _free_blob_context

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 7, 8, 9, 8191, 8192, 8193, 16383])
def test_sizes(lib, n):
    import torch
    rng = np.random.default_rng(n)
    r = rng.uniform(0.0, 2.5 * n ** (1.0 / 3.0), size=(n, 3)) + np.array([1e5, -3e4, 2e5])
    lam = rng.standard_normal(3 * n)
    ref = _free_blob_context(lib, r).rpy_apply(lam, lib.FP64)
    u = lib.rpy_apply_noalloc(torch.as_tensor(r.reshape(-1), device="cuda"), torch.as_tensor(lam, device="cuda"))
    assert ((u - ref).norm() / ref.norm()).item() < 2e-6
