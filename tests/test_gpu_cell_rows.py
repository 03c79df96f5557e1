"""GPU: cell-list rows against the all-pairs tiles, where a row of cells can go wrong.

The three x-neighbours of a blob's cell are adjacent hash buckets, read as one range; a row
whose buckets wrap past the last one is read cell by cell.  Bodies scattered far apart in
close pairs put their cells at arbitrary keys: of the about 250 occupied cells' nine rows each,
2 in 1,024 wrap, so four seeds hold about 18 such rows.  Body counts 1, 256, 257 and 2,047-2,049 are the edges
of the reference point's sum (one block or eight, four bodies per thread)."""
import dataclasses

import numpy as np
import pytest

from synthetic import workloads as WL

pytestmark = pytest.mark.gpu


def _scattered(n, seed, extent):
    wl = WL.mixed_small(n, seed=seed)
    rng = np.random.default_rng(100 + seed)
    Y = rng.uniform(-extent, extent, wl.Y.shape)
    m = len(Y) // 2
    d = rng.standard_normal((m, 3))
    Y[m:2 * m] = Y[:m] + 2.2 * d / np.linalg.norm(d, axis=1, keepdims=True)
    return dataclasses.replace(wl, Y=Y)


def _both(lib, wl, prec):
    return [lib.context_from_workload(wl, precision=prec, force_method=m).forces().cpu().numpy() for m in (1, 2)]


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("seed", range(4))
def test_scattered_pairs(lib, prec, seed):
    # a blob sums at most some 100 terms, a body 15 blobs; the all-pairs sum differs in order only:
    # 1,500 roundings of terms no larger than 100 times the largest result
    a, b = _both(lib, _scattered(32, seed, 60.0 * 2 ** seed), prec)
    unit = 2.0 ** -53 if prec == 0 else 2.0 ** -24
    assert np.abs(a).max() > 0
    assert np.abs(a - b).max() <= 1500 * unit * 100 * np.abs(a).max()


@pytest.mark.parametrize("n", [1, 256, 257, 2047, 2048, 2049])
def test_reference_point_edges(lib, n):
    wl = _scattered(n, 7, 400.0)
    a, b = _both(lib, wl, 0)
    assert np.abs(a - b).max() <= 1500 * 2.0 ** -53 * 100 * max(np.abs(a).max(), 1.0)
    # the same bodies far from the origin: positions are taken relative to the mean centre, which
    # a wrong mean would leave far away and FP32 coordinates without digits
    far = dataclasses.replace(wl, Y=wl.Y + 2.0 ** 20)
    c = lib.context_from_workload(far, precision=1, force_method=2).forces().cpu().numpy()
    d = lib.context_from_workload(wl, precision=1, force_method=2).forces().cpu().numpy()
    # coordinates within 1,024 of the mean: FP32 spacing 2^-13 at most, of a force whose range
    # is a tenth of the radius; a lost mean would give spacings of 2^-3
    assert np.abs(c - d).max() <= 2.0 ** -13 * 2 * 2 * 100 * max(np.abs(d).max(), 1.0)
