"""The workspace that gdc_workspace_bytes asks for, over the sizes in use (no GPU calls).

The partial sums of the pair kernels live in one array for all of them, since an epilogue takes a
kernel's sums before the next kernel starts.  Limits in MiB: the sizes that this gives (restart
50, 128 Lanczos vectors, autotuner on), rounded up by 3%; an array per kernel asks for 1.2 to
1.8 times as much.
"""
import ctypes
import os

import numpy as np
import pytest

C4 = np.random.default_rng(0).integers(8, 129, 512).tolist()


@pytest.fixture(scope="module")
def lib():
    from paper_2106_00449_gb300 import build
    if not os.path.exists(build.LIB):
        build.build()
    import paper_2106_00449_gb300 as g
    return g


@pytest.mark.parametrize("templates,bodies,mib", [
    ([12], [4], 0.5), ([10], [256], 28), ([42, 15, 21], [351], 219), ([42, 15, 21], [777], 317),
    ([42, 15, 21], [2520], 595), ([20], [8192], 2227), ([12, 10, 42], C4[:64], 777), ([12, 10, 42], C4, 4548)])
def test_workspace_bytes(lib, templates, bodies, mib):
    n = np.array(templates, dtype=np.int32)
    off = np.concatenate([[0], np.cumsum(bodies)]).astype(np.int64)
    bt = (np.arange(off[-1]) % len(n)).astype(np.int32)
    p = lib.Params(lanczos_max_iter=128)._c()
    need = lib.load_library().gdc_workspace_bytes(ctypes.byref(p), len(n), lib._np_ptr(n), len(bodies),
                                                  lib._np_ptr(off), lib._np_ptr(bt))
    assert 0 < need <= mib * 2 ** 20, need / 2 ** 20
