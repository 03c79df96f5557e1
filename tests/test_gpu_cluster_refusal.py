"""GPU: cluster launches that the device refuses, by a fake of the CUDA runtime calls.

A small library, preloaded into a child process, stands in front of the runtime: it refuses
clusters above a given size in the attribute call, in the occupancy query and at the launch, or
at the launch alone.  No kernel is made to fail; a refused one is not launched.
"""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

FAKE = r"""
#include <dlfcn.h>
#include <stdlib.h>
#include <cuda_runtime_api.h>

static int largest = 16, asked = 1;   /* largest cluster granted; asked: by the queries too */

void fake_limit(int clusters, int queries) { largest = clusters; asked = queries; }

static void* real(const char* name) {
    static void* lib;
    if (!lib) lib = dlopen(getenv("FAKE_CUDART"), RTLD_LAZY | RTLD_NOLOAD);
    if (!lib) abort();
    return dlsym(lib, name);
}

static int width(const cudaLaunchConfig_t* cfg) {
    for (unsigned i = 0; i < cfg->numAttrs; ++i)
        if (cfg->attrs[i].id == cudaLaunchAttributeClusterDimension) return (int)cfg->attrs[i].val.clusterDim.x;
    return 1;
}

cudaError_t cudaFuncSetAttribute(const void* f, enum cudaFuncAttribute a, int v) {
    if (a == cudaFuncAttributeNonPortableClusterSizeAllowed && asked && largest <= 8) return cudaErrorNotSupported;
    return ((cudaError_t (*)(const void*, enum cudaFuncAttribute, int))real("cudaFuncSetAttribute"))(f, a, v);
}

cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void* f, const cudaLaunchConfig_t* cfg) {
    if (asked && width(cfg) > largest) {
        *n = 0;
        return cudaSuccess;
    }
    return ((cudaError_t (*)(int*, const void*, const cudaLaunchConfig_t*))real("cudaOccupancyMaxActiveClusters"))(
        n, f, cfg);
}

cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* cfg, const void* f, void** args) {
    if (width(cfg) > largest) return cudaErrorInvalidClusterSize;
    return ((cudaError_t (*)(const cudaLaunchConfig_t*, const void*, void**))real("cudaLaunchKernelExC"))(cfg, f, args);
}
"""

# 144 rods of 10 blobs: 5,184 saddle and 4,320 blob entries, which clusters of 16 blocks take
SETUP = """
import ctypes, os, sys
import numpy as np, torch
import paper_2106_00449_gb300 as g
from synthetic import workloads as WL
wl = WL.c2(n_rods=144, box=52.0)
def context(**kw):
    return g.context_from_workload(wl, precision=g.FP64, autotune=0, gmres_tol=1e-9, lanczos_tol=1e-9,
                                   lanczos_max_iter=100, **kw)
rng = np.random.default_rng(3)
FT = np.zeros((wl.n_bodies, 6)); FT[:, :3] = rng.standard_normal((wl.n_bodies, 3))
W = rng.standard_normal(3 * wl.n_blobs)
def results(c):
    return np.concatenate([c.mobility_solve(FT.reshape(-1))[0].cpu().numpy(), c.brownian_slip(W)[0].cpu().numpy()])
"""


@pytest.fixture(scope="module")
def child(lib, tmp_path_factory):
    """Runs code after SETUP in a child process with the fake in front of the runtime."""
    lib.load_library()
    d = tmp_path_factory.mktemp("fake")
    (d / "fake.c").write_text(FAKE)
    subprocess.run(["gcc", "-shared", "-fPIC", "-I/usr/local/cuda/include", "-o", str(d / "fake.so"), str(d / "fake.c"),
                    "-ldl"], check=True)
    with open("/proc/self/maps") as f:
        cudart = next(line.split()[-1] for line in f if "libcudart.so" in line)

    def run(code):
        env = dict(os.environ, LD_PRELOAD=str(d / "fake.so"), FAKE_CUDART=cudart, PYTHONPATH=ROOT, OUT=str(d / "out.npy"))
        full = SETUP + "fake = ctypes.CDLL(%r)\n" % str(d / "fake.so") + code
        r = subprocess.run([sys.executable, "-c", full], env=env, cwd=ROOT, capture_output=True, text=True, timeout=300)
        assert r.returncode == 0, r.stderr[-2000:]
        return r.stdout, d / "out.npy"
    return run


@pytest.mark.parametrize("graph", [0, 1])
def test_refused_launch_is_an_error_and_the_context_recovers(child, graph):
    out, _ = child("""
c = context(graph=%d)
before = results(c)
Y0, q0, s0 = c.get_state()
fake.fake_limit(1, 0)
for call in (lambda: c.mobility_solve(FT.reshape(-1)), lambda: c.brownian_slip(W), lambda: c.step(1)):
    try:
        call()
        print("no error")
    except g.GdcError as e:
        print("status", e.status, "kernel launch" in str(e))
Y1, q1, s1 = c.get_state()
print("state", bool(np.array_equal(Y0, Y1) and np.array_equal(q0, q1) and s0 == s1))
fake.fake_limit(16, 0)
print("again", bool(np.array_equal(before, results(c))))
c.step(1)
print("stepped", c.get_state()[2] == s0 + 1)
""" % graph)
    assert out.split("\n")[:6] == ["status 2 True"] * 3 + ["state True", "again True", "stepped True"], out


@pytest.mark.parametrize("largest", [8, 2, 1])
def test_smaller_clusters_where_the_device_refuses_16(child, largest):
    """8 and 2 blocks, and the separate kernels where no cluster holds a suspension."""
    _, f = child("np.save(os.environ['OUT'], results(context()))")
    full = np.load(f)
    _, f = child("fake.fake_limit(%d, 1)\nnp.save(os.environ['OUT'], results(context()))" % largest)
    # converged to 1e-9 of the right-hand side and of the root; the block-preconditioned operators'
    # condition numbers are below 1e3
    few = np.load(f)
    assert np.linalg.norm(few - full) < 1e-6 * np.linalg.norm(full)
