"""A first call whose scratch cannot be made says so, and the next one makes what
is missing: streaming and network training, each of their allocations failing
once, in a build whose cudaMalloc fails on request (needs a GB300)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2604_24627_gb300 import _lib, build  # noqa: E402
from paper_2604_24627_gb300.mlp import LAYOUT  # noqa: E402
from test_gpu_stream import C, make  # noqa: E402

SHIM = """
#include <cuda_runtime.h>
static int left = 0;
extern "C" void fail_malloc_after(int n) { left = n; }
extern "C" cudaError_t malloc_or_fail(void** p, size_t bytes) {
  if (left > 0 && --left == 0) return cudaErrorMemoryAllocation;
  return cudaMalloc(p, bytes);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = str(tmp_path_factory.mktemp("alloc"))
    with open(os.path.join(d, "shim.cu"), "w") as f:
        f.write(SHIM)
    own = ("api.cu", "mlp.cu")
    procs = [subprocess.Popen([build.nvcc()] + build.ARCH + build.FLAGS + ["-DcudaMalloc=malloc_or_fail", "-c",
                              os.path.join(build.CSRC, s), "-o", os.path.join(d, s + ".o")]) for s in own]
    procs.append(subprocess.Popen([build.nvcc()] + build.ARCH + build.FLAGS + ["-c", os.path.join(d, "shim.cu"), "-o",
                                  os.path.join(d, "shim.o")]))
    assert all(p.wait() == 0 for p in procs)
    rest = [os.path.join(build.BUILD, s + ".o") for s in build.SOURCES if s not in own]
    if not all(os.path.exists(o) for o in rest):
        build.build()
    out = os.path.join(d, "libaxpic_alloc.so")
    subprocess.run([build.nvcc()] + build.ARCH + ["-shared", "-o", out, os.path.join(d, "shim.o")] +
                   [os.path.join(d, s + ".o") for s in own] + rest + ["-lcudart"], check=True)
    return ctypes.CDLL(out)


def test_streaming_after_a_failed_allocation(lib):
    dims, n, cap = (5, 4, 1), 20, 36
    ref = make(n, cap)
    ref.sample(0, 0, 20)
    ref.stream_axions(dims, 1e-4, 0.7e-4 / C)
    want = [ref.cell(c)["a"] for c in range(n)]
    for which in (1, 2, 3, 4):
        pl = make(n, cap)
        pl.sample(0, 0, 20)
        torch.cuda.synchronize()
        h = ctypes.c_void_p()
        assert lib.axpic_init_plasma(ctypes.byref(h), ctypes.byref(pl.desc), ctypes.byref(pl.params), None) == 0
        args = (h, 5, 4, 1, ctypes.c_double(1e-4), ctypes.c_double(0.7e-4 / C), ctypes.c_double(0.0), 0)
        lib.fail_malloc_after(which)
        assert lib.axpic_stream_axions(*args) == _lib.AXPIC_E_CUDA
        assert lib.axpic_stream_axions(*args) == _lib.AXPIC_OK
        assert lib.axpic_destroy(h) == _lib.AXPIC_OK
        for c in range(n):
            got = pl.cell(c)["a"]
            assert all(np.array_equal(got[f], want[c][f]) for f in got), (which, c)
        pl.close()
    ref.close()


def test_training_after_a_failed_allocation(lib):
    P = np.random.default_rng(1).uniform(-0.1, 0.1, sum(int(np.prod(s)) for _, s in LAYOUT)).astype(np.float32)
    X, Z = torch.rand((300, 4), device="cuda"), torch.rand((300, 96), device="cuda")
    torch.cuda.synchronize()
    ptr = P.ctypes.data_as(ctypes.c_void_p)
    outs = []
    for which in (0, 1, 2):
        h = ctypes.c_void_p()
        assert lib.axpic_mlp_create(ctypes.byref(h), None) == _lib.AXPIC_OK
        assert lib.axpic_mlp_set_params(h, ptr) == _lib.AXPIC_OK
        args = (h, ctypes.c_void_p(X.data_ptr()), ctypes.c_void_p(Z.data_ptr()), 300, ctypes.c_float(1e-3), None)
        if which:
            lib.fail_malloc_after(which)
            assert lib.axpic_mlp_train_step(*args) == _lib.AXPIC_E_CUDA
        assert lib.axpic_mlp_train_step(*args) == _lib.AXPIC_OK
        got = np.zeros_like(P)
        assert lib.axpic_mlp_get_params(h, got.ctypes.data_as(ctypes.c_void_p)) == _lib.AXPIC_OK
        assert lib.axpic_mlp_destroy(h) == _lib.AXPIC_OK
        outs.append(got)
    assert not np.array_equal(outs[0], P)
    assert np.array_equal(outs[1], outs[0]) and np.array_equal(outs[2], outs[0])
