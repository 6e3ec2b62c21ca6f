"""The network kernel when a tensor-core wait runs out for some of a block's
threads and not for others: the block leaves its tiles as one, releases its
tensor memory and the call reports the time-out, in a build of mlp.cu whose
bound is zero for half of the warps of some blocks at one wait of every tile
(needs a GB300).
Nothing hangs or faults: the products themselves complete as ever."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import surrogate as S

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2604_24627_gb300 import _lib, build  # noqa: E402
from paper_2604_24627_gb300.mlp import LAYOUT, SurrogateNet  # noqa: E402
from test_gpu_mlp import forward_bound, seeded  # noqa: E402

PARAMS = sum(int(np.prod(s)) for _, s in LAYOUT)


@pytest.fixture(scope="module", params=[0, 1])
def variant(request, tmp_path_factory):
    """The library with mlp.cu's waits on phases of this parity cut short in the warps 2, 3, 6, 7, ... of the blocks
    from the third on."""
    out = str(tmp_path_factory.mktemp("wait") / "libaxpic_wait.so")
    obj = out + ".o"
    polls = "AXPIC_WAIT_POLLS=((threadIdx.x & 64) && blockIdx.x > 1 && parity == %du ? 0 : kWaitPolls)" % request.param
    src = os.path.join(build.CSRC, "mlp.cu")
    subprocess.run([build.nvcc()] + build.ARCH + build.FLAGS + ["-D" + polls, "-c", src, "-o", obj], check=True)
    rest = [os.path.join(build.BUILD, s + ".o") for s in build.SOURCES if s != "mlp.cu"]
    if not all(os.path.exists(o) for o in rest):
        build.build()
    subprocess.run([build.nvcc()] + build.ARCH + ["-shared", "-o", out, obj] + rest + ["-lcudart"], check=True)
    return out


# the third block's tile a part of one; more than one tile for every block
# (two blocks an SM in inference, one in training)
@pytest.mark.parametrize("rows", [300, 120000])
@pytest.mark.parametrize("call", ["forward", "train"])
def test_partial_time_out_ends_cleanly(variant, rows, call):
    lib = ctypes.CDLL(variant)
    P = np.random.default_rng(1).uniform(-0.1, 0.1, PARAMS).astype(np.float32)
    X = torch.rand((rows, 4), device="cuda")
    Z = torch.rand((rows, 96), device="cuda")
    h = ctypes.c_void_p()
    assert lib.axpic_mlp_create(ctypes.byref(h), None) == _lib.AXPIC_OK
    assert lib.axpic_mlp_set_params(h, P.ctypes.data_as(ctypes.c_void_p)) == _lib.AXPIC_OK

    def run(n):
        if call == "forward":
            return lib.axpic_mlp_forward(h, ctypes.c_void_p(X.data_ptr()), n, ctypes.c_void_p(Z.data_ptr()))
        return lib.axpic_mlp_train_step(h, ctypes.c_void_p(X.data_ptr()), ctypes.c_void_p(Z.data_ptr()), n,
                                        ctypes.c_float(1e-3), None)

    before, got = np.zeros_like(P), np.zeros_like(P)
    assert run(200) == _lib.AXPIC_OK  # two blocks: no wait is cut short
    assert lib.axpic_mlp_get_params(h, before.ctypes.data_as(ctypes.c_void_p)) == _lib.AXPIC_OK
    assert np.array_equal(before, P) == (call == "forward")
    for _ in range(2):
        assert run(rows) == _lib.AXPIC_OK  # asynchronous
    assert lib.axpic_mlp_get_params(h, got.ctypes.data_as(ctypes.c_void_p)) == _lib.AXPIC_E_TIMEOUT
    assert np.array_equal(got, before)  # a step that did not finish leaves the parameters as they were
    assert lib.axpic_mlp_destroy(h) == _lib.AXPIC_E_TIMEOUT
    # the device is as usable as before, its tensor memory free again
    Pd, Xs, _ = seeded(7, 300)
    net = SurrogateNet()
    net.set_params(Pd)
    out = net.forward(torch.as_tensor(np.asarray(Xs, np.float32), device="cuda")).cpu().numpy()
    want, _ = S.forward(Pd, Xs, bf16_mma=True)
    assert np.all(np.abs(out - want) <= forward_bound(Pd, Xs) + 1e-7)
    net.close()
