"""Launch shapes: what axpic_launch_shape reports can be asked for, and tuning
replaces a shape by a faster one only (needs a GB300)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2604_24627_gb300 import _lib  # noqa: E402
from test_gpu_batch import assert_same, base_params, make, state  # noqa: E402


# capacities for which the rule takes 1, 2, 4 and 8 cells a chunk
@pytest.mark.parametrize("caps,chunk", [((64, 192, 1024), 1), ((64, 192, 512), 2), ((64, 96, 192), 4), ((64, 64, 64), 8)])
def test_a_reported_shape_can_be_asked_for(caps, chunk):
    a = make(29, base_params(dt_phys_s=1e11), caps=caps, counts=(61, 37, 13))
    assert a.launch_shape()[0] == chunk
    b = make(29, base_params(dt_phys_s=1e11, decide_chunk=chunk), caps=caps, counts=(61, 37, 13))
    assert b.launch_shape() == a.launch_shape()
    for s in range(2):
        a.step(s, _lib.CH_ALL)
        b.step(s, _lib.CH_ALL)
    torch.cuda.synchronize()
    assert_same(state(a), state(b), "chunk %d" % chunk)
    a.close()
    b.close()


@pytest.mark.parametrize("chunk", [-1, 3, 12, 33, 64])
def test_other_chunks_are_refused(chunk):
    with pytest.raises(_lib.AxpicError) as e:
        make(2, base_params(decide_chunk=chunk))
    assert "INVALID" in str(e.value)


def test_tuning_leaves_no_slower_shape():
    """4,096 cells of 512 electrons and 256 photons: the rule takes 1 cell a
    chunk, which none of the shapes that the tuner tries comes near (a step 7 %
    slower at 4, 26 % at 8). And a shape slower than a tried one is replaced."""
    kw = dict(T=np.full(4096, 3.0), caps=(512, 384, 384), counts=(512, 256, 16))
    prm = base_params(dt_phys_s=8.8e11, g_ae=1e-13, w_a=1e12, tally_enable=0, diag_enable=0)
    pl = make(4096, prm, **kw)
    assert pl.launch_shape()[0] == 1
    before = pl.launch_shape()
    ms, chunk, warps = pl.autotune(0, 8)
    assert ms > 0 and chunk in (4, 8, 16, 32) and warps in (2, 4)
    assert pl.launch_shape() == before
    pl.close()
    pl = make(4096, dict(prm, decide_chunk=32), **kw)  # 128 warps' work at once: far too few
    pl.autotune(0, 8)
    assert pl.launch_shape()[0] in (4, 8)
    pl.close()
