"""Launch shapes: what axpic_launch_shape reports can be asked for (needs a
GB300)."""
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
