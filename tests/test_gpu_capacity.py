"""The largest slab capacities that the entry points take, and the first that
they refuse: the events' shared-memory scratch is the limit. A plasma with such
slabs steps as one with small slabs does, slot for slot (needs a GB300)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2604_24627_gb300 import _lib  # noqa: E402
from test_gpu_parity import base_params, make  # noqa: E402

PRM = base_params(dt_phys_s=6e12, T_mode=2)  # some cells with more events than a lane takes, some with fewer
FIELDS = ("w", "px", "py", "pz", "x", "y", "z")


def assert_close(ref, big, bits):
    """bits: photons and axions are the same bits (the records are); the sums
    behind the electrons' and the temperatures' update may be in another order."""
    torch.cuda.synchronize()
    np.testing.assert_allclose(big.temperatures(), ref.temperatures(), rtol=1e-5)
    for c in range(ref.ncells):
        a, b = ref.cell(c), big.cell(c)
        for k in "ega":
            for f in FIELDS:
                if bits and k != "e":
                    assert np.array_equal(a[k][f], b[k][f]), (c, k, f)
                else:
                    np.testing.assert_allclose(b[k][f], a[k][f], rtol=1e-5,
                                               atol=1e-6 * np.abs(a[k][f]).max(initial=0), err_msg=str((c, k, f)))


@pytest.mark.parametrize("cap", [1024, 1028, 8864, 36512, 36704])
@pytest.mark.parametrize("calls", ["step", "separate"])
def test_large_slabs_step_like_small_ones(cap, calls):
    T = np.array([1.5, 3.0, 4.5])
    ref, big = make(3, T, PRM), make(3, T, PRM, caps=(cap,) * 3)
    for pl in (ref, big):
        if calls == "step":
            pl.step(0)
        else:
            pl.absorb(0)
            pl.emit(0)
            pl.feedback(0)
    assert_close(ref, big, True)
    assert ref.tally()[1]["events_c"] > 0
    ref.close()
    big.close()


def test_init_refuses_beyond():
    with pytest.raises(_lib.AxpicError) as e:
        make(1, 3.0, PRM, caps=(36764,) * 3)
    assert "INVALID" in str(e.value)


@pytest.mark.parametrize("cap,ok", [(8636, True), (8640, True), (8864, True), (8884, False)])
def test_noalloc_range(cap, ok):
    prm = dict(PRM, tally_enable=0, diag_enable=0)
    ref, big = make(2, np.array([2.0, 4.0]), prm), make(2, np.array([2.0, 4.0]), prm, caps=(cap,) * 3)
    carry = torch.zeros(8, dtype=torch.float64, device="cuda")
    st = _lib.lib().axpic_step_noalloc(big.desc, big.params, 0, 7, carry.data_ptr(),
                                       torch.cuda.current_stream().cuda_stream)
    assert st == (_lib.AXPIC_OK if ok else _lib.AXPIC_E_INVALID)
    if ok:
        ref.step(0)
        assert_close(ref, big, False)
    ref.close()
    big.close()
