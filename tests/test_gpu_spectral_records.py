"""Spectral records as they are read and saved under the surrogate model: the
table's for every cell, whether the network is trusted for it or not, from its
current temperature and composition (needs a GB300)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2604_24627_gb300 import _lib  # noqa: E402
from test_gpu_records import load_net, make, params, seeded_net  # noqa: E402

KW = dict(counts=(8, 8, 4), caps=(16, 64, 64))


def mixed(model, T, ne):
    """A plasma of the model; under the surrogate the colder cells take the network."""
    pl = make(T, ne, params(model), **KW)
    if model == 2:
        net = load_net(*seeded_net(6))
        err = np.ones((2, 4, 4, 3), dtype=np.float32)
        err[:, :, :3] = 0.0
        _lib.axpic_set_surrogate(pl.ctx, net.h, err, 4, 4, 1e-3, 1e-3)
        net.close()
    return pl


@pytest.mark.parametrize("n", [1, 33, 300])
def test_every_cell_has_the_tables_record(n):
    rng = np.random.default_rng(n)
    T, ne = np.exp(rng.uniform(np.log(0.6), np.log(9.5), n)), 10 ** rng.uniform(23.3, 25.9, n)
    T[0] = 0.7  # the network's
    ref, pl = mixed(1, T, ne), mixed(2, T, ne)
    _, src = _lib.axpic_get_cell_records(pl.ctx, 0, n)
    assert src[0] == 0 and (n == 1 or src.any())
    for scale in (1.0, 1.1):  # at set-up, and for temperatures the caller set later
        for p in (ref, pl):
            p.T.copy_(torch.as_tensor(T * scale))
            p.update_cells()
        a, b = (_lib.axpic_get_spectral_records(p.ctx, 0, n) for p in (pl, ref))
        assert np.array_equal(a, b)
        assert np.array_equal(_lib.axpic_get_spectral_records(pl.ctx, n // 2, n - n // 2), b[n // 2:])
    # two contexts in the same state save the same bytes
    other = mixed(2, T, ne)
    other.T.copy_(torch.as_tensor(T * 1.1))
    other.update_cells()
    assert np.array_equal(pl.save_state(), other.save_state())
    for p in (ref, pl, other):
        p.close()
