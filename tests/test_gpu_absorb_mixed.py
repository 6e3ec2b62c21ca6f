"""The absorb phase of a separate call where about half of a warp's cells have
more than 64 axions flagged and the others any number up to that, against the
oracle (needs a GB300)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from test_gpu_parity import base_params, make  # noqa: E402
from test_gpu_remap_groups import _compare_separate  # noqa: E402


@pytest.mark.parametrize("heavy", [15, 16, 25])
def test_mixed_warps_match_oracle(heavy):
    ncells = 35  # a warp and a part of one
    prm = base_params(absorb_mode=1, T_mode=2)
    pl = make(ncells, np.linspace(1.5, 4.5, ncells), prm, caps=(64, 192, 512), counts=(61, 37, 110))
    rng = np.random.default_rng(heavy)
    na = rng.choice([0, 1, 15, 16, 17, 18, 40, 63, 64], ncells)
    na[rng.permutation(32)[:heavy]] = rng.integers(65, 111, heavy)
    na[32:] = (110, 16, 65)
    pl.slabs["axions"].count.copy_(torch.from_numpy(na.astype(np.int32)))
    for step in range(2):
        before = [pl.cell(c) for c in range(ncells)]
        T_before, res_before = pl.temperatures().copy(), pl.residuals()
        pl.absorb(step)
        pl.emit(step)
        pl.feedback(step)
        _compare_separate(pl, ncells, before, T_before, prm, step, res_before, "%d heavy" % heavy)
    pl.close()
