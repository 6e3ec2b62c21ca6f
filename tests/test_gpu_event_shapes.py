"""The full-step event kernel with 4, 8 and 32 cells a warp, and cells on both
sides of the flagged slots a lane takes (16 axions or photons, 8 electrons):
ranges of one plasma stepped apart give the state of one step over all of it,
bit for bit (needs a GB300)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from test_gpu_batch import assert_same, base_params, make, state  # noqa: E402


# 49,155 cells: 32 a warp as a whole, in ranges of 12,290 cells 8, of 1,001 4.
# g_ae and dt set how many slots are flagged: few, and often more than a lane takes
@pytest.mark.parametrize("dt", [5e11, 3e12])
@pytest.mark.parametrize("part", [12290, 1001])
def test_ranges_equal_the_whole(dt, part):
    n = 49155
    prm = base_params(dt_phys_s=dt, diag_enable=0)
    whole, parts = (make(n, prm, caps=(24, 256, 512), counts=(21, 37, 30)) for _ in range(2))
    for step in range(2):
        whole.step(step)
        for first in range(0, n, part):
            parts.step_cells(step, first, min(part, n - first))
    torch.cuda.synchronize()
    a, b = state(whole), state(parts)
    assert_same(a, b, "ranges of %d" % part)
    ta, tb = whole.tally()[1], parts.tally()[1]
    for k in ("events_p", "events_c", "events_b", "events_pinv", "absorbed_c", "absorbed_b", "dropped"):
        assert ta[k] == tb[k] > 0 or k == "dropped" and ta[k] == tb[k], k
    whole.close()
    parts.close()
