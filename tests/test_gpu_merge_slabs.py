"""Merging at the slab sizes where the kernel changes how many passes of 32 slots
it keeps in registers (1, 2 and 5), full, partly full and beyond them, against
the oracle bit for bit (needs a GB300)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from oracle import merge as MG  # noqa: E402
from test_gpu_merge import EDGES, FIELDS, assert_cell_equal, gpu_cell, make, random_axions  # noqa: E402


@pytest.mark.parametrize("cap", [4, 32, 36, 64, 68, 160, 164, 260])
@pytest.mark.parametrize("edges", [0, 3, 16])
def test_slab_sizes_match_oracle(cap, edges):
    rng = np.random.default_rng(cap + edges)
    counts = [k for k in (0, 1, 3, 31, 32, 33, 63, 64, 65, 159, 160, 161, 193) if k <= cap]
    counts += [cap] + list(rng.integers(0, cap + 1, 9))
    cells = [random_axions(rng, int(k)) for k in counts]
    pl = make(len(cells), cap)
    for c, sp in enumerate(cells):
        pl.slabs["axions"].set_cell(c, {f: getattr(sp, f) for f in FIELDS})
    removed = 0
    for n_target in (cap // 2, 2):
        pl.merge_axions(n_target, EDGES[:edges])
        cells, r = MG.merge(cells, n_target, EDGES[:edges])
        removed += r
    torch.cuda.synchronize()
    for c, sp in enumerate(cells):
        assert_cell_equal(gpu_cell(pl.slabs["axions"], c), sp, c)
    assert pl.merge_stats() == removed and (removed > 0 or cap == 4)
    pl.close()
