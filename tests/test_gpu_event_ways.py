"""Cells that the events' lanes take and cells that a warp takes, where the choice
depends on how many there are: few cells, with axions flagged on both sides of
their limit; axions with events on both sides of a lane's and more removed
than the tail fill loads at once, against the oracle; and the time of one
such cell (needs a GB300)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from oracle import step as ostep  # noqa: E402
from oracle.plasma import cell_state  # noqa: E402
from parity_util import assert_species_close, oracle_params, to_species  # noqa: E402
from test_gpu_parity import MIX_A, MIX_Z, base_params, make  # noqa: E402
from test_gpu_remap_groups import _compare_separate  # noqa: E402


@pytest.mark.parametrize("ncells", [1, 2, 7, 33, 60])
@pytest.mark.parametrize("most", [9, 36, 65, 166, 300])
def test_weight_reduction_matches_oracle(ncells, most):
    prm = base_params(absorb_mode=1, T_mode=2)
    pl = make(ncells, np.linspace(1.5, 4.5, ncells), prm, caps=(64, 192, 512), counts=(61, 37, 300))
    na = np.random.default_rng(most).integers(0, min(most, 17), ncells)
    na[0] = most
    if ncells > 4:
        na[3], na[-1] = most - 1, most
    pl.slabs["axions"].count.copy_(torch.from_numpy(na.astype(np.int32)))
    for step in range(2):
        before = [pl.cell(c) for c in range(ncells)]
        T_before, res_before = pl.temperatures().copy(), pl.residuals()
        pl.absorb(step)
        pl.emit(step)
        pl.feedback(step)
        _compare_separate(pl, ncells, before, T_before, prm, step, res_before, "%d cells" % ncells)
    pl.close()


@pytest.mark.parametrize("dt,na", [(1e13, 60), (1e13, 250), (5e13, 30)])
def test_axions_with_events_match_oracle(dt, na):
    ncells = 34
    prm = base_params(dt_phys_s=dt, T_mode=1, g_ae=1e-13)
    pl = make(ncells, np.linspace(2.0, 4.5, ncells), prm, caps=(24, 1000, 600), counts=(23, 10, na))
    n0 = np.linspace(0, na, ncells).astype(np.int32)
    pl.slabs["axions"].count.copy_(torch.from_numpy(n0))
    op, T = oracle_params(prm), pl.temperatures()
    n_ion = pl.n_ion.reshape(ncells, -1).cpu().numpy()
    before = [pl.cell(c) for c in range(ncells)]
    pl.absorb(0)
    gone = n0 - pl.counts()["axions"]
    assert gone.max() > 8 and np.count_nonzero((gone > 0) & (gone <= 8)) > 3
    for c in range(ncells):
        parts = {k: to_species(before[c][k]) for k in "ega"}
        ostep.absorb_cell(cell_state(T[c], n_ion[c], MIX_Z, MIX_A, op), parts, op, 0, c, 7, ostep.StepTally())
        got = pl.cell(c)
        assert_species_close(got["a"], parts["a"], "cell %d axions" % c)
        assert_species_close(got["g"], parts["g"], "cell %d photons" % c)
    pl.close()


def test_one_cells_axions_are_absorbed_side_by_side():
    """A cell alone in its warp: 60 axions take no longer than twice 8 of them
    (20 us; one after the other in a lane they took 60)."""
    us = {}
    for na in (8, 60):
        pl = make(1, 3.0, base_params(absorb_mode=1, dt_phys_s=1e11), caps=(64, 192, 128), counts=(61, 37, na))
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        t = []
        for step in range(30):
            torch.cuda._sleep(200000)  # both kernels are queued before the first starts
            ev[0].record()
            pl.absorb(step)
            ev[1].record()
            torch.cuda.synchronize()
            t.append(ev[0].elapsed_time(ev[1]))
        us[na] = 1e3 * np.median(t)
        pl.close()
    assert us[60] < 2 * us[8], us
