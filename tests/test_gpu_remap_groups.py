"""Weight reduction, where every axion is flagged and every cell remapped: the
remap's groups of 8, 16 and 32 lanes a cell and the absorb phase's lane and
warp paths, at uneven counts, against the oracle (needs a GB300)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2604_24627_gb300 import _lib  # noqa: E402
from oracle import step as ostep  # noqa: E402
from oracle.plasma import cell_state  # noqa: E402
from parity_util import assert_electron_remap_close, assert_species_close, oracle_params, to_species  # noqa: E402
from test_gpu_parity import MIX_A, MIX_Z, _compare_step, base_params, make  # noqa: E402


# the most electrons a cell of a warp holds: at most 32 (8 lanes a cell), 64
# (16) and more (the warp); one quad over each limit too
@pytest.mark.parametrize("most", [4, 32, 33, 64, 65, 200])
@pytest.mark.parametrize("calls", ["step", "separate"])
def test_uneven_cells_match_oracle(most, calls):
    ncells = 39  # a full warp of cells and a part of one
    rng = np.random.default_rng(most)
    prm = base_params(absorb_mode=1, T_mode=2)
    cap = (most + 3) // 4 * 4
    pl = make(ncells, np.linspace(1.5, 4.5, ncells), prm, caps=(cap, 192, 512), counts=(most, 37, 110))
    # (at least two: one electron has no variance to compare)
    ne = rng.integers(2, most + 1, ncells)
    ne[:3], ne[-1] = (most, 2, most), 0  # the last cell has no electrons: its exchange is carried
    na = rng.integers(0, 111, ncells)  # none to one more than a lane takes, and on to the warp's
    na[:6] = (0, 1, 63, 64, 65, 110)
    pl.slabs["electrons"].count.copy_(torch.from_numpy(ne.astype(np.int32)))
    pl.slabs["axions"].count.copy_(torch.from_numpy(na.astype(np.int32)))
    pl.update_cells()
    for step in range(2):
        before = [pl.cell(c) for c in range(ncells)]
        T_before = pl.temperatures().copy()
        res_before = pl.residuals()
        if calls == "step":
            pl.step(step)
        else:
            pl.absorb(step)
            pl.emit(step)
            pl.feedback(step)
        assert pl.temperatures()[-1] == T_before[-1]
        if calls == "step":
            _compare_step(_FirstCells(pl, ncells - 1), before, T_before, prm, step, _lib.CH_ALL, res_before,
                          "step %d" % most)
        else:
            _compare_separate(pl, ncells - 1, before, T_before, prm, step, res_before, "separate %d" % most)
    assert pl.tally()[1]["remaps"] > 0
    pl.close()


def _compare_separate(pl, n, before, T_before, prm, step, res_before, label):
    """The separate calls' slot rule (each phase closes its own holes), and
    the feedback fed the GPU's own exchange."""
    op = oracle_params(prm)
    n_ion = pl.n_ion.reshape(pl.ncells, -1).cpu().numpy()
    diag, Tn = pl.cell_diag(), pl.temperatures()
    for c in range(n):
        got, what = pl.cell(c), "%s cell %d" % (label, c)
        parts = {k: to_species(before[c][k]) for k in "ega"}
        cs = cell_state(T_before[c], n_ion[c], MIX_Z, MIX_A, op)
        tally = ostep.StepTally()
        ostep.absorb_cell(cs, parts, op, step, c, _lib.CH_ALL, tally)
        ostep.emit_cell(cs, parts, op, step, c, _lib.CH_ALL, tally, n_g0=tally.n_g0)
        assert_species_close(got["a"], parts["a"], what + " axions")
        assert_species_close(got["g"], parts["g"], what + " photons")
        d = diag[c]
        assert abs(d[0] - tally.dE) <= 1e-5 * tally.gross_E + 1e-30, (what, d[0], tally.dE)
        assert np.all(np.abs(d[1:4] - tally.dP) <= 1e-5 * tally.gross_P + 1e-30), what
        e_parts = {"e": to_species(before[c]["e"])}
        fb = ostep.feedback_cell(cs, e_parts, op, ostep.StepTally(dE=d[0], dP=np.array(d[1:4])), res_before[c][0],
                                 np.array(res_before[c][1:4]))
        assert_electron_remap_close(before[c]["e"], got["e"], e_parts["e"], what + " electrons")
        assert abs(Tn[c] - fb.T_new) <= 1e-5 * fb.T_new, (what, Tn[c], fb.T_new)


class _FirstCells:
    """The first n cells of a plasma, as _compare_step reads them."""

    def __init__(self, pl, n):
        self.pl, self.ncells = pl, n
        self.n_ion = pl.n_ion.reshape(pl.ncells, -1)[:n].reshape(-1)
        self.cell_diag, self.temperatures, self.cell = pl.cell_diag, pl.temperatures, pl.cell
