"""The no-event bounds of the decision kernel over the range of their
arguments: photons and axions from far below kappa to far above it (s = 4
omega^2 / kappa^2 from 1e-14 to 1e5), weights on both sides of the product
weight, capped and uncapped means, both absorption targets; and electrons in
equal and unequal numbers a cell. A bound that cleared a slot with an event
would lose it against the oracle (needs a GB300)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2604_24627_gb300 import _lib  # noqa: E402
from parity_util import oracle_step  # noqa: E402
from test_gpu_parity import MIX_A, MIX_Z, base_params, make  # noqa: E402


def spread(rng, n, w_a, decades):
    """n particles with log-uniform energies and weights, isotropic."""
    E = 10.0 ** rng.uniform(-6.5, 2.5, n) / 510.99895
    u, ph = rng.uniform(-1, 1, n), rng.uniform(0, 2 * np.pi, n)
    st = np.sqrt(1 - u * u)
    return {"w": w_a * 10.0 ** rng.uniform(-decades, decades, n), "px": E * st * np.cos(ph), "py": E * st * np.sin(ph),
            "pz": E * u, "x": rng.uniform(0, 1, n), "y": rng.uniform(0, 1, n), "z": rng.uniform(0, 1, n)}


@pytest.mark.parametrize("case", [dict(lambda_cap=0.3), dict(lambda_cap=2.5, eq_stats=1),
                                  dict(dt_phys_s=2e10), dict(dt_phys_s=2e13, lambda_cap=0.05, brems_gamma_shape=2.2)])
@pytest.mark.parametrize("n_el", [3, 8, 60])  # one quad a cell, two, and fifteen
def test_bounds_lose_no_event(case, n_el):
    rng = np.random.default_rng(int(case.get("dt_phys_s", 1) / 1e9) + n_el)
    prm = base_params(T_mode=2, **case)
    ncells = 37
    pl = make(ncells, np.linspace(0.7, 8.0, ncells), prm, caps=(64, 1024, 1024), counts=(n_el, 1, 1))
    decades = 3 if "lambda_cap" in case else 1
    for c in range(ncells):
        pl.set_cell(c, {"g": spread(rng, 41, prm["w_a"], decades), "a": spread(rng, 43, prm["w_a"], decades)})
    if n_el == 8:
        pl.slabs["electrons"].count[5::7] = 7  # unequal numbers: the chunk's quads are searched
        pl.update_cells()
    for step in range(2):
        before = [pl.cell(c) for c in range(ncells)]
        T_before = pl.temperatures().copy()
        res_before = pl.residuals()
        pl.step(step)
        n_ion = pl.n_ion.reshape(ncells, -1).cpu().numpy()
        for c in range(ncells):
            parts, _, _ = oracle_step(before[c], T_before[c], n_ion[c], MIX_Z, MIX_A, prm, step, c, _lib.CH_ALL,
                                      res=res_before[c])
            got = pl.cell(c)
            for k in "ga":
                assert len(got[k]["w"]) == len(parts[k]), (c, k)
                # the same events: a remainder w - K w_prod is exact to a few
                # roundings of the heaviest particle, whatever is left of it
                top = max(before[c]["g"]["w"].max(), before[c]["a"]["w"].max() if len(before[c]["a"]["w"]) else 0)
                assert np.all(np.abs(got[k]["w"] - parts[k].w) <= 1e-5 * parts[k].w + 2.0 ** -20 * top), (c, k)
    tot = pl.tally()[1]
    assert tot["dropped"] == 0
    if "lambda_cap" in case:  # the short uncapped step hardly has any
        assert tot["events_p"] > 0 and tot["events_pinv"] > 0
    pl.close()
