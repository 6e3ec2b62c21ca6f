"""A carried exchange just below and just above what binary32 momenta can take
(2^-22 of the cell's kinetic energy, or of its momentum spread): below it the
electrons and the carry keep their bits, above it the cell is remapped. Through
the entry point whose carry the caller owns (needs a GB300)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2604_24627_gb300 import AxionPlasma, _lib  # noqa: E402

MC2 = 510.99895
# the moments are binary32 sums of 48 weights of one sign, a few 2^-24 off at
# most: 5e-5 from the threshold is told apart, and lies inside the kernel's
# first test's margin of 1e-4
BELOW, ABOVE = (1e-310, 1e-12, 0.5, 0.999, 1 - 5e-5), (1 + 5e-5, 1.001, 4.0)
WAYS = [(1, 0, 0, 0), (-1, 0, 0, 0), (0, 1, 0, 0), (0, 0, -1, 0), (0, 0, 0, 1), (0, 0.6, -0.64, 0.48)]


@pytest.mark.parametrize("scale", [1.0, 1e-9])  # of the weights
def test_carry_about_the_threshold(scale):
    f = np.array(BELOW + ABOVE)
    ncells = len(f) * len(WAYS)
    pl = AxionPlasma(ncells, np.linspace(1.5, 4.5, ncells), np.full((ncells, 1), 6e25), [1.0], [1.00794], 1e-12,
                     (48, 8, 8), dict(g_agg_GeV_inv=1e-10, g_ae=1e-12, dt_phys_s=1.0, w_a=3e9, T_mode=2, relax_r=0.0,
                                      tally_enable=0, diag_enable=0))
    pl.sample(48, 0, 0)
    pl.slabs["electrons"].storage["wp"].view(-1, 4)[:, 0] *= scale
    want = np.zeros((ncells, 4))
    before = []
    for c in range(ncells):
        e = pl.cell(c)["e"]
        before.append({k: np.array(e[k]) for k in ("px", "py", "pz")})
        w, p = np.array(e["w"], np.float64), np.stack([np.array(e[k], np.float64) for k in ("px", "py", "pz")])
        U2 = (w * (p ** 2).sum(0)).sum()
        lim = 2.0 ** -22 * np.array([0.5 * U2 * MC2] + [np.sqrt(U2 * w.sum())] * 3)
        want[c] = f[c % len(f)] * lim * np.array(WAYS[c // len(f)])
    buf = torch.zeros(4 * ncells + 1, dtype=torch.float64, device="cuda")
    carry = buf[1:]  # aligned to 8 bytes only
    carry.copy_(torch.from_numpy(want.reshape(-1)))
    _lib.axpic_step_noalloc(pl.desc, pl.params, 0, _lib.CH_PRIMAKOFF, carry.data_ptr(),
                            torch.cuda.current_stream().cuda_stream)
    got = carry.reshape(ncells, 4).cpu().numpy()
    for c in range(ncells):
        e = pl.cell(c)["e"]
        moved = any(np.any(np.array(e[k]) != before[c][k]) for k in ("px", "py", "pz"))
        above = c % len(f) >= len(BELOW)
        assert moved == above, (c, f[c % len(f)], WAYS[c // len(f)])
        assert np.any(got[c] != want[c]) == above, (c, got[c], want[c])
    pl.close()
