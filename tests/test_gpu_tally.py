"""The totals and the folded spectrum rows of axpic_tally_spectrum against
64-bit sums of the slabs, at the sizes where the totals kernel's cell groups,
passes and number range end (needs a GB300 and the built library)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2604_24627_gb300 import AxionPlasma, _lib  # noqa: E402

ME = 510.99895


def make(ncells, caps, **kw):
    prm = dict(g_agg_GeV_inv=1e-10, g_ae=1e-12, dt_phys_s=2e12, w_a=3.0e9, seed=5, T_mode=2)
    prm.update(kw)
    return AxionPlasma(ncells, 3.0, np.full((ncells, 1), 6e25), [1.0], [1.00794], 1e-12, caps, prm)


# cells below, at and beyond a warp's group of 8 and a full grid's; slabs from
# empty to several passes; weights whose binary32 sums overflow (1e38) or whose
# products leave the range of exact remainders (1e-30)
@pytest.mark.parametrize("ncells", [1, 7, 8, 9, 1300])
@pytest.mark.parametrize("caps,scale", [((4, 4, 4), 1e9), ((132, 68, 36), 1e9), ((64, 64, 64), 1e38),
                                        ((64, 64, 64), 1e-30), ((0, 32, 0), 1.0)])
def test_totals_equal_64_bit_sums(ncells, caps, scale):
    pl = make(ncells, caps)
    rng = np.random.default_rng(ncells * 7 + caps[0])
    want = {}
    for (name, key), cap in zip((("electrons", "e"), ("photons", "g"), ("axions", "a")), caps):
        cnt = rng.integers(0, cap + 1, ncells).astype(np.int32)
        wp = rng.uniform(0.5, 1.5, (ncells, cap, 4)).astype(np.float32)
        wp[..., 0] *= np.float32(scale)
        wp[..., 1:] = (wp[..., 1:] - np.float32(1.0)) * np.float32(0.02)
        slab = pl.slabs[name]
        if cap:
            slab.storage["wp"][:wp.size].copy_(torch.from_numpy(wp.reshape(-1)))
        slab.count[:ncells].copy_(torch.from_numpy(cnt))
        live = np.arange(cap)[None, :] < cnt[:, None]
        w, p = wp[..., 0].astype(np.float64), wp[..., 1:].astype(np.float64)
        p2 = (p ** 2).sum(-1)
        want[key] = (np.sum(w[live]), np.sum((w * np.sqrt(p2))[live]), 0.5 * np.sum((w * p2)[live]), cnt.sum())
    torch.cuda.synchronize()
    _, tot = pl.tally()
    # the particle's |p| or p^2 is formed in binary32 (3 roundings and a root:
    # below 4 2^-24); the sums are 64-bit or better
    for k, v in (("n_axions", want["a"][0]), ("n_photons", want["g"][0])):
        assert abs(tot[k] - v) <= 1e-13 * v, k
    for k, v in (("u_axions", want["a"][1] * ME), ("u_photons", want["g"][1] * ME), ("u_electrons", want["e"][2] * ME)):
        assert abs(tot[k] - v) <= 4 * 2.0 ** -24 * v, k
    assert tot["macro_axions"] == want["a"][3] and tot["macro_photons"] == want["g"][3]
    pl.close()


# one row (few cells), many rows, and a histogram long enough to limit them
@pytest.mark.parametrize("ncells,nbins", [(20, 160), (3000, 160), (3000, 1), (3000, 50000)])
def test_folded_rows_hold_every_emitted_axion(ncells, nbins):
    a = make(ncells, (64, 64, 128), tally_nbins=nbins, tally_Emax_keV=4000.0)
    b = make(ncells, (64, 64, 128), tally_nbins=nbins, tally_Emax_keV=4000.0)
    a.sample(64, 32, 0)
    a.emit(0, _lib.CH_ALL)
    b.load_state(a.save_state())
    H, tot = a.tally()
    n, u = sum(tot["nemit_" + c] for c in "pcb"), [tot["uemit_" + c] for c in "pcb"]
    assert tot["macro_axions"] > 0
    assert abs(n - tot["n_axions"]) <= 1e-12 * n  # nothing was there before
    assert abs(sum(u) - tot["u_axions"]) <= 8 * 2.0 ** -24 * sum(u)  # E and |p| rounded apart
    assert np.allclose(H.sum(1), u, rtol=1e-12, atol=0)
    Hb, tb = b.tally()  # the saved state carries the folded rows
    assert np.allclose(Hb, H, rtol=1e-12, atol=0) and all(tb["uemit_" + c] == tot["uemit_" + c] for c in "pcb")
    H2, t2 = a.tally()  # cleared by the read
    assert not H2.any() and t2["nemit_p"] == 0 and t2["n_axions"] == tot["n_axions"]
    a.close()
    b.close()
