"""The work that users of the library have it do, as cases that can be timed.

Each case is one call sequence of a host code on one plasma, at a size of the
synthetic workloads (paper_2604_24627_gb300/workloads.py), of the benchmark
or of the tests:

* "steps": the Monte-Carlo steps themselves, by single calls or by graph
  replays, with or without the axions' transport, under one of the three
  rate models;
* "separate": a host code that interleaves its own work with the operators:
  absorption by weight reduction, emission, feedback and merging as four calls;
* "monitor": one step, the transport and the spectrum read back, every cycle;
* "transport", "merge", "composition": these operators alone;
* "train", "forward": the surrogate network's training and evaluation.

prepare() builds the plasma with its slabs (or the network) from a seed,
run() makes one pass, exact() gives the 64-bit result where the outputs are
functions of the inputs. The products of Monte-Carlo decisions have no such
value (a draw is compared with a binary32 threshold): None there.
"""
import math

import numpy as np
import torch

from paper_2604_24627_gb300 import AxionPlasma, _lib
from paper_2604_24627_gb300 import workloads as wl
from paper_2604_24627_gb300.mlp import LAYOUT, SurrogateNet, flatten

DEV = "cuda:0"
MC2 = 510.99895  # keV
C_CM_S = 2.99792458e10
STEP_DT = 9.93e11  # s: the step of the 3 keV workloads
H_CM = 1e-4        # edge of a 1 um cell


# ------------------------------------------------------------------ the cases
def _steps(name, dims, el, ph, ax, caps, **kw):
    c = {"name": name, "kind": "steps", "nx": dims[0], "ny": dims[1], "nz": dims[2], "el": el, "ph": ph, "ax": ax,
         "cap_e": caps[0], "cap_g": caps[1], "cap_a": caps[2], "field": "uniform", "T": 3.0, "n_e": 6e25,
         "helium": False, "dt": STEP_DT, "mask": 7, "T_mode": 2, "model": 0, "calls": "graph", "steps": 4,
         "ratio": 1.0, "stream": "", "mass": 0.0, "absorb": 0}
    c.update(kw)
    return c


def listed():
    return [
        # the smallest box: 1-D Primakoff exchange on 64 cells, step by step; launches and latency
        _steps("primakoff-1d-64", (64, 1, 1), 0, 128, 0, (4, 640, 512), T=1.3, dt=9.02e10, mask=1, T_mode=0,
               calls="step", steps=1, ratio=0.25),
        # the 2-D relaxation with all channels, hydrogen and helium, many particles a cell, replayed
        _steps("relax-2d-256", (256, 256, 1), 512, 256, 128, (512, 384, 384), helium=True, dt=8.763e11, steps=32),
        # a prescribed temperature bump whose axions stream out of an open box after every step
        _steps("bump-2d-512", (512, 512, 1), 256, 128, 16, (256, 768, 384), field="bump", T_mode=1, steps=8,
               stream="open"),
        # many small independent boxes of uneven cell counts batched in one context
        _steps("boxes-512", (0, 512, 1), 128, 64, 24, (128, 384, 256), field="boxes", steps=16),
        # the operators as separate calls, absorption by weight reduction, Bose-Einstein targets, then merging
        {"name": "separate-3d-47", "kind": "separate", "nx": 47, "ny": 53, "nz": 45, "el": 64, "ph": 32, "ax": 24,
         "cap_e": 64, "cap_g": 96, "cap_a": 128, "T": 5.0, "n_e": 6e25, "n_target": 24},
        # the 3-D plasma under the exact table rate model
        _steps("table-3d-96", (96, 96, 96), 64, 32, 13, (64, 64, 64), T=5.0, dt=5.448e11, model=1),
        # the benchmark's plasma: 3-D, the network rate model, more cells than fit the branches
        _steps("surrogate-3d-160", (160, 160, 160), 64, 32, 13, (64, 64, 64), T=5.0, dt=5.448e11, model=2),
        # a host loop that moves the axions and reads the emitted spectrum and the totals every cycle
        {"name": "monitor-3d-64", "kind": "monitor", "nx": 64, "ny": 64, "nz": 64, "el": 64, "ph": 32, "ax": 13,
         "cap_e": 64, "cap_g": 64, "cap_a": 64, "T": 5.0, "n_e": 6e25},
        # the transport alone, about half of the axions changing cell
        {"name": "transport-2d-256", "kind": "transport", "nx": 256, "ny": 256, "nz": 1, "ax": 128, "cap_a": 384,
         "cfl": 0.6, "mass": 0.0},
        # population control: every cell of a relaxed plasma merged after its axions were handed over
        {"name": "merge-2d-256", "kind": "merge", "cells": 65536, "ax": 128, "cap_a": 192, "n_target": 64,
         "edges": 16},
        # the composition from the electrons that the host code deposited
        {"name": "composition-2d-256", "kind": "composition", "cells": 65536, "el": 512, "cap_e": 512, "species": 2,
         "bind": -1},
        # the surrogate's training at the benchmark's batch: 8 steps, then the weights
        {"name": "train-8192", "kind": "train", "rows": 8192, "steps": 8},
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def up4(n):
        return (int(n) + 3) // 4 * 4

    kind = rng.choice(["steps", "steps", "steps", "steps", "separate", "monitor", "transport", "merge",
                       "composition", "train", "forward"])
    if kind == "steps":
        flavour = rng.choice(["small", "relax", "bump", "boxes", "cube"])
        if flavour == "small":
            n = log(33, 6000)
            return _draw_steps(rng, (n, 1, 1), 64, 48, 12, (64, 192, 160), calls=rng.choice(["step", "graph"]),
                               steps=1 + rng.randrange(4), T_mode=rng.choice([0, 1, 2]),
                               absorb=0, mass=rng.choice([0.0, 0.0, 1.0]), helium=rng.random() < 0.3)
        if flavour == "relax":
            nx = log(60, 250)
            el = 4 * log(16, 128)
            return _draw_steps(rng, (nx, nx + rng.randrange(7), 1), el, el // 2, el // 4,
                               (up4(el), up4(0.75 * el + 32), up4(0.75 * el + 32)), helium=rng.random() < 0.7,
                               steps=rng.choice([5, 8, 32]), dt=8.763e11)
        if flavour == "bump":
            nx = log(100, 500)
            return _draw_steps(rng, (nx, nx - rng.randrange(9), 1), 256, 128, 16, (256, 768, 384), field="bump",
                               T_mode=1, steps=rng.choice([1, 3, 8]), stream=rng.choice(["open", "periodic", ""]),
                               model=rng.choice([0, 0, 1]))
        if flavour == "boxes":
            return _draw_steps(rng, (0, log(24, 500), rng.randrange(1, 1000)), 128, 64, 24, (128, 384, 256),
                               field="boxes", steps=rng.choice([4, 16, 33]))
        n = log(40, 140)
        return _draw_steps(rng, (n, n + rng.randrange(5), n - rng.randrange(5)), 64, 32, 13, (64, 64, 64), T=5.0,
                           dt=5.448e11, model=rng.choice([0, 1, 2, 2]), calls=rng.choice(["step", "graph"]),
                           steps=1 + rng.randrange(4))
    if kind in ("separate", "monitor"):
        n = log(16, 60)
        c = {"kind": kind, "nx": n, "ny": n + rng.randrange(6), "nz": n - rng.randrange(6), "el": 64, "ph": 32,
             "ax": 13, "cap_e": 64, "cap_g": 64, "cap_a": 64, "T": 5.0, "n_e": 6e25}
        if kind == "separate":
            c.update(ax=24, cap_g=96, cap_a=128, n_target=16 + rng.randrange(16))
        return c
    if kind == "transport":
        if rng.random() < 0.5:
            ax, dims = 4 * log(4, 32), (log(90, 256), log(90, 256), 1)
        else:
            n = log(24, 110)
            ax, dims = rng.randrange(5, 24), (n, n + rng.randrange(6), n - rng.randrange(6))
        return {"kind": "transport", "nx": dims[0], "ny": dims[1], "nz": dims[2], "ax": ax, "cap_a": up4(2.5 * ax + 40),
                "cfl": round(rng.uniform(0.1, 0.95), 3), "mass": rng.choice([0.0, 2.0])}
    if kind == "merge":
        ax = log(30, 128)
        return {"kind": "merge", "cells": log(900, 65536), "ax": ax, "cap_a": up4(1.5 * ax + 8),
                "n_target": rng.randrange(8, ax), "edges": rng.randrange(0, 25)}
    if kind == "composition":
        el = log(24, 512)
        ns = rng.randrange(1, 4)
        return {"kind": "composition", "cells": log(1500, 65536), "el": el, "cap_e": up4(el + el // 4), "species": ns,
                "bind": rng.randrange(-1, ns)}
    rows = log(200, 30000) if kind == "train" else log(500, 1000000)
    return {"kind": kind, "rows": rows, "steps": 8 if kind == "train" else 1}


def _draw_steps(rng, *a, **kw):
    c = _steps("", *a, **kw)
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs
def _fields(c):
    """(ncells, T [ncells], n_ion, Z, A) of a steps case."""
    Z, A = np.array([1.0]), np.array([wl.A_H])
    if c["field"] == "boxes":
        w = wl.config4(c["ny"], seed=c["nz"])
        return w.ncells, w.T_keV, w.n_ion, w.Z, w.A
    n = c["nx"] * c["ny"] * c["nz"]
    if c["field"] == "bump":
        i, j = np.arange(c["nx"]) + 0.5 - c["nx"] / 2, np.arange(c["ny"]) + 0.5 - c["ny"] / 2
        T = 1.0 + 4.0 * np.exp(-(j[:, None] ** 2 + i[None, :] ** 2) / (2 * (c["nx"] / 8.0) ** 2))
        T = T.reshape(-1)
    else:
        T = np.full(n, c["T"])
        if c["model"] == 2:  # a few colder cells, outside the network's trusted region
            T[:: 512] = 0.4 * c["T"]
    if c["helium"]:
        tot = c["n_e"] / 1.1
        return n, T, np.tile([[0.9 * tot, 0.1 * tot]], (n, 1)), np.array([1.0, 2.0]), np.array([wl.A_H, wl.A_HE])
    return n, T, np.full((n, 1), c["n_e"]), Z, A


def _network(seed):
    """A network for the region around the 5 keV plasma: the model's constants and linear map fitted to the library's
    targets there, and small weights. Returns (SurrogateNet, error map, nT, nne)."""
    rng = np.random.default_rng(seed)
    m = 384
    T, ne = rng.uniform(3.0, 8.0, m), 10.0 ** rng.uniform(25.4, 26.0, m)
    hc, alpha = 1.973269804e-8, 1.0 / 137.035999084
    kT = np.sqrt(4 * math.pi * alpha * hc ** 3 * 2 * ne / T) / T  # Debye screening of hydrogen
    rows = np.stack([np.ones(m), kT, ne, np.ones(m)], 1)
    y = _lib.axpic_surrogate_targets(rows)
    f = _lib.axpic_surrogate_features(rows).astype(np.float64)
    s = 4.0 / kT ** 2
    y[:, 0] -= -math.log(math.e - 1.0) + np.log((1 + 1 / s) * np.log1p(s) - 1)
    y[:, 32] -= -math.log(math.e - 1.0)
    y[:, 64] -= -1.0
    D = np.stack([np.ones(m), f[:, 1], f[:, 2]], 1)
    sol = np.linalg.solve(D.T @ D, D.T @ y)
    mu, skip, sigma = sol[0].copy(), np.zeros((96, 4)), np.full(96, 1e-5)
    skip[:, 1], skip[:, 2] = sol[1], sol[2]
    sigma[[0, 32, 64]] = 1e-4
    for k in range(32, 96):  # the quantiles that do not depend on the cell
        if k % 32:
            mu[k], skip[k], sigma[k] = y[0, k], 0.0, 0.0
    net = SurrogateNet()
    net.set_params(_weights(rng))
    _lib.axpic_mlp_set_norm(net.h, mu, sigma)
    _lib.axpic_mlp_set_skip(net.h, skip)
    nT, nne = 65, 49
    Tg, ng = 0.5 * 20.0 ** (np.arange(nT) / (nT - 1)), 10.0 ** (23 + 3 * np.arange(nne) / (nne - 1))
    ok = ((Tg > 2.8) & (Tg < 8.2))[None, :] & ((ng > 2e25) & (ng < 1.01e26))[:, None]
    err = np.where(ok[None, :, :, None], 1e-4, 1.0) * np.ones((2, 1, 1, 3))
    return net, err, nT, nne


def _weights(rng):
    P = {}
    for k, shp in LAYOUT:
        lim = math.sqrt(6.0 / sum(shp)) if len(shp) == 2 else 0.1
        P[k] = rng.uniform(-lim, lim, shp)
    return flatten(P)


def _plasma(c, n, T, n_ion, Z, A, seed, extra):
    prm = dict(g_agg_GeV_inv=1e-10, g_ae=1e-13, relax_r=0.1, seed=seed, dt_phys_s=c.get("dt", 5.448e11),
               T_mode=c.get("T_mode", 2))
    prm["w_a"] = c.get("ratio", 1.0) * wl.photon_weight(3.0 if c.get("field") in ("bump", "boxes") else c["T"],
                                                        wl.VOLUME_1UM3, c["ph"])
    prm.update(extra)
    pl = AxionPlasma(n, T, n_ion, Z, A, wl.VOLUME_1UM3, (c["cap_e"], c["cap_g"], c["cap_a"]), prm, device=DEV)
    pl.sample(c["el"], c["ph"], c["ax"])
    return pl


def _momenta(gen, shape, T):
    """Isotropic momenta with a x^2 e^-x energy spectrum at T keV, in m_e c: [..., 3] float32."""
    u = torch.rand((*shape, 5), generator=gen, device=DEV)
    E = -T * torch.log((u[..., 0] + 1e-7) * (u[..., 1] + 1e-7) * (u[..., 2] + 1e-7))
    ct, ph = 2 * u[..., 3] - 1, 2 * math.pi * u[..., 4]
    st = torch.sqrt(torch.clamp(1 - ct * ct, min=0))
    return torch.stack([st * torch.cos(ph), st * torch.sin(ph), ct], -1) * (E / MC2)[..., None]


def _axions(c, n, seed):
    """wp, xyz [n, cap, 4] and count [n] (ragged) of an axion slab."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    cap, m = c["cap_a"], c["ax"]
    cnt = torch.randint(max(1, (3 * m) // 4), min(cap, (5 * m) // 4) + 1, (n,), generator=gen, device=DEV,
                        dtype=torch.int32)
    used = (torch.arange(cap, device=DEV)[None, :] < cnt[:, None])[..., None]
    wp = torch.zeros((n, cap, 4), device=DEV)
    wp[..., 0] = 1e9 * (0.5 + torch.rand((n, cap), generator=gen, device=DEV))
    wp[..., 1:] = _momenta(gen, (n, cap), 3.0)
    xyz = torch.zeros((n, cap, 4), device=DEV)
    xyz[..., :3] = torch.rand((n, cap, 3), generator=gen, device=DEV)
    return wp * used, xyz * used, cnt


def _axion_plasma(c, n, seed):
    pl = AxionPlasma(n, 3.0, np.full((n, 1), 6e25), [1.0], [wl.A_H], wl.VOLUME_1UM3, (4, 4, c["cap_a"]),
                     dict(w_a=1e9), device=DEV)
    src = _axions(c, n, seed)
    _hand_over(pl, src)
    return pl, src


def _hand_over(pl, src):
    """The host code's axions copied into the slab."""
    slab = pl.slabs["axions"]
    slab.storage["wp"].copy_(src[0].view(-1))
    slab.storage["xyz"].copy_(src[1].view(-1))
    slab.count.copy_(src[2])


def _electrons(c, seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    n, cap, m = c["cells"], c["cap_e"], c["el"]
    cnt = torch.randint((3 * m) // 4, min(cap, (5 * m) // 4) + 1, (n,), generator=gen, device=DEV, dtype=torch.int32)
    wp = torch.zeros((n, cap, 4), device=DEV)
    wp[..., 0] = (6e13 / m) * (0.5 + torch.rand((n, cap), generator=gen, device=DEV))
    wp[..., 1:] = 0.08 * torch.randn((n, cap, 3), generator=gen, device=DEV)
    return wp, cnt


_ION_Z, _ION_A = [1.0, 2.0, 6.0], [wl.A_H, wl.A_HE, 12.011]


def _fractions(ns):
    x = np.array([0.7, 0.28, 0.02][:ns])
    return x / x.sum()


def _rows(c, seed):
    """Cell features and normalised targets of a training or validation set."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    X = 2 * torch.rand((c["rows"], 4), generator=gen, device=DEV) - 1
    X[:, 0] = 0.0
    X[:, 3] = torch.where(X[:, 3] > 0, 0.5, -0.5)
    B = torch.randn((4, 96), generator=gen, device=DEV)
    return X, torch.sin(2 * X @ B) + 0.05 * torch.randn((c["rows"], 96), generator=gen, device=DEV)


def _edges(k):
    return (np.geomspace(0.5, 50.0, k) / MC2).astype(np.float32) ** 2 if k else np.zeros(0, dtype=np.float32)


def prepare(case, seed):
    c, k = case, case["kind"]
    s = {"case": c, "step": 0}
    if k == "steps":
        n, T, n_ion, Z, A = _fields(c)
        extra = dict(absorb_mode=c["absorb"], axion_mass_keV=c["mass"], rate_model=c["model"])
        if c["model"]:
            extra.update(sr_table_nkt=64, sr_table_nne=32)
        s["pl"] = _plasma(c, n, T, n_ion, Z, A, seed, extra)
        if c["model"] == 2:
            net, err, nT, nne = _network(11)
            _lib.axpic_set_surrogate(s["pl"].ctx, net.h, err, nT, nne, 3e-4, 1e-3)
            net.close()
    elif k in ("separate", "monitor"):
        n = c["nx"] * c["ny"] * c["nz"]
        extra = dict(absorb_mode=1, eq_stats=1) if k == "separate" else {}
        s["pl"] = _plasma(c, n, np.full(n, c["T"]), np.full((n, 1), c["n_e"]), [1.0], [wl.A_H], seed, extra)
        s["edges"] = _edges(4)
    elif k == "transport":
        s["pl"], _ = _axion_plasma(c, c["nx"] * c["ny"] * c["nz"], seed)
        s["dt"] = c["cfl"] * H_CM / C_CM_S
    elif k == "merge":
        s["pl"], s["src"] = _axion_plasma(c, c["cells"], seed)
        s["edges"] = _edges(c["edges"])
    elif k == "composition":
        ns = c["species"]
        s["pl"] = AxionPlasma(c["cells"], 3.0, np.full((c["cells"], ns), 1e25), _ION_Z[:ns], _ION_A[:ns],
                              wl.VOLUME_1UM3, (c["cap_e"], 4, 4), dict(w_a=1e9), device=DEV)
        wp, cnt = _electrons(c, seed)
        slab = s["pl"].slabs["electrons"]
        slab.storage["wp"].copy_(wp.view(-1))
        slab.count.copy_(cnt)
        s["pl"].update_cells()
        s["x"] = _fractions(ns) if c["bind"] < 0 else None
    else:
        s["net"] = SurrogateNet()
        s["net"].set_params(_weights(np.random.default_rng(seed)))
        s["X"], s["Zt"] = _rows(c, seed)
    return s


# ------------------------------------------------------------------ one pass
def _slabs(pl, names=("electrons", "photons", "axions")):
    out = {}
    for n in names:
        slab = pl.slabs[n]
        out[n] = [slab.storage["wp"], slab.storage["xyz"], slab.count]
    return out


def run(s):
    c, k = s["case"], s["case"]["kind"]
    if k in ("train", "forward"):
        if k == "forward":
            return s["net"].forward(s["X"])
        for _ in range(c["steps"]):  # the end of a cosine schedule, where the rate is a hundredth of its start
            s["net"].train_step(s["X"], s["Zt"], 2e-5)
        return {n: v.astype(np.float32) for n, v in s["net"].get_params().items()}
    pl = s["pl"]
    if k == "steps":
        first, m = s["step"], c["steps"]
        s["step"] += m
        if c["stream"]:
            pl.run_steps_streamed(first, m, c["mask"], (c["nx"], c["ny"], c["nz"]), H_CM, 0.6 * H_CM / C_CM_S,
                                  c["stream"] == "periodic", c["mass"])
        elif c["calls"] == "graph":
            pl.run_steps(first, m, c["mask"])
        else:
            for i in range(m):
                pl.step(first + i, c["mask"])
        return {**_slabs(pl), "T": pl.T}
    if k == "separate":
        pl.absorb(s["step"])
        pl.emit(s["step"])
        pl.feedback(s["step"])
        pl.merge_axions(c["n_target"], s["edges"])
        s["step"] += 1
        return {**_slabs(pl), "T": pl.T}
    if k == "monitor":
        pl.step(s["step"])
        pl.stream_axions((c["nx"], c["ny"], c["nz"]), H_CM, 0.6 * H_CM / C_CM_S)
        s["step"] += 1
        H, tot = pl.tally()
        return {**_slabs(pl), "T": pl.T, "H": H, "totals": tot}
    if k == "transport":
        pl.stream_axions((c["nx"], c["ny"], c["nz"]), H_CM, s["dt"], mass_keV=c["mass"])
        return _slabs(pl, ("axions",))
    if k == "merge":
        _hand_over(pl, s["src"])
        pl.merge_axions(c["n_target"], s["edges"])
        return _slabs(pl, ("axions",))
    return pl.deposit_composition(s["x"], c["bind"])


# ------------------------------------------------------------------ work
def work(case):
    """Bytes: per step the weight and momentum (16 B) of every photon and axion, the cells' rate constants and
    temperatures; per moved or merged axion its two records in and out; per electron of a deposit its weight; per
    network row its inputs, targets or outputs. Operations: the draws' and rates' arithmetic, or the network's
    products."""
    c, k = case, case["kind"]
    if k in ("steps", "separate", "monitor"):
        n = len(_fields(c)[1]) if c.get("field") == "boxes" else c["nx"] * c["ny"] * c["nz"]
        steps = c.get("steps", 1)
        b, f = n * (16 * (c["ph"] + c["ax"]) + 96), n * (25 * c["el"] + 60 * (c["ph"] + 2 * c["ax"]))
        if k == "monitor" or c.get("stream"):
            b += n * 56 * c["ax"]
        if k == "monitor":
            b += n * 16 * c["el"]
        if k == "separate":
            b += n * 56 * c["ax"]
        return {"bytes": b * steps, "flops": f * steps}
    if k in ("transport", "merge"):
        n = c["ax"] * (c["cells"] if k == "merge" else c["nx"] * c["ny"] * c["nz"])
        if k == "merge":  # handed over, then merged
            return {"bytes": 56 * n + 64 * c["cells"] * c["cap_a"], "flops": 40 * n}
        return {"bytes": 56 * n, "flops": 20 * n}
    if k == "composition":
        return {"bytes": c["cells"] * (4 * c["el"] + 8 * c["species"] + 64), "flops": 8 * c["cells"] * c["el"]}
    macs = 4 * 64 + 64 * 64 + 64 * 96
    if k == "forward":
        return {"bytes": 400 * c["rows"], "flops": 2 * macs * c["rows"]}
    return {"bytes": c["steps"] * (400 * c["rows"] + 7 * 4 * 10720), "flops": 6 * macs * c["rows"] * c["steps"]}


# ------------------------------------------------------------------ 64-bit results
def exact(case, seed):
    k = case["kind"]
    if k == "transport":
        return _exact_transport(case, seed)
    if k == "merge":
        return _exact_merge(case, seed)
    if k == "composition":
        wp, cnt = _electrons(case, seed)
        live = torch.arange(case["cap_e"], device=DEV)[None, :] < cnt[:, None]
        ne = (wp[..., 0].double() * live).sum(1) / wl.VOLUME_1UM3
        ns, Z, A = case["species"], _ION_Z, _ION_A
        if case["bind"] >= 0:
            coef = [1.0 / Z[i] if i == case["bind"] else 0.0 for i in range(ns)]
        else:
            x = _fractions(ns)
            zxa = sum(Z[i] * x[i] / A[i] for i in range(ns))
            coef = [x[i] / A[i] / zxa for i in range(ns)]
        return (ne[:, None] * torch.tensor(coef, dtype=torch.float64, device=DEV)[None, :]).reshape(-1)
    if k in ("train", "forward"):
        return _exact_network(case, seed)
    return None  # Monte-Carlo decisions


def _exact_network(case, seed):
    flat = torch.tensor(_weights(np.random.default_rng(seed)), dtype=torch.float64, device=DEV)
    P, o = {}, 0
    for n, shp in LAYOUT:
        m = int(np.prod(shp))
        P[n] = flat[o:o + m].reshape(shp).clone().requires_grad_(case["kind"] == "train")
        o += m
    X, Zt = (t.double() for t in _rows(case, seed))

    def net():
        h = torch.tanh(X @ P["W1"] + P["b1"])
        return torch.tanh(h @ P["W2"] + P["b2"]) @ P["W3"] + P["b3"]

    if case["kind"] == "forward":
        return net()
    mom = {n: (torch.zeros_like(v), torch.zeros_like(v)) for n, v in P.items()}
    for t in range(1, case["steps"] + 1):
        loss = ((net() - Zt) ** 2).sum() / X.shape[0]
        grads = torch.autograd.grad(loss, list(P.values()))
        with torch.no_grad():
            for (n, v), g in zip(P.items(), grads):
                m1 = 0.9 * mom[n][0] + 0.1 * g
                m2 = 0.999 * mom[n][1] + 0.001 * g * g
                mom[n] = (m1, m2)
                v -= 2e-5 * (m1 / (1 - 0.9 ** t)) / (torch.sqrt(m2 / (1 - 0.999 ** t)) + 1e-8)
    return {n: v.detach().float().double().cpu().numpy() for n, v in P.items()}


def _fill(keep, wp, xyz):
    """The tail fill: per cell the free slots below the new count take, in order, the kept slots at or beyond it."""
    n, cap = keep.shape
    slot = torch.arange(cap, device=DEV)[None, :]
    ns = keep.sum(1, keepdim=True)
    hole, mover = (~keep) & (slot < ns), keep & (slot >= ns)
    hc, hs = torch.nonzero(hole, as_tuple=True)  # both ascending by cell and slot, equally many per cell
    mc, ms = torch.nonzero(mover, as_tuple=True)
    wp[hc, hs], xyz[hc, hs] = wp[mc, ms], xyz[mc, ms]
    return ns.reshape(-1).to(torch.int32)


def _exact_transport(case, seed):
    nx, ny, nz, cap = case["nx"], case["ny"], case["nz"], case["cap_a"]
    n = nx * ny * nz
    wp32, xyz32, cnt = _axions(case, n, seed)
    wp, xyz = wp32.double(), xyz32.double()
    slot = torch.arange(cap, device=DEV)[None, :]
    live = slot < cnt[:, None]
    p = wp[..., 1:]
    E = torch.sqrt((p * p).sum(-1) + (case["mass"] / MC2) ** 2)
    step = torch.where((E > 0) & live, case["cfl"] / torch.clamp(E, min=1e-300), 0.0)
    shift = torch.zeros((n, cap, 3), dtype=torch.int64, device=DEV)
    for d, m in enumerate((nx, ny, nz)):
        if m > 1:
            t = xyz[..., d] + step * p[..., d]
            fl = torch.floor(t)
            xyz[..., d] = torch.where(live, t - fl, xyz[..., d])
            shift[..., d] = torch.where(live, fl.long(), 0)
    stay = live & (shift == 0).all(-1)
    c, s = torch.nonzero(live & ~stay, as_tuple=True)
    sh = shift[c, s]
    i, j, k = c % nx, (c // nx) % ny, c // (nx * ny)
    dest = (((k + sh[:, 2]) % nz) * ny + (j + sh[:, 1]) % ny) * nx + (i + sh[:, 0]) % nx
    r = (1 - sh[:, 2]) * 9 + (1 - sh[:, 1]) * 3 + (1 - sh[:, 0])  # the source seen from the destination
    order = torch.argsort((dest * 27 + r) * cap + s)
    c, s, dest = c[order], s[order], dest[order]
    rank = torch.arange(len(dest), device=DEV)
    first = torch.zeros(n, dtype=torch.int64, device=DEV)
    arr = torch.bincount(dest, minlength=n)
    first[1:] = torch.cumsum(arr, 0)[:-1]
    rank = rank - first[dest]
    free = live & ~stay
    H = free.sum(1)
    fslot = torch.argsort((~free).to(torch.int8), dim=1, stable=True)  # the freed slots first, ascending
    place = torch.where(rank < H[dest], fslot[dest, torch.clamp(rank, max=cap - 1)], cnt[dest].long() + rank - H[dest])
    ok = place < cap
    c, s, dest, place = c[ok], s[ok], dest[ok], place[ok]
    mw, mx = wp[c, s], xyz[c, s]
    keep = stay.clone()
    wp[dest, place], xyz[dest, place] = mw, mx
    keep[dest, place] = True
    out = _fill(keep, wp, xyz)
    return {"axions": [wp.reshape(-1), xyz.reshape(-1), out]}


def _exact_merge(case, seed):
    n, cap = case["cells"], case["cap_a"]
    wp32, xyz32, cnt = _axions(case, n, seed)
    wp, xyz = wp32.double(), xyz32.double()
    slot = torch.arange(cap, device=DEV)[None, :].expand(n, cap)
    live = slot < cnt[:, None]
    p32 = wp32[..., 1:]
    p2 = (p32[..., 0] * p32[..., 0] + p32[..., 1] * p32[..., 1]) + p32[..., 2] * p32[..., 2]
    bins = torch.zeros((n, cap), dtype=torch.int64, device=DEV)
    for e in _edges(case["edges"]):
        bins += p2 >= float(e)
    neg = p32 < 0
    g = bins * 8 + neg[..., 0] + 2 * neg[..., 1] + 4 * neg[..., 2]
    G = (case["edges"] + 1) * 8
    key = torch.arange(n, device=DEV)[:, None] * G + g
    take = live & (cnt > case["n_target"])[:, None]
    size = torch.bincount(key[take], minlength=n * G)
    take &= size[key] >= 3
    kk, ss = key[take], slot[take]
    order = torch.argsort(kk * cap + ss)
    kk, ss = kk[order], ss[order]
    cc = kk // G
    head = torch.ones_like(kk, dtype=torch.bool)
    head[1:] = kk[1:] != kk[:-1]
    gid = torch.cumsum(head, 0) - 1
    ng = int(gid[-1]) + 1 if len(gid) else 0
    w, p, x = wp[cc, ss, 0], wp[cc, ss, 1:], xyz[cc, ss, :3]
    E = torch.sqrt((p * p).sum(-1))
    vals = torch.cat([w[:, None], w[:, None] * p, (w * E)[:, None], w[:, None] * x], 1)
    sums = torch.zeros((ng, 8), dtype=torch.float64, device=DEV).index_add_(0, gid, vals)
    W, P, Es, X = sums[:, :1], sums[:, 1:4], sums[:, 4:5], sums[:, 5:8]
    Pn = torch.sqrt((P * P).sum(-1, keepdim=True))
    e = P / Pn
    ct = torch.clamp(Pn / Es, max=1.0)
    st = torch.sqrt(1 - ct * ct)
    ax = torch.nn.functional.one_hot(torch.argmin(e.abs(), 1), 3).double()
    u = torch.linalg.cross(e, ax)
    u = u / torch.sqrt((u * u).sum(-1, keepdim=True))
    pa, pb = Es / W * (ct * e + st * u), Es / W * (ct * e - st * u)
    at = torch.nonzero(head).reshape(-1)
    zero = torch.zeros_like(W)
    for off, q in ((0, pa), (1, pb)):
        wp[cc[at], ss[at + off]] = torch.cat([0.5 * W, q], 1)
        xyz[cc[at], ss[at + off]] = torch.cat([X / W, zero], 1)
    freed = torch.arange(len(kk), device=DEV) - at[gid] >= 2 if ng else torch.zeros(0, dtype=torch.bool, device=DEV)
    keep = live.clone()
    keep[cc[freed], ss[freed]] = False
    out = _fill(keep, wp, xyz)
    return {"axions": [wp.reshape(-1), xyz.reshape(-1), out]}
