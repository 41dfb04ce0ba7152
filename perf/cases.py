"""Performance cases of the radiative transfer library: the calls a simulation
makes, through the package's public entry points (``paper_1705_04702_gb300.skirt``
and ``selfabsorb``), over the sizes at which it makes them.

A case is a dict of plain values; ``kind`` says which call it stands for:

* ``trace``      the photon-packet life cycle (``skirt_trace``) on one of the
                 four problem families of ``workloads``: the dust sphere with a
                 central point source, the exponential-disk galaxy, the clumpy
                 torus with many wavelengths of uneven packet counts, and the
                 disk galaxy on an adaptive octree; mixed or FP64 form;
* ``reemit``     the dust emission phase's trace: packets start in the dust
                 cells in proportion to an emission table;
* ``selfabs``    whole dust self-absorption cycles (two-field emission, source
                 totals, dust trace);
* ``exact``      exact equilibrium emission of cells from one absorbed table,
                 or from a stellar and a dust table (``n_dust`` > 0);
* ``surrogate``  dust emission through the network, the exact solver for the
                 cells it does not cover;
* ``train``      training of the network.

Every input is made from the seed alone, on the GPU where it is large.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1705_04702_gb300 import selfabsorb
from paper_1705_04702_gb300 import skirt as S
from paper_1705_04702_gb300 import workloads as W

DEV = "cuda"
NOUT, NBANDS, NHID = 100, 32, 128


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest whole run: a central star in a dust sphere, 32^3 cells, 1e5 packets; launches,
        # synchronisations and the tail of the packet queue count
        {"name": "trace_sphere_small", "kind": "trace", "grid": "sphere", "n": 32, "nlambda": 1, "packets": 100_000,
         "npx": 64, "precision": "mixed", "graph": False},
        # the headline workload: an exponential-disk galaxy at one optical wavelength with three instruments
        # (a tenth of the benchmark's packets, so that a pass stays well below a second)
        {"name": "trace_disk_galaxy", "kind": "trace", "grid": "disk", "n": 256, "nlambda": 1, "packets": 10_000_000,
         "npx": 512, "precision": "mixed", "graph": True},
        # a panchromatic run: the clumpy torus, 200 wavelengths with uneven packet counts in one launch
        {"name": "trace_torus_200_lambda", "kind": "trace", "grid": "torus", "n": 128, "nlambda": 200,
         "packets": 8_000_000, "npx": 256, "precision": "mixed", "graph": True},
        # the adaptive grid: the disk galaxy on a mass-refined octree of some 8e5 leaves
        {"name": "trace_disk_octree", "kind": "trace", "grid": "octree", "n": 12, "nlambda": 1, "packets": 3_000_000,
         "npx": 512, "precision": "mixed", "graph": False},
        # the plain FP64 form, which a user takes to check the mixed one: the disk galaxy, ragged grid
        {"name": "trace_disk_fp64", "kind": "trace", "grid": "disk", "n": 97, "nlambda": 3, "packets": 300_000,
         "npx": 200, "precision": "fp64", "graph": False},
        # the dust emission phase: 100 infrared wavelengths from the dust cells of the torus, with peel-off
        {"name": "reemit_torus", "kind": "reemit", "n": 128, "packets": 2_000_000, "npx": 256, "precision": "mixed"},
        # two dust self-absorption cycles on a small torus (20 stellar wavelengths)
        {"name": "selfabs_two_cycles", "kind": "selfabs", "n": 64, "n_in": 20, "packets": 200_000},
        # the exact solver on a training set's worth of cells
        {"name": "exact_emission_1m", "kind": "exact", "ncell": 1_000_000, "n_in": 200, "n_dust": 0},
        # the exact solver on a handful of cells (a user probing a model)
        {"name": "exact_emission_small", "kind": "exact", "ncell": 2_000, "n_in": 41, "n_dust": 0},
        # a self-absorption cycle's emission on a full grid: stellar and dust field together
        {"name": "exact_emission_pair", "kind": "exact", "ncell": 2_097_152, "n_in": 200, "n_dust": 100},
        # the learned emission step on a full grid whose cells are mostly empty space
        {"name": "surrogate_torus", "kind": "surrogate", "n": 200, "n_in": 200},
        # the network's training on one emission step's labels, the default batch
        {"name": "train_surrogate", "kind": "train", "rows": 300_000, "batch": 2048, "epochs": 4},
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["trace", "trace", "trace", "reemit", "selfabs", "exact", "exact", "surrogate", "train"])
    if kind == "trace":
        grid = rng.choice(["sphere", "disk", "torus", "octree", "disk"])
        if grid == "sphere":
            return {"kind": "trace", "grid": grid, "n": rng.randint(16, 64), "nlambda": 1,
                    "packets": int(_log_uniform(rng, 2e4, 4e6)), "npx": rng.randint(32, 128), "precision": "mixed",
                    "graph": rng.random() < 0.5}
        if grid == "disk":
            fp64 = rng.random() < 0.3
            return {"kind": "trace", "grid": grid, "n": rng.randint(48, 128 if fp64 else 256),
                    "nlambda": rng.choice([1, 1, 3, 7]), "packets": int(_log_uniform(rng, 5e4, 2e5 if fp64 else 8e6)),
                    "npx": rng.randint(64, 512), "precision": "fp64" if fp64 else "mixed", "graph": rng.random() < 0.5}
        if grid == "torus":
            return {"kind": "trace", "grid": grid, "n": rng.randint(40, 128), "nlambda": rng.randint(20, 200),
                    "packets": int(_log_uniform(rng, 2e5, 6e6)), "npx": rng.randint(64, 256), "precision": "mixed",
                    "graph": rng.random() < 0.5}
        return {"kind": "trace", "grid": grid, "n": rng.randint(7, 12), "nlambda": rng.choice([1, 1, 5]),
                "packets": int(_log_uniform(rng, 5e4, 3e6)), "npx": rng.randint(64, 512), "precision": "mixed",
                "graph": False}
    if kind == "reemit":
        return {"kind": kind, "n": rng.randint(40, 128), "packets": int(_log_uniform(rng, 1e5, 2e6)),
                "npx": rng.randint(64, 256), "precision": "mixed"}
    if kind == "selfabs":
        return {"kind": kind, "n": rng.randint(24, 80), "n_in": rng.randint(10, 60),
                "packets": int(_log_uniform(rng, 5e4, 5e5))}
    if kind == "exact":
        return {"kind": kind, "ncell": int(_log_uniform(rng, 500, 2e6)), "n_in": rng.randint(20, 240),
                "n_dust": rng.choice([0, 0, 100])}
    if kind == "surrogate":
        return {"kind": kind, "n": rng.randint(30, 200), "n_in": rng.randint(40, 220)}
    return {"kind": kind, "rows": int(_log_uniform(rng, 2e4, 3e5)), "batch": rng.choice([512, 1024, 2048, 2048, 4096]),
            "epochs": rng.randint(1, 4)}


# ----------------------------------------------------------------- the inputs
@functools.lru_cache(maxsize=8)
def _octree(level):
    # 8.3e5 leaves from level 11 on; eight times the mass bound per level below that
    return W.disk_octree(max_level=level, delta=1.35e-5 * 8.0 ** max(0, 11 - level))


def _packets(case, n, seed, uneven):
    """Packets per wavelength that add up to about case["packets"]."""
    if not uneven:
        return np.full(n, max(1, case["packets"] // n), dtype=np.uint64)
    p = W.uneven_packet_counts(n, seed=seed).astype(np.float64)
    return np.maximum(np.round(p * (case["packets"] / p.sum())), 1).astype(np.uint64)


def _trace_problem(case, seed):
    rng = np.random.default_rng(seed)
    nl = case["nlambda"]
    if case["grid"] == "sphere":
        prob = W.sphere_problem(1, n=case["n"], albedo=0.5, seed=seed)
        prob.grid.kr = (prob.grid.kr * np.float32(rng.uniform(0.7, 1.4))).astype(np.float32)
        prob.instruments = [W.Instrument(100.0, 0.0, 0.0, 2.0, case["npx"])]
    elif case["grid"] == "disk":
        prob = W.disk_problem(1, n=case["n"], nlambda=nl, npx=case["npx"], seed=seed)
        prob.grid.kr = (prob.grid.kr * np.float32(rng.uniform(0.7, 1.4))).astype(np.float32)
    elif case["grid"] == "torus":
        prob = W.torus_problem(n=case["n"], nlambda=nl, npx=case["npx"], seed=seed)
    else:
        prob = W.octree_problem(_octree(case["n"]), 1, nlambda=nl, npx=case["npx"], seed=seed)
    return prob.with_packets(_packets(case, nl, seed, case["grid"] == "torus"))


def _outputs(ncell, nl, instruments):
    img = sum(i.npx * i.npx for i in instruments) * nl
    return (torch.zeros((ncell, nl), dtype=torch.float64, device=DEV),
            torch.zeros(max(img, 1), dtype=torch.float64, device=DEV),
            torch.zeros((max(len(instruments), 1), nl), dtype=torch.float64, device=DEV))


def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _spectra(n, lam, gen, rows=1 << 18):
    """Absorbed spectra and dust masses with the distributions of
    ``workloads.absorbed_spectra``, made on the GPU: a power law attenuated by
    dust, log-normal power per unit mass."""
    lam = torch.as_tensor(lam, dtype=torch.float32, device=DEV)
    out = torch.empty((n, lam.numel()), dtype=torch.float64, device=DEV)
    mass = torch.empty(n, dtype=torch.float32, device=DEV)
    for a in range(0, n, rows):
        b = min(n, a + rows)
        u = torch.rand((b - a, 3), device=DEV, generator=gen)
        alpha = -2.0 + 2.5 * u[:, :1]
        tau = 10.0 ** (-3.0 + 5.0 * u[:, 1:2])
        s = lam ** alpha * torch.exp(-tau * (lam / 0.55) ** -1.2)
        m = 10.0 ** (-7.0 + 3.0 * u[:, 2])
        per_mass = 10.0 ** torch.randn(b - a, device=DEV, generator=gen)
        out[a:b] = (s / s.sum(dim=1, keepdim=True)).double()
        out[a:b] *= (per_mass * m).double()[:, None]
        mass[a:b] = m
    return out, mass


def _torus_mask(n):
    """Which cells of the n^3 torus grid hold dust (flat, x fastest)."""
    x = -1.0 + (torch.arange(n, device=DEV) + 0.5) * (2.0 / n)
    z, y, x = torch.meshgrid(x, x, x, indexing="ij")
    r = torch.sqrt(x * x + y * y + z * z)
    inside = (r >= 0.05) & (r <= 1.0) & (z.abs() <= math.sin(math.radians(50.0)) * r)
    return inside.reshape(-1), r.reshape(-1)


def _emission_table(n, gen):
    """A dust emission table of the torus: modified black bodies whose
    temperature falls with the distance from the centre, no emission outside
    the dust."""
    inside, r = _torus_mask(n)
    lam, wt = S.skirt_emission_grid()
    lam = torch.as_tensor(lam, dtype=torch.float64, device=DEV)
    wt = torch.as_tensor(wt, dtype=torch.float64, device=DEV)
    out = torch.zeros((n ** 3, NOUT), dtype=torch.float64, device=DEV)
    idx = torch.nonzero(inside).flatten()
    for a in range(0, idx.numel(), 1 << 19):
        k = idx[a:a + (1 << 19)]
        T = 300.0 * (r[k] / 0.05) ** -0.5 * (0.7 + 0.6 * torch.rand(k.numel(), device=DEV, generator=gen))
        m = 10.0 ** (-2.0 + 2.0 * torch.rand(k.numel(), device=DEV, generator=gen))
        x = torch.clamp(14387.768775 / (lam[None, :] * T[:, None].double()), max=80.0)
        out[k] = m[:, None].double() * wt * (lam / 100.0) ** -1.8 * (lam ** -5.0) / torch.expm1(x)
    return out


class _State:
    pass


def prepare(case, seed):
    st = _State()
    st.case = case
    kind = case["kind"]
    if kind == "trace":
        st.prob = _trace_problem(case, seed)
        st.grid = S.Grid(st.prob.grid)
        st.out = _outputs(st.grid.ncell, st.prob.wl.n, st.prob.instruments)
        st.kw = {"precision": S.PREC_MIXED if case["precision"] == "mixed" else S.PREC_FP64,
                 "use_graph": case["graph"]}
        st.emission = None
    elif kind == "reemit":
        g = W.torus_grid(case["n"], seed=seed)
        wl = selfabsorb.dust_wavelengths()
        wl.lsrc = None  # the emission table's column sums
        st.prob = W.Problem("reemit", g, W.Source(W.SRC_DUST), wl, _packets(case, NOUT, seed, False),
                            W.galaxy_instruments(case["npx"], fov=2.0), seed=seed, phase=1)
        st.grid = S.Grid(g)
        st.emission = _emission_table(case["n"], _generator(seed))
        st.out = _outputs(st.grid.ncell, NOUT, st.prob.instruments)
        st.kw = {"precision": S.PREC_MIXED}
    elif kind == "selfabs":
        st.grid = S.Grid(W.torus_grid(case["n"], seed=seed))
        st.lam = np.geomspace(0.09, 10.0, case["n_in"])
        st.mass = torch.empty(st.grid.ncell, dtype=torch.float32, device=DEV)
        S.skirt_dust_mass(st.grid.h, st.mass)
        st.absorbed, m = _spectra(st.grid.ncell, st.lam, _generator(seed))
        # the same power per unit mass, in the grid's own dust masses (nothing absorbs outside the dust)
        st.absorbed *= (st.mass.double() / m.double())[:, None]
        st.wl = selfabsorb.dust_wavelengths()
        st.wl.kscale = st.wl.kscale * 20.0  # infrared extinction that re-absorbs some of the emission
        st.per_lambda = max(1, case["packets"] // NOUT)
        st.seed = seed
    elif kind == "exact":
        gen = _generator(seed)
        st.lam = np.geomspace(0.09, 10.0, case["n_in"])
        st.a, st.mass = _spectra(case["ncell"], st.lam, gen)
        st.b = st.lam_b = None
        if case["n_dust"]:
            st.lam_b = np.geomspace(1.0, 1000.0, case["n_dust"])
            st.b, m = _spectra(case["ncell"], st.lam_b, gen)
            st.b *= (0.1 * st.mass.double() / m.double())[:, None]
        st.emission = torch.empty((case["ncell"], NOUT), dtype=torch.float64, device=DEV)
        st.temperature = torch.empty((case["ncell"], 3), dtype=torch.float32, device=DEV)
    elif kind == "surrogate":
        gen = _generator(seed)
        st.lam = np.geomspace(0.09, 10.0, case["n_in"])
        ncell = case["n"] ** 3
        st.a, st.mass = _spectra(ncell, st.lam, gen)
        inside, _ = _torus_mask(case["n"])
        for a in range(0, ncell, 1 << 20):
            st.a[a:a + (1 << 20)] *= inside[a:a + (1 << 20), None].double()
        st.mass *= inside.float()
        st.host = _network(gen, st, inside)
        st.net = S.MLP(seed=1)
        st.net.set_params(*st.host[:5])
        st.net.set_guard(st.host[5])
        st.emission = torch.empty((ncell, NOUT), dtype=torch.float64, device=DEV)
        st.temperature = torch.empty((ncell, 3), dtype=torch.float32, device=DEV)
    else:
        gen = _generator(seed)
        n = case["rows"]
        lam = np.geomspace(0.09, 10.0, 64)
        a, mass = _spectra(n, lam, gen)
        st.features, _ = _features64(a, lam, mass)
        st.features = st.features.float().contiguous()
        # labels: modified black bodies whose temperature follows the absorbed power per unit mass
        le, wt = S.skirt_emission_grid()
        le = torch.as_tensor(le, dtype=torch.float64, device=DEV)
        wt = torch.as_tensor(wt, dtype=torch.float64, device=DEV)
        T = 30.0 * (a.sum(dim=1) / mass.double()).clamp(1e-4, 1e6) ** (1.0 / 6.0)
        x = torch.clamp(14387.768775 / (le[None, :] * T[:, None]), max=80.0)
        st.labels = (a.sum(dim=1)[:, None] * wt * (le / 100.0) ** -1.8 * le ** -5.0 / torch.expm1(x)).contiguous()
        st.seed = seed
        st.params = _random_params(gen)
        st.net = S.MLP(seed=1)
    return st


def _random_params(gen):
    """Network parameters: uniform weights of the usual fan-in scale, zero biases."""
    out = []
    for rows, cols in ((NHID, NBANDS), (NHID, NHID), (NOUT, NHID)):
        b = math.sqrt(6.0 / cols)
        out.append(((2.0 * torch.rand((rows, cols), device=DEV, generator=gen) - 1.0) * b).reshape(-1))
        out.append(torch.zeros(rows, device=DEV))
    return torch.cat(out).float().cpu().numpy()


def _network(gen, st, inside):
    """Parameters, standardisation, range and guard of a network that covers
    all but about a hundredth of the heated cells, as a trained one does."""
    idx = torch.nonzero(inside).flatten()
    pick = idx[torch.randint(0, idx.numel(), (50_000,), device=DEV, generator=gen)]
    f, _ = _features64(st.a[pick], st.lam, st.mass[pick])
    lo, hi = f.min(dim=0).values, f.max(dim=0).values
    share = 1.0 / (10.0 ** (f - f.max(dim=1, keepdim=True).values)).sum(dim=1)
    guard = float(torch.sort(share).values[int(0.99 * (share.numel() - 1))])
    host = [v.float().cpu().numpy() for v in (f.mean(dim=0), f.std(dim=0), lo - 1e-3, hi + 1e-3)]
    return (_random_params(gen), *host, guard)


# -------------------------------------------------------------------- the pass
def run(st):
    case = st.case
    kind = case["kind"]
    if kind in ("trace", "reemit"):
        r = S.run_problem(st.prob, grid=st.grid, outputs=st.out, emission=st.emission, **st.kw)
        led = r["ledger"]
        return {"absorbed": r["absorbed"], "images": r["images_flat"], "sed": r["sed"],
                "ledger_per_lambda": r["ledger_per_lambda"],
                "ledger": [led[k] for k in ("emitted", "absorbed", "escaped", "residual")],
                "counts": [int(led[k]) for k in ("scatterings", "deposit_steps", "locate_steps", "peel_steps")]}
    if kind == "selfabs":
        r = selfabsorb.self_absorption(st.grid, st.absorbed, st.lam, st.mass, st.per_lambda, st.seed, tol=0.0,
                                       max_cycles=2, wl=st.wl)
        return {"absorbed_dust": r["absorbed_dust"], "emission": r["emission"], "cycles": r["cycles"],
                "history": [[h["emitted"], h["absorbed"]] for h in r["history"]]}
    if kind == "exact":
        if st.b is None:
            S.skirt_dust_emission(st.a, case["ncell"], case["n_in"], st.lam, st.mass, S.EMIT_EXACT, None, st.emission,
                                  st.temperature)
        else:
            S.skirt_dust_emission_pair(st.a, case["ncell"], st.lam, st.b, st.lam_b, st.mass, st.emission,
                                       st.temperature)
        return {"emission": st.emission, "temperature": st.temperature}
    if kind == "surrogate":
        r = S.skirt_dust_emission(st.a, st.a.shape[0], case["n_in"], st.lam, st.mass, S.EMIT_SURROGATE, st.net,
                                  st.emission, st.temperature)
        return {"emission": st.emission, "temperature": st.temperature, "n_fallback": int(r["n_fallback"])}
    # the same start for every pass: training goes on from the network's parameters
    st.net.set_params(st.params)
    hist = st.net.train(st.features, st.labels, case["rows"], epochs=case["epochs"], batch=case["batch"],
                        seed=st.seed)
    params, mean, std, lo, hi = st.net.get_params()
    return {"loss": hist, "params": params, "mean": mean, "std": std, "lo": lo, "hi": hi}


# -------------------------------------------------------------- what it cannot do without
# cell crossings per packet and cell along an axis, summed over the deposit, search and peel-off paths
# (measured with the ledger's counters), at roughly 12 operations each
_CROSSINGS = {"sphere": 8.0, "disk": 11.0, "torus": 10.0, "octree": 0.7, "reemit": 2.5}


def work(case):
    kind = case["kind"]
    if kind in ("trace", "reemit"):
        g = "reemit" if kind == "reemit" else case["grid"]
        nl = NOUT if kind == "reemit" else case["nlambda"]
        if g == "octree":
            ncell, side = _octree(case["n"]).ncell, 2 ** case["n"]
        else:
            ncell, side = case["n"] ** 3, case["n"]
        nins = 1 if g == "sphere" else 3
        out = ncell * nl + nins * case["npx"] ** 2 * nl
        read = ncell * 4 + (ncell * nl * 8 if kind == "reemit" else 0)
        return {"bytes": read + 8 * out, "flops": 12.0 * _CROSSINGS[g] * side * case["packets"]}
    if kind == "selfabs":
        n = case["n"] ** 3
        return {"bytes": n * (8 * case["n_in"] + 4 + 2 * 8 * 2 * NOUT),
                "flops": 2 * (n * 300 * 20.0 + 12.0 * 2.0 * case["n"] * case["packets"])}
    if kind == "exact":
        n = case["ncell"]
        nin = case["n_in"] + case["n_dust"]
        return {"bytes": n * (8.0 * nin + 4 + 8 * NOUT + 12), "flops": n * (6.0 * nin + 300 * 20.0)}
    if kind == "surrogate":
        n = float(case["n"] ** 3)
        return {"bytes": n * (8.0 * case["n_in"] + 4 + 8 * NOUT + 12),
                "flops": n * (case["n_in"] + 0.4 * 2 * (NBANDS * NHID + NHID * NHID + NHID * NOUT))}
    steps = (case["rows"] // case["batch"]) * case["epochs"]
    npar = NBANDS * NHID + NHID + NHID * NHID + NHID + NHID * NOUT + NOUT
    return {"bytes": case["rows"] * (4.0 * NBANDS + 8 * NOUT) + steps * case["batch"] * 4.0 * (NBANDS + NOUT),
            "flops": steps * (6.0 * npar * case["batch"])}


# ------------------------------------------------------------------- 64-bit values
def _band_index(lam):
    lam = np.asarray(lam, dtype=np.float64)
    b = np.floor(NBANDS * np.log(lam / lam[0]) / np.log(lam[-1] / lam[0])) if lam[-1] > lam[0] else np.zeros(lam.size)
    return torch.as_tensor(np.clip(b, 0, NBANDS - 1).astype(np.int64), device=DEV)


def _features64(a, lam, mass):
    idx = _band_index(lam)
    B = torch.zeros((a.shape[0], NBANDS), dtype=torch.float64, device=DEV).index_add_(1, idx, a)
    tot = B.sum(dim=1)
    M = mass.double()
    ok = (M > 0) & (tot > 0)
    x = torch.where(ok[:, None], torch.maximum(B, 1e-6 * tot[:, None] / NBANDS) / torch.where(ok, M, 1.0)[:, None], 0.0)
    return torch.log10(x.clamp_min(1e-30)), tot


def _model64():
    """Emission grid, terms a_l = hc/(k lambda_l) and K_il of the three grain populations."""
    lam = 10.0 ** (3.0 * np.arange(NOUT) / (NOUT - 1))
    d = np.diff(lam)
    wt = 0.5 * (np.concatenate([[0.0], d]) + np.concatenate([d, [0.0]]))
    hck = 6.62607015e-34 * 299792458.0 / 1.380649e-23 * 1e6
    K = np.stack([wt * (lam / 100.0) ** -b * lam ** -5.0 for b in (1.5, 2.0, 2.0)])
    return (torch.as_tensor(hck / lam, dtype=torch.float64, device=DEV),
            torch.as_tensor(K, dtype=torch.float64, device=DEV))


def _shares64(lam):
    lam = np.asarray(lam, dtype=np.float64)
    r = np.stack([(lam / 0.55) ** d for d in (-0.5, 0.0, 0.5)])
    return torch.as_tensor((r / r.sum(axis=0)).T.copy(), dtype=torch.float64, device=DEV)


def _lnG(a, Ki, y):
    """ln G_i and its derivative by ln T at y = ln T."""
    x = a[None, :] * torch.exp(-y)[:, None]
    q = 1.0 / torch.expm1(x)
    g = (Ki * q).sum(dim=1)
    return torch.log(g), (Ki * q * x * (1.0 + q)).sum(dim=1) / g


def _emission64(P, mass):
    """Emission rows and temperatures from the populations' powers [n, 3]."""
    a, K = _model64()
    n = P.shape[0]
    em = torch.zeros((n, NOUT), dtype=torch.float64, device=DEV)
    T = torch.zeros((n, 3), dtype=torch.float64, device=DEV)
    ylo, yhi = math.log(3.0), math.log(2000.0)
    grid = torch.linspace(ylo, yhi, 2049, dtype=torch.float64, device=DEV)
    for i in range(3):
        table, _ = _lnG(a, K[i], grid)
        lnc = -_lnG(a, K[i], torch.full((1,), math.log(30.0), dtype=torch.float64, device=DEV))[0]
        ok = (P[:, i] > 0) & (mass > 0)
        target = torch.log(torch.where(ok, P[:, i] / torch.where(ok, mass.double(), 1.0), 1.0)) - lnc
        k = torch.searchsorted(table, target).clamp(1, 2048)
        u = ((target - table[k - 1]) / (table[k] - table[k - 1])).clamp(0.0, 1.0)
        y = grid[k - 1] + u * (grid[k] - grid[k - 1])
        for _ in range(4):
            f, df = _lnG(a, K[i], y)
            y = (y + (target - f) / df).clamp(ylo, yhi)
        q = K[i] / torch.expm1(a[None, :] * torch.exp(-y)[:, None])
        em += torch.where(ok[:, None], q * (torch.where(ok, P[:, i], 0.0) / q.sum(dim=1))[:, None], 0.0)
        T[:, i] = torch.where(ok, torch.exp(y), 0.0)
    return em, T


def _exact_rows(a, lam, mass, b=None, lam_b=None, rows=1 << 17):
    n = a.shape[0]
    em = torch.empty((n, NOUT), dtype=torch.float64, device=DEV)
    T = torch.empty((n, 3), dtype=torch.float64, device=DEV)
    wa = _shares64(lam)
    wb = None if b is None else _shares64(lam_b)
    for k in range(0, n, rows):
        s = slice(k, min(n, k + rows))
        P = a[s] @ wa
        if b is not None:
            P = P + b[s] @ wb
        em[s], T[s] = _emission64(P, mass[s])
    return em, T


def _forward64(net, f):
    params, mean, std = (torch.as_tensor(v, dtype=torch.float64, device=DEV) for v in net[:3])
    h, o = (f - mean) / std, 0
    for rows, cols, last in ((NHID, NBANDS, False), (NHID, NHID, False), (NOUT, NHID, True)):
        w = params[o:o + rows * cols].view(rows, cols)
        o += rows * cols
        h = h @ w.T + params[o:o + rows]
        o += rows
        if not last:
            h = h * torch.sigmoid(h)
    return torch.softmax(h, dim=1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "exact":
        st = prepare(case, seed)
        em, T = _exact_rows(st.a, st.lam, st.mass, st.b, st.lam_b)
        return {"emission": em, "temperature": T}
    if kind == "surrogate":
        st = prepare(case, seed)
        n = st.a.shape[0]
        lo, hi = (torch.as_tensor(v, dtype=torch.float64, device=DEV) for v in st.host[3:5])
        em = torch.zeros((n, NOUT), dtype=torch.float64, device=DEV)
        T = torch.zeros((n, 3), dtype=torch.float64, device=DEV)
        for k in range(0, n, 1 << 18):
            s = slice(k, min(n, k + (1 << 18)))
            f, tot = _features64(st.a[s], st.lam, st.mass[s])
            em[s] = _forward64(st.host, f) * tot[:, None]
            share = 1.0 / (10.0 ** (f - f.max(dim=1, keepdim=True).values)).sum(dim=1)
            out = ((f < lo) | (f > hi)).any(dim=1) | (share > st.host[5])
            j = torch.nonzero(out & (tot > 0)).flatten() + k
            if j.numel():
                em[j], T[j] = _exact_rows(st.a[j], st.lam, st.mass[j])
        return {"emission": em, "temperature": T, "n_fallback": None}
    return None
