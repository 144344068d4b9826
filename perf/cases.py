"""Workloads of the library as its users run them, each one pass through the public entry points.

Model families (seeded stand-ins of the same shapes as ``synth``'s, grown on the GPU so that inputs are made quickly):

* clump: uniform background plus a Gaussian clump, refined around it, a point source in the centre;
* cloud: lognormal density from a random field with P(k) ~ k^-4, refined where dense, an isotropic external field;
* disc:  flared circumstellar disc refined towards the midplane and the star, a blackbody star and warm dust.

A case holds plain values only; ``prepare`` makes what a program has in hand before the call (grid, sources, optics, output
buffers, tables, captured batch), ``run`` is one pass: outputs zeroed (the entry points add to them), then the call.  The
tree follows from the case; the seed gives the densities on it and the packages' random streams.
"""
import math

import numpy as np
import torch

from paper_1206_3710_gb300 import rt, synth

DEV = "cuda:0"
_CTX = []


def _ctx():
    """One context per process, as a program keeps it."""
    if not _CTX:
        _CTX.append(rt.Context(0))
    return _CTX[0]


def listed():
    return [
        # a first look at a model: 16^3 root cells, one map; latency and launches count
        dict(name="clump_map", call="peel", model="clump", nx=16, ny=16, nz=16, levels=1, n_lambda=1, packets=100_000,
             precision=32, obs="axis1", n_pix=64, per_lambda=True),
        # the FP64 mode: reference runs beside which FP32 results are checked
        dict(name="clump_fp64", call="peel", model="clump", nx=32, ny=32, nz=32, levels=2, n_lambda=4, packets=25_000,
             precision=64, obs="oblique1", n_pix=64, per_lambda=True),
        # a survey run on an odd box: external field and an embedded star, absorbed energy summed over the bins
        dict(name="ragged_trace", call="trace", model="cloud", nx=100, ny=75, nz=61, levels=2, scale=1.0, n_lambda=7,
             packets=150_001, precision=32, per_lambda=False, star=True),
        # heating of a cloud whose cells fit the L2: absorbed energy per wavelength
        dict(name="cloud128_trace", call="trace", model="cloud", nx=128, ny=128, nz=128, levels=3, scale=1.0, n_lambda=20,
             packets=200_000, precision=32, per_lambda=True, star=False),
        # the headline step: 256^3 root cells, three levels, absorbed energy, six maps, temperatures
        dict(name="cloud256_step", call="step", model="cloud", nx=256, ny=256, nz=256, levels=3, scale=1.0, n_lambda=20,
             packets=2_000_000, precision=32, obs="axis6", n_pix=256, per_lambda=True, star=False),
        # deeply refined cloud (8 % of the uniform cells) seen from directions off the axes
        dict(name="deep_maps", call="peel", model="cloud", nx=64, ny=64, nz=64, levels=3, scale=0.067, n_lambda=5,
             packets=200_000, precision=32, obs="oblique3", n_pix=129, per_lambda=True, star=False),
        # maps with precomputed extinction tables
        dict(name="maps_tables", call="tables", model="cloud", nx=96, ny=96, nz=96, levels=2, scale=1.0, n_lambda=5,
             packets=400_000, precision=32, obs="axis6", n_pix=96, per_lambda=True, star=False),
        # one dust re-emission trace on the full disc: emission, packages per cell, tracing
        dict(name="disc_dust", call="dust", model="disc", n_root=64, levels=10, thr=15.4, n_lambda=30, packets=10_000_000,
             precision=32),
        # the Lambda iteration on a medium disc
        dict(name="disc_lambda", call="lambda", model="disc", n_root=32, levels=8, thr=11.5, n_lambda=30,
             packets=1_000_000, steps=4, precision=32),
        # subiterations with the accelerated operator on a small disc
        dict(name="disc_subiter", call="subiter", model="disc", n_root=16, levels=6, thr=13.3, n_lambda=12,
             packets=200_000, steps=6, precision=32),
        # the dust solve alone: temperatures from absorbed energy, then emission per cell and bin
        dict(name="dust_solve", call="dust_solve", model="cloud", nx=128, ny=128, nz=128, levels=3, scale=1.0,
             n_lambda=20),
        # many small models in one captured launch
        dict(name="batch16", call="batch", models=16, n_lambda=16, packets=20_000, precision=32),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["clump", "cloud", "cloud", "cloud", "disc", "dust_solve", "batch"])
    if kind == "clump":
        n = rng.randint(12, 48)
        return dict(call="peel", model="clump", nx=n, ny=n, nz=n, levels=rng.randint(0, 3), n_lambda=rng.randint(1, 6),
                    packets=log(10_000, 200_000), precision=rng.choice([32, 32, 64]),
                    obs=rng.choice(["axis1", "axis6", "oblique1", "oblique3"]), n_pix=rng.randint(32, 160),
                    per_lambda=rng.random() < 0.5)
    if kind in ("cloud", "dust_solve"):
        scale = rng.choice([1.0, 1.0, 0.25, 0.067])
        top = {1.0: 200, 0.25: 110, 0.067: 64}[scale]
        c = dict(call="dust_solve", model="cloud", nx=log(24, top), ny=log(24, top), nz=log(24, top),
                 levels=rng.randint(0, 3), scale=scale, n_lambda=rng.randint(1, 24))
        if kind == "cloud":
            c.update(call=rng.choice(["trace", "trace", "peel", "tables", "step"]), packets=log(5_000, 500_000),
                     precision=rng.choice([32, 32, 32, 64]), per_lambda=rng.random() < 0.7, star=rng.random() < 0.3)
            if c["precision"] == 64:
                c["packets"] = min(c["packets"], 20_000)
            if c["call"] == "trace":
                c["option"] = rng.choice(["", "", "analog", "poly", "split"])
            else:
                c.update(obs=rng.choice(["axis1", "axis6", "oblique1", "oblique3"]), n_pix=rng.randint(32, 256))
        return c
    if kind == "disc":
        return dict(call=rng.choice(["dust", "lambda", "subiter"]), model="disc", n_root=rng.choice([16, 24, 32]),
                    levels=rng.randint(4, 8), thr=round(math.exp(rng.uniform(math.log(11.0), math.log(200.0))), 3),
                    n_lambda=rng.randint(6, 30), packets=log(50_000, 1_000_000), steps=rng.randint(2, 5),
                    precision=rng.choice([32, 32, 64]))
    return dict(call="batch", models=rng.randint(2, 24), n_lambda=rng.randint(4, 16), packets=log(2_000, 30_000),
                precision=32)


# ----------------------------------------------------------------------------------------------------------------------
# models
# ----------------------------------------------------------------------------------------------------------------------
RHO_UNIT = 70.0 * 2.8 * synth.MH_G   # n(H2) = 70 cm^-3
SIGMA = 1.5
FIELD_ERG = 2.0e36                   # erg/s entering a 2 pc box: grains of 10 to 20 K


def _rng(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _grow(root, h0, max_level, rho_fn, refine_fn, seed):
    """Level-ordered tree description (see ``synth.grow_tree``), built with torch; the seed roughens the densities."""
    rx, ry, rz = root
    i = torch.arange(rx * ry * rz, device=DEV)
    c = torch.stack([i % rx, (i // rx) % ry, i // (rx * ry)])
    octant = torch.arange(8, device=DEV)
    octant = torch.stack([octant & 1, (octant >> 1) & 1, octant >> 2])
    flags, dens, n_ref = [], [], []
    for lev in range(max_level + 1):
        rho = rho_fn(lev, c)
        f = refine_fn(lev, c, rho) if lev < max_level else torch.zeros(rho.numel(), dtype=torch.bool, device=DEV)
        flags.append(f.to(torch.uint8))
        dens.append(rho)
        n_ref.append(int(f.sum()))
        if n_ref[-1] == 0:
            break
        c = (2 * c[:, f, None] + octant[:, None, :]).reshape(3, -1)
    rho = torch.cat(dens)
    rho *= torch.exp(0.1 * torch.randn(rho.numel(), generator=_rng(seed), device=DEV, dtype=torch.float64))
    return synth.TreeDesc(root=tuple(root), box=tuple(n * h0 for n in root), n_refined=np.asarray(n_ref, dtype=np.int64),
                          refine_flags=torch.cat(flags).cpu().numpy(), density=rho.cpu().numpy())


def _cloud_tree(nx, ny, nz, levels, scale, seed):
    white = torch.randn((nz, ny, nx), generator=_rng(1002), device=DEV, dtype=torch.float64)
    k2 = (torch.fft.fftfreq(nz, device=DEV, dtype=torch.float64)[:, None, None] ** 2
          + torch.fft.fftfreq(ny, device=DEV, dtype=torch.float64)[None, :, None] ** 2
          + torch.fft.rfftfreq(nx, device=DEV, dtype=torch.float64)[None, None, :] ** 2)
    k2[0, 0, 0] = 1.0
    amp = 1.0 / k2
    amp[0, 0, 0] = 0.0
    g = torch.fft.irfftn(torch.fft.rfftn(white) * amp, s=(nz, ny, nx))
    g = ((g - g.mean()) / g.std()).reshape(-1)

    def rho_fn(lev, c):
        if lev == 0:
            v = g
        else:
            v = torch.zeros(c.shape[1], dtype=torch.float64, device=DEV)
            q = (c.to(torch.float64) + 0.5) * 0.5 ** lev - 0.5
            lo = torch.floor(q)
            w = q - lo
            lo = lo.to(torch.int64)
            for o in range(8):
                b = (o & 1, (o >> 1) & 1, o >> 2)
                ix, iy, iz = ((lo[a] + b[a]) % (nx, ny, nz)[a] for a in range(3))
                wt = 1.0
                for a in range(3):
                    wt = wt * (w[a] if b[a] else 1.0 - w[a])
                v += wt * g[ix + nx * (iy + ny * iz)]
        return RHO_UNIT * torch.exp(SIGMA * v - 0.5 * SIGMA * SIGMA)

    return _grow((nx, ny, nz), 2.0 * synth.PC_CM / max(nx, ny, nz), levels, rho_fn,
                 lambda lev, c, rho: rho > scale * 4.0 ** (lev + 1) * RHO_UNIT, seed)


def _clump_tree(n, levels, seed):
    L, bg = synth.PC_CM, 1.0e-21

    def rho_fn(lev, c):
        x = (c.to(torch.float64) + 0.5) / (n << lev) - 0.5
        return bg * (1.0 + 100.0 * torch.exp(-(x * x).sum(0) / (2.0 * 0.1 ** 2)))

    return _grow((n,) * 3, L / n, levels, rho_fn, lambda lev, c, rho: rho > 2.0 * 2.57 * bg * 4.0 ** lev, seed)


def _disc_tree(n, levels, thr, seed):
    L = 600.0 * synth.AU_CM
    integral = (0.1 ** -1.25 - 300.0 ** -1.25) / 1.25
    rho0 = 1.0e5 / (integral * synth.AU_CM)          # midplane optical depth 1e5 at 1 um (kappa 1 cm^2/g)

    def at(p):
        r = torch.sqrt(p[0] ** 2 + p[1] ** 2) / synth.AU_CM
        h = 0.05 * r.clamp_min(1e-30) ** 1.125 * synth.AU_CM
        rho = rho0 * r.clamp_min(1e-30) ** -2.25 * torch.exp(-0.5 * (p[2] / h) ** 2)
        return torch.where((r >= 0.1) & (r <= 300.0), rho, torch.zeros_like(rho))

    def rho_fn(lev, c):
        h = L / (n << lev)
        return at((c.to(torch.float64) + 0.5) * h - 0.5 * L)

    def refine_fn(lev, c, rho):
        h = L / (n << lev)
        top = rho
        for o in range(8):
            corner = torch.tensor([o & 1, (o >> 1) & 1, o >> 2], device=DEV)[:, None]
            top = torch.maximum(top, at((c + corner).to(torch.float64) * h - 0.5 * L))
        return (top * h > thr) | (c == (n << lev) // 2).all(0)

    return _grow((n,) * 3, L / n, levels, rho_fn, refine_fn, seed)


class _Star:
    kind = "point"

    def __init__(self, energy, pos):
        self.bin_energy, self.pos = energy, pos


def _field(n_lambda):
    return synth.Source("external", bin_energy=np.full(n_lambda, FIELD_ERG / n_lambda))


def _observers(kind, n_pix, box):
    fov = max(box)
    if kind == "axis6":
        return synth.axis_observers(n_pix, fov, "all6")
    if kind == "axis1":
        return synth.axis_observers(n_pix, fov, "+z")
    d = np.array([[0.36, 0.48, 0.8], [-0.6, 0.64, 0.48], [0.8, -0.36, -0.48]][:int(kind[-1])])
    return synth.Observers(dirs=d, ups=np.array([[0.0, 0.0, 1.0]] * len(d)), nx=n_pix, ny=max(1, n_pix * 3 // 4),
                           fov=(1.2 * fov, 0.9 * fov))


def _model(case, seed):
    """(tree, optics, sources) of a case."""
    nl = case["n_lambda"]
    lam = synth.log_lambda_grid(nl)
    if case["model"] == "clump":
        tree = _clump_tree(case["nx"], case["levels"], seed)
        L = tree.box[0]
        tau1 = 1.0e-21 * L * (0.5 + 100.0 * 0.1 * math.sqrt(math.pi / 2))   # centre to face, per cm^2/g
        return tree, synth.powerlaw_dust(lam, 1.0 / tau1, 0.55), [_Star(np.full(nl, 1.0e36 / nl), (0.5 * L,) * 3)]
    if case["model"] == "disc":
        tree = _disc_tree(case["n_root"], case["levels"], case["thr"], seed)
        star = _Star(synth.blackbody_star_bins(lam, 4000.0, 2.0 * synth.RSUN_CM), (0.5 * tree.box[0],) * 3)
        return tree, synth.powerlaw_dust(lam, 1.0, 1.0), [star]
    tree = _cloud_tree(case["nx"], case["ny"], case["nz"], case["levels"], case["scale"], seed)
    src = [_field(nl)]
    if case.get("star"):
        src.append(_Star(np.full(nl, 1.0e36 / nl), tuple(0.45 * b for b in tree.box)))
    return tree, synth.powerlaw_dust(lam, 0.4 / (RHO_UNIT * max(tree.box)), 0.55), src


def _dust(optics):
    return optics.lambda_um, (1.0 - optics.albedo) * optics.kappa_ext, optics.dnu


def _leaves(tree):
    """(leaf mask, mass per cell) on the device."""
    leaf = torch.from_numpy(tree.refine_flags == 0).to(DEV)
    h = tree.box[0] / tree.root[0] * 0.5 ** torch.from_numpy(tree.cell_levels().astype(np.float64)).to(DEV)
    return leaf, torch.from_numpy(tree.density).to(DEV) * h ** 3


def _emission(T, mass, lam, kabs, dnu):
    """4 pi rho V kappa B_nu(T) dnu per bin and cell, 64 bits."""
    nu = torch.tensor(synth.C_CGS / (np.asarray(lam) * synth.MICRON_CM), device=DEV, dtype=torch.float64)
    pre = torch.tensor(4.0 * math.pi * np.asarray(kabs) * np.asarray(dnu), device=DEV, dtype=torch.float64)
    for b in range(nu.numel()):
        x = synth.H_CGS * nu[b] / (synth.K_CGS * T)
        yield mass * pre[b] * (2.0 * synth.H_CGS * nu[b] ** 3 / synth.C_CGS ** 2) / torch.expm1(x)


def _solve_inputs(case, seed):
    """What the dust solve is given: the tree, its dust, temperatures of the grains and the energy they absorb per bin."""
    tree, optics, _ = _model(case, seed)
    dust = _dust(optics)
    leaf, mass = _leaves(tree)
    gen = _rng(seed + 1)
    T = torch.exp(torch.empty(tree.n_cells, device=DEV, dtype=torch.float64).uniform_(math.log(6.0), math.log(180.0), generator=gen))
    T = torch.where(leaf, T, torch.zeros_like(T))
    total = torch.zeros_like(T)
    for e in _emission(torch.where(leaf, T, torch.ones_like(T)), mass, *dust):
        total += e
    share = torch.rand((case["n_lambda"], tree.n_cells), generator=gen, device=DEV, dtype=torch.float64) + 0.05
    share *= torch.where(leaf, total, torch.zeros_like(total)) / share.sum(0)
    return tree, dust, leaf, mass, T, share


# ----------------------------------------------------------------------------------------------------------------------
# prepare / run
# ----------------------------------------------------------------------------------------------------------------------
def prepare(case, seed):
    ctx, call = _ctx(), case["call"]
    if call == "batch":
        rng = np.random.default_rng(1004)
        jobs = []
        for m in range(case["models"]):
            n, levels = int(rng.choice([24, 32, 48, 64])), int(rng.integers(0, 4))
            c = dict(model="clump" if m % 2 == 0 else "cloud", nx=n, ny=n, nz=n, levels=levels, scale=1.0,
                     n_lambda=case["n_lambda"])
            tree, optics, src = _model(c, 64 * seed + m)
            out = torch.zeros((case["n_lambda"], tree.n_cells), dtype=torch.float64, device=DEV)
            jobs.append(rt.Job(rt.Grid(ctx, tree), src, optics, absorbed=out, seed=seed, job=m,
                               precision=case["precision"], packets_per_bin=int(case["packets"] * rng.uniform(0.2, 3.0)),
                               rr_wmin=1e-4, rr_p=0.9))
        return dict(call=call, batch=rt.Batch(ctx, jobs), jobs=jobs)
    if call == "dust_solve":
        tree, dust, _, _, T, absorbed = _solve_inputs(case, seed)
        return dict(call=call, ctx=ctx, grid=rt.Grid(ctx, tree), dust=dust, T_in=T, absorbed=absorbed,
                    T=torch.zeros_like(T), emission=torch.empty_like(absorbed))
    tree, optics, src = _model(case, seed)
    grid = rt.Grid(ctx, tree)
    nl, n = case["n_lambda"], grid.n_cells
    bins = nl if case.get("per_lambda") else 1
    prm = dict(seed=seed, precision=case["precision"], rr_wmin=1e-4, rr_p=0.9)
    s = dict(call=call, ctx=ctx, grid=grid, optics=optics, src=src, prm=prm, T=torch.zeros(n, dtype=torch.float64, device=DEV))
    if call in ("lambda", "subiter"):
        prm.update(packets_total=case["packets"], dust_packets_total=case["packets"], min_hits=100.0, tol=0.0)
        s["steps"] = case["steps"]
        return s
    if call == "dust":
        # warm dust: T falls outwards as in an irradiated disc
        gen = _rng(seed + 1)
        leaf, mass = _leaves(tree)
        T = 8.0 + 60.0 * torch.rand(n, generator=gen, device=DEV, dtype=torch.float64)
        T = torch.where(leaf & (mass > 0), T, torch.zeros_like(T))
        s["src"] = [rt.DustSource(T, *_dust(optics))]
        prm.update(packets_total=case["packets"], per_lambda=False)
        s["absorbed"] = torch.zeros((1, n), dtype=torch.float64, device=DEV)
        return s
    prm.update(packets_per_bin=case["packets"], per_lambda=case["per_lambda"])
    option = case.get("option", "")
    if option == "analog":
        prm.update(estimator=rt.RT_EST_ANALOG, rr_wmin=0.0)
    elif option == "poly":
        prm.update(poly_group=4)
    elif option == "split":
        prm.update(split_factor=2, split_max_level=2)
    s["absorbed"] = torch.zeros((bins, n), dtype=torch.float64, device=DEV)
    if call != "trace":
        ob = _observers(case["obs"], case["n_pix"], tree.box)
        s["obs"] = ob
        s["images"] = torch.zeros((ob.n_obs, bins, ob.ny, ob.nx), dtype=torch.float64, device=DEV)
        if call == "tables":
            s["tables"] = rt.PeelTables(ctx, grid, ob, 16, 8)
        s["dust"] = _dust(optics)
        s["bins"] = bins
    return s


_ENERGIES = ["emitted", "absorbed", "escaped", "rr_gain", "rr_loss", "killed", "peeled"]
_COUNTS = ["n_packets", "n_cross", "n_scatter", "n_peel_cross", "n_killed", "n_peel_out"]


def _ledger(led):
    return dict(energies=np.array([led[k] for k in _ENERGIES]), counts=np.array([led[k] for k in _COUNTS], dtype=np.int64))


def run(s):
    call = s["call"]
    if call == "batch":
        leds = s["batch"].run()   # the captured graph zeroes the outputs itself
        return dict(absorbed=[j.absorbed for j in s["jobs"]],
                    counts=np.array([[led[k] for k in _COUNTS] for led in leds], dtype=np.int64))
    if call == "dust_solve":
        lam, kabs, dnu = s["dust"]
        rt.rt_dust_temperature(s["ctx"], s["grid"], s["absorbed"], int(s["absorbed"].shape[0]), lam, kabs, dnu, s["T"])
        totals = rt.rt_dust_emission(s["ctx"], s["grid"], s["T_in"], lam, kabs, dnu, s["emission"])
        return dict(T=s["T"], emission=s["emission"], totals=totals)
    if call == "lambda":
        r = rt.rt_lambda_iterate(s["ctx"], s["grid"], s["src"], s["optics"], s["T"], max_iter=s["steps"], **s["prm"])
        return dict(T=s["T"], history=np.array(r["history"]))
    if call == "subiter":
        r = rt.rt_lambda_subiterate(s["ctx"], s["grid"], s["src"], s["optics"], s["T"], sub_level=1,
                                    schedule=["full" if i % 3 == 0 else "sub" for i in range(s["steps"])], ali=True,
                                    **s["prm"])
        return dict(T=s["T"], history=np.array(r["history"]), imbalance=np.array(r["imbalance"]))
    s["absorbed"].zero_()
    if call in ("trace", "dust"):
        return dict(absorbed=s["absorbed"],
                    ledger=_ledger(rt.rt_trace(s["ctx"], s["grid"], s["src"], s["optics"], s["absorbed"], **s["prm"])))
    s["images"].zero_()
    if call == "tables":
        led = rt.rt_peel_tabulated(s["ctx"], s["grid"], s["src"], s["optics"], s["obs"], s["tables"], s["images"],
                                   s["absorbed"], **s["prm"])
    else:
        led = rt.rt_peel(s["ctx"], s["grid"], s["src"], s["optics"], s["obs"], s["images"], s["absorbed"], **s["prm"])
    out = dict(absorbed=s["absorbed"], images=s["images"], ledger=_ledger(led))
    if call == "step":
        rt.rt_dust_temperature(s["ctx"], s["grid"], s["absorbed"], s["bins"], *s["dust"], s["T"])
        out["T"] = s["T"]
    return out


# ----------------------------------------------------------------------------------------------------------------------
# exact / work
# ----------------------------------------------------------------------------------------------------------------------
def exact(case, seed):
    """The dust solve in 64 bits by bisection.  The traced fields are sums over random histories: no closed value."""
    if case["call"] != "dust_solve":
        return None
    _, dust, leaf, mass, T_in, absorbed = _solve_inputs(case, seed)
    emission = torch.stack(list(_emission(torch.where(leaf, T_in, torch.ones_like(T_in)), mass, *dust)))
    emission *= leaf
    A = absorbed.sum(0)
    lo = torch.full_like(T_in, math.log(2.7))
    hi = torch.full_like(T_in, math.log(3000.0))
    for _ in range(56):
        mid = 0.5 * (lo + hi)
        e = torch.zeros_like(A)
        for v in _emission(torch.exp(mid), mass, *dust):
            e += v
        low = e < A
        lo, hi = torch.where(low, mid, lo), torch.where(low, hi, mid)
    T = torch.where(leaf, torch.exp(0.5 * (lo + hi)), torch.zeros_like(lo))
    return dict(T=T, emission=emission, totals=emission.sum(1))


def _cells(case):
    """Expected number of cells and crossings per unit root length (relative), from the density's distribution."""
    if case.get("model") == "disc":
        n0 = case["n_root"] ** 3
        return n0 + 1.5e8 / case["thr"] * min(1.0, 4.0 ** (case["levels"] + math.log2(case["n_root"] / 16.0) - 12)), 1.0
    n0 = case["nx"] * case["ny"] * case["nz"]
    cells, dense, share = float(n0), 1.0, 1.0
    for lev in range(case["levels"]):
        if case["model"] == "clump":
            p = 0.03 * 0.5 ** lev
        else:
            p = 0.5 * math.erfc((math.log(case["scale"] * 4.0 ** (lev + 1)) + 0.5 * SIGMA ** 2) / SIGMA / math.sqrt(2.0))
        share = min(share, p)
        cells += n0 * 8.0 ** (lev + 1) * share
        dense += share * 2.0 ** lev
    return cells, dense


def work(case):
    """Bytes: the node words read once and the outputs written once.  Operations: about 30 per cell crossing of a package
    and 4 per crossing of a peel-off march, with the mean number of crossings expected from the geometry."""
    call = case["call"]
    if call == "batch":
        cells = case["models"] * 1.2e5
        packets = case["models"] * 1.6 * case["packets"] * case["n_lambda"]
        return dict(bytes=cells * (4 + 8 * case["n_lambda"]), flops=packets * 35.0 * 30)
    cells, dense = _cells(case)
    nl = case["n_lambda"]
    if call == "dust_solve":
        # temperatures: absorbed energy read, T written; emission: T read, a value per bin written; 40 per Planck term
        return dict(bytes=cells * (8.0 * nl + 8 + 8 + 8.0 * nl + 2 * 13), flops=cells * nl * 40.0 + cells * 60.0)
    if case["model"] == "disc":
        n = case["packets"] * (1 if call == "dust" else 1 + case["steps"])
        steps = 1 if call == "dust" else case["steps"]
        return dict(bytes=steps * cells * (8 + 13 + 4 + 8.0), flops=n * 30.0 * 30 + steps * cells * nl * 40.0)
    n3 = (case["nx"], case["ny"], case["nz"])
    area = 2.0 * (n3[0] * n3[1] + n3[1] * n3[2] + n3[0] * n3[2])
    chord = 4.0 * n3[0] * n3[1] * n3[2] / area if case["model"] == "cloud" else 0.5 * n3[0]
    packets = case["packets"] * nl * (2 if case.get("star") else 1)
    bins = nl if case["per_lambda"] else 1
    out = 8.0 * cells * bins
    flops = packets * 1.5 * chord * dense * 30
    if "obs" in case:
        n_obs = int(case["obs"][-1])
        out += 8.0 * n_obs * bins * case["n_pix"] ** 2
        flops += packets * 0.24 * n_obs * 0.5 * max(n3) * dense * 4
    return dict(bytes=4.0 * cells + out, flops=flops)
