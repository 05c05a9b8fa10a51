"""The workloads that this framework's speed is judged by: what its users run, from a thousand
protons to a million nuclei, through the public entry points only.

  propagate  a batch of particles injected into one or more field realisations, advanced to its
             observer distance in either form, and the observer's records read back
  scenario   the structured-universe run: sources drawn on the device at density-weighted
             positions, a modulated field in a reflective box, records and an arrival map
  sky        Eq. 1 sources of a nearby volume: sampling, a short propagation, the arrival map and
             the rigidity-binned maps that a lens takes
  adjoint    arrival directions and the gradients of a loss of them, through the autograd function
             or through a handle that is kept
  lens       a lens applied to one set of rigidity-binned maps, or to many at once
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch
import torch.utils.checkpoint

import paper_1410_5323_gb300 as crp
from paper_1410_5323_gb300 import inputs as I
from paper_1410_5323_gb300.adjoint import Adjoint, PropagateAdjoint

TOL, HMIN, HMAX = 1e-4, I.KPC, I.MPC
SPECIES = {"H": (("H", 1.0),), "pFe": (("H", 0.5), ("Fe", 0.5)),
           "mix": (("H", 0.4), ("He", 0.3), ("N", 0.2), ("Fe", 0.1))}
ARRIVAL_EMIN = 10 ** 18.7


# ---- the cases ----------------------------------------------------------------------------
def propagate_case(form, grid, particles, species, energy, distance, *, store="f32", tables=False, n_grids=1,
                   b_lo=1.0, b_hi=1.0, cell_mpc=0.25, lmax=32, slice_steps=0, e_lo=18.0, e_hi=20.5):
    return {"kind": "propagate", "form": form, "grid": grid, "particles": particles, "species": species,
            "energy": energy, "e_lo": e_lo, "e_hi": e_hi, "distance_mpc": distance, "store": store, "tables": tables,
            "n_grids": n_grids, "b_lo_ng": b_lo, "b_hi_ng": b_hi, "cell_mpc": cell_mpc, "lmax": lmax,
            "slice_steps": slice_steps}


def listed():
    def named(name, case):
        return dict(case, name=name)

    return [
        # the plain FP64 configuration: a first look at a field, one small batch
        named("protons_fp64_64cube", propagate_case("fp64", 64, 1024, "H", "fixed", 100.0, e_lo=19.0)),
        # a nearby source (a few Mpc away) in a field whose size is no power of two
        named("nearby_fp64_100cube", propagate_case("fp64", 100, 30011, "H", "power", 4.0, e_lo=18.5, b_lo=0.3, b_hi=0.3)),
        # the FP64 form on nuclei with losses, photo-disintegration and secondaries: the reference-grade run
        named("nuclei_fp64_256cube", propagate_case("fp64", 256, 200_000, "mix", "power", 100.0, tables=True)),
        # the same in the precision form at production size
        named("nuclei_mixed_256cube", propagate_case("mixed", 256, 1_000_000, "mix", "power", 100.0, tables=True)),
        # protons and iron through a large grid stored as BF16 with one scale
        named("pfe_bf16_512cube", propagate_case("mixed", 512, 1_000_000, "pFe", "power", 100.0, store="bf16", b_lo=0.5,
                                                 b_hi=0.5, lmax=128)),
        # many field realisations in one simulation, step counts that differ by 1000x, the device-side slice loop
        named("batched_64x128cube", propagate_case("mixed", 128, 64 * 8000, "H", "log", 100.0, n_grids=64, b_lo=0.1,
                                                   b_hi=10.0, e_lo=17.0, slice_steps=4000)),
        # the structured-universe run with an arrival map
        named("scenario_220cube_x_128cube", {"kind": "scenario", "mod": 220, "grid": 128, "particles": 100_000,
                                             "distance_mpc": 50.0, "nside": 64}),
        # sky maps of sources in a nearby volume
        named("sky_1M_eq1_sources", {"kind": "sky", "grid": 128, "particles": 1_000_000, "distance_mpc": 1.0,
                                     "nside": 64, "bins": 24}),
        # one optimisation step over the field and the momenta: the differentiation workload
        named("adjoint_128cube_4k", {"kind": "adjoint", "grid": 128, "chains": 4096, "steps": 2000, "through": "autograd"}),
        # a small fit with a handle that is kept between steps
        named("adjoint_48cube_300", {"kind": "adjoint", "grid": 48, "chains": 300, "steps": 40, "through": "handle"}),
        # a full-resolution lens (49 152 pixels, 24 rigidity bins) on one set of maps
        named("lens_nside64_1map", {"kind": "lens", "nside": 64, "bins": 24, "entries": 24, "maps": 1}),
        # a coarse lens on the maps of ten source models: the smallest call
        named("lens_nside16_10maps", {"kind": "lens", "nside": 16, "bins": 12, "entries": 20, "maps": 10}),
    ]


# Attempted steps per Mpc of a 0.25 Mpc-cell Kolmogorov field (tolerance 1e-4, 1 kpc to 1 Mpc) against
# log10 of rigidity / B_rms in units of 10^18 V / nG: measured, and close to R^-0.4 in between.
ATT_LG = (-2.0, -1.5, -1.0, -0.5, 0.0, 0.5, 1.0, 1.5, 2.0, 2.5)
ATT_PER_MPC = (127.0, 42.7, 19.2, 12.8, 8.0, 4.8, 3.1, 2.0, 1.14, 1.0)


def attempts_per_mpc(lg_rigidity, b_ng, cell_mpc):
    lg = lg_rigidity - 18.0 - math.log10(b_ng) + 1.43 * math.log10(cell_mpc / 0.25)
    return float(np.exp(np.interp(lg, ATT_LG, np.log(ATT_PER_MPC))))


def energy_quantiles(case, n=24):
    """log10 of n equally likely energies."""
    q = (np.arange(n) + 0.5) / n
    if case["energy"] == "fixed":
        return np.full(1, case["e_lo"])
    if case["energy"] == "log":
        return case["e_lo"] + q * (case["e_hi"] - case["e_lo"])
    lo, hi = 10.0 ** -case["e_lo"], 10.0 ** -case["e_hi"]
    return -np.log10(lo + q * (hi - lo))


def attempts(case):
    """(attempted steps of the whole batch, of its longest trajectory), roughly."""
    if case["kind"] == "scenario":
        case = propagate_case("mixed", case["grid"], case["particles"], "mix", "power", case["distance_mpc"],
                              tables=True, cell_mpc=0.05)
    if case["kind"] == "sky":
        case = propagate_case("mixed", case["grid"], case["particles"], "H", "power", case["distance_mpc"])
    mean = longest = 0.0
    bs = np.exp(np.linspace(math.log(case["b_lo_ng"]), math.log(case["b_hi_ng"]), 5))
    names = SPECIES[case["species"]]
    for name, part in names:
        z = I.SPECIES[name][1]
        for b in bs:
            a = [attempts_per_mpc(lg - math.log10(z), b, case["cell_mpc"]) for lg in energy_quantiles(case)]
            mean += part * float(np.mean(a)) / len(bs)
            longest = max(longest, attempts_per_mpc(case["e_lo"] - math.log10(z), b, case["cell_mpc"]))
    return case["particles"] * case["distance_mpc"] * mean, case["distance_mpc"] * longest


def log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def even(v):
    return max(16, int(v) // 2 * 2)


def draw(rng):
    kind = rng.choice(["propagate", "propagate", "propagate", "scenario", "sky", "adjoint", "lens"])
    if kind == "propagate":
        form = rng.choice(["fp64", "mixed"])
        store = "bf16" if form == "mixed" and rng.random() < 0.3 else "f32"
        many = rng.random() < 0.25
        grid = rng.choice([32, 64, 128]) if rng.random() < 0.5 else even(log_int(rng, 24, 160))
        tables = rng.random() < 0.4
        species = "mix" if tables else rng.choice(["H", "pFe", "mix"])
        b = math.exp(rng.uniform(math.log(0.2), math.log(2.0)))
        c = propagate_case(form, grid, log_int(rng, 50, 1_000_000), species, rng.choice(["fixed", "power", "log"]),
                           round(math.exp(rng.uniform(math.log(1.0), math.log(200.0))), 2), store=store, tables=tables,
                           n_grids=rng.randint(2, 24) if many else 1, b_lo=round(b / 3 if many else b, 3),
                           b_hi=round(b * 3 if many else b, 3), lmax=rng.choice([8, 16, grid // 2]),
                           slice_steps=rng.choice([0, 0, 500, 4000]), e_lo=round(rng.uniform(18.0, 19.5), 2))
        # no dearer than the largest listed: the whole batch, then the longest trajectory
        most, chain = (1.0e8, 4500.0) if form == "fp64" else (8.0e8, 12000.0)
        if (long := attempts(c)[1]) > chain:
            c["distance_mpc"] = round(max(1.0, c["distance_mpc"] * chain / long), 2)
        if (all_ := attempts(c)[0]) > most:
            c["particles"] = max(50, int(c["particles"] * most / all_))
        return c
    if kind == "scenario":
        c = {"kind": "scenario", "mod": even(log_int(rng, 48, 220)), "grid": even(log_int(rng, 48, 160)),
             "particles": log_int(rng, 500, 100_000), "distance_mpc": round(rng.uniform(2.0, 50.0), 2),
             "nside": rng.choice([16, 32, 64])}
        return c
    if kind == "sky":
        return {"kind": "sky", "grid": even(log_int(rng, 32, 128)), "particles": log_int(rng, 200, 1_000_000),
                "distance_mpc": round(rng.uniform(0.5, 3.0), 2), "nside": rng.choice([8, 16, 32, 64, 128]),
                "bins": rng.randint(3, 30)}
    if kind == "adjoint":
        return {"kind": "adjoint", "grid": even(log_int(rng, 16, 128)), "chains": log_int(rng, 1, 4096),
                "steps": log_int(rng, 8, 2000), "through": rng.choice(["autograd", "handle"])}
    return {"kind": "lens", "nside": rng.choice([8, 16, 32, 64]), "bins": rng.randint(3, 24), "entries": rng.randint(6, 24),
            "maps": 1 if rng.random() < 0.4 else rng.choice([2, 3, 5, 8, 13, 16, 24])}


# ---- inputs -------------------------------------------------------------------------------
def generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) % (1 << 62) + 17)


def rand(n, g):
    return torch.rand(n, generator=g, device="cuda", dtype=torch.float64)


def directions(n, g):
    """Isotropic unit vectors, as three columns."""
    w = 2.0 * rand(n, g) - 1.0
    phi = 2.0 * math.pi * rand(n, g)
    s = torch.sqrt(1.0 - w * w)
    return s * torch.cos(phi), s * torch.sin(phi), w


def turbulent(n, lmax, b_ng, seed):
    return I.kolmogorov_grid_torch(n, 2.0, float(min(lmax, n // 2)), b_ng * I.NANOGAUSS, int(seed) % (1 << 31))


def field_of(grid, case, spacing):
    if case.get("store") == "bf16":
        q, scale = I.quantize_bf16(grid)
        return crp.Field(q, spacing, scale=scale)
    return crp.Field(grid, spacing)


def grids_of(case, seed):
    n = case["n_grids"]
    bs = np.exp(np.linspace(math.log(case["b_lo_ng"]), math.log(case["b_hi_ng"]), n))
    return [turbulent(case["grid"], case["lmax"], float(b), seed * 1009 + k) for k, b in enumerate(bs)]


def particles_of(case, seed):
    """Columns of the injected batch (device tensors): isotropic emission from the origin."""
    g, n = generator(seed), case["particles"]
    names = SPECIES[case["species"]]
    part = torch.tensor([p for _, p in names], dtype=torch.float64, device="cuda").cumsum(0)
    pick = torch.searchsorted(part / part[-1], rand(n, g)).clamp(max=len(names) - 1)
    az = torch.tensor([I.SPECIES[s] for s, _ in names], dtype=torch.int32, device="cuda")[pick]
    if case["energy"] == "fixed":
        E = torch.full((n,), 10.0 ** case["e_lo"], dtype=torch.float64, device="cuda")
    elif case["energy"] == "log":
        E = 10.0 ** (case["e_lo"] + (case["e_hi"] - case["e_lo"]) * rand(n, g))
    else:
        lo, hi = 10.0 ** -case["e_lo"], 10.0 ** -case["e_hi"]
        E = 1.0 / (lo + rand(n, g) * (hi - lo))
    zero = torch.zeros(n, dtype=torch.float64, device="cuda")
    gid = torch.arange(n, device="cuda", dtype=torch.int32) % case["n_grids"]
    return {"x": (zero, zero.clone(), zero.clone()), "u": directions(n, g), "E": E, "A": az[:, 0].contiguous(),
            "Z": az[:, 1].contiguous(), "uid": torch.arange(n, device="cuda"), "grid_id": gid}


@functools.lru_cache(maxsize=1)
def tables():
    return I.synthetic_tables()


@functools.lru_cache(maxsize=4)
def lens_arrays(nside, bins, entries):
    return I.synthetic_lens(nside, I.lens_edges(bins), seed=1, k=entries)


def density(n, seed):
    """Log-normal matter density [n, n, n] with power |k|^-2 on 2 to n/4 cells, mean 1."""
    g = generator(seed)
    F = torch.fft.rfftn(torch.randn((n, n, n), generator=g, device="cuda", dtype=torch.float32))
    k1 = torch.fft.fftfreq(n, 1.0 / n, device="cuda")
    kz = torch.fft.rfftfreq(n, 1.0 / n, device="cuda")
    k = torch.sqrt(k1.view(n, 1, 1) ** 2 + k1.view(1, n, 1) ** 2 + kz.view(1, 1, -1) ** 2)
    F *= torch.where((k >= 4.0) & (k <= n / 2), 1.0 / k.clamp(min=1.0), torch.zeros_like(k))
    G = torch.fft.irfftn(F, s=(n, n, n))
    rho = torch.exp(G / G.std())
    return rho / rho.mean()


def momenta_of(case, seed):
    """10^19.5 eV protons from random points of the box: x0, p0, Z."""
    g, n = generator(seed + 5), case["chains"]
    x0 = torch.stack([rand(n, g) for _ in range(3)], 1) * (case["grid"] * 0.25 * I.MPC)
    p0 = torch.stack(directions(n, g), 1) * 10 ** 19.5
    return x0, p0, torch.ones(n, dtype=torch.int32, device="cuda")


def prepare(case, seed):
    kind = case["kind"]
    if kind == "propagate":
        spacing = case["cell_mpc"] * I.MPC
        fields = [field_of(g, case, spacing) for g in grids_of(case, seed)]
        cols = particles_of(case, seed)
        room = case["particles"] * (12 if case["tables"] else 1)   # a nucleus of the mix has ten nucleons in the mean
        sim = crp.Simulation(fields, crp.Tables(tables()) if case["tables"] else None, seed=seed + 1, capacity=room)
        return {"case": case, "sim": sim, "cols": cols, "out": crp.Simulation.observe_buffers(room, device="cuda"), "rows": rows_of(case)}
    if kind == "scenario":
        n, spacing = case["mod"], 0.3 * I.MPC
        rho = density(n, seed)
        mod = rho ** (2.0 / 3.0)
        mod = mod / torch.sqrt(torch.mean(mod * mod))
        field = crp.Field(turbulent(case["grid"], 44, 1.0, seed), 0.05 * I.MPC).modulate(mod, spacing)
        g, m = generator(seed + 3), case["particles"]
        cell = torch.searchsorted(rho.flatten().double().cumsum(0), rand(m, g) * float(rho.double().sum())).clamp(max=n ** 3 - 1)
        ijk = (cell // (n * n), cell // n % n, cell % n)
        x = tuple((i.double() + rand(m, g)) * spacing for i in ijk)
        room = m * 20      # Eq. 1's composition above 10^18 eV is about a third iron
        sim = crp.Simulation(field, crp.Tables(tables()), seed=seed + 1, capacity=room)
        sim.set_boundary(((0.0, 0.0, 0.0), (n * spacing,) * 3))
        return {"case": case, "sim": sim, "x": x, "spectrum": crp.Spectrum.of(*I.EQ1_SPECTRUM),
                "out": crp.Simulation.observe_buffers(room, device="cuda"), "rows": rows_of(case)}
    if kind == "sky":
        n, m = case["grid"], case["particles"]
        g = generator(seed)
        sim = crp.Simulation(crp.Field(turbulent(n, 32, 1.0, seed), 0.25 * I.MPC), None, seed=seed + 1, capacity=m)
        npix = 12 * case["nside"] ** 2
        edges = I.lens_edges(case["bins"], 10 ** 17.5, 10 ** 20.5)
        rp = np.zeros((case["bins"], npix + 1), dtype=np.int64)
        lens = crp.Lens(npix, rp, np.zeros(0, np.int32), np.zeros(0, np.float32), edges)
        return {"case": case, "sim": sim, "x": tuple(rand(m, g) * (n * 0.25 * I.MPC) for _ in range(3)),
                "spectrum": crp.Spectrum.of(*I.EQ1_SPECTRUM), "lens": lens}
    if kind == "adjoint":
        grid = turbulent(case["grid"], 32, 1.0, seed)
        x0, p0, Z = momenta_of(case, seed)
        bar = torch.stack(directions(case["chains"], generator(seed + 9)), 1)
        st = {"case": case, "x0": x0, "Z": Z, "bar": bar}
        if case["through"] == "handle":
            st["field"] = crp.Field(grid, 0.25 * I.MPC)
            st["adj"] = Adjoint(st["field"], case["chains"], case["steps"])
            return dict(st, p0=p0)
        return dict(st, grid=grid.requires_grad_(), p0=p0.requires_grad_())
    rp, col, val = lens_arrays(case["nside"], case["bins"], case["entries"])
    g, npix = generator(seed), 12 * case["nside"] ** 2
    shape = (case["bins"], npix) if case["maps"] == 1 else (case["bins"], npix, case["maps"])
    x = torch.poisson(torch.full(shape, 3.0, dtype=torch.float64, device="cuda"), generator=g)
    return {"case": case, "lens": crp.Lens(npix, rp, col, val), "x": x}


# ---- one pass -----------------------------------------------------------------------------
def rows_of(case):
    """Rows of the record table: the primaries and as many secondaries as these flights release at most."""
    return case["particles"] if not case.get("tables", True) else 3 * case["particles"] + 200


def records(sim, out, rows):
    """The observer's records in order of particle id (they come in finishing order), as a table of a
    fixed number of rows, zero after the last record."""
    r = sim.observe(out=out)
    order = torch.argsort(r["uid"])
    n, table = len(order), {k: v.new_zeros(rows) for k, v in r.items()}
    for k, v in r.items():
        torch.index_select(v, 0, order, out=table[k][:n])
    return table


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "propagate":
        sim, c = state["sim"], state["cols"]
        form = crp.FORM_FP64 if case["form"] == "fp64" else crp.FORM_MIXED
        sim.reset()
        sim.inject(**c)
        if case["slice_steps"]:
            sim.propagate_loop(TOL, HMIN, HMAX, case["distance_mpc"] * I.MPC, max_steps=case["slice_steps"], form=form)
        else:
            sim.propagate(TOL, HMIN, HMAX, case["distance_mpc"] * I.MPC, form=form)
        sim.sync()
        return records(sim, state["out"], state["rows"])
    if kind == "scenario":
        sim = state["sim"]
        sim.reset()
        sim.sample_sources(state["spectrum"], state["x"])
        sim.propagate(TOL, HMIN, HMAX, case["distance_mpc"] * I.MPC, form=crp.FORM_MIXED)
        sim.sync()
        return {"map": sim.arrival_map(case["nside"], ARRIVAL_EMIN), "records": records(sim, state["out"], state["rows"])}
    if kind == "sky":
        sim = state["sim"]
        sim.reset()
        sim.sample_sources(state["spectrum"], state["x"])
        sim.propagate(TOL, HMIN, HMAX, case["distance_mpc"] * I.MPC, form=crp.FORM_MIXED)
        sim.sync()
        n = case["particles"]
        cols = {k: sim.read(k, 0, n, out=torch.empty(n, dtype=torch.int32 if k in "AZ" else torch.float64, device="cuda"))
                for k in ("A", "Z", "E", "ux", "uy", "uz")}
        return {"map": sim.arrival_map(case["nside"], ARRIVAL_EMIN), "bins": state["lens"].bin(sim, case["nside"], 1e18),
                "columns": cols}
    if kind == "adjoint":
        if case["through"] == "handle":
            xT, uT = state["adj"].forward(state["x0"], state["p0"], state["Z"], TOL, HMIN, HMAX)
            grid_bar, p0_bar, x0_bar = state["adj"].backward(state["bar"], (case["grid"],) * 3)
            return {"xT": xT, "uT": uT, "grid_bar": grid_bar, "p0_bar": p0_bar, "x0_bar": x0_bar}
        uT = PropagateAdjoint.apply(state["grid"], state["p0"], state["x0"], state["Z"], 0.25 * I.MPC, case["steps"], 64,
                                    TOL, HMIN, HMAX)
        grid_bar, p0_bar = torch.autograd.grad(uT, (state["grid"], state["p0"]), state["bar"])
        return {"uT": uT.detach(), "grid_bar": grid_bar, "p0_bar": p0_bar}
    return {"y": state["lens"].apply(state["x"])}


# ---- what a pass cannot do without --------------------------------------------------------
def work(case):
    kind = case["kind"]
    record, injected = crp.Simulation.observe_bytes(1), 76
    if kind == "propagate":
        nodes = case["n_grids"] * case["grid"] ** 3
        return {"bytes": nodes * (6 if case["store"] == "bf16" else 12) + case["particles"] * (injected + record),
                "flops": 950.0 * attempts(case)[0]}
    if kind == "scenario":
        return {"bytes": 12 * case["grid"] ** 3 + 4 * case["mod"] ** 3 + case["particles"] * (24 + record) + 96 * case["nside"] ** 2,
                "flops": 1150.0 * attempts(case)[0]}
    if kind == "sky":
        return {"bytes": 12 * case["grid"] ** 3 + case["particles"] * (24 + 40) + 96 * case["nside"] ** 2 * (1 + case["bins"]),
                "flops": 950.0 * attempts(case)[0] + 600.0 * case["particles"]}
    if kind == "adjoint":
        # 1.5 attempts a step recorded, the stages formed again, and their reverse
        return {"bytes": (12 + 12) * case["grid"] ** 3 + case["chains"] * (24 + 24 + 4 + 24 + 24 + 24),
                "flops": (1.5 * 950.0 + 2400.0) * case["chains"] * case["steps"]}
    npix = 12 * case["nside"] ** 2
    nnz = npix * case["bins"] * case["entries"]
    return {"bytes": 8 * nnz + 8 * case["maps"] * npix * (case["bins"] + 1), "flops": 2.0 * nnz * case["maps"]}


# ---- the same in plain torch, 64 bits -----------------------------------------------------
C_LIGHT = 299792458.0
CK_A = ((), (1 / 5,), (3 / 40, 9 / 40), (3 / 10, -9 / 10, 6 / 5), (-11 / 54, 5 / 2, -70 / 27, 35 / 27),
        (1631 / 55296, 175 / 512, 575 / 13824, 44275 / 110592, 253 / 4096))
CK_B = (37 / 378, 0.0, 250 / 621, 125 / 594, 0.0, 512 / 1771)
CK_BS = (2825 / 27648, 0.0, 18575 / 48384, 13525 / 55296, 277 / 14336, 1 / 4)


def lookup(grid, n, spacing, x, gid=None):
    """Trilinear periodic B at x [m, 3]; grid [fields * n^3, 3]."""
    r = x / spacing
    i0 = torch.floor(r)
    f = r - i0
    i0 = i0.long()
    i1 = torch.remainder(i0 + 1, n)
    i0 = torch.remainder(i0, n)
    base = 0 if gid is None else gid * n ** 3
    B = 0.0
    for a in (0, 1):
        for b in (0, 1):
            for c in (0, 1):
                ix, iy, iz = (i1 if q else i0 for q in (a, b, c))
                w = (f[:, 0] if a else 1 - f[:, 0]) * (f[:, 1] if b else 1 - f[:, 1]) * (f[:, 2] if c else 1 - f[:, 2])
                B = B + w[:, None] * grid[base + (ix[:, 0] * n + iy[:, 1]) * n + iz[:, 2]]
    return B


def stages(grid, n, spacing, kappa, x, u, h, gid=None):
    """The Cash-Karp stage derivatives (position and direction) of one step of size h."""
    kx, ku = [], []
    for row in CK_A:
        xs, us = x, u
        if row:
            xs = x + h[:, None] * sum(a * k for a, k in zip(row, kx))
            us = u + h[:, None] * sum(a * k for a, k in zip(row, ku))
        B = lookup(grid, n, spacing, xs, gid)
        kx.append(us)
        ku.append(kappa[:, None] * torch.linalg.cross(us, B))
    return kx, ku


def combine(cs, k):
    return sum(c * v for c, v in zip(cs, k) if c)


def controlled(grid, n, spacing, kappa, x, u, dmax=None, n_steps=None, gid=None):
    """Adaptive integration to a path length or for a number of accepted steps; returns x, u and the
    accepted steps (the latter with n_steps only)."""
    m = len(kappa)
    inf = torch.full((m,), math.inf, dtype=torch.float64, device=x.device)
    s, count, hprop = torch.zeros_like(inf), torch.zeros(m, dtype=torch.long, device=x.device), inf.clone()
    hs = torch.zeros((n_steps or 1, m), dtype=torch.float64, device=x.device)
    h, fresh, rejected, first, bid = inf.clone(), torch.ones(m, dtype=torch.bool, device=x.device), None, inf, inf
    rejected = torch.zeros_like(fresh)
    left = torch.arange(m, device=x.device)
    while len(left):
        at = left
        new_bid = hprop[at].clamp(HMIN, HMAX)
        start = new_bid if dmax is None else torch.minimum(new_bid, dmax - s[at])
        bid = bid.clone(); first = first.clone()
        bid[at] = torch.where(fresh[at], new_bid, bid[at])
        first[at] = torch.where(fresh[at], start, first[at])
        h[at] = torch.where(fresh[at], start, h[at])
        rejected[at] &= ~fresh[at]
        hh, xa, ua = h[at], x[at], u[at]
        kx, ku = stages(grid, n, spacing, kappa[at], xa, ua, hh, None if gid is None else gid[at])
        E = [b - bs for b, bs in zip(CK_B, CK_BS)]
        r = torch.maximum(torch.linalg.norm(combine(E, kx), dim=1), torch.linalg.norm(hh[:, None] * combine(E, ku), dim=1)) / TOL
        ok = (r <= 1.0) | (hh <= HMIN)
        bad, good = at[~ok], at[ok]
        h[bad] = torch.clamp(hh[~ok] * torch.clamp(0.95 * r[~ok] ** -0.25, 0.1, 1.0), min=HMIN)
        rejected[bad] = True
        x = x.index_copy(0, good, xa[ok] + hh[ok, None] * combine(CK_B, [k[ok] for k in kx]))
        u = u.index_copy(0, good, ua[ok] + hh[ok, None] * combine(CK_B, [k[ok] for k in ku]))
        grown = hh[ok] * torch.clamp(0.95 * r[ok] ** -0.2, 0.2, 5.0)
        keep = ~rejected[good] & (first[good] < bid[good])
        grown = torch.where(keep, torch.maximum(grown, bid[good]), grown)
        hprop[good] = grown.clamp(HMIN, HMAX)
        if dmax is None:
            hs[count[good], good] = hh[ok]
            done = count[good] + 1 >= n_steps
        else:
            done = hh[ok] == dmax - s[good]
        s[good] = s[good] + hh[ok]
        count[good] += 1
        fresh[at] = ok
        gone = torch.zeros(m, dtype=torch.bool, device=x.device)
        gone[good[done]] = True
        left = left[~gone[left]]
    return x, u, hs


def exact_propagate(case, seed):
    """Arrival positions, directions and energies of a short flight without interactions; beyond a few
    Mpc two valid integrations part by themselves (one e-fold per ~20 Mpc and less), and none is exact."""
    if case["tables"] or case["distance_mpc"] > (4.5 if case["form"] == "fp64" else 2.0):
        return None
    grids = grids_of(case, seed)
    if case["store"] == "bf16":
        grids = [q.double() * s for q, s in (I.quantize_bf16(g) for g in grids)]
    grid = torch.cat([g.double().reshape(-1, 3) for g in grids])
    c = particles_of(case, seed)
    kappa = c["Z"].double() * C_LIGHT / c["E"]
    u0 = torch.stack(c["u"], 1)
    x, u, _ = controlled(grid, case["grid"], case["cell_mpc"] * I.MPC, kappa, torch.stack(c["x"], 1), u0,
                         dmax=case["distance_mpc"] * I.MPC, gid=c["grid_id"].long())
    full = torch.full_like(c["E"], case["distance_mpc"] * I.MPC)
    got = {"E": c["E"], "s": full, "uid": None, "A": None, "Z": None, "n_int": None, "status": None, "n_steps": None,
           "n_att": None}
    for k, q in enumerate("xyz"):
        got[q], got["u" + q], got["u0" + q] = x[:, k], u[:, k], u0[:, k]
    return got


def exact_adjoint(case, seed):
    """The gradients by automatic differentiation of the frozen steps. The step sizes feed back on
    themselves through the error estimate: a difference of 10^-7 in one doubles every other step, and
    after some ten steps two valid sequences have parted and neither is exact."""
    if case["steps"] > 12:
        return None
    n, spacing = case["grid"], 0.25 * I.MPC
    grid = turbulent(n, 32, 1.0, seed).double().reshape(-1, 3)
    x0, p0, Z = momenta_of(case, seed)
    bar = torch.stack(directions(case["chains"], generator(seed + 9)), 1)
    E = torch.linalg.norm(p0, dim=1)
    _, _, hs = controlled(grid, n, spacing, Z.double() * C_LIGHT / E, x0, p0 / E[:, None], n_steps=case["steps"])
    gr, p, xs = grid.clone().requires_grad_(), p0.clone().requires_grad_(), x0.clone().requires_grad_()
    E = torch.linalg.norm(p, dim=1)
    kappa = Z.double() * C_LIGHT / E

    def some(x, u, gr, kappa, h):
        for hm in h:
            kx, ku = stages(gr, n, spacing, kappa, x, u, hm)
            x = x + hm[:, None] * combine(CK_B, kx)
            u = u + hm[:, None] * combine(CK_B, ku)
        return x, u

    x, u = xs, p / E[:, None]
    for m in range(0, case["steps"], 8):
        x, u = torch.utils.checkpoint.checkpoint(some, x, u, gr, kappa, hs[m:m + 8], use_reentrant=False)
    g_bar, p_bar, x_bar = torch.autograd.grad(u, (gr, p, xs), bar)
    g_bar = g_bar.reshape(n, n, n, 3)
    if case["through"] == "handle":
        return {"xT": x.detach(), "uT": u.detach(), "grid_bar": g_bar, "p0_bar": p_bar, "x0_bar": x_bar}
    return {"uT": u.detach(), "grid_bar": g_bar, "p0_bar": p_bar}


def exact(case, seed):
    if case["kind"] == "propagate":
        return exact_propagate(case, seed)
    if case["kind"] == "adjoint":
        return exact_adjoint(case, seed)
    if case["kind"] == "lens":
        rp, col, val = lens_arrays(case["nside"], case["bins"], case["entries"])
        x = prepare(case, seed)["x"]
        npix = 12 * case["nside"] ** 2
        x = x.reshape(case["bins"], npix, case["maps"])
        y = torch.zeros((npix, case["maps"]), dtype=torch.float64, device="cuda")
        for m in range(case["bins"]):
            rows = torch.from_numpy(np.repeat(np.arange(npix), np.diff(rp[m]))).cuda()
            lo, hi = int(rp[m, 0]), int(rp[m, -1])
            c = torch.from_numpy(col[lo:hi]).cuda().long()
            v = torch.from_numpy(val[lo:hi]).cuda().double()
            y.index_add_(0, rows, v[:, None] * x[m][c])
        return {"y": y[:, 0] if case["maps"] == 1 else y}
    return None   # sampled species, splits and counts: no closed value
