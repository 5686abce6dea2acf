"""The measured work: calls a user's program makes through the public entry
points, over the sizes the repository's own workloads, tests and bench use.

`prepare` makes what a program has in hand before a call (line lists, cells,
ray sets, coefficient tables, contexts), `run` is one such call and its
outputs, `exact` the same outputs in 64 bits from plain torch.

Line lists and cell states come from the seeded generators of `synth`; the
coefficient tables of the march cases are drawn here (lognormal spectra, about
a percent of the columns optically thick over the whole path, emission
kappa times a Planck function), so that they do not depend on the code that
is measured.

The results of the FP32 path are returned in 32 bits, the wall flux among
them: it is summed in 64 bits, but from 32-bit spectra.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2604_11856_gb300 import rapral as R
from paper_2604_11856_gb300 import solver, synth

KB, CL, H, ME, QE = 1.380e-16, 2.998e10, 6.626e-27, 9.109e-28, 4.803e-10   # printed constants, cgs
C2 = H * CL / KB
N_A = 6.022e23
E_H = 109678.77


# ---------------------------------------------------------------- the cases

def listed():
    return [
        # one small request, start to finish: the uniform slab of the tests and the bench at the low end
        # of its grid; launches, the planning read-back and host work decide it
        dict(name="solve_slab_small", do="solve", precision=32, gas="uniform", cells=20, atomic=1500, molecular=0,
             points=20_001),
        # the stagnation-line step at full size (200 cells, 1e6 points, 320k lines): one whole FP32 solve
        dict(name="solve_stagnation", do="solve", precision=32, gas="stagnation", cells=200, atomic=20_000,
             molecular=300_000, points=1_000_000),
        # the loop body of the afterbody solve (coefficients, march, flux of one spectral chunk; populations
        # done) on its full mesh, points and rays, over a part of a chunk
        dict(name="chunk_afterbody", do="chunk", nx=400, nr=200, surface=200, n_mu=16, n_phi=32, atomic=20_000,
             molecular=300_000, points=1_000_000, k0=131_072, nk=4096),
        # coefficients of an ordinary chunk of the stagnation line (the autotuner's sample: 48 cells)
        dict(name="coeffs_chunk", do="coeffs", precision=32, broad=False, cells=48, atomic=20_000, molecular=300_000,
             points=1_000_000, k0=196_608, nk=65_536),
        # the default precision of solver.solve, on a ragged range of a test-sized problem
        dict(name="coeffs_fp64", do="coeffs", precision=64, broad=False, cells=24, atomic=4000, molecular=60_000,
             points=200_001, k0=30_001, nk=50_001),
        # the paper's full Lorentz width (Stark from the ionisation gap, resonance, van der Waals)
        dict(name="coeffs_full_lorentz", do="coeffs", precision=32, broad=True, cells=96, atomic=20_000,
             molecular=60_000, points=500_000, k0=20_000, nk=100_001),
        # the tangent slab of the stagnation line: 16 directions and the normal ray
        dict(name="march_slab", do="march_slab", precision=32, cells=200, n_mu=16, points=1_000_000, k0=0,
             nk=262_144, wall=False),
        # lines of sight of a reduced afterbody (the profiles' 100 x 50 mesh), 512 rays a point
        dict(name="march_afterbody", do="march_axisym", precision=32, nx=100, nr=50, surface=20, n_mu=16, n_phi=32,
             points=1_000_000, k0=65_536, nk=16_384),
        # the default precision of solver.solve: a slab of many directions from a hot wall, odd sizes
        dict(name="march_slab_fp64", do="march_slab", precision=64, cells=61, n_mu=24, points=100_001, k0=0,
             nk=100_001, wall=True),
        # partition functions of a field of cells with the whole level database
        dict(name="populations", do="populations", cells=5000, atomic=20_000, molecular=300_000),
        # the atomic continuum of N and O (100 levels each) added to a chunk of the stagnation line
        dict(name="continuum", do="continuum", precision=32, cells=200, levels=100, points=1_000_000, k0=0,
             nk=250_000),
        # collisional-radiative populations of N in the cells of a reduced afterbody
        dict(name="qss", do="qss", cells=20_000, levels=32, lumped=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    do = rng.choice(["solve", "solve", "chunk", "coeffs", "coeffs", "march_slab", "march_axisym", "populations",
                     "continuum", "qss"])
    if do == "solve":
        precision = rng.choice([32, 32, 64])
        cells = _log(rng, 8, 200 if precision == 32 else 24)
        points = _log(rng, 5_000, 1_000_000 if precision == 32 else 60_000)
        if rng.random() < 0.4:
            return dict(do=do, precision=precision, gas="uniform", cells=cells, atomic=_log(rng, 200, 3000),
                        molecular=0, points=points)
        return dict(do=do, precision=precision, gas="stagnation", cells=cells, atomic=4 * _log(rng, 250, 5000),
                    molecular=_log(rng, 3000, 280_000 if precision == 32 else 30_000), points=points)
    if do == "chunk":
        n = _log(rng, 100_000, 1_000_000)
        nk = _log(rng, 500, 2048)
        return dict(do=do, nx=_log(rng, 60, 400), nr=_log(rng, 40, 200), surface=_log(rng, 4, 200),
                    n_mu=rng.randrange(4, 17), n_phi=rng.randrange(7, 33), atomic=4 * _log(rng, 500, 5000),
                    molecular=_log(rng, 10_000, 300_000), points=n, k0=rng.randrange(n // 20, n - nk), nk=nk)
    if do == "coeffs":
        precision = rng.choice([32, 32, 64])
        cells = _log(rng, 8, 200 if precision == 32 else 24)
        n = _log(rng, 60_000, 1_000_000)
        nk = min(n // 2, _log(rng, 2_000, 120_000 if precision == 32 else 20_000))
        return dict(do=do, precision=precision, broad=rng.random() < 0.3, cells=cells, atomic=4 * _log(rng, 500, 5000),
                    molecular=_log(rng, 3000, 300_000 if precision == 32 else 60_000), points=n,
                    k0=rng.randrange(n - nk), nk=nk)
    if do == "march_slab":
        precision = rng.choice([32, 32, 64])
        n = _log(rng, 60_000, 1_000_000)
        nk = min(n, _log(rng, 5_000, 300_000 if precision == 32 else 60_000))
        return dict(do=do, precision=precision, cells=_log(rng, 8, 300), n_mu=rng.randrange(1, 33), points=n,
                    k0=rng.randrange(n - nk + 1), nk=nk, wall=rng.random() < 0.3)
    if do == "march_axisym":
        precision = rng.choice([32, 32, 64])
        nk = _log(rng, 1_000, 8_192 if precision == 32 else 2_000)
        return dict(do=do, precision=precision, nx=_log(rng, 40, 200), nr=_log(rng, 20, 100), surface=_log(rng, 2, 40),
                    n_mu=rng.randrange(4, 17), n_phi=rng.randrange(8, 33), points=1_000_000,
                    k0=rng.randrange(1_000_000 - nk), nk=nk)
    if do == "populations":
        return dict(do=do, cells=_log(rng, 50, 10_000), atomic=4 * _log(rng, 500, 5000),
                    molecular=_log(rng, 5_000, 300_000))
    if do == "continuum":
        precision = rng.choice([32, 32, 64])
        nk = _log(rng, 5_000, 300_000 if precision == 32 else 50_000)
        return dict(do=do, precision=precision, cells=_log(rng, 8, 200), levels=rng.randrange(20, 101),
                    points=1_000_000, k0=rng.randrange(1_000_000 - nk), nk=nk)
    return dict(do=do, cells=_log(rng, 500, 40_000), levels=rng.randrange(8, 33), lumped=rng.randrange(0, 6))


# ------------------------------------------------------------ what they need

def _device():
    return torch.device("cuda", torch.cuda.current_device())


@functools.lru_cache(maxsize=8)
def _air(seed, atomic, molecular):
    """The air line database of a seed (lines and species)."""
    p = synth.stagnation_line(seed=seed % (1 << 31), n_cells=2, n_atomic=atomic, n_molecular=molecular, n_grid=11)
    return p.species, p.lines


def _grid(c):
    return synth.Grid(50.0, 1000.0 if c.get("gas") == "uniform" else 2000.0, int(c["points"]))


def _rng(seed):
    return np.random.default_rng((int(seed), 77))


def _stagnation_cells(n, seed):
    """The stagnation line's profiles, with the seed's peak temperatures and density."""
    rng = _rng(seed)
    x = (np.arange(n) + 0.5) * 3.0 / n
    Ttr, Tve = synth.stagnation_profiles(x)
    Ttr = Ttr * rng.uniform(0.9, 1.1)
    Tve = Tve * rng.uniform(0.9, 1.1)
    return synth.Cells(Ttr=Ttr, Tve=Tve, n=synth.composition(Tve, 1e17 * rng.uniform(0.5, 1.5)))


def _slab(n, n_mu, dx, wall=False):
    mu, w = synth.gauss_legendre_01(n_mu)
    return synth.SlabGeometry(cell_order=np.arange(n, dtype=np.int64), dx=np.full(n, dx), mu=mu, wmu=w,
                              wall_start=wall, T_wall=8000.0 if wall else 0.0)


def _axisym(c, seed):
    """Mesh, surface points and directions around the afterbody's cylinder."""
    xf = np.linspace(0.0, 200.0, c["nx"] + 1)
    rf = np.linspace(33.5, 183.5, c["nr"] + 1)
    mu, w = synth.gauss_legendre_01(c["n_mu"])
    surf = np.sort(_rng(seed).uniform(1.0, 199.0, c["surface"]))
    return synth.AxisymGeometry(xf=xf, rf=rf, surf_x=surf, r_body=33.5, mu=mu, wmu=w, n_phi=c["n_phi"])


def _afterbody_cells(geo, seed):
    xc = 0.5 * (geo.xf[1:] + geo.xf[:-1])
    yc = 0.5 * (geo.rf[1:] + geo.rf[:-1]) - geo.r_body
    Ttr, Tve, nt = synth.afterbody_fields(xc, yc)
    f = _rng(seed).uniform(0.9, 1.1)
    Ttr, Tve = (Ttr * f).ravel(), (Tve * f).ravel()
    return synth.Cells(Ttr=Ttr, Tve=Tve, n=synth.composition(Tve, nt.ravel()))


def _field_cells(n, seed):
    """States of a field's cells, drawn over the range the workloads have."""
    rng = _rng(seed)
    Ttr = rng.uniform(3000.0, 30000.0, n)
    Tve = np.minimum(rng.uniform(3000.0, 15000.0, n), Ttr)
    return synth.Cells(Ttr=Ttr, Tve=Tve, n=synth.composition(Tve, 10.0 ** rng.uniform(15.0, 17.0, n)))


def _problem(c, seed):
    """The problem of a solve / chunk / coeffs / populations case."""
    if c["do"] == "solve" and c["gas"] == "uniform":
        rng = _rng(seed)
        return synth.uniform_slab(seed=int(seed), n_lines=c["atomic"], n_cells=c["cells"], n_grid=c["points"],
                                  T=rng.uniform(9000.0, 11000.0))
    species, lines = _air(int(seed), c["atomic"], c["molecular"])
    if c["do"] == "chunk":
        geo = _axisym(c, seed)
        cells = _afterbody_cells(geo, seed)
    elif c["do"] == "populations":
        geo, cells = None, _field_cells(c["cells"], seed)
    else:
        geo, cells = _slab(c["cells"], 16, 3.0 / c["cells"]), _stagnation_cells(c["cells"], seed)
    grid = _grid(c) if "points" in c else synth.Grid(50.0, 2000.0, 11)
    return synth.Problem(c["do"], species, lines, cells, grid, geo)


def _smooth(x, width):
    """x [n] convolved with a Gaussian of `width` samples, unit variance again."""
    r = 3 * width
    w = torch.exp(-0.5 * (torch.arange(-r, r + 1, device=x.device, dtype=x.dtype) / width) ** 2)
    w = w / w.square().sum().sqrt()
    return torch.nn.functional.conv1d(torch.nn.functional.pad(x, (r, r))[None, None], w[None, None])[0, 0]


def _spectra(c, C, path, seed, dtype):
    """kappa, j [C, nk]: lognormal spectra in narrow lines, smooth over the
    cells; the median optical depth of `path` cm is 3e-4."""
    dev = _device()
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed) + 5)
    nk, grid = c["nk"], _grid(c)
    z = _smooth(torch.randn(nk, generator=g, device=dev), 3)
    z2 = _smooth(torch.randn(nk, generator=g, device=dev), 200)
    y = _smooth(torch.randn(C, generator=g, device=dev), 8)
    y2 = _smooth(torch.randn(C, generator=g, device=dev), 20)
    T = 9000.0 + 2500.0 * torch.tanh(y2)
    lam = torch.arange(c["k0"], c["k0"] + nk, device=dev, dtype=torch.float64) * (
        (grid.lam_max - grid.lam_min) / (grid.n - 1)) + grid.lam_min
    col = 3.0 * z + 0.5 * z2 + math.log(3e-4 / path)
    x = (H * CL * 1e7 / KB / lam).float()
    pre = (1e-7 * 2.0 * H * CL * CL / (1e4 * (lam * 1e-7) ** 5)).float()
    kap = torch.empty((C, nk), dtype=dtype, device=dev)
    em = torch.empty_like(kap)
    for a in range(0, C, 4096):
        b = min(C, a + 4096)
        k = torch.exp(col[None] + 0.5 * y[a:b, None])
        kap[a:b] = k
        em[a:b] = k * pre[None] / torch.expm1((x[None] / T[a:b, None]).clamp(max=80.0))
    return kap, em


def _precision(c):
    return R.FP64 if c.get("precision", 32) == 64 else R.FP32


def _dtype(c):
    return torch.float64 if c.get("precision", 32) == 64 else torch.float32


def _models(c, seed):
    return [synth.continuum_model(seed=int(seed) + k, species=s, n_levels=c["levels"]) for k, s in
            enumerate(("N", "O"))]


def prepare(case, seed):
    c, do, dev = case, case["do"], _device()
    ctx = R.Context(dev.index)
    s = dict(c=c, ctx=ctx)
    if do in ("solve", "chunk", "coeffs", "populations"):
        p = _problem(c, seed)
        s["problem"] = p
        if do in ("solve", "chunk"):
            s["dp"] = solver.DeviceProblem(p, ctx)
            s["sp"], s["ln"], s["cells"] = s["dp"].species, s["dp"].lines, s["dp"].cells
        else:
            s["sp"] = R.DeviceSpecies(p.species, dev)
            s["ln"] = R.DeviceLines(p.lines, dev)
            s["cells"] = R.DeviceCells(p.cells, s["sp"].S, dev)
        if do in ("chunk", "coeffs"):
            R.populations(ctx, s["sp"], s["cells"])
            s["kap"] = torch.empty((s["cells"].C, c["nk"]), dtype=_dtype(c), device=dev)
            s["em"] = torch.empty_like(s["kap"])
        if do == "chunk":
            s["qlam"] = torch.empty((s["dp"].P, c["nk"]), dtype=torch.float32, device=dev)
            s["q"] = torch.zeros(s["dp"].P, dtype=torch.float64, device=dev)
        if do == "coeffs" and c["broad"]:
            ctx.set_broadening(R.BROAD_STARK_IONIZE | R.BROAD_RESONANCE | R.BROAD_VDW, synth.RAD_E_IONIZE,
                               synth.FLOW_MASS)
    elif do == "march_slab":
        s["rays"] = R.slab_rays(ctx, _slab(c["cells"], c["n_mu"], 3.0 / c["cells"], c["wall"]), dev)
        s["kap"], s["em"] = _spectra(c, c["cells"], 3.0, seed, _dtype(c))
        s["qlam"] = torch.empty((1, c["nk"]), dtype=_dtype(c), device=dev)
        s["I"] = torch.empty((s["rays"].n_dirs, c["nk"]), dtype=_dtype(c), device=dev)
    elif do == "march_axisym":
        geo = _axisym(c, seed)
        s["rays"] = R.axisym_rays(ctx, geo, dev)
        s["kap"], s["em"] = _spectra(c, c["nx"] * c["nr"], 100.0, seed, _dtype(c))
        s["qlam"] = torch.empty((c["surface"], c["nk"]), dtype=_dtype(c), device=dev)
    elif do == "continuum":
        species, _lines = _air(int(seed), 400, 2000)
        cells = _stagnation_cells(c["cells"], seed)
        s["sp"] = R.DeviceSpecies(species, dev)
        s["cells"] = R.DeviceCells(cells, s["sp"].S, dev)
        R.populations(ctx, s["sp"], s["cells"])
        s["models"] = R.DeviceContinuum(_models(c, seed), dev)
        s["kap0"], s["em0"] = _spectra(c, c["cells"], 3.0, seed, _dtype(c))
        s["kap"], s["em"] = torch.empty_like(s["kap0"]), torch.empty_like(s["em0"])
    elif do == "qss":
        model = synth.cr_model(seed=int(seed), n_levels=c["levels"], n_lumped=c["lumped"])
        s["model"] = R.DeviceCrModel(model, dev)
        s["cells"] = R.DeviceCells(_field_cells(c["cells"], seed), 8, dev)
        s["out"] = torch.empty((c["cells"], c["levels"]), dtype=torch.float64, device=dev)
    if "points" in c:
        s["grid"] = _grid(c)
    return s


def run(s):
    c, do, ctx = s["c"], s["c"]["do"], s["ctx"]
    if do == "solve":
        out = solver.solve(s["dp"], ctx, _precision(c), keep_coeffs=True)
        return {"q": out["q"].to(_dtype(c)), "q_lambda": out["q_lambda"], "kappa": out["kappa"], "emis": out["emis"]}
    if do == "chunk":
        dp = s["dp"]
        s["q"].zero_()
        R.spectral_coeffs(ctx, s["sp"], s["ln"], s["cells"], s["grid"], c["k0"], c["nk"], R.FP32, s["kap"], s["em"])
        R.trace_rays(ctx, dp.rays, dp.C, s["kap"], s["em"], s["grid"], c["k0"], c["nk"], R.FP32, s["qlam"])
        R.wall_flux(ctx, s["qlam"], R.FP32, s["grid"], c["k0"], c["nk"], dp.P, s["q"])
        return {"q": s["q"].float(), "q_lambda": s["qlam"], "kappa": s["kap"], "emis": s["em"]}
    if do == "coeffs":
        R.spectral_coeffs(ctx, s["sp"], s["ln"], s["cells"], s["grid"], c["k0"], c["nk"], _precision(c), s["kap"],
                          s["em"])
        return {"kappa": s["kap"], "emis": s["em"]}
    if do == "march_slab":
        R.trace_rays(ctx, s["rays"], c["cells"], s["kap"], s["em"], s["grid"], c["k0"], c["nk"], _precision(c),
                     s["qlam"], s["I"])
        return {"q_lambda": s["qlam"], "I": s["I"]}
    if do == "march_axisym":
        R.trace_rays(ctx, s["rays"], c["nx"] * c["nr"], s["kap"], s["em"], s["grid"], c["k0"], c["nk"],
                     _precision(c), s["qlam"])
        return {"q_lambda": s["qlam"]}
    if do == "populations":
        return {"lnpref": R.populations(ctx, s["sp"], s["cells"])}
    if do == "continuum":   # adds to the tables of the lines: they are put back first
        s["kap"].copy_(s["kap0"])
        s["em"].copy_(s["em0"])
        R.continuum_coeffs(ctx, s["models"], s["sp"].S, s["cells"], s["grid"], c["k0"], c["nk"], _precision(c),
                           s["kap"], s["em"])
        return {"kappa": s["kap"], "emis": s["em"]}
    R.qss_populations(ctx, s["model"], s["cells"], s["out"])
    return {"n": s["out"]}


# --------------------------------------------------------------------- work

def work(case):
    """Bytes: inputs once, outputs once.  Operations: the profile's about 25
    an in-window (line, cell, point), where a line of the air database spans
    about 0.8 nm; a march step's 15; a level's 20 (its exponential)."""
    c, do = case, case["do"]
    esz = 8 if c.get("precision", 32) == 64 else 4
    lines = c.get("atomic", 0) + c.get("molecular", 0)
    if do in ("solve", "chunk", "coeffs"):
        C = c["nx"] * c["nr"] if do == "chunk" else c["cells"]
        nk = c.get("nk", c["points"])
        g = _grid(c)
        span = g.lam_max - g.lam_min
        evals = C * lines * (nk / c["points"]) * 0.8 * c["points"] / span
        b = lines * 92 + C * (13 * 8 + 64) + 2.0 * C * nk * esz
        f = 25.0 * evals
        if do == "solve":
            b += nk * esz
            f += 15.0 * C * 17 * nk
        if do == "chunk":
            segs = c["surface"] * c["n_mu"] * c["n_phi"] * 0.65 * c["nr"] * 2
            b += c["surface"] * nk * 4.0 + segs * 12
            f += 15.0 * segs * nk
        return {"bytes": b, "flops": f}
    if do == "march_slab":
        nd = c["n_mu"] + 1
        return {"bytes": (2.0 * c["cells"] + nd + 1) * c["nk"] * esz, "flops": 15.0 * c["cells"] * nd * c["nk"]}
    if do == "march_axisym":
        segs = c["surface"] * c["n_mu"] * c["n_phi"] * 0.65 * c["nr"] * 2
        return {"bytes": (2.0 * c["nx"] * c["nr"] + c["surface"]) * c["nk"] * esz + segs * 12,
                "flops": 15.0 * segs * c["nk"]}
    if do == "populations":
        levels = 1.7 * c["atomic"] + 11 * 11 * 152
        return {"bytes": c["cells"] * (13 + 8) * 8.0 + levels * 16, "flops": 20.0 * c["cells"] * levels}
    if do == "continuum":
        return {"bytes": 4.0 * c["cells"] * c["nk"] * esz,
                "flops": c["cells"] * c["nk"] * (4.0 * 2 * c["levels"] * 0.2 + 40)}
    l = c["levels"]
    return {"bytes": c["cells"] * (13.0 + l) * 8, "flops": c["cells"] * (2 * l ** 3 / 3 + l * (l - 1) / 2 * 60.0)}


# ----------------------------------------------------- the same in 64 bits

def _d(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=_device())


def _lam(grid, k0, nk):
    k = torch.arange(k0, k0 + nk, device=_device(), dtype=torch.float64)
    return grid.lam_min + k * ((grid.lam_max - grid.lam_min) / (grid.n - 1))


def _exact_lnpref(sp, cells):
    """ln(N_s / Z_s) [C, S], two-temperature Boltzmann."""
    Ttr, Tve, n = _d(cells.Ttr), _d(cells.Tve), _d(cells.n)
    C, S = len(Ttr), len(sp.names)
    out = torch.empty((C, S), dtype=torch.float64, device=_device())
    for a in range(0, C, 512):
        bve, btr = C2 / Tve[a:a + 512, None], C2 / Ttr[a:a + 512, None]
        for s in range(S):
            if sp.kind[s] == 0:
                i0, i1 = sp.atom_off[s], sp.atom_off[s + 1]
                Z = (torch.exp(-bve * _d(sp.atom_E[i0:i1])) * _d(sp.atom_g[i0:i1])).sum(1)
            else:
                Z = torch.zeros_like(bve[:, 0])
                for i in range(sp.st_off[s], sp.st_off[s + 1]):
                    nv, nj = int(sp.st_nv[i]), int(sp.st_nj[i])
                    rot = _d(sp.rot_E[sp.st_rot_off[i]:sp.st_rot_off[i] + nv * nj])
                    vib = _d(sp.vib_E[sp.st_vib_off[i]:sp.st_vib_off[i] + nv])
                    J = torch.arange(nj, device=_device(), dtype=torch.float64)
                    alt = _d(sp.st_Lalt[i])[J.long() % 2] * (2.0 * J + 1.0)
                    zr = (torch.exp(-btr * rot).reshape(-1, nv, nj) * alt).sum(2)
                    Z = Z + float(sp.st_g[i] / sp.st_sigma[i]) * torch.exp(-bve[:, 0] * float(sp.st_E[i])) * (
                        torch.exp(-bve * vib) * zr).sum(1)
            N = n[a:a + 512, int(sp.density_col[s])]
            out[a:a + 512, s] = torch.where(N > 0, torch.log(N) - torch.log(Z), -math.inf)   # -inf: no particles
    return out


def _exact_coeffs(p, k0, nk, broad):
    """kappa, j [C, nk]: Whiting's profile of every line within 100 Voigt
    half widths, cell by cell, lines grouped by the length of their window."""
    dev, g = _device(), p.grid
    ln, sp, cells = p.lines, p.species, p.cells
    h = (g.lam_max - g.lam_min) / (g.n - 1)
    lnp = _exact_lnpref(sp, cells)
    s = torch.as_tensor(ln.species.astype(np.int64), device=dev)
    lam0, A, gu, gl = _d(ln.lam0), _d(ln.A), _d(ln.gu), _d(ln.gl)
    Eve_u, Er_u = _d(ln.Eu_el) + _d(ln.Eu_v), _d(ln.Eu_j)
    Eve_l, Er_l = _d(ln.El_el) + _d(ln.El_v), _d(ln.El_j)
    mass, kind = _d(sp.mass)[s], torch.as_tensor(sp.kind.astype(np.int64), device=dev)[s]
    lamS0 = _d(ln.lamS0)
    lcm = lam0 * 1e-7
    cR = cW = torch.zeros_like(lam0)
    atom = kind == 0
    if broad:
        gap = (_d(synth.RAD_E_IONIZE)[s] - _d(ln.Eu_el)).clamp(min=E_H / 25.0)
        lamS0 = torch.where(atom, 1.69e3 * lam0 ** 2 / gap ** 2.623, lamS0)
        f = ME * CL * lcm ** 2 / (8.0 * math.pi ** 2 * QE ** 2) * gu / gl * A
        ground = atom & (Eve_l == 0) & (Er_l == 0)
        cR = torch.where(ground, 4.3e-28 * lam0 * f * torch.sqrt(gl / gu) * lam0 ** 2, 0.0)
        cW = torch.where(atom, lam0 ** 2, 0.0)
    kap = torch.zeros((len(cells.Ttr), nk), dtype=torch.float64, device=dev)
    em = torch.zeros_like(kap)
    lk = _lam(g, k0, nk)
    for c in range(len(cells.Ttr)):
        Ttr, Tve, n = float(cells.Ttr[c]), float(cells.Tve[c]), np.asarray(cells.n[c], np.float64)
        lamG = (7.16233e-7 / 2.0) * lam0 * torch.sqrt(Ttr / mass)
        lamL = 5.9e-6 + lamS0 * ((Tve / 1e4) ** 0.33 * (n[cells.ne_col] / 1e16))
        if broad:
            N0, W = np.zeros(len(sp.names)), np.zeros(len(sp.names))
            for q in range(len(sp.names)):
                if sp.kind[q] != 0:
                    continue
                i0, i1 = sp.atom_off[q], sp.atom_off[q + 1]
                g0 = sp.atom_g[i0:i1][sp.atom_E[i0:i1] == 0.0].sum()
                N0[q] = math.exp(float(lnp[c, q])) * g0
                col = int(sp.density_col[q])
                other = (np.arange(len(n)) != col) & (synth.FLOW_MASS > 0)
                No, NoM = n[other].sum(), (n[other] * synth.FLOW_MASS[other]).sum()
                W[q] = 6.65e-29 * n[col] * math.sqrt(2.0 * Ttr / sp.mass[q])
                if No > 0:
                    W[q] += 2.925e-29 * No * math.sqrt(2.0 * Ttr / (NoM / No))
            lamL = lamL + cR * _d(N0)[s] + cW * _d(W)[s]
        d = (lamL - lamG) / (lamL + lamG)
        lamV = (1.0 - 0.18121 * (1.0 - d * d) - (0.023665 * torch.exp(0.6 * d) + 0.00418 * torch.exp(-1.9 * d)) *
                torch.sin(math.pi * d)) * (lamL + lamG)
        lo = (torch.ceil((lam0 - 100.0 * lamV - g.lam_min) / h) - 1.0).clamp(min=k0)
        hi = (torch.floor((lam0 + 100.0 * lamV - g.lam_min) / h) + 1.0).clamp(max=k0 + nk - 1)
        idx = torch.nonzero(lo <= hi)[:, 0]
        size = (hi - lo + 1)[idx]
        idx = idx[torch.argsort(size)]
        lnNu = lnp[c][s] + torch.log(gu) - C2 * (Eve_u / Tve + Er_u / Ttr)
        x = C2 * ((Eve_u - Eve_l) / Tve + (Er_u - Er_l) / Ttr)
        Sj = torch.exp(torch.log(1e-7 * (H * CL / (4.0 * math.pi)) * A / lcm) + lnNu)
        Sk = torch.exp(torch.log(1e4 * A * lcm ** 4 / (8.0 * math.pi * CL)) + lnNu) * torch.expm1(x)
        r = lamL / lamV
        pre = 1e3 / (2.0 * lamV * (1.065 + 0.447 * r + 0.058 * r * r))
        sizes = (hi - lo + 1)[idx].long().cpu().numpy()
        a = 0
        while a < len(sizes):
            b = min(len(sizes), a + max(1, 8_000_000 // int(sizes[min(len(sizes) - 1, a + 20_000)])))
            L = idx[a:b]
            k = lo[L, None].long() - k0 + torch.arange(int(sizes[b - 1]), device=dev)[None]
            inside = k <= (hi[L, None].long() - k0)
            k = k.clamp(max=nk - 1)
            dl = (lk[k] - lam0[L, None]).abs()
            inside &= dl <= 100.0 * lamV[L, None]
            u = dl / (2.0 * lamV[L, None])
            rr, v = r[L, None], u ** 2.25
            br = (1.0 - rr) * torch.exp(-2.772 * u * u) + rr / (1.0 + 4.0 * u * u) + 0.016 * rr * (1.0 - rr) * (
                torch.exp(-0.4 * v) - 1.0 / (1.0 + 0.1 * v))
            br = torch.where(inside, br * pre[L, None], 0.0).reshape(-1)
            k = k.reshape(-1)
            n_k = int(sizes[b - 1])
            em[c].index_add_(0, k, br * Sj[L].repeat_interleave(n_k))
            kap[c].index_add_(0, k, br * Sk[L].repeat_interleave(n_k))
            a = b
    return kap, em


def _step(I, kf, ds, jf, jn):
    """One segment: kappa at its far node, emission linear between the nodes."""
    t = kf * ds
    thin = t.abs() < 4e-4
    em1 = torch.expm1(-t)
    ts, ks = torch.where(thin, 1.0, t), torch.where(thin, 1.0, kf)
    f = -em1 / ts
    ca = torch.where(thin, ds * (0.5 - t / 3.0 + t * t / 8.0), (f - 1.0 - em1) / ks)
    cb = torch.where(thin, ds * (0.5 - t / 6.0 + t * t / 24.0), (1.0 - f) / ks)
    return I + I * em1 + ca * jf + cb * jn


def _planck(lam, T):
    lcm = lam * 1e-7
    return 1e-7 * 2.0 * H * CL * CL / (1e4 * lcm ** 5 * torch.expm1(H * CL / (lcm * KB * T)))


def _exact_slab(geo, kap, em, lam):
    """I [n_dirs, nk] (the normal ray first) and q_lambda [1, nk]."""
    nk, dev = len(lam), _device()
    scale = _d(np.concatenate([[1.0], 1.0 / geo.mu]))
    weight = _d(np.concatenate([[0.0], 2.0 * np.pi * geo.wmu * geo.mu]))
    I = torch.empty((len(scale), nk), dtype=torch.float64, device=dev)
    m = len(geo.cell_order)
    for a in range(0, nk, 65_536):
        K, J = kap[:, a:a + 65_536].double(), em[:, a:a + 65_536].double()
        x = torch.zeros((len(scale), K.shape[1]), dtype=torch.float64, device=dev)
        if geo.wall_start:
            x += _planck(lam[a:a + 65_536], geo.T_wall)[None]
        kf, jf = K[0], J[0]
        for i in range(m):
            kn, jn = (0.5 * (K[i] + K[i + 1]), 0.5 * (J[i] + J[i + 1])) if i + 1 < m else (K[i], J[i])
            x = _step(x, kf[None], float(geo.dx[i]) * scale[:, None], jf[None], jn[None])
            kf, jf = kn, jn
        I[:, a:a + 65_536] = x
    return I, (weight[:, None] * I).sum(0, keepdim=True)


def _exact_rays(geo, p):
    """Cells and lengths [rays, pieces] of the lines of sight of surface point
    p, far piece first, short lists led by pieces of length 0."""
    dev = _device()
    mu = _d(geo.mu).repeat_interleave(geo.n_phi)
    psi = ((torch.arange(geo.n_phi, device=dev, dtype=torch.float64) + 0.5) * (2.0 * math.pi / geo.n_phi)).repeat(
        len(geo.mu))
    st = torch.sqrt(1.0 - mu * mu)
    dx, dn, dt = st * torch.cos(psi), mu, st * torch.sin(psi)
    xf, rf, rb, x0 = _d(geo.xf), _d(geo.rf), float(geo.rf[0]), float(geo.surf_x[p])
    tx = (xf[None] - x0) / dx[:, None]
    A, B = (dn * dn + dt * dt)[:, None], (2.0 * rb * dn)[:, None]
    cq = (rb * rb - rf * rf)[None]
    tr = -2.0 * cq / (B + torch.sqrt(B * B - 4.0 * A * cq))
    end = torch.minimum(torch.maximum(tx[:, :1], tx[:, -1:]), tr[:, -1:])
    t = torch.cat([tx, tr], 1)
    t = torch.where((t > 0) & (t <= end), t, 0.0).sort(1)[0]
    t = torch.cat([torch.zeros_like(end), t], 1)
    ds = t[:, 1:] - t[:, :-1]
    mid = 0.5 * (t[:, 1:] + t[:, :-1])
    ix = (torch.searchsorted(xf, x0 + mid * dx[:, None], right=True) - 1).clamp(0, len(xf) - 2)
    r = torch.sqrt((rb + mid * dn[:, None]) ** 2 + (mid * dt[:, None]) ** 2)
    jr = (torch.searchsorted(rf, r, right=True) - 1).clamp(0, len(rf) - 2)
    cell = ix * (len(rf) - 1) + jr
    n = int((ds > 0).sum(1).max())
    ds, cell = ds[:, -n:].flip(1), cell[:, -n:].flip(1)           # far piece first, pieces of length 0 last
    order = torch.argsort((ds > 0).int(), dim=1, stable=True)       # pieces of length 0 first
    ds, cell = ds.gather(1, order), cell.gather(1, order)
    first = (ds > 0).int().argmax(1, keepdim=True)
    at = torch.arange(n, device=dev)[None]
    return torch.where(at < first, cell.gather(1, first), cell), ds


def _exact_axisym(geo, kap, em, nk):
    dev = _device()
    w = _d(geo.mu * geo.wmu).repeat_interleave(geo.n_phi) * (2.0 * math.pi / geo.n_phi)
    q = torch.empty((len(geo.surf_x), nk), dtype=torch.float64, device=dev)
    for p in range(len(geo.surf_x)):
        cell, ds = _exact_rays(geo, p)
        n = cell.shape[1]
        for a in range(0, nk, 8192):
            K, J = kap[:, a:a + 8192], em[:, a:a + 8192]
            I = torch.zeros((cell.shape[0], K.shape[1]), dtype=torch.float64, device=dev)
            kc, jc = K[cell[:, 0]].double(), J[cell[:, 0]].double()
            kf, jf = kc, jc
            for i in range(n):
                kx, jx = (K[cell[:, i + 1]].double(), J[cell[:, i + 1]].double()) if i + 1 < n else (kc, jc)
                kn, jn = 0.5 * (kc + kx), 0.5 * (jc + jx)
                I = _step(I, kf, ds[:, i, None], jf, jn)
                kf, jf, kc, jc = kn, jn, kx, jx
            q[p, a:a + 8192] = (w[:, None] * I).sum(0)
    return q


def _exact_continuum(c, models, cells, lnp, lam, kap, em):
    Tve, n = _d(cells.Tve), _d(cells.n)
    kap, em = kap.double(), em.double()
    B = _planck(lam[None], Tve[:, None])
    for m in models:
        T = Tve
        Qp = (_d(m["ion_g"]) * torch.exp(-C2 * _d(m["ion_E"])[None] / T[:, None])).sum(1)
        lnQ = 1.5 * torch.log(H * H / (2.0 * math.pi * ME * KB * T))
        pe = n[:, m["ion_col"]] * n[:, cells.ne_col]
        for i in range(len(m["E"])):
            a, b = int(m["node_off"][i]), int(m["node_off"][i + 1])
            x, y = _d(m["node_lam"][a:b]), _d(m["node_sigma"][a:b])
            on = torch.nonzero((lam >= x[0]) & (lam <= x[-1]))[:, 0]
            if not len(on):
                continue
            sl = slice(int(on[0]), int(on[-1]) + 1)
            j = (torch.searchsorted(x, lam[sl], right=True) - 1).clamp(0, len(x) - 2)
            sg = y[j] + (y[j + 1] - y[j]) / (x[j + 1] - x[j]) * (lam[sl] - x[j])
            lng = math.log(m["g"][i])
            kap[:, sl] += torch.exp(lnp[:, m["species"]] + lng - C2 * float(m["E"][i]) / T)[:, None] * sg[None]
            S = pe * torch.exp(lnQ + lng + C2 * float(m["E_ion"] - m["E"][i]) / T) / (2.0 * Qp)
            em[:, sl] += S[:, None] * sg[None] * B[:, sl]
        F = torch.exp(lnp[:, m["species"]] + torch.log(2.0 * Qp) - lnQ - C2 * m["E_ion"] / T)
        cc, sig = m["ff_c"], 91.1267 / lam
        A1 = cc[0] + cc[1] * torch.exp(-cc[2] * T)
        A2 = cc[3] + cc[4] * torch.exp(-cc[5] * T) + cc[6] * torch.exp(-cc[7] * T)
        xs, ts, D = _d(m["D_sigma"]), _d(m["D_T"]), _d(m["D"])
        sc, Tc = sig.clamp(float(xs[0]), float(xs[-1])), T.clamp(float(ts[0]), float(ts[-1]))
        j = (torch.searchsorted(xs, sc, right=True) - 1).clamp(0, len(xs) - 2)
        it = (torch.searchsorted(ts, Tc, right=True) - 1).clamp(0, len(ts) - 2)
        w, v = (sc - xs[j]) / (xs[j + 1] - xs[j]), (Tc - ts[it]) / (ts[it + 1] - ts[it])
        Dc = (1.0 - v)[:, None] * D[it] + v[:, None] * D[it + 1]
        Dv = (1.0 - w)[None] * Dc[:, j] + w[None] * Dc[:, j + 1]
        kff = F[:, None] * (A1[:, None] / sig[None] + A2[:, None]) / (sig[None] ** 3 * 1e40) * (1.0 + Dv)
        kap += kff
        em += B * kff
    return kap, em


def _exact_qss(m, cells):
    dev = _device()
    C, l = len(cells.Ttr), int(m["l"])
    Ttr, Tve, n = _d(cells.Ttr)[:, None], _d(cells.Tve)[:, None], _d(cells.n)
    ne, nion = n[:, cells.ne_col, None], n[:, m["ion_col"], None]
    nM = (n.sum(1) - n[:, cells.ne_col])[:, None]
    E, g = _d(m["E"]), _d(m["g"])
    Qh, Qv = g * torch.exp(-C2 * E / Ttr), g * torch.exp(-C2 * E / Tve)
    lo, up = torch.as_tensor(m["lo"], device=dev).long(), torch.as_tensor(m["up"], device=dev).long()
    theta = C2 * (E[up] - E[lo])
    kh = _d(m["hp_C"]) * Ttr ** _d(m["hp_n"]) * torch.exp(-theta / Ttr)
    ke = _d(m["e_C"]) * Tve ** _d(m["e_n"]) * torch.exp(-theta / Tve)
    rad = _d(m["A"]) * (_d(m["lam"]) >= 200.0)
    ru = (kh * nM + ke * ne) / N_A
    rd = (kh * Qh[:, lo] / Qh[:, up] * nM + ke * Qv[:, lo] / Qv[:, up] * ne) / N_A + rad
    M = torch.zeros((C, l, l), dtype=torch.float64, device=dev)
    M[:, lo, up] = rd
    M[:, up, lo] = ru
    loss = torch.zeros((C, l), dtype=torch.float64, device=dev)
    loss.index_add_(1, lo, ru)
    loss.index_add_(1, up, rd)
    kf = _d(m["ii_C"]) * Tve ** _d(m["ii_n"]) * torch.exp(-C2 * (m["E_ion"] - E[:l]) / Tve)
    Qp, Qe = m["g_ion"] * torch.exp(-C2 * m["E_ion"] / Tve), 2.0 * (2.0 * math.pi * ME * KB * Tve / (H * H)) ** 1.5
    i = torch.arange(l, device=dev)
    M[:, i, i] = -(loss + kf * ne / N_A)
    b = -kf * Qv[:, :l] / (Qp * Qe) * nion * ne * ne / N_A
    M[:, 0, :] = 1.0
    M[:, 0, l - 1] += Qv[:, l:].sum(1) / Qv[:, l - 1]
    b[:, 0] = n[:, m["col"]]
    return torch.linalg.solve(M, b)


def exact(case, seed):
    c, do = case, case["do"]
    if do == "populations":
        p = _problem(c, seed)
        return {"lnpref": _exact_lnpref(p.species, p.cells)}
    if do == "qss":
        model = synth.cr_model(seed=int(seed), n_levels=c["levels"], n_lumped=c["lumped"])
        return {"n": _exact_qss(model, _field_cells(c["cells"], seed))}
    grid = _grid(c)
    if do in ("solve", "coeffs"):
        k0, nk = c.get("k0", 0), c.get("nk", c["points"])
        evals = c["cells"] * (c["atomic"] + c["molecular"]) * 0.8 * nk / (grid.lam_max - grid.lam_min)
        if evals > 3e9 or c["cells"] * nk > 3e7:
            return None
        p = _problem(c, seed)
        kap, em = _exact_coeffs(p, k0, nk, c.get("broad", False))
        if do == "coeffs":
            return {"kappa": kap, "emis": em}
        lam = _lam(grid, 0, nk)
        _I, ql = _exact_slab(p.geometry, kap, em, lam)
        h = (grid.lam_max - grid.lam_min) / (grid.n - 1) * 1e-3
        q = (ql.sum(1) - 0.5 * (ql[:, 0] + ql[:, -1])) * h
        return {"q": q, "q_lambda": ql, "kappa": kap, "emis": em}
    if do == "march_slab":
        kap, em = _spectra(c, c["cells"], 3.0, seed, _dtype(c))
        I, q = _exact_slab(_slab(c["cells"], c["n_mu"], 3.0 / c["cells"], c["wall"]), kap, em,
                           _lam(grid, c["k0"], c["nk"]))
        return {"q_lambda": q, "I": I}
    if do == "march_axisym":
        kap, em = _spectra(c, c["nx"] * c["nr"], 100.0, seed, _dtype(c))
        return {"q_lambda": _exact_axisym(_axisym(c, seed), kap, em, c["nk"])}
    if do == "continuum":
        species, _lines = _air(int(seed), 400, 2000)
        cells = _stagnation_cells(c["cells"], seed)
        kap, em = _spectra(c, c["cells"], 3.0, seed, _dtype(c))
        kap, em = _exact_continuum(c, _models(c, seed), cells, _exact_lnpref(species, cells),
                                   _lam(grid, c["k0"], c["nk"]), kap, em)
        return {"kappa": kap, "emis": em}
    return None
