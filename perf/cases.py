"""Performance cases of the library: what its users have it do, through the Python binding.

A case is a dict of plain values; ``kind`` says which entry point it goes through:

  opacity   Context.synth_opacity of rows of a (T, P) table on a log-lambda grid
  spectrum  Context.synth_spectrum of one grey model atmosphere on a wavelength window
  batch     Batch.run: rows on uneven wavelength windows, prepared and captured once
  serve     Server: a burst of spectrum requests of different sizes, submitted and waited for
  odf       Context.build_odf of an opacity array
  bins      Context.odf_intensity of many rays through an ODF table
  plasma    Context.set_atmosphere_grid_eos, the populations read back, and synth_continuum

Line lists are uniform in ln lambda with the distributions of workloads.linelist; the sizes
are those of the workloads, the benchmark and the tests.  ``exact`` restates each path in
FP64 with torch and numpy alone.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import workloads as wl
from paper_2105_13611_gb300 import binding

WIDTHS = [float(w) for w in wl.ODF_WIDTHS_12]
MUS = [1.0, 0.8, 0.6, 0.4, 0.2]
CUT, KC_FACTOR = 1e-3, 1e-2
DEV = "cuda"


def listed():
    return [
        # one (T, P) point of a handful of lines on a fraction of a nanometre: the smallest call,
        # as made in a loop over narrow features
        dict(name="opacity_40_lines", kind="opacity", n_lines=40, list_lo=300.0, list_hi=300.6, n_metals=5,
             lam0=300.0, lam1=300.6, R=2e6, nT=4, nP=1, n_rows=1, vturb=0.0),
        # the plain method's workload: 20,000 lines, 100 nm at R = 2e6, four points
        dict(name="opacity_20k_lines", kind="opacity", n_lines=20000, list_lo=300.0, list_hi=400.0, n_metals=5,
             lam0=300.0, lam1=400.0, R=2e6, nT=4, nP=1, n_rows=4, vturb=0.0),
        # rows of the full ODF table: 5e6 lines, 9-10000 nm at R = 2e6, spread over the 57 x 25 grid
        dict(name="opacity_table_rows", kind="opacity", n_lines=5_000_000, list_lo=9.0, list_hi=10000.0, n_metals=15,
             lam0=9.0, lam1=10000.0, R=2e6, nT=57, nP=25, n_rows=2, vturb=0.0),
        # a line profile study: a short list and a window of one nanometre through one atmosphere
        dict(name="spectrum_20k_1nm", kind="spectrum", n_lines=20000, list_lo=480.0, list_hi=520.0, n_metals=5,
             lam0=500.0, dlam=1.0, R=5e5, depths=40, teff=5772.0, logg=4.44, continuum=0, vturb=1e5),
        # a spectrum request of ordinary size over the full list, solar-like
        dict(name="spectrum_5M_7nm", kind="spectrum", n_lines=5_000_000, list_lo=9.0, list_hi=10000.0, n_metals=15,
             lam0=500.0, dlam=7.3, R=5e5, depths=80, teff=5772.0, logg=4.44, continuum=0, vturb=0.0),
        # a long window of a hotter star with the closed-form continuum: the largest requests
        dict(name="spectrum_5M_150nm", kind="spectrum", n_lines=5_000_000, list_lo=9.0, list_hi=10000.0, n_metals=15,
             lam0=350.0, dlam=150.0, R=5e5, depths=63, teff=8500.0, logg=4.0, continuum=15, vturb=2e5),
        # rows of many compositions on uneven windows (1-500 nm), replayed as one captured batch
        dict(name="batch_24_windows", kind="batch", n_lines=1_000_000, list_lo=9.0, list_hi=10000.0, n_metals=15,
             groups=24, comps=8, dlam_hi=500.0, R=5e5),
        # a burst of spectrum requests arriving together at the request server
        dict(name="serve_8_spectra", kind="serve", n_lines=500_000, list_lo=9.0, list_hi=10000.0, n_metals=15,
             requests=8, dlam_hi=100.0, R=5e5),
        # the ODFs of table rows: 328 intervals x 12 steps over 14 M points
        dict(name="odf_328x12", kind="odf", n_rows=4, N=14_025_881, K=328, n_steps=12, geom=False),
        # ten wide intervals with the paper's default (geometric) mean
        dict(name="odf_10x12_geometric", kind="odf", n_rows=2, N=14_025_881, K=10, n_steps=12, geom=True),
        # bin intensities of the rays of a model cube through the 57 x 25 x 328 x 12 table
        dict(name="bins_1024_rays", kind="bins", rays=1024, depths=80, nT=57, nP=25, K=328, n_steps=12, n_mu=5),
        # the plasma of several compositions on the table's grid, and the continuum of some rows
        dict(name="plasma_8_comps", kind="plasma", n_metals=15, nT=57, nP=25, comps=8, n_rows=8,
             lam0=100.0, lam1=3000.0, R=5e5),
    ]


def draw(rng):
    log_u = lambda a, b: math.exp(rng.uniform(math.log(a), math.log(b)))  # noqa: E731
    kind = rng.choice(["opacity", "opacity", "spectrum", "spectrum", "batch", "serve", "odf", "odf", "bins", "plasma"])
    if kind == "opacity":
        while True:
            lo = log_u(9.0, 5000.0)
            c = dict(kind=kind, n_lines=int(log_u(40, 5e6)), list_lo=9.0, list_hi=10000.0, n_metals=rng.randint(1, 15),
                     lam0=round(lo, 3), lam1=round(lo * math.exp(log_u(2e-3, 7.0)), 3), R=rng.choice([5e5, 1e6, 2e6]),
                     nT=rng.choice([4, 19, 57]), nP=rng.choice([1, 25]), n_rows=rng.randint(1, 4),
                     vturb=rng.choice([0.0, 1e5]))
            if c["lam1"] <= 10000.0 and c["n_rows"] <= c["nT"] * c["nP"] and c["n_rows"] * c["n_lines"] * c["R"] <= 1.5e13:
                return c
    if kind == "spectrum":
        while True:
            c = dict(kind=kind, n_lines=int(log_u(1e3, 5e6)), list_lo=9.0, list_hi=10000.0, n_metals=rng.randint(2, 15),
                     lam0=round(log_u(120.0, 4000.0), 3), dlam=round(log_u(0.5, 400.0), 3), R=5e5,
                     depths=rng.randint(40, 120), teff=round(rng.uniform(3500.0, 9000.0), 1),
                     logg=round(rng.uniform(1.0, 5.0), 2), continuum=rng.choice([0, 0, 15, 3]),
                     vturb=rng.choice([0.0, 1.5e5]))
            if c["depths"] * c["n_lines"] * (c["dlam"] + 5.0) <= 2.5e10 and c["depths"] * c["n_lines"] <= 4e8:
                return c
    if kind == "batch":
        return dict(kind=kind, n_lines=int(log_u(5e4, 1e6)), list_lo=9.0, list_hi=10000.0, n_metals=rng.randint(5, 15),
                    groups=rng.randint(3, 24), comps=rng.randint(1, 8), dlam_hi=rng.choice([50.0, 200.0, 500.0]), R=5e5)
    if kind == "serve":
        return dict(kind=kind, n_lines=int(log_u(2e4, 5e5)), list_lo=9.0, list_hi=10000.0, n_metals=rng.randint(5, 15),
                    requests=rng.randint(2, 8), dlam_hi=rng.choice([5.0, 30.0, 100.0]), R=5e5)
    if kind == "odf":
        N = int(log_u(2000, 1.4e7))
        K = max(rng.choice([1, 3, 10, 100, 328]), N // 2_000_000 + 1)
        return dict(kind=kind, n_rows=rng.randint(1, 4), N=N, K=min(K, N // 20), n_steps=rng.choice([4, 10, 12, 12, 12, 20]),
                    geom=rng.random() < 0.5)
    if kind == "bins":
        return dict(kind=kind, rays=int(log_u(1, 1024)), depths=rng.randint(40, 80), nT=57, nP=25,
                    K=rng.choice([40, 328]), n_steps=rng.choice([4, 12]), n_mu=rng.randint(1, 5))
    return dict(kind=kind, n_metals=rng.randint(1, 15), nT=rng.choice([5, 57]), nP=25, comps=rng.randint(1, 8),
                n_rows=rng.randint(1, 8), lam0=100.0, lam1=round(log_u(110.0, 3000.0), 2), R=5e5)


# ---------------------------------------------------------------------------
# Inputs

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _lines(c, seed):
    """The line list of workloads.linelist's distributions, drawn on the GPU."""
    g, n = _gen(seed), c["n_lines"]
    uni = lambda lo, hi: lo + (hi - lo) * torch.rand(n, generator=g, device=DEV, dtype=torch.float64)  # noqa: E731
    nrm = lambda m, s: (m + s * torch.randn(n, generator=g, device=DEV, dtype=torch.float64)).float()  # noqa: E731
    lam = torch.exp(uni(math.log(c["list_lo"]), math.log(c["list_hi"]))).sort().values
    gf, E = nrm(-3.0, 1.5), uni(0.0, 10.0).float()
    sp = torch.randint(0, 2 * c["n_metals"], (n,), generator=g, device=DEV, dtype=torch.int32)
    return wl.LineList(*(t.cpu().numpy() for t in (lam, gf, E, sp, nrm(-8.0, 0.5), nrm(-8.0, 0.5), nrm(-8.0, 0.5))))


def _points(c):
    """(T, P) of the table grid; four solar-type points when the grid is 4 x 1."""
    if (c["nT"], c["nP"]) == (4, 1):
        return np.array([4000.0, 6000.0, 9000.0, 15000.0]), np.full(4, 1e4)
    if c["nP"] == 1:
        return wl.tp_grid_dfsynthe(c["nT"], 2)[0][::2].copy(), np.full(c["nT"], 1e4)
    return wl.tp_grid_dfsynthe(c["nT"], c["nP"])


def _rows(c, n):
    """n_rows rows spread evenly over a table of n rows."""
    return np.array([(2 * k + 1) * n // (2 * c["n_rows"]) for k in range(c["n_rows"])], dtype=np.int32)


def _context(c, lines, T, P, abund=None, vturb=0.0):
    ctx = binding.Context(torch.cuda.current_device())
    ctx.load_linelist(lines, *wl.species_table(c["n_metals"]))
    ctx.set_atmosphere_grid(wl.elements(c["n_metals"]), T, P, abund_scale=abund, vturb=vturb)
    return ctx


def _batch_groups(c):
    """Windows, compositions and rows of the batch (the row of a group is one of comps x 57 x 25)."""
    r = np.random.default_rng(c["groups"])
    out = []
    for k in range(c["groups"]):
        # lengths spread over 1 nm .. dlam_hi in steps of equal ratio
        d = math.exp(math.log(c["dlam_hi"]) * (k + 0.5) / c["groups"])
        lam0 = math.exp(r.uniform(math.log(150.0), math.log(3000.0)))
        iT, iP = int(r.integers(5, 40)), int(r.integers(6, 20))
        out.append((lam0, d, int(r.integers(0, c["comps"])) * 1425 + iT * 25 + iP))
    return out


def _requests(c):
    """Spectrum requests: windows, depths and atmospheres of a burst."""
    r = np.random.default_rng(c["requests"])
    out = []
    for k in range(c["requests"]):
        d = math.exp(math.log(c["dlam_hi"]) * (k + 0.5) / c["requests"])
        lam0 = math.exp(r.uniform(math.log(200.0), math.log(2000.0)))
        D = 40 + (37 * k) % 81
        out.append((lam0, d, D, r.uniform(4500.0, 7500.0), r.uniform(2.0, 5.0)))
    return out


def _opacity_like(c, seed):
    """An opacity array with the structure of line opacities: every 64 points a line of log-normal
    strength and width on a slowly varying floor, and a stretch without lines (zeros)."""
    g, n, N = _gen(seed), c["n_rows"], c["N"]
    cells = N // 64 + 3
    amp = torch.pow(10.0, -1.0 + 1.5 * torch.randn((n, cells), generator=g, device=DEV))
    wid = torch.pow(10.0, 0.5 + 0.4 * torch.randn((n, cells), generator=g, device=DEV))
    off = 64.0 * torch.rand((n, cells), generator=g, device=DEV)
    j = torch.arange(N, device=DEV)
    cell, pos = j // 64, (j % 64).float()
    k = torch.empty((n, N), device=DEV)
    for r in range(n):
        k[r] = 1e-4 * torch.exp(3.0 * torch.sin(j * (6.0 / N) + r))
        for d in (0, 1, 2):
            q = cell + d
            k[r] += amp[r][q] / (1.0 + ((pos + (64.0 - 64.0 * d) - off[r][q]) / wid[r][q]) ** 2)
    k[:, : N // 50] = 0.0
    return k


def _bins_inputs(c, seed):
    g = _gen(seed)
    T, P = wl.tp_grid_dfsynthe(c["nT"], c["nP"])
    lt, lp = np.log10(T.reshape(c["nT"], c["nP"])[:, 0]).copy(), np.log10(P.reshape(c["nT"], c["nP"])[0]).copy()
    n, K, ns = c["nT"] * c["nP"], c["K"], c["n_steps"]
    rnd = lambda *s: torch.rand(s, generator=g, device=DEV, dtype=torch.float64)  # noqa: E731
    odf = torch.pow(10.0, -2.0 + 4.0 * rnd(n, K, 1) + torch.randn((n, K, ns), generator=g, device=DEV, dtype=torch.float64))
    odf = odf.sort(dim=-1).values.contiguous()
    kc = torch.pow(10.0, -3.0 + 3.0 * rnd(n)).float()
    edges = np.exp(np.linspace(math.log(9.0), math.log(10000.0), K + 1))
    m, Tr, Pr = (torch.from_numpy(a).to(DEV) for a in wl.ray_atmospheres(c["rays"], c["depths"], seed))
    w = WIDTHS if ns == 12 else [1.0 / ns] * ns
    return lt, lp, odf, kc, 0.5 * (edges[:-1] + edges[1:]), w, m, Tr, Pr, MUS[: c["n_mu"]]


def _odf_args(c):
    w = WIDTHS if c["n_steps"] == 12 else [1.0 / c["n_steps"]] * c["n_steps"]
    return wl.equal_intervals(c["N"], c["K"]), w


def prepare(case, seed):
    c = case
    if c["kind"] == "opacity":
        T, P = _points(c)
        ctx = _context(c, _lines(c, seed), T, P, vturb=c["vturb"])
        N, sel = binding.grid_size(c["lam0"], c["lam1"], c["R"]), _rows(c, len(T))
        return dict(kind="opacity", ctx=ctx, grid=wl.Grid(c["lam0"], c["lam1"], c["R"]), sel=sel,
                    kappa=torch.empty((len(sel), N), device=DEV), kappa_c=torch.empty(len(sel), device=DEV),
                    evals=torch.empty(len(sel), dtype=torch.int64, device=DEV), opts=binding.make_opts(CUT, KC_FACTOR))
    if c["kind"] == "spectrum":
        ctx = _context(c, _lines(c, seed), np.array([5000.0]), np.array([1e4]), vturb=c["vturb"])
        win = wl.Grid(c["lam0"], c["lam0"] + c["dlam"], c["R"])
        I = torch.empty((len(MUS), binding.grid_size(win.lam0_nm, win.lam1_nm, win.R)), device=DEV)
        return dict(kind="spectrum", ctx=ctx, win=win, atm=wl.grey_atmosphere(c["depths"], c["teff"], c["logg"]), I=I,
                    opts=binding.make_opts(CUT, KC_FACTOR, continuum=c["continuum"]))
    if c["kind"] == "batch":
        T, P = wl.tp_grid_dfsynthe()
        ab = wl.abundance_scales(c["comps"], 2 + c["n_metals"], seed)
        ctx = _context(c, _lines(c, seed), T, P, abund=ab)
        groups = []
        for lam0, d, row in _batch_groups(c):
            g = wl.Grid(lam0, lam0 + d, c["R"])
            groups.append(dict(grid=g, sel=np.array([row], dtype=np.int32),
                               kappa=torch.empty((1, binding.grid_size(g.lam0_nm, g.lam1_nm, g.R)), device=DEV),
                               kappa_c=torch.empty(1, device=DEV)))
        return dict(kind="batch", batch=binding.Batch(ctx, groups), ctx=ctx, groups=groups)
    if c["kind"] == "serve":
        ctx = _context(c, _lines(c, seed), np.array([5000.0]), np.array([1e4]))
        req = [(wl.grey_atmosphere(D, teff, logg), wl.Grid(lam0, lam0 + d, c["R"]))
               for lam0, d, D, teff, logg in _requests(c)]
        return dict(kind="serve", server=binding.Server(ctx, 64 << 30, max_inflight=8), req=req)
    if c["kind"] == "odf":
        b, w = _odf_args(c)
        return dict(kind="odf", ctx=binding.Context(torch.cuda.current_device()), kappa=_opacity_like(c, seed), bounds=b,
                    widths=w, odf=torch.empty((c["n_rows"], c["K"], c["n_steps"]), dtype=torch.float64, device=DEV),
                    mean=binding.MEAN_GEOM if c["geom"] else binding.MEAN_ARITH)
    if c["kind"] == "bins":
        a = _bins_inputs(c, seed)
        return dict(kind="bins", ctx=binding.Context(torch.cuda.current_device()), args=a,
                    I=torch.empty((c["rays"], c["n_mu"], c["K"]), device=DEV))
    T, P = wl.tp_grid_dfsynthe(c["nT"], c["nP"])
    ab = wl.abundance_scales(c["comps"], 2 + c["n_metals"], seed)
    N = binding.grid_size(c["lam0"], c["lam1"], c["R"])
    return dict(kind="plasma", ctx=binding.Context(torch.cuda.current_device()), eos=wl.eos_table(c["n_metals"]), T=T, P=P,
                ab=ab, n=c["comps"] * len(T), sel=_rows(c, c["comps"] * len(T)), grid=wl.Grid(c["lam0"], c["lam1"], c["R"]),
                kappa=torch.empty((c["n_rows"], N), device=DEV))


# ---------------------------------------------------------------------------
# One pass

def run(state):
    s = state
    if s["kind"] == "opacity":
        s["ctx"].synth_opacity(s["grid"], s["sel"], s["kappa"], s["kappa_c"], s["evals"], opts=s["opts"])
        return dict(kappa=s["kappa"], kappa_c=s["kappa_c"], evals=s["evals"])
    if s["kind"] == "spectrum":
        s["ctx"].synth_spectrum(*s["atm"], s["win"], MUS, s["I"], opts=s["opts"])
        return s["I"]
    if s["kind"] == "batch":
        s["batch"].run()
        return [dict(kappa=g["kappa"], kappa_c=g["kappa_c"]) for g in s["groups"]]
    if s["kind"] == "serve":
        tickets = [s["server"].submit_spectrum(*atm, win, MUS) for atm, win in s["req"]]
        return [s["server"].wait(t)[0] for t in tickets]
    if s["kind"] == "odf":
        s["ctx"].build_odf(s["kappa"], s["bounds"], s["widths"], s["odf"], s["mean"])
        return s["odf"]
    if s["kind"] == "bins":
        lt, lp, odf, kc, lam, w, m, T, P, mus = s["args"]
        s["ctx"].odf_intensity(lt, lp, odf, kc, lam, w, m, T, P, mus, s["I"])
        return s["I"]
    s["ctx"].set_atmosphere_grid_eos(s["eos"], s["T"], s["P"], abund_scale=s["ab"])
    pop = s["ctx"].get_populations(0, s["n"])
    s["ctx"].synth_continuum(s["grid"], s["sel"], s["kappa"])
    return dict(populations=pop, continuum=s["kappa"])


# ---------------------------------------------------------------------------
# Work

LINE_BYTES = 32      # lambda (8), log gf, E, three damping constants (20) and the species (4)
LINE_FLOPS = 60      # line strength, damping and cut window of one (row, line)
CORE_FLOPS = 20      # one profile value


def _grid_points(lam0, lam1, R):
    return int(math.log(lam1 / lam0) / math.log1p(1.0 / R)) + 1


def _synthesis_flops(c, rows, lam0, lam1):
    """Line terms of every (row, line), and the profile over the cores (six Doppler widths of 2 km/s
    on either side) of the lines centred on the grid; the wings are smooth, and how many operations
    they take is the implementation's business."""
    span = math.log(c["list_hi"] / c["list_lo"])
    inside = max(0.0, min(math.log(lam1 / lam0), math.log(c["list_hi"] / lam0))) / span
    core = min(12.0 * 2.0e3 / 2.998e8 * c["R"], _grid_points(lam0, lam1, c["R"]))
    return rows * c["n_lines"] * (LINE_FLOPS + min(1.0, inside) * core * CORE_FLOPS)


def work(case):
    c = case
    if c["kind"] == "opacity":
        N = _grid_points(c["lam0"], c["lam1"], c["R"])
        return dict(bytes=c["n_lines"] * LINE_BYTES + c["n_rows"] * N * 4,
                    flops=_synthesis_flops(c, c["n_rows"], c["lam0"], c["lam1"]))
    if c["kind"] == "spectrum":
        N = _grid_points(c["lam0"], c["lam0"] + c["dlam"], c["R"])
        return dict(bytes=c["n_lines"] * LINE_BYTES + 5 * N * 4,
                    flops=_synthesis_flops(c, c["depths"], c["lam0"], c["lam0"] + c["dlam"]) + c["depths"] * N * 5 * 15)
    if c["kind"] == "batch":
        g = _batch_groups(c)
        return dict(bytes=c["n_lines"] * LINE_BYTES + sum(4 * _grid_points(a, a + d, c["R"]) for a, d, _ in g),
                    flops=sum(_synthesis_flops(c, 1, a, a + d) for a, d, _ in g))
    if c["kind"] == "serve":
        q = _requests(c)
        pts = [(_grid_points(a, a + d, c["R"]), a, d, D) for a, d, D, _, _ in q]
        return dict(bytes=c["n_lines"] * LINE_BYTES + sum(20 * n for n, _, _, _ in pts),
                    flops=sum(_synthesis_flops(c, D, a, a + d) + D * n * 75 for n, a, d, D in pts))
    if c["kind"] == "odf":
        n = c["n_rows"] * c["N"]
        return dict(bytes=4 * n + 8 * c["n_rows"] * c["K"] * c["n_steps"], flops=n * (10 if c["geom"] else 1))
    if c["kind"] == "bins":
        u = c["rays"] * c["depths"] * c["K"] * c["n_steps"]
        return dict(bytes=8 * c["nT"] * c["nP"] * c["K"] * c["n_steps"] + 24 * c["rays"] * c["depths"] +
                    4 * c["rays"] * c["n_mu"] * c["K"], flops=u * (10 + 15 * c["n_mu"]))
    n, el = c["comps"] * c["nT"] * c["nP"], 2 + c["n_metals"]
    N = _grid_points(c["lam0"], c["lam1"], c["R"])
    return dict(bytes=8 * n * (5 + 5 * el) + 4 * c["n_rows"] * N, flops=n * el * 5 * 40 * 10 + c["n_rows"] * N * 30)


# ---------------------------------------------------------------------------
# FP64 restatement

C_CGS, H_CGS, K_CGS = 2.99792458e10, 6.62607015e-27, 1.380649e-16
ME, QE, AMU, EV = 9.1093837015e-28, 4.803204712570263e-10, 1.66053906660e-24, 1.602176634e-12
MAX_EVALS = 6e10     # profile values an exact opacity may take (some ten seconds)


def _eos(c, multi):
    """mass, log eps, stages, chi [n, 4], lnU [n, 5, 3] of the element table."""
    if multi:
        e = wl.eos_table(c["n_metals"])
        return e.mass_amu, e.log_eps, np.asarray(e.n_stages), e.chi_eV, e.lnU
    e = wl.elements(c["n_metals"])
    chi, lnU = np.zeros((e.n, 4)), np.zeros((e.n, 5, 3))
    chi[:, 0], lnU[:, 0, 0], lnU[:, 1, 0] = e.chi_eV, np.log(e.U1), np.log(e.U2)
    return e.mass_amu, e.log_eps, np.full(e.n, 2), chi, lnU


def _populations(eos, T, P, abund):
    """Rows T, P, n_e, n_HI, rho, N/U of five stages per element, for every (T, P) and scale row."""
    mass, log_eps, ns, chi, lnU = eos
    T, P = np.asarray(T, np.float64)[:, None], np.asarray(P, np.float64)[:, None]
    kT = K_CGS * T
    eps = 10.0 ** (log_eps - 12.0) * abund
    a = eps / eps.sum(axis=1, keepdims=True)
    x = np.log(T / 5040.0)[:, :, None]
    lu = lnU[None, :, :, 0] + x * (lnU[None, :, :, 1] + x * lnU[None, :, :, 2])            # [r, e, 5]
    lsaha = 1.5 * np.log(2.0 * math.pi * ME * kT / H_CGS ** 2)[:, :, None]
    lphi = math.log(2.0) + lu[:, :, 1:] - lu[:, :, :-1] + lsaha - chi[None] * EV / kT[:, :, None]
    on = np.arange(5)[None, None, :] < ns[None, :, None]
    j = np.arange(5)[None, None, :]
    n_tot = P / kT

    def weights(y):
        lp = np.concatenate([np.zeros_like(lphi[:, :, :1]), np.cumsum(lphi - y[:, :, None], axis=2)], axis=2)
        lp = np.where(on, lp, -np.inf)
        w = np.exp(lp - lp.max(axis=2, keepdims=True))
        return w / w.sum(axis=2, keepdims=True)

    lo, hi = np.full_like(n_tot, math.log(1e-300)), np.log(n_tot)
    for it in range(120):
        y = 0.5 * (lo + hi)
        ne = np.exp(y)
        q = (a * (weights(y) * j).sum(axis=2)).sum(axis=1, keepdims=True)
        up = ne - (n_tot - ne) * q > 0
        hi, lo = np.where(up, y, hi), np.where(up, lo, y)
    y = 0.5 * (lo + hi)
    ne = np.exp(y)
    nj = a[:, :, None] * (n_tot - ne)[:, :, None] * weights(y)
    rho = (n_tot - ne) * (a * mass).sum(axis=1, keepdims=True) * AMU
    nu = np.where(on, nj / np.exp(np.where(on, lu, 0.0)), 0.0)
    return np.concatenate([T, P, ne, nj[:, 0, :1], rho, nu.reshape(len(T), -1)], axis=1)


_WEIDEMAN = {}


def _w_core(z):
    """Faddeeva function by Weideman's rational expansion (1994, N = 64)."""
    if "a" not in _WEIDEMAN:
        N = 64
        M = 2 * N
        k = np.arange(-M + 1, M)
        L = math.sqrt(N / math.sqrt(2.0))
        t = L * np.tan(k * math.pi / M / 2.0)
        f = np.concatenate([[0.0], np.exp(-t * t) * (L * L + t * t)])
        _WEIDEMAN.update(a=[float(v) for v in np.real(np.fft.fft(np.fft.fftshift(f)))[1:N + 1][::-1] / (2 * M)], L=L)
    L, iz = _WEIDEMAN["L"], 1j * z
    d = 1.0 / (L - iz)
    Z, p = (L + iz) * d, torch.zeros_like(z)
    for a in _WEIDEMAN["a"]:
        p = p * Z + a
    return 2.0 * p * d * d + d / math.sqrt(math.pi)


def _h_inner(v, a):
    """H(v, a) where |z| < 40: Laplace's continued fraction outside |z| = 6 (with the Gaussian it
    leaves out), Weideman's expansion inside."""
    z = torch.complex(v, a)
    t = z
    for k in range(24, 0, -1):
        t = z - 0.5 * k / t
    h = (1j / t).real / math.sqrt(math.pi)
    h = h + torch.where(a < 1e-2, torch.exp(a * a - v * v) * torch.cos(2.0 * v * a), torch.zeros_like(v))
    core = v * v + a * a < 36.0
    if bool(core.any()):
        h[core] = _w_core(z[core]).real
    return h


def _h(v, a):
    """H(v, a) of a [n, 1] of damping constants and a [n, points] of arguments."""
    V, A = v * v, a * a
    r = 1.0 / (V + A)
    # w ~ i / (sqrt(pi) z) (1 + u + 3 u^2 + 15 u^3 + 105 u^4), u = 1 / (2 z^2): below 1e-13 for |z| >= 40
    ur, ui = 0.5 * (V - A) * r * r, -(v * a) * r * r
    pr, pi = torch.full_like(v, 105.0), torch.zeros_like(v)
    for k in (15.0, 3.0, 1.0, 1.0):
        pr, pi = pr * ur - pi * ui + k, pr * ui + pi * ur
    h = (a * pr - v * pi) * r / math.sqrt(math.pi)
    at = (V + A < 1600.0).nonzero(as_tuple=True)
    if len(at[0]):
        h[at] = _h_inner(v[at].abs(), a.expand_as(v)[at])
    return h


def _exact_opacity(c, lines, pops, grid, abund_elements, vturb):
    """kappa [rows, N] and kappa_c [rows] in FP64, or None where that takes too many profile values."""
    dev = lambda x: torch.from_numpy(np.asarray(x, dtype=np.float64)).to(DEV)  # noqa: E731
    lam = dev(lines.lam_nm) * 1e-7
    gf, E, gR, gS, gW = (torch.pow(10.0, dev(lines.log_gf)), dev(lines.E_eV), torch.pow(10.0, dev(lines.log_gR)),
                         torch.pow(10.0, dev(lines.log_gS)), torch.pow(10.0, dev(lines.log_gW)))
    sp = torch.from_numpy(lines.species.astype(np.int64)).to(DEV)
    se, ss = wl.species_table(c["n_metals"])
    N = _grid_points(grid.lam0_nm, grid.lam1_nm, grid.R)
    lnq, lam0 = math.log1p(1.0 / grid.R), grid.lam0_nm * 1e-7
    nu_j = C_CGS / (lam0 * torch.exp(torch.arange(N, device=DEV, dtype=torch.float64) * lnq))
    nu0, evals, out, kcs = C_CGS / lam, 0.0, [], []
    for row in pops:
        T, ne, nHI, rho = row[0], row[2], row[3], row[4]
        u = dev(np.sqrt(2.0 * K_CGS * T / (abund_elements[se] * AMU) + vturb ** 2))[sp]
        NU = dev(row[5 + 5 * se + ss])[sp]
        dnu = nu0 * u / C_CGS
        a = (gR + gS * ne + gW * nHI) / (4.0 * math.pi * dnu)
        S = (math.sqrt(math.pi) * QE ** 2 / (ME * C_CGS) / rho) * gf * NU / dnu * torch.exp(-E * EV / (K_CGS * T)) * \
            -torch.expm1(-H_CGS * nu0 / (K_CGS * T))
        k0 = S * torch.special.erfcx(a)
        kc = KC_FACTOR * float(k0.sort().values[(len(k0) - 1) // 2])
        t = CUT * kc
        s = S / t
        # no |v| beyond vb passes the cut: H <= 4 a / (sqrt(pi) v^2) + exp(-v^2 / 4)
        vb = torch.sqrt(8.0 * a * s / math.sqrt(math.pi)) + 2.0 * torch.sqrt(torch.log(2.0 * s).clamp(min=0.0)) + 1.0
        lo = (torch.log(C_CGS / (nu0 + vb * dnu) / lam0) / lnq).floor()
        low = nu0 - vb * dnu
        hi = torch.where(low > 0, torch.log(C_CGS / low.clamp(min=1.0) / lam0) / lnq, torch.full_like(low, 1e18)).ceil()
        keep = (k0 >= t) & (hi >= 0) & (lo < N)
        evals += float((torch.minimum(hi, torch.full_like(hi, N - 1.0)) - lo.clamp(min=0) + 1)[keep].sum())
        if evals > MAX_EVALS:
            return None
        at = keep.nonzero().flatten()
        q = [x[at] for x in (lo, hi, s, a, nu0, 1.0 / dnu)]
        acc = torch.zeros(N, device=DEV, dtype=torch.float64)
        G = 4096
        for j0 in range(0, N, G):
            j1 = min(N, j0 + G)
            hit = ((q[0] < j1) & (q[1] >= j0)).nonzero().flatten()
            for i in range(0, len(hit), 8192):
                h = hit[i:i + 8192]
                l = q[2][h, None] * _h((nu_j[None, j0:j1] - q[4][h, None]) * q[5][h, None], q[3][h, None])
                acc[j0:j1] += torch.where(l >= 1.0, l, torch.zeros_like(l)).sum(dim=0)
        out.append(acc * t)
        kcs.append(kc)
    return torch.stack(out), torch.tensor(kcs, device=DEV, dtype=torch.float64)


def _formal(tau, B, mus):
    """Emergent intensity for tau and B [D, ...] (linear source, diffusion below), stacked over mus."""
    out = []
    for mu in mus:
        I = B[-1] + mu * (B[-1] - B[-2]) / (tau[-1] - tau[-2])
        for d in range(len(tau) - 2, -1, -1):
            x = (tau[d + 1] - tau[d]) / mu
            e = torch.exp(-x)
            small = x < 1e-3
            xs = torch.where(small, torch.ones_like(x), x)
            f = torch.where(small, x * (0.5 - x * (1 / 3.0 - x * (0.125 - x / 30.0))), (-torch.expm1(-xs) - xs * e) / xs)
            I = I * e - B[d] * torch.expm1(-x) + (B[d + 1] - B[d]) * f
        x = tau[0] / mu
        out.append(I * torch.exp(-x) - B[0] * torch.expm1(-x))
    return torch.stack(out)


def _planck(lam_cm, T):
    return 2.0 * H_CGS * C_CGS ** 2 / lam_cm ** 5 / torch.expm1(H_CGS * C_CGS / (lam_cm * K_CGS * T))


def _continuum(pops, eos, lam_cm, sources):
    """Closed-form continuum [rows, N]."""
    chi = 13.598 * EV
    kbf = 64.0 * math.pi ** 4 * ME * QE ** 10 / (3.0 * math.sqrt(3.0) * C_CGS * H_CGS ** 6)
    kff = 4.0 * QE ** 6 / (3.0 * ME * H_CGS * C_CGS) * math.sqrt(2.0 * math.pi / (3.0 * K_CGS * ME))
    nu, out = C_CGS / lam_cm, []
    L2 = (lam_cm * 1e8).clamp(min=1300.0) ** 2
    ray = (5.799e-13 + (1.422e-6 + 2.784 / L2) / L2) / (L2 * L2)
    lnU = eos[4][0]
    for row in pops:
        T, ne, nHI, rho = row[0], row[2], row[3], row[4]
        x = math.log(T / 5040.0)
        U1, U2 = (math.exp(lnU[i][0] + x * (lnU[i][1] + x * lnU[i][2])) for i in (0, 1))
        kT, k = K_CGS * T, torch.zeros_like(nu)
        stim = -torch.expm1(-H_CGS * nu / kT)
        if sources & 1:
            k = k + ne * 6.6524587321e-25
        if sources & 2:
            for n in range(1, 9):
                Nn = nHI * 2.0 * n * n / U1 * math.exp(-chi * (1.0 - 1.0 / (n * n)) / kT)
                k = k + torch.where(nu >= chi / (H_CGS * n * n), Nn * kbf / (n ** 5 * nu ** 3), torch.zeros_like(nu)) * stim
        if sources & 4:
            k = k + kff * ne * row[6] * U2 / (math.sqrt(T) * nu ** 3) * stim
        if sources & 8:
            k = k + nHI * ray
        out.append(k / rho)
    return torch.stack(out)


def _grid_lam(lam0, lam1, R):
    return lam0 * 1e-7 * torch.exp(torch.arange(_grid_points(lam0, lam1, R), device=DEV, dtype=torch.float64) * math.log1p(1.0 / R))


def _exact_spectrum(c, lines, atm, win, vturb, sources):
    m, T, P = atm
    eos = _eos(c, False)
    pops = _populations(eos, T, P, np.ones((len(T), len(eos[0]))))
    got = _exact_opacity(c, lines, pops, win, eos[0], vturb)
    if got is None:
        return None
    kappa, kc = got
    lam = _grid_lam(win.lam0_nm, win.lam1_nm, win.R)
    k = kappa + (_continuum(pops, eos, lam, sources) if sources else kc[:, None])
    tau = [k[0] * m[0]]
    for d in range(1, len(m)):
        tau.append(tau[-1] + 0.5 * (k[d - 1] + k[d]) * (m[d] - m[d - 1]))
    B = [_planck(lam, t) for t in T]
    return _formal(torch.stack(tau), torch.stack(B), MUS)


def _exact_odf(c, seed):
    b, w = _odf_args(c)
    x = _opacity_like(c, seed)
    cw = [0.0]
    for v in w:
        cw.append(cw[-1] + v)
    cw[-1] = 1.0
    out = torch.empty((c["n_rows"], c["K"], c["n_steps"]), dtype=torch.float64, device=DEV)
    for k in range(c["K"]):
        y = x[:, int(b[k]):int(b[k + 1])].sort(dim=1).values.double()
        n = y.shape[1]
        zeros = (y == 0).sum(dim=1)
        if c["geom"]:
            y = torch.where(y > 0, torch.log(y), torch.zeros_like(y))
        cum = torch.cat([torch.zeros_like(y[:, :1]), y.cumsum(dim=1)], dim=1)
        S = []
        for u in (v * n for v in cw):
            i = min(int(math.floor(u)), n)
            S.append(cum[:, i] + ((u - i) * y[:, i] if i < n else 0.0))
        for s in range(c["n_steps"]):
            v = (S[s + 1] - S[s]) / (w[s] * n)
            out[:, k, s] = torch.where(cw[s] * n < zeros, torch.zeros_like(v), torch.exp(v)) if c["geom"] else v
    return out


def _exact_bins(c, seed):
    lt, lp, odf, kc, lam, w, m, T, P, mus = _bins_inputs(c, seed)
    ltd, lpd = torch.from_numpy(lt).to(DEV), torch.from_numpy(lp).to(DEV)
    odf, kc = odf.reshape(len(lt), len(lp), c["K"], c["n_steps"]), kc.double().reshape(len(lt), len(lp))
    lam_cm = torch.from_numpy(lam).to(DEV) * 1e-7
    wt = torch.tensor(w, dtype=torch.float64, device=DEV)

    def cell(ax, x):
        x = x.clamp(min=float(ax[0]), max=float(ax[-1]))
        i = (torch.searchsorted(ax, x, right=True) - 1).clamp(0, len(ax) - 2)
        return i, (x - ax[i]) / (ax[i + 1] - ax[i])

    out = []
    for r in range(0, c["rays"], 8):
        iT, fT = cell(ltd, torch.log10(T[r:r + 8]))
        iP, fP = cell(lpd, torch.log10(P[r:r + 8]))

        def mix(tab):
            e = (slice(None),) * 2 + (None,) * (tab.dim() - 2)
            return ((1 - fT) * (1 - fP))[e] * tab[iT, iP] + ((1 - fT) * fP)[e] * tab[iT, iP + 1] + \
                (fT * (1 - fP))[e] * tab[iT + 1, iP] + (fT * fP)[e] * tab[iT + 1, iP + 1]

        k = (mix(odf) + mix(kc)[:, :, None, None]).transpose(0, 1)                           # [D, ray, K, ns]
        mr, Tr = m[r:r + 8].T, T[r:r + 8].T
        dt = 0.5 * (k[1:] + k[:-1]) * (mr[1:] - mr[:-1])[:, :, None, None]
        tau = torch.cat([k[:1] * mr[:1, :, None, None], dt]).cumsum(dim=0)
        B = _planck(lam_cm[None, None, :], Tr[:, :, None])[..., None].expand_as(tau)
        out.append((_formal(tau, B, mus) * wt).sum(dim=-1).transpose(0, 1))                 # [ray, mu, K]
    return torch.cat(out)


def exact(case, seed):
    c = case
    if c["kind"] == "opacity":
        T, P = _points(c)
        rows, eos = _rows(c, len(T)), _eos(c, False)
        pops = _populations(eos, T[rows], P[rows], np.ones((len(rows), len(eos[0]))))
        got = _exact_opacity(c, _lines(c, seed), pops, wl.Grid(c["lam0"], c["lam1"], c["R"]), eos[0], c["vturb"])
        return None if got is None else dict(kappa=got[0], kappa_c=got[1], evals=None)
    if c["kind"] == "spectrum":
        return _exact_spectrum(c, _lines(c, seed), wl.grey_atmosphere(c["depths"], c["teff"], c["logg"]),
                               wl.Grid(c["lam0"], c["lam0"] + c["dlam"], c["R"]), c["vturb"], c["continuum"])
    if c["kind"] == "batch":
        T, P = wl.tp_grid_dfsynthe()
        ab, eos, lines, out = wl.abundance_scales(c["comps"], 2 + c["n_metals"], seed), _eos(c, False), _lines(c, seed), []
        for n, (lam0, d, row) in enumerate(_batch_groups(c)):
            if n % 4:            # a few of the windows: all of them would take too long
                out.append(dict(kappa=None, kappa_c=None))
                continue
            pops = _populations(eos, T[row % 1425:row % 1425 + 1], P[row % 1425:row % 1425 + 1], ab[row // 1425][None])
            got = _exact_opacity(c, lines, pops, wl.Grid(lam0, lam0 + d, c["R"]), eos[0], 0.0)
            out.append(dict(kappa=None, kappa_c=None) if got is None else dict(kappa=got[0], kappa_c=got[1]))
        return out
    if c["kind"] == "serve":
        lines, out = _lines(c, seed), []
        for n, (lam0, d, D, teff, logg) in enumerate(_requests(c)):
            got = None if n > 1 else _exact_spectrum(c, lines, wl.grey_atmosphere(D, teff, logg),
                                                     wl.Grid(lam0, lam0 + d, c["R"]), 0.0, 0)
            out.append(got)
        return out
    if c["kind"] == "odf":
        return _exact_odf(c, seed)
    if c["kind"] == "bins":
        return _exact_bins(c, seed)
    T, P = wl.tp_grid_dfsynthe(c["nT"], c["nP"])
    ab, eos = wl.abundance_scales(c["comps"], 2 + c["n_metals"], seed), _eos(c, True)
    pops = np.concatenate([_populations(eos, T, P, np.repeat(ab[k:k + 1], len(T), axis=0)) for k in range(c["comps"])])
    return dict(populations=pops, continuum=_continuum(pops[_rows(c, len(pops))], eos, _grid_lam(c["lam0"], c["lam1"], c["R"]), 15))
