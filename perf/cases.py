"""Cases of the library's main paths for timing: what a program that uses it calls, over its range of sizes.

A case is a dict of plain values; ``kind`` names the path:

  kappa   rt_build_kappa, the line-by-line table of absorption coefficients over (T, nu);
  trace   rt_trace, the Monte-Carlo walk of rays through a grid of finite volumes with that table;
  batch   rt_batch_trace, many enclosures of uneven size in one launch;
  march   rt_march, the intensity along given rays at every wavenumber;
  train   rt_mlp_train_steps_nets, training steps of a spectral-band ensemble of surrogate networks;
  bands   rt_trace_mlp_bands, the walk with such an ensemble in place of the table.

Inputs come from the seed alone.  The walks' tables are made here (line strengths on the grid, convolved
with a Lorentz profile by FFT), not by the library's own line sum, so that a walk's inputs do not depend
on it.  ``exact`` restates each path in 64 bits with plain torch: Eqs. (S), (tau), (I) and (planck) of the
method, the Philox draws and the binary32 walk that the library specifies for its rays.
"""
import ctypes as ct
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_cs_0703028_gb300 as rt

H, C, KB, AMU, ATM = 6.62607015e-34, 299792458.0, 1.380649e-23, 1.66053906660e-27, 101325.0
C2 = 100.0 * H * C / KB  # second radiation constant, cm K
MASS, N_T, Q_EXP, T_REF = 44.0, 0.75, 1.0, 296.0
WIDTH, N_PARAM = 128, 50305
DEV = "cuda"


# ---------------------------------------------------------------- the cases
def listed():
    box32 = dict(nx=32, ny=32, nz=32, n_nu=100000, nu_min=2000.0, dnu=0.01, n_lines=20000, nT=64, T_min=800.0, T_max=2000.0)
    box128 = dict(nx=128, ny=128, nz=128, n_nu=400000, nu_min=1500.0, dnu=0.005, n_lines=100000, nT=64, T_min=500.0, T_max=2500.0)
    spec32 = {k: v for k, v in box32.items() if k not in ("nx", "ny", "nz")}
    spec128 = {k: v for k, v in box128.items() if k not in ("nx", "ny", "nz")}
    return [
        # one isothermal row of a 64-cell slab: 500 Lorentz lines from host memory, the smallest table a user
        # builds (a gas that is changed and rebuilt interactively): launches and copies
        dict(name="kappa_slab", kind="kappa", profile="lorentz", memory="host", n_nu=25000, nu_min=2000.0, dnu=0.02, n_lines=500,
             nT=1, T_min=1000.0, T_max=1000.0, cutoff=25.0, kappa_min=0.0),
        # the table of the 32^3 box: 20k Voigt lines, host line list through the Python call
        dict(name="kappa_box32", kind="kappa", profile="voigt", memory="host", cutoff=25.0, kappa_min=0.0, **spec32),
        # the table of the 128^3 box, the largest: 100k Voigt lines that stay on the GPU
        dict(name="kappa_box128", kind="kappa", profile="voigt", memory="device", cutoff=25.0, kappa_min=0.0, **spec128),
        # the same 20k lines with points per line adapted to temperature and intensity (the user trades the far wings)
        dict(name="kappa_adaptive", kind="kappa", profile="voigt", memory="device", cutoff=25.0, kappa_min=1e-3, **spec32),
        # the 64-cell slab traced and read back to the host, the smallest whole estimate
        dict(name="trace_slab", kind="trace", nx=64, ny=1, nz=1, n_nu=25000, nu_min=2000.0, dnu=0.02, n_lines=500, nT=1, T_min=1000.0,
             T_max=1000.0, n_rays=100000, x=0.1, px=False, tau_cut=False, slab=True, read=True),
        # the 32^3 box's 1e7 rays in its opaque gas
        dict(name="trace_box32", kind="trace", n_rays=10000000, x=0.1, px=False, tau_cut=False, slab=False, read=False, **box32),
        # an uneven grid of a thin gas with pressure and mole-fraction fields: most rays reach a wall with some of their power
        dict(name="trace_thin", kind="trace", nx=75, ny=52, nz=61, n_nu=60001, nu_min=2000.0, dnu=0.01, n_lines=12000, nT=33, T_min=500.0,
             T_max=2200.0, n_rays=8000000, x=2e-6, px=True, tau_cut=False, slab=False, read=False),
        # the 128^3 box with its pressure field, part of the 1e9 rays of its estimate: the largest walk
        dict(name="trace_box128", kind="trace", n_rays=400000000, x=0.1, px=True, tau_cut=False, slab=False, read=False, **box128),
        # enclosures of 8 to 48 cells a side that share one table, 200 rays a cell
        dict(name="batch_48", kind="batch", n_encl=48, side_lo=8, side_hi=48, rays_per_cell=200, x=0.1, n_nu=100000, nu_min=2000.0, dnu=0.01,
             n_lines=20000, nT=64, T_min=600.0, T_max=2000.0),
        # the intensity along 512 paths at all 100k wavenumbers of the 32^3 box, and what each beam loses
        dict(name="march_512", kind="march", n_paths=512, x=1e-3, incoming=True, **box32),
        # eight training steps, late in a schedule of 24000, of a group of spectral-band networks, 128 samples a step
        # and network
        dict(name="train_bands", kind="train", n_nets=1024, batch=128, n_batches=4, n_steps=8),
        # the 64^3 box walked with an ensemble of one network per 16 wavenumbers
        dict(name="walk_bands", kind="bands", nx=64, ny=64, nz=64, n_nu=100000, nu_min=2000.0, dnu=0.01, band_pts=16, T_min=600.0,
             T_max=2200.0, n_rays=10000000, log_kappa=5.0, tau_cut=False),
    ]


def draw(rng):
    def lg(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    def fl(a, b):
        return math.exp(rng.uniform(math.log(a), math.log(b)))

    kind = rng.choice(["kappa", "kappa", "kappa", "trace", "trace", "trace", "batch", "march", "train", "bands"])
    dnu = fl(0.005, 0.02)
    nT = lg(2, 64)
    T_min = rng.uniform(400.0, 900.0)
    T_max = T_min + rng.uniform(400.0, 1600.0)
    nu_min = rng.uniform(1500.0, 3000.0)
    spec = dict(nu_min=nu_min, dnu=dnu, nT=nT, T_min=T_min, T_max=T_max)
    if kind == "kappa":
        n_nu = lg(5000, 300000)
        per_cm = fl(1.0, 50.0)  # lines per cm^-1
        adaptive = rng.random() < 0.25
        return dict(kind=kind, profile=rng.choice(["lorentz", "voigt", "voigt"]), memory=rng.choice(["host", "device"]), n_nu=n_nu,
                    n_lines=max(50, int(per_cm * n_nu * dnu)), cutoff=rng.choice([5.0, 10.0, 25.0, 25.0]),
                    kappa_min=fl(1e-4, 1e-1) if adaptive else 0.0, **spec)
    if kind == "march":
        n_nu = lg(5000, 100000)
        return dict(kind=kind, nx=lg(8, 64), ny=lg(8, 64), nz=lg(8, 64), n_nu=n_nu, n_lines=max(50, int(20 * n_nu * dnu)),
                    n_paths=min(lg(32, 2000), 50000000 // n_nu), x=fl(1e-6, 0.1), incoming=rng.random() < 0.5, **spec)
    if kind == "train":
        n_nets = lg(1, 1024)
        return dict(kind=kind, n_nets=n_nets, batch=min(lg(64, 512), 131072 // n_nets), n_batches=rng.randint(1, 5), n_steps=rng.randint(2, 8))
    n_nu = lg(5000, 400000)
    x = fl(1e-6, 0.1)
    if kind == "batch":
        lo = lg(4, 16)
        return dict(kind=kind, n_encl=lg(4, 60), side_lo=lo, side_hi=lg(lo, 44), rays_per_cell=lg(10, 200), x=x, n_nu=n_nu,
                    n_lines=max(50, int(20 * n_nu * dnu)), **spec)
    sides = dict(nx=lg(8, 128), ny=lg(8, 128), nz=lg(8, 128))
    if kind == "bands":
        n_nu = lg(2000, 100000)
        return dict(kind=kind, n_nu=n_nu, nu_min=nu_min, dnu=dnu, band_pts=rng.choice([16, 16, 32, 64]), T_min=T_min, T_max=T_max,
                    n_rays=lg(200000, 5000000), log_kappa=rng.uniform(1.0, 6.0), tau_cut=rng.random() < 0.25, **sides)
    n_rays = lg(100000, 100000000)
    if x < 1e-3:  # a thin gas: every visit of a ray counts
        n_rays = min(n_rays, 8000000)
    return dict(kind=kind, n_nu=n_nu, n_lines=max(50, int(20 * n_nu * dnu)), n_rays=n_rays, x=x, px=rng.random() < 0.5, tau_cut=rng.random() < 0.25,
                slab=False, read=rng.random() < 0.25, **sides, **spec)


# ---------------------------------------------------------------- inputs
def _lines(case, rng):
    n = case["n_lines"]
    hi = case["nu_min"] + case["n_nu"] * case["dnu"]
    nu0 = np.sort(rng.uniform(case["nu_min"], hi, n))
    S = np.exp(rng.uniform(math.log(1e-22), math.log(1e-19), n))
    return SimpleNamespace(nu0=nu0, S_ref=S, gamma_ref=rng.uniform(0.05, 0.1, n), E_lower=rng.uniform(0.0, 5000.0, n), T_ref=T_REF,
                           n_T=N_T, q_exp=Q_EXP, mass_amu=MASS)


def _spec(case, x=0.1):
    return SimpleNamespace(nu_min=case["nu_min"], dnu=case["dnu"], n_nu=case["n_nu"], cutoff=case.get("cutoff", 25.0),
                           profile=case.get("profile", "voigt"), nT=case.get("nT", 2), T_min=case["T_min"], T_max=case["T_max"],
                           p_ref_atm=1.0, x_ref=x, points_per_line=0, accumulate=0, kappa_min=case.get("kappa_min", 0.0))


def _nodes(case):
    n = case["nT"]
    return np.array([case["T_min"]]) if n == 1 else case["T_min"] + np.arange(n) * ((case["T_max"] - case["T_min"]) / (n - 1))


def _strength(L, T, x):
    """u(T) S(T) of Eq. (S) and (tau) in 64 bits, [lines] at temperature T and 1 atm."""
    q = (T_REF / T) ** Q_EXP
    boltz = np.exp(-C2 * L.E_lower * (1.0 / T - 1.0 / T_REF))
    stim = np.expm1(-C2 * L.nu0 / T) / np.expm1(-C2 * L.nu0 / T_REF)
    return x * ATM / (KB * T) * 1e-6 * L.S_ref * q * boltz * stim


def _table(case, rng, x):
    """A spectrum of the workload's lines on the grid, [nT, n_nu] float32 on the GPU: the lines' strengths at
    each node on their grid points, convolved with the node's mean Lorentz profile."""
    L, n, dnu = _lines(case, rng), case["n_nu"], case["dnu"]
    at = np.clip(np.rint((L.nu0 - case["nu_min"]) / dnu).astype(np.int64), 0, n - 1)
    T = _nodes(case)
    hist = np.stack([np.bincount(at, weights=_strength(L, t, x), minlength=n) for t in T]) / dnu
    gam = np.maximum(0.075 * (T_REF / T) ** N_T, 2.5 * dnu)
    f = torch.arange(n // 2 + 1, dtype=torch.float64, device=DEV) / (n * dnu)
    damp = torch.exp(-2.0 * math.pi * torch.from_numpy(gam).to(DEV)[:, None] * f[None, :])
    out = torch.fft.irfft(torch.fft.rfft(torch.from_numpy(hist).to(DEV)) * damp, n=n)
    return torch.maximum(out, 1e-2 * out.mean(1, keepdim=True)).float().contiguous()


def _field(n, h, rng, k, lo, hi):
    """A smooth field over the cells: k Gaussians, scaled to [lo, hi]; float32, x fastest."""
    ax = [(torch.arange(m, dtype=torch.float64, device=DEV) + 0.5) * h for m in n]
    size = [m * h for m in n]
    v = torch.zeros(n[2], n[1], n[0], dtype=torch.float64, device=DEV)
    for _ in range(k):
        c = [rng.uniform(0.0, s) for s in size]
        sg = rng.uniform(0.05, 0.3) * max(size)
        e = [torch.exp(-(ax[i] - c[i]) ** 2 / (2 * sg * sg)) for i in range(3)]
        v += e[2][:, None, None] * e[1][None, :, None] * e[0][None, None, :]
    a, b = v.min(), v.max()
    v = (v - a) / (b - a) if float(b - a) > 0 else v * 0.0
    return (lo + (hi - lo) * v).float().reshape(-1).contiguous()


def _grid(case, rng, x):
    n = (case["nx"], case["ny"], case["nz"])
    if case.get("slab"):
        T = torch.full((n[0],), case["T_min"], dtype=torch.float32, device=DEV)
        return SimpleNamespace(nx=n[0], ny=1, nz=1, hx=1.0 / n[0], hy=math.inf, hz=math.inf, T=T, p_atm=None, x=None, ncells=n[0])
    h = 1.0 / max(n)
    T = _field(n, h, rng, 8, case["T_min"], case["T_max"])
    p = _field(n, h, rng, 4, 1.0, 3.0) if case.get("px") else None
    xf = _field(n, h, rng, 4, 0.5 * x, 2.0 * x) if case.get("px") else None
    return SimpleNamespace(nx=n[0], ny=n[1], nz=n[2], hx=h, hy=h, hz=h, T=T, p_atm=p, x=xf, ncells=n[0] * n[1] * n[2])


def _enclosures(case, rng):
    grids, rays = [], []
    sides = np.random.default_rng(case["n_encl"])  # the sizes are the case's, the fields are the seed's
    for _ in range(case["n_encl"]):
        n = [int(v) for v in sides.integers(case["side_lo"], case["side_hi"] + 1, 3)]
        g = _grid(dict(case, nx=n[0], ny=n[1], nz=n[2]), rng, case["x"])
        g.hx = g.hy = g.hz = 1.0 / 32
        grids.append(g)
        rays.append(case["rays_per_cell"] * g.ncells)
    return grids, rays


def _paths(case, rng, g):
    n = case["n_paths"]
    size = np.array([g.nx * g.hx, g.ny * g.hy, g.nz * g.hz])
    pos = (rng.uniform(0.02, 0.98, (n, 3)) * size).astype(np.float32)
    d = rng.normal(size=(n, 3))
    d = (d / np.linalg.norm(d, axis=1, keepdims=True)).astype(np.float32)
    nu = 100.0 * (case["nu_min"] + np.arange(case["n_nu"]) * case["dnu"])
    I_in = (2 * H * C * C * nu ** 3 / np.expm1(H * C / KB * nu / 1500.0) * rng.uniform(0.5, 1.0, case["n_nu"])).astype(np.float32)
    return pos, d, I_in if case["incoming"] else None


def _networks(n_nets, seed):
    """Weights U(+-1/sqrt(fan in)) of n_nets networks, [n_nets, N_PARAM] float32."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    fan = torch.full((N_PARAM,), WIDTH ** -0.5, dtype=torch.float32, device=DEV)
    fan[:640] = 0.5
    return (torch.rand(n_nets, N_PARAM, generator=gen, device=DEV) * 2.0 - 1.0) * fan


def _band_norms(case, n_nets, mean, scale):
    j0 = np.arange(n_nets) * case["band_pts"]
    j1 = np.minimum(j0 + case["band_pts"], case["n_nu"]) - 1
    lo = np.log(case["nu_min"] + j0 * case["dnu"])
    hi = np.maximum(np.log(case["nu_min"] + j1 * case["dnu"]), lo + 1e-6)
    one = np.ones(n_nets)
    return np.stack([lo, case["T_min"] * one, 0.5 * one, 0.01 * one, hi, case["T_max"] * one, 5.0 * one, 0.3 * one, mean * one,
                     scale * one], 1).astype(np.float32)


def _samples(case, seed):
    """Training samples of each network's band: log nu, T, p, x and the log kappa of a few lines there."""
    n_nets, n = case["n_nets"], case["batch"] * case["n_batches"]
    gen = torch.Generator(device=DEV).manual_seed(seed + 1)
    u = torch.rand(n_nets, n, 4, generator=gen, device=DEV, dtype=torch.float64)
    c = torch.rand(n_nets, 1, 12, generator=gen, device=DEV, dtype=torch.float64)
    band = dict(nu_min=2000.0, dnu=0.01, n_nu=16 * n_nets, band_pts=16, T_min=600.0, T_max=2200.0)
    norms = torch.from_numpy(_band_norms(band, n_nets, 4.0, 1.2)).to(DEV)
    lo, hi = norms[:, None, 0:4].double(), norms[:, None, 4:8].double()
    raw = lo + (hi - lo) * u
    g = 0.15 * (T_REF / raw[..., 1]) ** N_T * raw[..., 2]
    y = torch.zeros_like(raw[..., 0])
    for i in range(6):
        y += (0.1 + c[..., 6 + i]) * g / ((u[..., 0] - c[..., i]) ** 2 + g * g)
    return raw.float().contiguous(), (4.0 + 0.6 * torch.log(y * raw[..., 3] / 0.1)).float().contiguous(), norms


def prepare(case, seed):
    kind = case["kind"]
    rng = np.random.default_rng(seed)
    s = SimpleNamespace(case=case, seed=seed)
    if kind == "kappa":
        s.lines, s.spec = _lines(case, rng), _spec(case)
        s.out = torch.empty(case["nT"], case["n_nu"], dtype=torch.float32, device=DEV)
        if case["memory"] == "device":  # the program keeps the list on the GPU and counts the evaluations
            s.L, s.keep = rt.make_lines(s.lines, "device")
            s.S = rt.make_spectral(s.spec)
            s.evals = torch.zeros(1, dtype=torch.int64, device=DEV)
            s.status = torch.zeros(1, dtype=torch.int32, device=DEV)
    elif kind in ("trace", "march"):
        s.spec = _spec(case, case["x"])
        s.table = _table(case, rng, case["x"])
        s.g = _grid(case, rng, case["x"])
        s.grid, s.keep = rt.make_grid(s.g)
        if kind == "trace":
            s.tally = rt.Tally(s.g.ncells)
        else:
            s.pos, s.dir, s.I_in = (None if v is None else torch.from_numpy(v).to(DEV) for v in _paths(case, rng, s.g))
    elif kind == "batch":
        s.spec = _spec(case, case["x"])
        s.table = _table(case, rng, case["x"])
        grids, rays = _enclosures(case, rng)
        s.batch = rt.Batch(grids, rays, s.spec, seed=seed)
    elif kind == "train":
        s.inputs, s.targets, s.norms = _samples(case, seed)
        s.trainer = rt.MlpEnsembleTrainer(_networks(case["n_nets"], seed).reshape(-1).contiguous(), s.norms)
        s.losses = torch.zeros(case["n_steps"], dtype=torch.float32, device=DEV)
    elif kind == "bands":
        s.spec = _spec(case)
        s.g = _grid(case, rng, 0.1)
        s.grid, s.keep = rt.make_grid(s.g)
        n_nets = -(-case["n_nu"] // case["band_pts"])
        s.params = _networks(n_nets, seed).reshape(-1).contiguous()
        s.norms = torch.from_numpy(_band_norms(case, n_nets, case["log_kappa"], 1.5)).to(DEV)
        s.tally = rt.Tally(s.g.ncells)
    return s


# ---------------------------------------------------------------- one pass
def run(s):
    case, kind = s.case, s.case["kind"]
    if kind == "kappa":
        if case["memory"] == "host":
            return rt.build_kappa(s.lines, s.spec, out=s.out)
        s.evals.zero_()
        stream = ct.c_void_p(torch.cuda.current_stream().cuda_stream)
        st = rt.rt_build_kappa(ct.byref(s.L), ct.byref(s.S), s.out.data_ptr(), s.evals.data_ptr(), s.status.data_ptr(), stream)
        if st:
            raise rt.RtError(st, "rt_build_kappa", "")
        return [s.out, s.evals]
    if kind == "trace":
        s.tally.zero()
        rt.trace(s.grid, s.table, s.spec, s.tally, case["n_rays"], seed=s.seed, flags=rt.RT_TAU_CUT if case["tau_cut"] else 0)
        if case["read"]:
            absorbed, scalars, _ = s.tally.read()
            return [absorbed, scalars[:3], s.tally.steps]
        return [s.tally.absorbed, s.tally.scalars[:3], s.tally.steps]
    if kind == "batch":
        s.batch.zero()
        s.batch.trace(s.table)
        return [torch.cat([t.flat for t in s.batch.tallies]), torch.cat([t.steps for t in s.batch.tallies])]
    if kind == "march":
        I_out, power = rt.march(s.grid, s.table, s.spec, s.pos, s.dir, I_in=s.I_in)
        return [I_out, power]
    if kind == "train":
        t = s.trainer
        t.steps(s.inputs, s.targets, case["batch"], 3e-3, 1e-5, 18001, case["n_steps"], 24000, losses=s.losses)
        return [t.params, t.m, t.v, t.grad, s.losses]
    s.tally.zero()
    rt.trace_mlp_bands(s.grid, case["band_pts"], s.params, s.norms, s.spec, s.tally, case["n_rays"], seed=s.seed,
                       flags=rt.RT_TAU_CUT if case["tau_cut"] else 0)
    return [s.tally.absorbed, s.tally.scalars[:3], s.tally.steps]


# ---------------------------------------------------------------- what a pass cannot do without
def _evals(case):
    """(line, point) pairs within the cutoff (or the mean adaptive window) of a table, over its T nodes."""
    width = 2.0 * case["cutoff"]
    if case["kappa_min"] > 0:
        L = _lines(case, np.random.default_rng(0))
        w = [np.sqrt(_strength(L, T, 0.1) * L.gamma_ref * (T_REF / T) ** N_T / (math.pi * case["kappa_min"])) for T in _nodes(case)]
        width = 2.0 * float(np.mean(np.minimum(np.stack(w), case["cutoff"])))
    span = case["n_nu"] * case["dnu"]
    inside = max(0.25, 1.0 - 0.25 * width / span) if width < 2 * span else 0.5
    return case["n_lines"] * case["nT"] * min(width * inside / case["dnu"], float(case["n_nu"]))


def _visits(case, n, h, x):
    """Mean number of cells a ray crosses before a wall or before nothing is left of it."""
    to_wall = 0.67 * sum(n) / 3.0 if not case.get("slab") else 0.5 * n[0]
    kappa = 1e4 * x if "log_kappa" not in case else math.exp(case["log_kappa"])
    return min(to_wall, 1.0 + 104.0 / max(1e-9, kappa * 100.0 * h))


def work(case):
    kind = case["kind"]
    if kind == "kappa":
        # lines in, table out; one reciprocal and six operations an evaluation were every line summed at every point
        return {"bytes": 32.0 * case["n_lines"] + 4.0 * case["nT"] * case["n_nu"], "flops": 7.0 * _evals(case)}
    if kind == "train":
        n, p = case["n_nets"] * case["n_steps"], 4.0 * N_PARAM
        return {"bytes": n * (6.0 * p + 20.0 * case["batch"]), "flops": n * case["batch"] * 3.0 * 2.0 * 3 * WIDTH * WIDTH}
    if kind == "batch":
        m = 0.5 * (case["side_lo"] + case["side_hi"])
        cells = case["n_encl"] * m ** 3
        v = _visits(case, (m, m, m), 1.0 / 32, case["x"])
        return {"bytes": 4.0 * case["nT"] * case["n_nu"] + 20.0 * cells, "flops": cells * case["rays_per_cell"] * (250.0 + 40.0 * v)}
    n = (case["nx"], case["ny"], case["nz"])
    cells, h = n[0] * n[1] * n[2], 1.0 / max(n)
    if kind == "march":
        u = case["n_paths"] * case["n_nu"] * 0.67 * sum(n) / 3.0
        return {"bytes": 4.0 * case["n_nu"] * (case["nT"] + case["n_paths"]) + 12.0 * cells, "flops": 13.0 * u}
    v = _visits(case, n, h, case.get("x", 0.1))
    if kind == "bands":
        nets = -(-case["n_nu"] // case["band_pts"])
        return {"bytes": 4.0 * N_PARAM * nets + 20.0 * cells, "flops": case["n_rays"] * (250.0 + v * 2.0 * 3 * WIDTH * WIDTH)}
    return {"bytes": 4.0 * case["nT"] * case["n_nu"] + 20.0 * cells, "flops": case["n_rays"] * (250.0 + 40.0 * v)}


# ---------------------------------------------------------------- the same in 64 bits
def _weideman(n=48):
    """Weideman's (1994) rational series of the Faddeeva function: L and the n coefficients, highest power first."""
    m = 2 * n
    k = np.arange(-m + 1, m)
    L = math.sqrt(n / math.sqrt(2.0))
    t = L * np.tan(k * math.pi / m / 2)
    f = np.concatenate([[0.0], np.exp(-t * t) * (L * L + t * t)])
    a = np.real(np.fft.fft(np.fft.fftshift(f))) / (2 * m)
    return L, a[1:n + 1][::-1].copy()


def _voigt_h(x, y):
    """Re w(x + iy) in 64 bits: the asymptotic series (Abramowitz and Stegun 7.1.23) for |z| >= 20, Weideman's inside."""
    r2 = x * x + y * y
    t = 1.0 / r2
    s = y * y * t
    v = 1.0 + t * (1.5 - 2.0 * s + t * (3.75 + s * (12.0 * s - 15.0) + t * (13.125 + s * (-105.0 + s * (210.0 - 120.0 * s))
                   + t * (59.0625 + s * (-787.5 + s * (2835.0 + s * (1680.0 * s - 3780.0)))))))
    v *= y * t / math.sqrt(math.pi)
    near = (r2 < 400.0).nonzero(as_tuple=True)
    if near[0].numel():
        L, a = _weideman()
        z = torch.complex(x[near], y.expand_as(x)[near])
        d = 1.0 / (L - 1j * z)
        Z = (L + 1j * z) * d
        p = torch.full_like(Z, a[0])
        for c in a[1:]:
            p = p * Z + c
        v[near] = (2.0 * p * d * d + d / math.sqrt(math.pi)).real
    return v


def _exact_kappa(case, seed):
    if _evals(case) > 8e10:
        return None
    L = _lines(case, np.random.default_rng(seed))
    n, dnu, cut = case["n_nu"], case["dnu"], case["cutoff"]
    T = _nodes(case)
    out = torch.zeros(case["nT"], n, dtype=torch.float64, device=DEV)
    A = torch.from_numpy(np.stack([_strength(L, t, 0.1) for t in T])).to(DEV)
    gam = torch.from_numpy(np.stack([L.gamma_ref * (T_REF / t) ** N_T for t in T])).to(DEV)
    dop = torch.from_numpy(np.stack([L.nu0 / C * math.sqrt(2.0 * math.log(2.0) * KB * t / (MASS * AMU)) for t in T])).to(DEV)
    win = torch.full_like(A, cut)
    if case["kappa_min"] > 0:
        win = torch.minimum(win, torch.sqrt(A * gam / (math.pi * case["kappa_min"])))
    nu0 = torch.from_numpy(L.nu0).to(DEV)
    nu = case["nu_min"] + torch.arange(n, dtype=torch.float64, device=DEV) * dnu
    block = 1024
    for j0 in range(0, n, block):
        v = nu[j0:j0 + block]
        a, b = np.searchsorted(L.nu0, [float(v[0]) - cut - dnu, float(v[-1]) + cut + dnu])
        if a == b:
            continue
        step = max(1, int(6e7 / (v.numel() * (b - a))))
        for k in range(0, case["nT"], step):
            ks = slice(k, k + step)
            d = (v[None, :, None] - nu0[None, None, a:b]).expand(A[ks].shape[0], -1, -1)
            g = gam[ks, None, a:b]
            if case["profile"] == "lorentz":
                f = g / math.pi / (d * d + g * g)
            else:
                sc = math.sqrt(math.log(2.0)) / dop[ks, None, a:b]
                f = sc / math.sqrt(math.pi) * _voigt_h(sc * d, sc * g)
            out[ks, j0:j0 + block] = torch.where(d.abs() <= win[ks, None, a:b], A[ks, None, a:b] * f, 0.0).sum(2)
    return out


def _philox(c, seed):
    """Philox4x32-10 (Salmon et al., SC'11) of counters c = [4] int64 tensors with values below 2^32."""
    m = 0xFFFFFFFF
    k0, k1 = seed & m, (seed >> 32) & m

    def mul(a, b):  # high and low words of a * b
        p = a * (b >> 16)
        q = a * (b & 0xFFFF)
        return (p + (q >> 16)) >> 16, (((p & 0xFFFF) << 16) + q) & m

    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & m, (k1 + 0xBB67AE85) & m
    return c


def _u24(v):
    return (v >> 8).float() * 2.0 ** -24


def _marsaglia(a, b):
    a, b = 2.0 * _u24(a) - 1.0, 2.0 * _u24(b) - 1.0
    s = a * a + b * b
    ok = (s < 1.0) & (s != 0.0)
    q = torch.sqrt(torch.clamp(1.0 - s, min=0.0))
    return ok, 2.0 * a * q, 2.0 * b * q, 1.0 - 2.0 * s


class _Walk:
    """The rays r0 .. r1 of an estimate: their draws and the binary32 walk."""

    def __init__(self, g, n_nu, r0, r1, seed, enclosure=0):
        r = torch.arange(r0, r1, dtype=torch.int64, device=DEV)
        ctr = lambda q, call: [q & 0xFFFFFFFF, q >> 32, torch.full_like(q, call), torch.full_like(q, enclosure)]  # noqa: E731
        v = _philox(ctr(r, 0), seed)
        self.cell = (v[0] * g.ncells) >> 32
        self.j = (v[1] * n_nu) >> 32
        w = _philox(ctr(r, 1), seed)
        f = [_u24(v[2]), _u24(v[3]), _u24(w[0])]
        ok, dx, dy, dz = _marsaglia(w[1], w[2])
        for call in range(2, 64):
            left = (~ok).nonzero(as_tuple=True)[0]
            if not left.numel():
                break
            w = _philox(ctr(r[left], call), seed)
            o1, x1, y1, z1 = _marsaglia(w[0], w[1])
            o2, x2, y2, z2 = _marsaglia(w[2], w[3])
            ok[left] = o1 | o2
            for t, p, q in ((dx, x1, x2), (dy, y1, y2), (dz, z1, z2)):
                t[left] = torch.where(o1, p, q)
        d = [dx, dy, dz]
        self.n = [g.nx, g.ny, g.nz]
        h = [g.hx, g.hy, g.hz]
        self.stride = [1, g.nx, g.nx * g.ny]
        self.i = [self.cell % g.nx, self.cell // g.nx % g.ny, self.cell // (g.nx * g.ny)]
        self.h = [torch.tensor(v if math.isfinite(v) else 0.0, dtype=torch.float32, device=DEV) for v in h]
        self.p = [(self.i[a].float() + f[a]) * self.h[a] for a in range(3)]
        self.iv, self.t = [], []
        for a in range(3):
            fin = (d[a] != 0.0) & math.isfinite(h[a])
            iv = torch.where(fin, 1.0 / d[a], 0.0)
            self.iv.append(iv)
            t = ((self.i[a] + (iv > 0)).float() * self.h[a] - self.p[a]) * iv
            self.t.append(torch.where(fin, t, math.inf))
        self.at = torch.zeros_like(dx)

    def keep(self, m):
        for name in ("cell", "j", "at"):
            setattr(self, name, getattr(self, name)[m])
        for name in ("i", "p", "iv", "t"):
            setattr(self, name, [v[m] for v in getattr(self, name)])

    def step(self):
        """The visit's length (float32) and cell, and whether the ray leaves; the walk goes to the next cell."""
        t, c = self.t, self.cell
        a0 = (t[0] <= t[1]) & (t[0] <= t[2])
        a1 = ~a0 & (t[1] <= t[2])
        sel = [a0, a1, ~a0 & ~a1]
        pick = lambda v: torch.where(a0, v[0], torch.where(a1, v[1], v[2]))  # noqa: E731
        tn, iv, i, p = pick(t), pick(self.iv), pick(self.i), pick(self.p)
        st = torch.where(iv > 0, 1, -1)
        i = i + st
        n = pick([torch.full_like(i, m) for m in self.n])
        out = torch.isinf(tn) | (i < 0) | (i >= n)
        ds = tn - self.at
        tm = ((i + (st > 0)).float() * pick([v.expand_as(p) for v in self.h]) - p) * iv
        self.at = tn
        self.cell = c + st * pick([torch.full_like(i, m) for m in self.stride])
        self.i = [torch.where(sel[a], i, self.i[a]) for a in range(3)]
        self.t = [torch.where(sel[a], tm, t[a]) for a in range(3)]
        return ds, c, out


def _tally(g, n_nu, n_rays, seed, spec, kappa, enclosure=0, chunk=20000000):
    """[absorbed | emitted, 0, escaped, 0] of n_rays rays; kappa(walk, cell): each ray's coefficient in a cell, 64 bits."""
    flat = torch.zeros(g.ncells + 4, dtype=torch.float64, device=DEV)
    V = math.prod(v for v in (g.hx, g.hy, g.hz) if math.isfinite(v))
    scale = 4.0 * math.pi * V * 100.0 * 100.0 * spec.dnu * g.ncells * n_nu / n_rays
    for r0 in range(0, n_rays, chunk):
        W = _Walk(g, n_nu, r0, min(n_rays, r0 + chunk), seed, enclosure)
        nu = 100.0 * (spec.nu_min + W.j.double() * spec.dnu)
        ib = 2.0 * H * C * C * nu ** 3 / torch.expm1(H * C / KB * nu / g.T[W.cell].double())
        w = tau = None
        while W.cell.numel():
            k = kappa(W, W.cell)
            if w is None:
                w, tau = scale * k * ib, torch.zeros_like(k)
                flat[g.ncells] += w.sum()
            ds, cell, out = W.step()
            a = torch.clamp(k * 100.0 * ds.double(), max=1e30)
            flat.index_add_(0, cell, w * torch.exp(-tau) * -torch.expm1(-a))
            tau = tau + a
            flat[g.ncells + 2] += (w * torch.exp(-tau) * out).sum()
            go = ~out & (tau < 200.0)
            w, tau = w[go], tau[go]
            W.keep(go)
    return flat


def _table_kappa(case, table, g, x):
    """The table's coefficient of a ray in a cell: linear in T, its bracket in binary32 as specified, times the density scale."""
    n = case["nT"]
    scale = torch.ones(g.ncells, dtype=torch.float64, device=DEV)
    if g.p_atm is not None:
        scale = g.p_atm.double() * g.x.double() / x
    if n == 1:
        return lambda W, c: scale[c] * table[0, W.j].double()
    dT = torch.tensor((case["T_max"] - case["T_min"]) / (n - 1), dtype=torch.float32, device=DEV)
    u = (g.T - torch.tensor(case["T_min"], dtype=torch.float32, device=DEV)) / dT
    k = torch.clamp(torch.floor(u), 0, n - 2)
    f, k = torch.clamp(u - k, 0.0, 1.0).double(), k.long()
    return lambda W, c: scale[c] * ((1.0 - f[c]) * table[k[c], W.j].double() + f[c] * table[k[c] + 1, W.j].double())


def _exact_march(case, seed):
    rng = np.random.default_rng(seed)
    table = _table(case, rng, case["x"])
    g = _grid(case, rng, case["x"])
    pos, d, I_in = _paths(case, rng, g)
    n, dnu = case["n_nu"], case["dnu"]
    nu = 100.0 * (case["nu_min"] + torch.arange(n, dtype=torch.float64, device=DEV) * dnu)
    I0 = torch.zeros(n, dtype=torch.float64, device=DEV) if I_in is None else torch.from_numpy(I_in).to(DEV).double()
    W = _Walk.__new__(_Walk)  # the given paths in place of drawn rays
    W.n, W.stride = [g.nx, g.ny, g.nz], [1, g.nx, g.nx * g.ny]
    W.h = [torch.tensor(v, dtype=torch.float32, device=DEV) for v in (g.hx, g.hy, g.hz)]
    W.p = [torch.from_numpy(pos[:, a].copy()).to(DEV) for a in range(3)]
    d = [torch.from_numpy(d[:, a].copy()).to(DEV) for a in range(3)]
    W.i = [torch.clamp(torch.floor(W.p[a] / W.h[a]).long(), 0, W.n[a] - 1) for a in range(3)]
    W.iv = [torch.where(v != 0, 1.0 / v, 0.0) for v in d]
    W.t = [torch.where(d[a] != 0, ((W.i[a] + (W.iv[a] > 0)).float() * W.h[a] - W.p[a]) * W.iv[a], math.inf) for a in range(3)]
    W.cell = W.i[0] + g.nx * (W.i[1] + g.ny * W.i[2])
    W.j, W.at = torch.zeros_like(W.cell), torch.zeros_like(W.p[0])
    visits, alive = [], torch.ones_like(W.cell, dtype=torch.bool)
    while bool(alive.any()):
        ds, cell, out = W.step()
        visits.append((torch.where(alive, ds, 0.0).double(), torch.where(alive, cell, 0)))
        alive = alive & ~out
        W.cell = torch.clamp(W.cell, 0, g.ncells - 1)
    kap = _table_kappa(case, table, g, case["x"])
    I_out = torch.empty(case["n_paths"], n, dtype=torch.float64, device=DEV)
    step = max(1, 20000000 // n)
    every = SimpleNamespace(j=torch.arange(n, device=DEV)[None, :])
    for a in range(0, case["n_paths"], step):
        I = I0.expand(min(step, case["n_paths"] - a), n)
        for ds, cell in visits:
            ds, c = ds[a:a + step, None], cell[a:a + step, None]
            if not bool((ds > 0).any()):
                continue
            att = -torch.expm1(-kap(every, c) * 100.0 * ds)
            I = I + att * (2.0 * H * C * C * nu ** 3 / torch.expm1(H * C / KB * nu / g.T[c].double()) - I)
        I_out[a:a + step] = I
    return [I_out, ((I0 - I_out) * (100.0 * dnu)).sum(1)]


def _layers(P):
    """W1, b1, W2, b2, W3, b3, W4, b4, w5, b5 of networks P [n, N_PARAM] (views)."""
    out, at = [], 0
    for shape in ((WIDTH, 4), (WIDTH,), (WIDTH, WIDTH), (WIDTH,), (WIDTH, WIDTH), (WIDTH,), (WIDTH, WIDTH), (WIDTH,), (1, WIDTH), (1,)):
        m = math.prod(shape)
        out.append(P[:, at:at + m].reshape(P.shape[0], *shape))
        at += m
    return out


def _exact_train(case, seed):
    if case["n_nets"] * case["batch"] * case["n_steps"] > 4000000:
        return None
    raw, target, norms = _samples(case, seed)
    nm = norms.double()
    P = _networks(case["n_nets"], seed).double()
    m, v, n = torch.zeros_like(P), torch.zeros_like(P), case["batch"]
    losses = []
    for i in range(case["n_steps"]):
        step = 18000 + i
        b = step % case["n_batches"] * n
        u = 2.0 * (raw[:, b:b + n].double() - nm[:, None, 0:4]) / (nm[:, None, 4:8] - nm[:, None, 0:4]) - 1.0
        y0 = (target[:, b:b + n].double() - nm[:, 8:9]) / nm[:, 9:10]
        L = _layers(P)
        h, z = [u], []
        for k in range(4):
            z.append(torch.baddbmm(L[2 * k + 1][:, None, :], h[-1], L[2 * k].transpose(1, 2)))
            h.append(z[-1] * torch.sigmoid(z[-1]))
        y = torch.baddbmm(L[9][:, None, :], h[4], L[8].transpose(1, 2))[..., 0]
        losses.append(float((0.5 * (y - y0) ** 2).mean()))
        dz = ((y - y0) / n)[..., None]
        grads = [dz.sum(1), torch.bmm(dz.transpose(1, 2), h[4])]
        for k in range(3, -1, -1):
            s = torch.sigmoid(z[k])
            dz = torch.bmm(dz, L[2 * k + 2]) * s * (1.0 + z[k] * (1.0 - s))
            grads += [dz.sum(1), torch.bmm(dz.transpose(1, 2), h[k])]
        G = torch.cat([q.reshape(P.shape[0], -1) for q in grads[::-1]], 1)
        lr = 1e-5 + 0.5 * (3e-3 - 1e-5) * (1.0 + math.cos(math.pi * step / 23999))
        m, v = 0.9 * m + 0.1 * G, 0.999 * v + 0.001 * G * G
        P = P - lr * (m / (1 - 0.9 ** (step + 1))) / (torch.sqrt(v / (1 - 0.999 ** (step + 1))) + 1e-8)
    return [P.reshape(-1), m.reshape(-1), v.reshape(-1), G.reshape(-1), torch.tensor(losses, dtype=torch.float64)]


def _exact_bands(case, seed):
    n = (case["nx"], case["ny"], case["nz"])
    if case["n_rays"] * _visits(case, n, 1.0 / max(n), 0.1) > 3e7:
        return None
    g = _grid(case, np.random.default_rng(seed), 0.1)
    n_nets = -(-case["n_nu"] // case["band_pts"])
    P = _networks(n_nets, seed)
    nm = torch.from_numpy(_band_norms(case, n_nets, case["log_kappa"], 1.5)).to(DEV).double()

    def kappa(W, c):
        band, order = torch.sort(W.j // case["band_pts"])
        one = torch.ones_like(band, dtype=torch.float64)
        raw = torch.stack([torch.log(case["nu_min"] + W.j[order].double() * case["dnu"]), g.T[c[order]].double(), one, 0.1 * one], 1)
        u = 2.0 * (raw - nm[band, 0:4]) / (nm[band, 4:8] - nm[band, 0:4]) - 1.0
        out = torch.empty_like(one)
        ends = torch.searchsorted(band, torch.arange(n_nets + 1, device=DEV)).tolist()
        group = 256
        for b0 in range(0, n_nets, group):  # the rays of up to 256 networks, padded to the same number each
            b1 = min(n_nets, b0 + group)
            s, e = ends[b0], ends[b1]
            if s == e:
                continue
            first = torch.tensor(ends[b0:b1], device=DEV)
            m = max(ends[b + 1] - ends[b] for b in range(b0, b1))
            place = (band[s:e] - b0) * m + torch.arange(s, e, device=DEV) - first[band[s:e] - b0]
            h = torch.zeros((b1 - b0) * m, 4, dtype=torch.float64, device=DEV)
            h[place] = u[s:e]
            h = h.reshape(b1 - b0, m, 4)
            L = _layers(P[b0:b1].double())
            for k in range(4):
                z = torch.baddbmm(L[2 * k + 1][:, None, :], h, L[2 * k].transpose(1, 2))
                h = z * torch.sigmoid(z)
            y = torch.baddbmm(L[9][:, None, :], h, L[8].transpose(1, 2)).reshape(-1)
            out[s:e] = torch.exp(nm[band[s:e], 8] + nm[band[s:e], 9] * y[place])
        back = torch.empty_like(out)
        back[order] = out
        return back

    flat = _tally(g, case["n_nu"], case["n_rays"], seed, _spec(case), kappa, chunk=5000000)
    return [flat[:g.ncells], flat[g.ncells:g.ncells + 3], None]


def exact(case, seed):
    kind = case["kind"]
    if kind == "kappa":
        out = _exact_kappa(case, seed)
        return out if out is None or case["memory"] == "host" else [out, None]
    if kind == "march":
        return _exact_march(case, seed)
    if kind == "train":
        return _exact_train(case, seed)
    if kind == "bands":
        return _exact_bands(case, seed)
    rng = np.random.default_rng(seed)
    table, spec = _table(case, rng, case["x"]), _spec(case, case["x"])
    if kind == "batch":
        grids, rays = _enclosures(case, rng)
        flats = [_tally(g, case["n_nu"], n, seed, spec, _table_kappa(case, table, g, case["x"]), enclosure=e) for e, (g, n) in enumerate(zip(grids, rays))]
        return [torch.cat(flats), None]
    g = _grid(case, rng, case["x"])
    if case["n_rays"] * _visits(case, (g.nx, g.ny, g.nz), g.hx, case["x"]) > 3e9:
        return None
    flat = _tally(g, case["n_nu"], case["n_rays"], seed, spec, _table_kappa(case, table, g, case["x"]))
    if case["read"]:
        flat[g.ncells + 1] = flat[:g.ncells].sum()
    return [flat[:g.ncells], flat[g.ncells:g.ncells + 3], None]
