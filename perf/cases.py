"""The work that a user of the library has it do, as cases that can be timed.

Each case is one call, or one job of a few calls, through the public Python
entry points on inputs that already lie on the GPU: Monte Carlo packet runs
(``Grid.run`` and the tallies it fills), the camera-directed emissivity fill,
the channel-map ray trace, the Lambda iteration, the batched launch of many
models, and the set-up of a grid with its line tables. Geometries, sizes and
physical constants are those of this repository's workloads, tests and
benchmark, scaled where a full job takes longer than a second or two.

Fields are made on the GPU from the case and the seed; the seed is also the
packets' random-number key.
"""
import math
from types import SimpleNamespace as NS

import numpy as np
import torch

import paper_2608_09340_gb300 as krl

DEV = "cuda"
AU = 1.495978707e13
G_CGS = 6.67430e-8
M_SUN = 1.98892e33
KB = 1.380649e-16
C_CGS = 2.99792458e10
AMU = 1.66053906660e-24
PARSEC = 3.0856775814913673e18

# arithmetic operations of one scattering and of one face crossing (two
# counter-based random blocks, the profile and sampler lookups, the new
# direction and frequency; the face distances and the step)
OPS_SCATTER, OPS_CROSS = 242, 32


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # the paper's Table 1 box with its fewest packets: the smallest
        # Monte Carlo call, set by latency
        dict(name="box32_1e3", kind="box", n=32, tau0=1e3, a=4.73e-3, packets=1_000),
        # the same box with a million packets: the ordinary run
        dict(name="box32_1e6", kind="box", n=32, tau0=1e3, a=4.73e-3, packets=1_000_000),
        # the static slab of the analytic test: 64 cells, tau0 = 1e4, 1e4 packets
        dict(name="slab64_1e4", kind="slab", n=64, tau0=1e4, a=1e-2, packets=10_000),
        # the benchmark's static sphere with its scattering map, at a depth
        # whose full job fits a second: the largest Monte Carlo job
        dict(name="sphere64_static", kind="sphere", n=64, tau0=3e4, a=4.7e-4, vmax=0.0, packets=500_000),
        # the benchmark's outflow at its depth: moving cells, escape in the wing
        dict(name="sphere64_outflow", kind="sphere", n=64, tau0=1e6, a=4.7e-4, vmax=200.0, packets=100_000),
        # the slab with dust: the packets carry a weight (rich walk, absorbed
        # weight per cell), (a tau0)^(1/3) tau_a = 1
        dict(name="dusty64", kind="dusty", n=64, tau0=1e4, a=0.015, zeta=1.0, packets=100_000),
        # first step of the two-step imaging: excitation, mean intensity and
        # the emissivity toward three cameras in 64 channels
        dict(name="fill128", kind="fill", n=128, channels=64, cameras=3, packets=1_000_000),
        # second step at full size: one inclination of 1024^2 pixels x 64
        # channels through 256^3 cells
        dict(name="trace256", kind="trace", n=256, channels=64, pixels=1024, theta=45.0, phi=0.0),
        # the molecular-cloud map: 128^2 pixels x 5 channels through 128^3
        # cells, channel count off the vector width
        dict(name="trace128_5ch", kind="trace", n=128, channels=5, pixels=128, theta=90.0, phi=30.0),
        # one cycle of the Lambda iteration on the 128^3 cloud: 4 lines of
        # 1e7 packets, tables per line, the per-cell solves
        dict(name="lambda128", kind="lambda", n=128, cycles=1, packets=10_000_000),
        # 64 spheres of uneven size and depth in one launch
        dict(name="batch64", kind="batch", models=64, tau_hi=1e5, packets=300_000),
        # what comes before a first run: grid, line tables with R_IIA, CDF
        dict(name="setup64", kind="setup", n=64, channels=16, cameras=3, emiss=True),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _count(rng, lo, hi):
    return int(round(_log(rng, lo, hi)))


def draw(rng):
    kind = rng.choice(["box", "slab", "sphere", "outflow", "dusty", "fill", "trace", "trace", "lambda", "batch", "setup"])
    if kind == "box":
        tau0 = _log(rng, 1e2, 3e3)
        return dict(kind="box", n=rng.randint(16, 64), tau0=tau0, a=_log(rng, 4e-4, 5e-3),
                    packets=min(_count(rng, 1e3, 1e6), int(1.5e9 / tau0)))
    if kind == "slab":
        tau0 = _log(rng, 1e3, 2e4)
        return dict(kind="slab", n=rng.randint(32, 128), tau0=tau0, a=_log(rng, 1e-3, 0.149),
                    packets=min(_count(rng, 1e3, 2e5), int(3e9 / tau0)))
    if kind == "sphere":
        tau0 = _log(rng, 1e3, 2e4)
        return dict(kind="sphere", n=rng.randint(32, 96), tau0=tau0, a=_log(rng, 1e-4, 1e-2), vmax=0.0,
                    packets=min(_count(rng, 1e3, 5e5), int(1e10 / tau0)))
    if kind == "outflow":
        tau0 = _log(rng, 1e4, 1e6)
        return dict(kind="sphere", n=rng.randint(32, 96), tau0=tau0, a=_log(rng, 1e-4, 1e-2),
                    vmax=rng.choice([-1.0, 1.0]) * rng.uniform(150.0, 300.0),
                    packets=min(_count(rng, 1e3, 5e5), int(5e10 / tau0)))
    if kind == "dusty":
        tau0 = _log(rng, 1e3, 1e4)
        return dict(kind="dusty", n=rng.randint(32, 96), tau0=tau0, a=_log(rng, 5e-3, 0.05), zeta=_log(rng, 0.01, 10.0),
                    packets=min(_count(rng, 1e3, 1e5), int(1e9 / tau0)))
    if kind == "fill":
        return dict(kind="fill", n=rng.randint(32, 128), channels=rng.randint(5, 64), cameras=rng.randint(1, 3),
                    packets=_count(rng, 1e4, 1e6))
    if kind == "trace":
        return dict(kind="trace", n=_count(rng, 32, 200), channels=rng.choice([5, 10, 16, 32, 64, rng.randint(1, 100)]),
                    pixels=_count(rng, 64, 700), theta=rng.choice([0.0, 45.0, 90.0, rng.uniform(0.0, 180.0)]),
                    phi=rng.uniform(0.0, 360.0))
    if kind == "lambda":
        return dict(kind="lambda", n=rng.randint(32, 128), cycles=1, packets=_count(rng, 1e5, 1e7))
    if kind == "batch":
        return dict(kind="batch", models=rng.randint(4, 64), tau_hi=_log(rng, 1e4, 1e5), packets=_count(rng, 1e4, 3e5))
    return dict(kind="setup", n=rng.randint(32, 128), channels=rng.randint(5, 32), cameras=rng.randint(1, 3),
                emiss=rng.random() < 0.5)


# ------------------------------------------------------------------ inputs

def _centres(n):
    k = torch.arange(n, device=DEV, dtype=torch.float64) + 0.5 - 0.5 * n
    z, y, x = torch.meshgrid(k, k, k, indexing="ij")
    return x, y, z


def _problem(shape, cell_cm, opacity, T_K, line, source, **more):
    p = dict(shape=shape, cell_cm=cell_cm, periodic=(False, False, False), opacity_kind="tau", opacity=opacity, T_K=T_K,
             line=line, source=source, vel_cms=None, n_coll=None, tau_abs=None, spectrum=(-30.0, 30.0, 200),
             channels=None, cameras=(), tallies=(), n_packets=1, seed=0)
    p.update(more)
    return NS(**p)


def _hydrogen(a):
    return NS(nu0_hz=2.466e15, mass_amu=1.00794, A_ul=6.265e8, g_u=6.0, g_l=2.0, k_ul=0.0, a_fixed=a, ph_mode=2)


def _rotor():
    return NS(nu0_hz=115.27e9, mass_amu=28.0, A_ul=1e-7, g_u=3.0, g_l=1.0, k_ul=1e-11, a_fixed=0.0, ph_mode=2)


def _source(kind, profile="line_centre", pos=(0.0, 0.0, 0.0), plane=0.0, rate=None):
    return NS(kind=kind, pos=pos, axis=2, plane=plane, band_axis=-1, band=(0.0, 0.0), profile=profile, luminosity=1.0,
              rate=rate)


def _box(c):
    n = c["n"]
    full = torch.full((n, n, n), c["tau0"] / (n / 2), device=DEV)
    return _problem((n, n, n), 1e15, full, 100.0, _hydrogen(c["a"]),
                    _source("volume", "gaussian", rate=torch.ones_like(full)), spectrum=(-20.0, 20.0, 200))


def _slab(c, T_K=1e4, **more):
    n = c["n"]
    return _problem((n, 1, 1), 1e13, torch.full((n, 1, 1), c["tau0"] / (n / 2), device=DEV), T_K, _hydrogen(c["a"]),
                    _source("plane", plane=n / 2), periodic=(True, True, False), **more)


def _dusty(c):
    n, tau_a = c["n"], c["zeta"] / (c["a"] * c["tau0"]) ** (1.0 / 3.0)
    return _slab(c, 10.0, tau_abs=torch.full((n, 1, 1), tau_a / (n / 2), device=DEV), spectrum=(-60.0, 60.0, 240))


def _sphere(c, tallies=("scatmap",)):
    n = c["n"]
    R = n / 2
    x, y, z = _centres(n)
    op = torch.where(x * x + y * y + z * z < R * R, c["tau0"] / R, 0.0).float()
    vel = torch.stack([x, y, z]).mul(c["vmax"] * 1e5 / R).float() if c["vmax"] else None
    return _problem((n, n, n), 1e15, op, 1e4, _hydrogen(c["a"]), _source("point", pos=(R, R, R)), vel_cms=vel,
                    spectrum=(-60.0, 60.0, 400), tallies=tallies)


def _envelope(n, channels, angles, tallies):
    """Rotating, infalling envelope around one solar mass: density r^-1.5
    outside a 100 AU cavity, free fall plus Keplerian rotation, a rotor's
    J = 1-0 line, thermal emission proportional to the emitters' density."""
    cell = 2000.0 * AU / n
    x, y, z = (q * cell for q in _centres(n))
    r = (x * x + y * y + z * z).sqrt()
    r_in = 100.0 * AU
    out = r >= r_in
    nH2 = torch.where(out, 1e6 * (r.clamp(min=r_in) / r_in) ** -1.5, 0.0)
    rs = r.clamp(min=0.5 * cell)
    v_k = (G_CGS * M_SUN / rs).sqrt()
    v_ff = v_k * math.sqrt(2.0)
    vel = torch.stack([torch.where(out, v, 0.0).float() for v in
                       ((-v_ff * x - v_k * y) / rs, (-v_ff * y + v_k * x) / rs, -v_ff * z / rs)])
    mol = 1e-4 * nH2
    half = 5e5
    return _problem((n, n, n), cell, (0.09 * mol).float(), 30.0, _rotor(),
                    _source("volume", "gaussian", rate=mol.float()), opacity_kind="n_l", vel_cms=vel,
                    n_coll=nH2.float(), spectrum=(-40.0, 40.0, 160), channels=(-half, 2.0 * half / channels, channels),
                    cameras=angles, tallies=tallies)


def _inclinations(k):
    return tuple((math.radians(t), 0.0) for t in (0.0, 45.0, 90.0)[:k])


def _random_field(n, slope, gen):
    k = torch.fft.fftfreq(n, device=DEV, dtype=torch.float64)
    kr = torch.fft.rfftfreq(n, device=DEV, dtype=torch.float64)
    kk = (k[:, None, None] ** 2 + k[None, :, None] ** 2 + kr[None, None, :] ** 2).sqrt()
    amp = torch.where(kk > 0, kk.clamp(min=1e-9) ** (slope / 2.0), 0.0)
    w = torch.randn((n, n, n), generator=gen, device=DEV, dtype=torch.float64)
    f = torch.fft.irfftn(torch.fft.rfftn(w) * amp, s=(n, n, n))
    return (f - f.mean()) / f.std()


LEVELS = 5


def _rotor_levels():
    J = np.arange(LEVELS, dtype=np.float64)
    A, k = np.zeros((LEVELS, LEVELS)), np.zeros((LEVELS, LEVELS))
    for u in range(1, LEVELS):
        A[u, u - 1] = 1e-7 * u ** 3
        k[u, :u] = 1e-11
    return 2.77 * J * (J + 1.0), 2.0 * J + 1.0, A, k


def _cloud(n, seed):
    """Turbulent molecular cloud: log-normal density, 1 km/s velocity field."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    rho = torch.exp(1.5 * _random_field(n, -11.0 / 3.0, gen))
    dens = 1e3 * rho / rho.mean()
    vel = torch.stack([1e5 * _random_field(n, -4.0, gen) for _ in range(3)]).float()
    mol = (1e-4 * dens).float()
    return _problem((n, n, n), 0.04 * PARSEC / n, mol, 20.0, _rotor(), _source("volume", "gaussian", rate=mol),
                    opacity_kind="n_l", vel_cms=vel, n_coll=dens.float(), spectrum=(-20.0, 20.0, 80), tallies=("exc",))


def _emissivity(p, c, seed):
    """Camera-directed emissivity [ncell][channels]: the emitters' density
    times a line profile around each cell's line-of-sight velocity, with the
    cell-to-cell scatter of a Monte Carlo estimate."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    th, ph = math.radians(c["theta"]), math.radians(c["phi"])
    n = (math.sin(th) * math.cos(ph), math.sin(th) * math.sin(ph), math.cos(th))
    vlos = sum(w * v for w, v in zip(n, p.vel_cms)).reshape(-1, 1)
    v0, dv, k = p.channels
    vk = (v0 + (torch.arange(k, device=DEV, dtype=torch.float32) + 0.5) * dv)
    em = ((vk - vlos) / 4e4).square_().neg_().exp_()
    noise = torch.rand(em.shape[0], generator=gen, device=DEV).add_(0.5)
    return em.mul_((p.source.rate.reshape(-1) / p.source.rate.max() * noise)[:, None])


# ------------------------------------------------------------------ prepare and run

def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind in ("box", "slab", "dusty", "sphere"):
        p = {"box": _box, "slab": _slab, "dusty": _dusty, "sphere": _sphere}[kind](c)
        return NS(case=c, seed=seed, grid=krl.Grid(p))
    if kind == "fill":
        p = _envelope(c["n"], c["channels"], _inclinations(c["cameras"]), ("exc", "J", "emiss"))
        return NS(case=c, seed=seed, grid=krl.Grid(p))
    if kind == "trace":
        p = _envelope(c["n"], c["channels"], (), ())
        return NS(case=c, grid=krl.Grid(p), emiss=_emissivity(p, c, seed))
    if kind == "lambda":
        p = _cloud(c["n"], seed)
        E, g, A, k = _rotor_levels()
        mol = p.opacity.reshape(-1).clone()
        pops = torch.zeros((mol.numel(), LEVELS), dtype=torch.float64, device=DEV)
        return NS(case=c, seed=seed, grid=krl.Grid(p), mol=mol, pops=pops, desc=krl.levels_desc(E, g, A, k, 28.0, mol))
    if kind == "batch":
        rng = np.random.default_rng(4)
        m = c["models"]
        side = rng.choice(np.array([32, 48, 64, 96, 128]), size=m)
        tau = np.exp(rng.uniform(math.log(1e3), math.log(c["tau_hi"]), m))
        a = np.exp(rng.uniform(math.log(1e-4), math.log(1e-2), m))
        vmax = rng.uniform(-300.0, 300.0, m)
        grids = [krl.Grid(_sphere(dict(n=int(side[i]), tau0=float(tau[i]), a=float(a[i]), vmax=float(vmax[i])), ()))
                 for i in range(m)]
        packets = [max(1, int(w)) for w in tau / tau.sum() * c["packets"]]
        return NS(case=c, seed=seed, grids=grids, batch=krl.Batch(grids), packets=packets)
    # set-up: the fields of one model among many, each with its own density
    p = _envelope(c["n"], c["channels"], _inclinations(c["cameras"]), ("exc", "J", "emiss") if c["emiss"] else ("exc",))
    gen = torch.Generator(device=DEV).manual_seed(seed)
    p.opacity = p.opacity * torch.rand(p.shape, generator=gen, device=DEV).add_(0.5)
    p.line.a_fixed = 1e-4 * (1.0 + seed % 97)
    return NS(case=c, problem=p)


def run(state):
    c, kind = state.case, state.case["kind"]
    if kind == "trace":
        return state.grid.raytrace(-1, c["pixels"], c["pixels"], float(c["n"]), emiss=state.emiss,
                                   theta=math.radians(c["theta"]), phi=math.radians(c["phi"]))
    if kind == "lambda":
        change = state.grid.levels_iterate(state.desc, c["cycles"], c["packets"], state.seed, state.pops)
        return {"pops": state.pops, "change": change}
    if kind == "batch":
        for g in state.grids:
            g.reset()
        state.batch.run(state.packets, seed=state.seed)
        return {k: torch.stack([g.tally(k) for g in state.grids]) for k in ("spec_w", "spec_n", "stats")}
    if kind == "setup":
        g = krl.Grid(state.problem)
        out = {k: g.tally(k) for k in _SETUP_OUT if c["emiss"] or k != "rtab"}
        g.close()
        return out
    state.grid.reset()
    state.grid.run(n=c["packets"], seed=state.seed, want_stats=False)
    out = {k: state.grid.tally(k) for k in ("spec_w", "spec_n", "stats") + _MORE_OUT.get(kind, ())}
    return out


_MORE_OUT = {"sphere": ("scatmap",), "dusty": ("absw",), "fill": ("exc", "J", "emiss")}
_SETUP_OUT = ("voigt", "us_lncdf", "rtab", "cells", "eps", "src_cdf")


# ------------------------------------------------------------------ what a pass cannot do without

def _scatterings(c):
    """Mean scatterings per packet: near tau0 in a static medium, fewer where
    the flow carries the photon out of the line's core."""
    if c["kind"] == "box":
        return 1.4 * c["tau0"]
    if c["kind"] == "sphere":
        return 2.0 * c["tau0"] / (1.0 + 0.11 * abs(c["vmax"]))
    return 1.6 * c["tau0"]


def work(case):
    c, kind = case, case["kind"]
    if kind in ("box", "slab", "dusty", "sphere"):
        ncell = c["n"] if kind in ("slab", "dusty") else c["n"] ** 3
        events = c["packets"] * _scatterings(c)
        per_cell = {"box": 24, "slab": 16, "dusty": 28, "sphere": 24}[kind]
        return {"bytes": ncell * per_cell + 70e3, "flops": events * OPS_SCATTER + c["packets"] * c["n"] * OPS_CROSS}
    if kind == "fill":
        ncell, segments = c["n"] ** 3, c["packets"] * 0.4 * c["n"]
        touched = segments * c["cameras"] * 0.3 * c["channels"]
        return {"bytes": ncell * (24 + 8 + c["channels"] * (8 + 4 * c["cameras"])), "flops": segments * 100 + touched * 12}
    if kind == "trace":
        ncell, rays = c["n"] ** 3, c["pixels"] ** 2
        return {"bytes": ncell * (16 + 4 * c["channels"]) + 4.0 * rays * c["channels"],
                "flops": rays * 1.2 * c["n"] * c["channels"] * 10}
    if kind == "lambda":
        ncell, lines = c["n"] ** 3, LEVELS - 1
        events = c["cycles"] * lines * c["packets"] * c["n"]
        return {"bytes": c["cycles"] * ncell * (lines * 36 + 16 * LEVELS), "flops": events * (OPS_CROSS + 40)}
    if kind == "batch":
        events = c["packets"] * 0.1 * c["tau_hi"]
        return {"bytes": c["models"] * 64.0 ** 3 * 16, "flops": events * OPS_SCATTER}
    ncell = c["n"] ** 3
    return {"bytes": ncell * (4 * 6 + 4 * 6 + 16 + 4 + 8) + (6.5e6 if c["emiss"] else 60e3),
            "flops": 48 * 8 * 5e3 + 40 * 250 * 60 + (1.6e6 * 250 * 8 if c["emiss"] else 0)}


# ------------------------------------------------------------------ 64-bit values

def _weideman(a, x, N=48):
    """Re w(x + i a) by Weideman's expansion (SIAM J. Numer. Anal. 31, 1497),
    the asymptotic series from |x| = 8 on."""
    L = math.sqrt(N / math.sqrt(2.0))
    M = 2 * N
    th = np.arange(-M + 1, M) * math.pi / M
    t = L * np.tan(th / 2)
    f = (L * L + t * t) * np.exp(-t * t)
    coef = np.array([(f * np.cos(k * th)).sum() / (2.0 * M) for k in range(1, N + 1)])
    z = np.minimum(x, 8.0) + 1j * a
    Z = (L + 1j * z) / (L - 1j * z)
    w = 2.0 * np.polyval(coef[::-1], Z) / (L - 1j * z) ** 2 + 1.0 / (math.sqrt(math.pi) * (L - 1j * z))
    zf = np.maximum(x, 8.0) + 1j * a
    term = np.ones_like(zf)
    s = np.ones_like(zf)
    for k in range(1, 25):
        term = term * (2 * k - 1) / (2.0 * zf * zf)
        s = s + term
    far = 1j / (math.sqrt(math.pi) * zf) * s
    return np.where(x >= 8.0, far.real, w.real)


def _slice(a):
    """ln H(a, x) at the 5000 nodes uniform in log10 x on [-4, 3]."""
    return np.log(_weideman(a, 10.0 ** np.linspace(-4.0, 3.0, 5000)))


def _masses(x, a):
    """Mass of exp(-u^2) / (a^2 + (x - u)^2) in the 250 u-cells of [-6, 6]:
    the Lorentz factor exactly, the Gaussian to second order."""
    u = -6.0 + 0.048 * np.arange(251)
    lo, hi, m = u[:-1], u[1:], 0.5 * (u[:-1] + u[1:])
    x = np.asarray(x)[:, None]
    dl, dh = lo - x, hi - x
    with np.errstate(all="ignore"):
        i0 = np.where(dl * dh > 0, np.arctan((hi - lo) * a / (a * a + dl * dh)), np.arctan(dh / a) - np.arctan(dl / a)) / a
    jx = 0.5 * np.log((a * a + dh * dh) / (a * a + dl * dl))
    i1 = jx + (x - m) * i0
    i2 = (hi - lo) - a * a * i0 + 2.0 * (x - m) * jx + (x - m) ** 2 * i0
    return np.exp(-m * m) * (i0 - 2.0 * m * i1 + (2.0 * m * m - 1.0) * i2)


def _line(p):
    b = math.sqrt(2.0 * KB * p.T_K / (p.line.mass_amu * AMU))
    a = p.line.a_fixed or p.line.A_ul / (4.0 * math.pi * p.line.nu0_hz * b / C_CGS)
    sigma0 = (p.line.g_u / p.line.g_l) * p.line.A_ul * C_CGS ** 3 / (8.0 * math.pi ** 1.5 * p.line.nu0_hz ** 3 * b)
    return b, a, sigma0


def _cells(p):
    b, _, sigma0 = _line(p)
    tau = p.opacity.double().reshape(-1) * (sigma0 * p.cell_cm)
    return torch.stack([tau] + [v.double().reshape(-1) / b for v in p.vel_cms], dim=1)


def _exact_setup(c, seed):
    p = prepare(c, seed).problem
    _, a, _ = _line(p)
    xs = np.where(np.arange(40) < 18, 8.0 * np.arange(40) / 18.0, 8.0 * 37.5 ** ((np.arange(40) - 18.0) / 21.0))
    cdf = np.concatenate([np.zeros((40, 1)), np.cumsum(_masses(xs, a), axis=1)], axis=1)
    cdf /= cdf[:, -1:]
    out = {"voigt": _slice(a), "us_lncdf": np.log(np.maximum(cdf, 1e-30)).reshape(-1), "cells": _cells(p).reshape(-1),
           "eps": None, "src_cdf": None}
    q = p.line.k_ul * p.n_coll.double().reshape(-1)
    out["eps"] = q / (p.line.A_ul + q)
    s = torch.cumsum(p.source.rate.double().reshape(-1), 0)
    out["src_cdf"] = s / s[-1]
    if c["emiss"]:
        w = _masses(np.linspace(0.0, 120.0, 200), a)
        w = torch.from_numpy(w / w.sum(axis=1, keepdims=True)).to(DEV)
        u = -6.0 + 0.048 * torch.arange(251, device=DEV, dtype=torch.float64)
        m = 0.5 * (u[:-1] + u[1:])
        D = -10.0 + 0.1 * torch.arange(201, device=DEV, dtype=torch.float64)
        rows = []
        for k in range(40):
            g = -1.0 + 2.0 * k / 39.0
            s = max(math.sqrt(max(0.0, 1.0 - g * g)) / math.sqrt(2.0), 0.1)
            kern = torch.exp(-(D[None, :] - m[:, None] * (g - 1.0)) ** 2 / (2.0 * s * s)) / (math.sqrt(2.0 * math.pi) * s)
            rows.append(w @ kern)
        out["rtab"] = torch.stack(rows).reshape(-1)
    return out


def _exact_trace(c, seed):
    """The formal solution along each ray in 64 bits: the profile slice of
    the line linear in log10|x| between its nodes, as the method defines it,
    and the segments from the planes that the ray crosses."""
    if c["pixels"] ** 2 * c["n"] * c["channels"] > 1.5e9:
        return None
    n, px, nch = c["n"], c["pixels"], c["channels"]
    p = _envelope(n, nch, (), ())
    em = _emissivity(p, c, seed)
    b, a, _ = _line(p)
    cells = _cells(p).float().double()
    lnH = torch.from_numpy(_slice(a)).to(DEV)
    th, ph = math.radians(c["theta"]), math.radians(c["phi"])
    d = np.array([math.sin(th) * math.cos(ph), math.sin(th) * math.sin(ph), math.cos(th)])
    eu = np.array([math.cos(th) * math.cos(ph), math.cos(th) * math.sin(ph), -math.sin(th)])
    ev = np.array([-math.sin(ph), math.cos(ph), 0.0])
    s = (torch.arange(px, device=DEV, dtype=torch.float64) + 0.5) * (n / px) - 0.5 * n
    vv, uu = torch.meshgrid(s, s, indexing="ij")
    P = [0.5 * n + uu.reshape(-1) * eu[k] + vv.reshape(-1) * ev[k] for k in range(3)]
    t_in, t_out = torch.full_like(P[0], -1e300), torch.full_like(P[0], 1e300)
    for k in range(3):
        if d[k] != 0.0:
            t0, t1 = -P[k] / d[k], (n - P[k]) / d[k]
            t_in, t_out = torch.maximum(t_in, torch.minimum(t0, t1)), torch.minimum(t_out, torch.maximum(t0, t1))
        else:
            t_out = torch.where((P[k] >= 0) & (P[k] < n), t_out, t_in)
    x0 = -(p.channels[0] + (torch.arange(nch, device=DEV, dtype=torch.float64) + 0.5) * p.channels[1]) / b
    I = torch.zeros((px * px, nch), dtype=torch.float64, device=DEV)
    tau = torch.zeros_like(I)
    t = t_out.clone()
    live = torch.nonzero(t_out > t_in).reshape(-1)
    # the cell on the camera's side, then one plane at a time away from it
    ci = [torch.floor(P[k] + t_out * d[k] - 1e-9 * np.sign(d[k])).clamp(0, n - 1) for k in range(3)]
    for _ in range(3 * n + 3):
        if live.numel() == 0:
            break
        nxt = torch.full_like(t[live], -1e300)
        axis = torch.zeros(live.numel(), dtype=torch.int64, device=DEV)
        for k in range(3):
            if abs(d[k]) > 1e-30:
                plane = ci[k][live] + (0.0 if d[k] > 0 else 1.0)
                tk = (plane - P[k][live]) / d[k]
                axis = torch.where(tk > nxt, k, axis)
                nxt = torch.maximum(nxt, tk)
        dl = (t[live] - nxt).clamp(min=0.0)[:, None]
        cell = ((ci[2][live] * n + ci[1][live]) * n + ci[0][live]).long()
        rec = cells[cell]
        xk = (x0[None, :] - (rec[:, 1:] @ torch.from_numpy(d).to(DEV))[:, None]).abs()
        q = ((torch.log10(xk.clamp(min=1e-300)) + 4.0) * (4999.0 / 7.0)).clamp(0.0, 4999.0)
        i = q.floor().clamp(max=4998.0).long()
        H = torch.exp(lnH[i] + (q - i) * (lnH[i + 1] - lnH[i]))
        H = torch.where(xk > 1e3, a / (math.sqrt(math.pi) * xk * xk) * (1.0 + 1.5 / (xk * xk)), H)
        dtau = rec[:, :1] * H * dl
        f = torch.where(dtau > 1e-12, -torch.expm1(-dtau) / dtau.clamp(min=1e-300), 1.0 - 0.5 * dtau)
        I[live] += torch.exp(-tau[live]) * em[cell].double() * dl * f
        tau[live] += dtau
        t[live] = nxt
        keep = torch.ones(live.numel(), dtype=torch.bool, device=DEV)
        for k in range(3):
            if abs(d[k]) > 1e-30:
                m = axis == k
                ci[k][live[m]] -= math.copysign(1.0, d[k])
                keep &= ~(m & ((ci[k][live] < 0) | (ci[k][live] > n - 1)))
        live = live[keep]
    return I.T.reshape(nch, px, px)


def exact(case, seed):
    if case["kind"] == "setup":
        return _exact_setup(case, seed)
    if case["kind"] == "trace":
        return _exact_trace(case, seed)
    return None     # a Monte Carlo walk in 64 bits takes minutes
