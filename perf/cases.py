"""Performance cases: what programs built on this library have it do, as calls of its public entry
points.

A case is a domain (mesh, bathymetry, forcing and boundary kinds of one of the workload families),
a discretisation (degree, flux, Runge-Kutta scheme, precision, limiter) and a use:

  "run"       advance the model some steps and take the state on device (dgswe_get_state_device);
  "monitor"   advance some steps, then read the mass ledger, the total volume, the wet/dry map and the state;
  "exchange"  one turn of a coupling loop on page-locked host arrays: state out, state in, one step;
  "ensemble"  advance several scenarios together and read every member's state.

The caller of the mixed-precision path takes the state on in float32, the type that path computes
its modal coefficients in (the library writes doubles); the FP64 path's state stays float64.

``exact`` advances the same problem in float64 torch operations over whole-mesh arrays, written
from the method (weak form, Dubiner modes, Roe / LLF flux, wet/dry closure, positive-depth
operator, SSP Runge-Kutta), without the library.
"""
from __future__ import annotations

import ctypes
import functools
import math

import numpy as np
import torch

from paper_2307_14302_gb300 import dgswe as D
from paper_2307_14302_gb300 import workloads as W

G, MMH = 9.81, 1.0 / 3.6e6
DOMAINS = ("basin", "flume", "river", "dam", "coastal", "hurricane", "graded")


def _case(name, domain, n, steps, use="run", p=1, precision="mixed", flux="roe", ssp=2, friction="manning",
          limiter=False, members=1):
    c = {"domain": domain, "n": n, "steps": steps, "use": use, "p": p, "precision": precision, "flux": flux,
         "ssp": ssp, "friction": friction, "limiter": limiter, "members": members}
    return {"name": name, **c} if name else c


def listed():
    return [
        # the smallest call: one step of the 400-triangle verification basin, driven step by step from outside
        _case("basin-400-step", "basin", 400, 1),
        # the paper's rain-on-a-plane flume (960 triangles, 1 ms steps, 86,400 of them): a stretch of its run
        _case("flume-960", "flume", 960, 200),
        # river inflow on a small estuary-sized mesh with the five-stage scheme and LLF, quadratic friction
        _case("river-4.8k-llf5", "river", 4800, 20, flux="llf", ssp=5, friction="quadratic"),
        # the flagship: coastal wet/dry mesh of 250k triangles, storm rain and tide
        _case("coastal-250k", "coastal", 250_000, 10),
        # the reference-precision run of the same family on a ragged mid-size mesh
        _case("coastal-61k-fp64", "coastal", 61_403, 2, precision="fp64"),
        # slope-limited dam-break bore (shocks) on a fine basin mesh
        _case("dam-100k-limiter", "dam", 100_003, 5, limiter=True),
        # a monitored run: ledger, volume and inundation map between stretches of steps
        _case("coastal-37k-monitor", "coastal", 37_001, 20, use="monitor"),
        # hurricane-scale basin with gridded hourly rain, far larger than L2
        _case("hurricane-2M", "hurricane", 2_000_000, 4),
        # the production discretisation of the paper's runs (LLF flux, five-stage SSPRK) on gridded rain
        _case("hurricane-500k-llf5", "hurricane", 501_231, 2, flux="llf", ssp=5),
        # degree 2 with pressure set-up on the graded mesh, SSP(3,3)
        _case("graded-300k-p2", "graded", 300_000, 4, p=2, ssp=3),
        # eight scenarios of 5k to 60k triangles batched, states read at the end of the stretch
        _case("ensemble-8", "coastal", 20_000, 20, use="ensemble", members=8),
        # coupling loop in FP64: state out and in over the host link every step
        _case("exchange-30k-fp64", "coastal", 30_011, 1, use="exchange", precision="fp64"),
    ]


def _loguni(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges above; sizes and steps log-uniform, at most the listed work."""
    dom = rng.choice(DOMAINS + ("coastal", "hurricane", "graded", "ensemble", "exchange", "monitor"))
    use = dom if dom in ("ensemble", "exchange", "monitor") else "run"
    dom = "coastal" if use != "run" else dom
    fp64 = rng.random() < 0.25
    lo, hi = {"basin": (50, 8000), "flume": (240, 3000), "river": (400, 20_000), "dam": (2000, 150_000), "coastal": (2000, 300_000),
              "hurricane": (20_000, 2_000_000), "graded": (5000, 300_000)}[dom]
    if use == "ensemble":
        lo, hi = 2000, 30_000
    if use in ("exchange", "monitor"):
        hi = 120_000
    if fp64:
        hi = min(hi, 60_000)
    n = _loguni(rng, lo, hi)
    p = 2 if dom == "graded" else 1
    flux = rng.choice(("roe", "roe", "llf"))
    ssp = rng.choice((3, 3, 2)) if p == 2 else rng.choice((2, 2, 2, 3, 5))
    friction = rng.choice(("manning", "manning", "manning", "quadratic"))
    limiter = dom == "dam"
    members = rng.randint(2, 10) if use == "ensemble" else 1
    most = max(1, min((100 if fp64 else 400) // ssp, int((2.0e6 if not fp64 else 1.2e5) / (n * members))))
    steps = 1 if use == "exchange" else _loguni(rng, 1, max(2, most))
    return _case("", dom, n, steps, use, p, "fp64" if fp64 else "mixed", flux, ssp, friction, limiter, members)


# ------------------------------------------------------------------------------------ inputs --
def _lattice(lx, ly, n, seed, jitter=0.2, xs=None, ocean=True):
    """Jittered lattice split along the shorter diagonals, ocean (segment 0) on x = 0, else land."""
    rng = np.random.default_rng(seed)
    if xs is None:
        xs = np.linspace(0.0, lx, max(2, int(round(lx / math.sqrt(2.0 * lx * ly / n)))) + 1)
    nx = len(xs) - 1
    ny = max(2, int(round(n / (2 * nx))))
    X, Y = np.meshgrid(xs, np.linspace(0.0, ly, ny + 1), indexing="xy")
    dx = np.diff(xs)
    HX = np.minimum(np.r_[dx[0], dx], np.r_[dx, dx[-1]])[None, :]
    jx = rng.uniform(-jitter, jitter, X.shape) * HX
    jy = rng.uniform(-jitter, jitter, X.shape) * (ly / ny)
    jx[:, [0, -1]] = 0.0
    jy[[0, -1], :] = 0.0
    x, y = (X + jx).ravel(), (Y + jy).ravel()
    a = (np.arange(ny)[:, None] * (nx + 1) + np.arange(nx)[None, :]).ravel()
    b, c, d = a + 1, a + nx + 2, a + nx + 1
    flip = np.hypot(x[b] - x[d], y[b] - y[d]) < np.hypot(x[a] - x[c], y[a] - y[c])
    tri = np.empty((2 * nx * ny, 3), np.int32)
    tri[0::2] = np.where(flip[:, None], np.stack([a, b, d], 1), np.stack([a, b, c], 1))
    tri[1::2] = np.where(flip[:, None], np.stack([b, c, d], 1), np.stack([a, c, d], 1))
    i, j = np.arange(nx), np.arange(ny)
    west = np.stack([(j + 1) * (nx + 1), j * (nx + 1)], 1)
    rest = np.concatenate([np.stack([i, i + 1], 1), np.stack([j * (nx + 1) + nx, (j + 1) * (nx + 1) + nx], 1),
                           np.stack([ny * (nx + 1) + i + 1, ny * (nx + 1) + i], 1)])
    bedge = np.concatenate([west, rest]).astype(np.int32)
    btype = np.full(len(bedge), W.LAND, np.int32)
    if ocean:
        btype[:ny] = W.OCEAN
    return W.Mesh(np.stack([x, y], 1), tri, bedge, btype, np.zeros(len(bedge), np.int32))


@functools.lru_cache(maxsize=64)
def _mesh(domain, n):
    """The mesh of a model domain: made once and kept for all the runs on it."""
    if domain == "flume":
        return W.inclined_plane(nx=max(2, n // 4)).mesh
    if domain in ("basin", "river"):
        ny = max(2, int(round(math.sqrt(n / 4))))
        nx = max(2, int(round(n / (2 * ny))))
        if domain == "basin":
            return W.basin_c1(nx=nx, ny=ny).mesh
        return W.river_basin(nx=nx, ny=ny).mesh
    if domain == "dam":
        return _lattice(1e4, 5e3, n, n, ocean=False)
    lx, ly = _extent(domain, n)
    return W.graded_c3(n).mesh if domain == "graded" else _lattice(lx, ly, n, n)


def _extent(domain, n):
    """Domain sides: those of the full-size workload; on the p = 1 lattices smaller for a smaller mesh,
    so that the element size (and the time step) is that of the full one."""
    lx, ly, full = {"hurricane": (1.5e6, 1.0e6, 8e6), "graded": (4.0e5, 3.0e5, 1)}.get(domain, (4.0e5, 3.0e5, 2.5e5))
    f = min(1.0, math.sqrt(n / full))
    return lx * f, ly * f


def _shelf(s, deep, s1, s2, shelf, top):
    """Depth along s in [0, 1]: deep ocean, shelf, then land rising to ``top`` above the geoid."""
    return np.where(s < s1, deep - (deep - shelf) * 0.5 * (1 - np.cos(np.pi * np.clip(s / s1, 0, 1))),
                    np.where(s < s2, shelf * (1 - (s - s1) / (s2 - s1)), -top * np.clip((s - s2) / (1 - s2), 0, None)))


def _inputs(c, n, seed):
    """Everything a run of one scenario needs, from the seed alone: mesh, nodal bathymetry and
    Manning field, forcing, and an initial state in motion (a surge, with films on dry land)."""
    rng = np.random.default_rng([seed, n])
    m = _mesh(c["domain"], n)
    x, y = m.xy[:, 0], m.xy[:, 1]
    q = {"mesh": m, "H0": 0.01, "storm": None, "grid": None, "nodal": None, "tide": None, "river": None,
         "press": None, "cf": 0.0025, "manning": rng.uniform(0.02, 0.06, m.n_tri)}
    ph = rng.uniform(0, 2 * np.pi, 8)
    if c["domain"] == "flume":
        w = W.inclined_plane("AB"[int(rng.integers(2))], nx=max(2, n // 4), sim_s=2.0)
        q.update(hb=w.hb, grid=w.rain_grid, tide=w.tide, H0=w.h0, manning=w.manning, dt=1e-3)
        film = 4e-4 * (1 + 0.5 * np.sin(2 * np.pi * x / 6 + ph[0])) * (x / 24.0) + 0.5 * w.h0
        q["zeta"] = film - w.hb  # a thin sheet already running off
        q["qx"], q["qy"] = film * 0.05 * np.clip(film / 1e-3, 0, 1), np.zeros_like(x)
        q["t0"] = float(rng.uniform(0.0, 1.0))
        return q
    if c["domain"] in ("basin", "river", "dam"):
        q["hb"] = 5.0 + 15.0 * x / 1e4 - np.sin(np.pi * x / 1e4) * np.sin(np.pi * y / 5e3)
        xc, yc = rng.uniform(0.3, 0.7) * 1e4, rng.uniform(0.3, 0.7) * 5e3
        q["zeta"] = 0.5 * np.exp(-((x - xc) ** 2 + (y - yc) ** 2) / (2 * 800.0**2))
        q["qx"] = q["hb"] * 0.2 * np.sin(2 * np.pi * y / 5e3 + ph[0])
        q["qy"] = q["hb"] * 0.2 * np.sin(2 * np.pi * x / 1e4 + ph[1])
        q["manning"] = np.full(m.n_tri, 0.025)
        if c["domain"] == "dam":
            q["zeta"] = np.where(x + 0.2 * y < xc, 1.5, 0.0)
        if c["domain"] != "river":
            q["nodal"] = np.full(m.n_nodes, rng.uniform(10, 80) * MMH)
        else:
            r = np.linspace(0, 1, 5)[:, None] * rng.uniform(0.5, 2.0, 2)[None, :]
            q["river"] = W.River(q=r, t0=0.0, dt=150.0)
        q["t0"] = float(rng.uniform(0.0, 300.0))
        q["dt"] = _cfl(c, q, 0.3)
        return q
    if c["domain"] == "hurricane":
        (lx, ly), top, s1, s2 = _extent("hurricane", n), 10.0, 0.4, 0.7
        g = lx / 135.0  # 0.1 degree on the full-size basin
        nx, ny, nt = int(lx / g) + 2, int(ly / g) + 2, 4
        k = np.stack(np.meshgrid(np.arange(nt), np.arange(ny), np.arange(nx), indexing="ij"))
        f = sum(np.sin(0.05 * (i + 1) * k[2] + ph[i]) * np.cos(0.07 * (i + 1) * k[1] + ph[i + 3] + 0.3 * k[0]) for i in range(3))
        q["grid"] = W.RainGrid(nx, ny, nt, 0.0, 0.0, g, g, 0.0, 3600.0,
                               np.clip(np.exp(1.0 + 1.2 * f), 0.0, 100.0).astype(np.float32))
    else:
        (lx, ly), top, s1, s2 = _extent(c["domain"], n), 2.0, 0.45, 0.78
        q["storm"] = W.Storm(x0=0.55 * lx, y0=rng.uniform(0.3, 0.7) * ly, heading=rng.uniform(0, 2 * np.pi), speed=5.0,
                             rpeak=rng.uniform(10, 80) * MMH, rm=lx / 8, re=lx / 4)
        if c["domain"] == "graded":
            q["press"] = (0.78 * lx, rng.uniform(0.35, 0.65) * ly, 6e4, 2.0)
    q["hb"] = hb = _shelf(x / lx + 0.02 * np.sin(6 * np.pi * y / ly + ph[6]), 3000.0, s1, s2, 200.0, top)
    q["tide"] = W.Tide(np.array([0.5]), np.array([12.42 * 3600.0]), np.array([rng.uniform(0, 2 * np.pi)]))
    kx, ky = 2 * np.pi / lx, 2 * np.pi / ly
    wave = 0.2 * np.sin(3 * kx * x + ky * y + ph[0]) + 0.1 * np.sin(5 * kx * x - 2 * ky * y + ph[1])
    wave *= np.clip(hb / 50.0, 0.0, 1.0)  # the surge has not reached the shore yet
    q["zeta"] = np.where(hb < 0.01, 0.005 - hb, wave)  # films of H0 / 2 on dry land
    c0 = np.sqrt(G * np.maximum(hb, 0.0))  # a long wave's transport, in a direction that wanders
    ang = 0.5 * np.sin(2 * kx * x + 3 * ky * y + ph[3])
    q["qx"], q["qy"] = c0 * wave * np.cos(ang), c0 * wave * np.sin(ang)
    q["t0"] = float(rng.uniform(0.0, 7000.0))
    q["dt"] = _cfl(c, q, 0.04)  # explicit Manning friction on films of about H0 needs dt tau < 1
    return q


def _cfl(c, q, cfl):
    """The fixed time step of the run: cfl times min 2 r_in / ((2p+1) (|u| + sqrt(g H)))."""
    xy, tri = q["mesh"].xy, q["mesh"].tri
    t = [xy[tri[:, (i + 1) % 3]] - xy[tri[:, i]] for i in range(3)]
    area = 0.5 * (t[0][:, 0] * -t[2][:, 1] + t[0][:, 1] * t[2][:, 0])
    H = np.maximum(q["hb"] + q["zeta"], q["H0"])
    lam = (np.hypot(q["qx"], q["qy"]) / H + np.sqrt(G * H))[tri].max(axis=1)
    return float(cfl * (4.0 * area / sum(np.hypot(v[:, 0], v[:, 1]) for v in t) / ((2 * c["p"] + 1) * lam)).min())


def _sizes(c):
    """Member sizes of an ensemble: spread over a factor of twelve around n, odd ones among them."""
    k = c["members"]
    return [int(c["n"] * 12.0 ** (i / max(k - 1, 1) - 0.5)) | 1 for i in range(k)] if c["use"] == "ensemble" else [c["n"]]


def _solver(c, q, stream=None):
    s = D.Solver(p=c["p"], flux=D.FLUX_LLF if c["flux"] == "llf" else D.FLUX_ROE, ssp_stages=c["ssp"],
                 precision=D.FP64 if c["precision"] == "fp64" else D.MIXED, H0=q["H0"], cfl=0.3, dt=q["dt"],
                 friction=D.QUADRATIC if c["friction"] == "quadratic" else D.MANNING, cf=q["cf"], limiter=c["limiter"],
                 stream=stream)
    s.set_mesh(q["mesh"])
    s.set_fields(q["hb"], q["manning"])
    if q["nodal"] is not None:
        s.set_rain_nodal(q["nodal"])
    if q["storm"] is not None:
        s.set_storm(q["storm"])
    if q["grid"] is not None:
        s.set_rain_grid(q["grid"])
    if q["tide"] is not None:
        s.set_tide(q["tide"])
    if q["river"] is not None:
        s.set_river(q["river"])
    if q["press"] is not None:
        s.set_pressure_setup(*q["press"])
    s.set_state(q["zeta"], q["qx"], q["qy"], t0=q["t0"])
    return s


# -------------------------------------------------------------------------------------- cases --
@functools.lru_cache(maxsize=1)
def _stream():
    """The program's working stream: its solvers' work and its own go in order on it."""
    return torch.cuda.Stream()


def prepare(case, seed):
    """Solver(s) with their mesh, fields, forcing and state, and the caller's output arrays."""
    c = case
    qs = [_inputs(c, n, seed + 1000 * i) for i, n in enumerate(_sizes(c))]
    stream = _stream()
    ss = [_solver(c, q, stream.cuda_stream) for q in qs]
    st = {"case": c, "solver": ss[0], "np": ss[0].np_, "stream": stream}
    f64 = torch.float64
    if c["use"] == "ensemble":
        st["ens"] = D.Ensemble(ss, stream=stream.cuda_stream)
        for s in ss:
            s.close()
        st["host"] = [torch.empty((3, st["np"], s.ne), dtype=f64, pin_memory=True) for s in ss]
    elif c["use"] == "exchange":
        st["out"] = torch.empty((3, st["np"], ss[0].ne), dtype=f64, pin_memory=True)
        st["in"] = torch.empty_like(st["out"], pin_memory=True)
        z = ss[0].state_arrays(*(st["in"][k].numpy() for k in range(3)))  # the coupled model's first answer
        for a in z:
            a[0] *= 1.0 + 1e-3
    else:
        with torch.cuda.stream(stream):
            st["dev"] = torch.empty((3, st["np"], ss[0].ne), dtype=f64, device="cuda")
    return st


def _f32(c, t):
    return t.float() if c["precision"] == "mixed" else t


def run(state):
    c = state["case"]
    if c["use"] == "ensemble":
        ens, L = state["ens"], D.lib()
        ens.step(c["steps"])
        dp = ctypes.POINTER(ctypes.c_double)
        for i, h in enumerate(state["host"]):
            rc = L.dgswe_ensemble_get_state(ens.h, i, *(ctypes.cast(h[k].data_ptr(), dp) for k in range(3)))
            if rc:
                raise RuntimeError("dgswe_ensemble_get_state: %d" % rc)
        return [_f32(c, h) for h in state["host"]]
    s = state["solver"]
    if c["use"] == "exchange":
        i, o = state["in"].numpy(), state["out"].numpy()
        s.step(c["steps"])
        s.exchange(i[0], i[1], i[2], o[0], o[1], o[2])
        return state["out"]
    s.step(c["steps"])
    d = state["dev"]
    s.state_device(d[0].data_ptr(), d[1].data_ptr(), d[2].data_ptr())
    if c["use"] == "monitor":
        led = s.ledger()
        with torch.cuda.stream(state["stream"]):
            f = _f32(c, d)
        return {"state": f, "dry": s.dry(), "volume": s.volume(),
                "ledger": {k: led[k] for k in ("t", "steps", "V0", "V", "rain_in", "bdry_in", "VH0", "wet_frac")}}
    with torch.cuda.stream(state["stream"]):
        return _f32(c, d)


def work(case):
    """Per element and stage: the state in and out (and the step-initial state in later stages that
    use it), connectivity, geometry, bathymetry and Manning read once; plus the state written for the
    caller.  Mixed: means 8 bytes, other modes 4.  Operations counted from the weak form: area points,
    each edge once, lift, combination, positive-depth operator."""
    c = case
    npm, w = (3, 4) if c["p"] == 1 else (6, 4)
    fp64 = c["precision"] == "fp64"
    state = 3 * npm * 8 if fp64 else 3 * (8 + (npm - 1) * w)
    static = (6 + 3 + 1) * (8 if fp64 else 4) + 12
    stages = c["ssp"]
    with_wn = {2: 1, 3: 2, 5: 1}[stages]
    e = sum(_mesh(c["domain"], n).n_tri for n in _sizes(c))
    per = stages * (2 * state + static) + with_wn * state
    out = 3 * npm * 8 * (2 if c["use"] == "exchange" else 1)
    flops = 7 * (55 if c["p"] == 1 else 110) + 1.5 * (c["p"] + 1) * (75 + 16 * npm) + 3 * (c["p"] + 1) * npm * 6 + 30 * npm
    return {"bytes": float(e * (c["steps"] * per + out)), "flops": float(e * c["steps"] * stages * flops)}


# ------------------------------------------------------------------ the method in 64 bits ----
def _basis(p, r, s):
    """Orthonormal Dubiner modes on the triangle (-1,-1), (1,-1), (-1,1) and their r, s gradients."""
    one = np.ones_like(r)
    f = [(np.sqrt(0.5) * one, 0 * one, 0 * one),
         (math.sqrt(3.0) * (r + 0.5 * (1 + s)), math.sqrt(3.0) * one, 0.5 * math.sqrt(3.0) * one),
         (0.5 * (1 + 3 * s), 0 * one, 1.5 * one)]
    if p == 2:
        a, b = r + 0.5 * (1 + s), 0.5 * (1 - s)  # modes (2,0), (1,1), (0,2)
        c20, c11, c02 = math.sqrt(7.5), math.sqrt(4.5), math.sqrt(1.5)
        f += [(c20 * (1.5 * a * a - 0.5 * b * b), c20 * 3 * a, c20 * (1.5 * a + 0.5 * b)),
              (c11 * a * (5 * s + 3) / 2, c11 * (5 * s + 3) / 2, c11 * ((5 * s + 3) / 4 + 2.5 * a)),
              (c02 * (5 * s * s + 2 * s - 1) / 2, 0 * one, c02 * (5 * s + 1))]
    return (np.stack([v[k] for v in f]) for k in range(3))


def _rules(p):
    """Barycentric area points with weights (sum 2) and Gauss points with weights (sum 2)."""
    L, w = [(1 / 3, 1 / 3, 1 / 3)], [27 / 60 if p == 1 else 9 / 40]
    r15 = math.sqrt(15.0)
    for a, wa in ([(0.5, 8 / 60), (0.0, 3 / 60)] if p == 1 else
                  [((6 - r15) / 21, (155 - r15) / 1200), ((6 + r15) / 21, (155 + r15) / 1200)]):
        for k in range(3):
            l = [a, a, a]
            l[k] = 1 - 2 * a
            L.append(tuple(l))
            w.append(wa)
    x = [-math.sqrt(1 / 3), math.sqrt(1 / 3)] if p == 1 else [-math.sqrt(0.6), 0.0, math.sqrt(0.6)]
    return np.array(L), 2 * np.array(w), np.array(x), np.array([1.0, 1.0] if p == 1 else [5 / 9, 8 / 9, 5 / 9])


def _rs(l):
    return -l[..., 0] + l[..., 1] - l[..., 2], -l[..., 0] - l[..., 1] + l[..., 2]


class _Model:
    """One scenario as float64 torch arrays, all elements at once (caller's element order)."""

    def __init__(self, c, q):
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        T = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=dev)  # noqa: E731
        self.T, self.c, self.q, self.p, self.H0 = T, c, q, c["p"], q["H0"]
        m = q["mesh"]
        tri = m.tri.astype(np.int64)
        self.ne, self.tri = len(tri), torch.as_tensor(tri, device=dev)
        x, y = m.xy[:, 0][tri].T, m.xy[:, 1][tri].T
        self.vx, self.vy, self.hv = T(x), T(y), T(q["hb"][tri].T)
        self.area = 0.5 * ((self.vx[1] - self.vx[0]) * (self.vy[2] - self.vy[0])
                           - (self.vx[2] - self.vx[0]) * (self.vy[1] - self.vy[0]))
        self.man = T(q["manning"])
        # neighbour of every (element, local edge) and boundary kinds by node pair
        a, b = tri, np.roll(tri, -1, axis=1)
        key = (np.minimum(a, b) * m.n_nodes + np.maximum(a, b)).ravel()
        o = np.argsort(key, kind="stable")
        same = key[o][1:] == key[o][:-1]
        nb = np.full(3 * self.ne, -1, np.int64)
        nb[o[:-1][same]], nb[o[1:][same]] = o[1:][same], o[:-1][same]
        kind, seg = np.zeros(3 * self.ne, np.int64), np.zeros(3 * self.ne, np.int64)
        be = m.bedge.astype(np.int64)
        bk = np.minimum(be[:, 0], be[:, 1]) * m.n_nodes + np.maximum(be[:, 0], be[:, 1])
        at = o[np.searchsorted(key[o], bk)]
        kind[at], seg[at] = m.btype, m.bseg
        I = lambda v: torch.as_tensor(v.reshape(-1, 3).T.copy(), device=dev)  # noqa: E731
        self.nb, self.nj, self.inner = I(np.maximum(nb, 0) // 3), I(np.maximum(nb, 0) % 3), I(nb >= 0)
        self.kind, self.seg = I(kind), I(seg)
        # tables
        L, qw, xg, self.gw = _rules(self.p)
        self.ql, self.qw = L, qw
        self.qphi, self.qr, self.qs = _basis(self.p, *_rs(L))
        l = np.zeros((3, len(xg), 3))
        for j in range(3):
            l[j, :, j], l[j, :, (j + 1) % 3] = 0.5 * (1 - xg), 0.5 * (1 + xg)
        self.el, self.ng = l, len(xg)
        self.ephi = np.stack([next(_basis(self.p, *_rs(l[j]))) for j in range(3)])  # [edge][mode][point]
        eye = np.eye(3)
        self.vphi = next(_basis(1, *_rs(eye)))  # [mode][vertex]
        self.vinv = np.linalg.inv(self.vphi.T)  # modes from vertex values
        self.mphi = next(_basis(1, *_rs(0.5 * (eye + np.roll(eye, -1, axis=0)))))
        # gradients of r and s
        xr, xs = 0.5 * (self.vx[1] - self.vx[0]), 0.5 * (self.vx[2] - self.vx[0])
        yr, ys = 0.5 * (self.vy[1] - self.vy[0]), 0.5 * (self.vy[2] - self.vy[0])
        self.det = xr * ys - xs * yr
        self.rx, self.ry, self.sx, self.sy = ys / self.det, -xs / self.det, -yr / self.det, xr / self.det
        hr, hs = 0.5 * (self.hv[1] - self.hv[0]), 0.5 * (self.hv[2] - self.hv[0])
        self.hbx, self.hby = hr * self.rx + hs * self.sx, hr * self.ry + hs * self.sy
        # initial state: the linear interpolant of the nodal values, then the positive-depth operator
        npm = 3 if self.p == 1 else 6
        self.w = torch.zeros((3, npm, self.ne), dtype=torch.float64, device=dev)
        for k, name in enumerate(("zeta", "qx", "qy")):
            f = T(q[name][tri].T)
            for mm in range(3):
                self.w[k, mm] = sum(self.vinv[mm][i] * f[i] for i in range(3))
        self.dry = torch.zeros(self.ne, dtype=torch.bool, device=dev)
        if c["limiter"]:
            self.limits()
        self.w = self.positive(self.w)
        self.n, self.rain, self.bdry = 0, 0.0, 0.0
        self.V0, self.VH0 = self.volume(), self.volume(True)

    def volume(self, depth=False):
        z = self.w[0, 0] * math.sqrt(0.5) + (self.hv.mean(0) if depth else 0.0)
        return float((self.area * z).sum())

    def linear(self, w, f):
        for m in (1, 2):
            w[m] = sum(self.vinv[m][i] * f[i] for i in range(3))

    def positive(self, w):
        H0 = self.H0
        ev = lambda a: torch.stack([sum(a[m] * self.vphi[m][i] for m in range(3)) for i in range(3)])  # noqa: E731
        H, qx, qy = ev(w[0]) + self.hv, ev(w[1]), ev(w[2])
        lo = H.min(0).values
        if self.p == 2:
            w[:, 3:] *= ((lo - H0) / H0).clamp(0.0, 1.0)
        low = lo < H0
        mean = H.sum(0) / 3.0
        flat = low & (mean <= H0)
        o = torch.sort(H, dim=0, stable=True).indices
        h = torch.gather(H, 0, o)
        d = H0 - h[0]
        share = h[1] - 0.5 * d >= H0
        ho = torch.stack([torch.full_like(d, H0), torch.where(share, h[1] - 0.5 * d, H0),
                          torch.where(share, h[2] - 0.5 * d, h[2] - d - (H0 - h[1]))])
        Ho = torch.where(flat, mean, torch.empty_like(H).scatter_(0, o, ho))
        Ho = torch.where(low, Ho, H)
        dv = torch.where(flat, True, (Ho < H0) & low)
        nd = dv.sum(0)
        z = w[0].clone()
        self.linear(z, Ho - self.hv)
        w[0] = torch.where(low, z, w[0])
        part = (nd > 0) & (nd < 3)
        for k, f in ((1, qx), (2, qy)):
            moved = torch.where(dv, f, 0.0).sum(0) / (3 - nd).clamp(min=1)
            z = w[k].clone()
            self.linear(z, torch.where(dv, 0.0, f + moved))
            w[k] = torch.where(nd == 3, 0.0, torch.where(part, z, w[k]))
        self.dry = nd > 0
        return w

    def limits(self):
        """Barycentric pairs of the minmod limiter: a, c and the second neighbour of every edge."""
        bx, by = self.vx.mean(0), self.vy.mean(0)
        nx = [bx[self.nb[j]] - bx for j in range(3)]
        ny = [by[self.nb[j]] - by for j in range(3)]
        self.lim, ok = [], self.inner.all(0) & (self.kind == 0).all(0)
        for i in range(3):
            mx = 0.5 * (self.vx[i] + self.vx[(i + 1) % 3]) - bx
            my = 0.5 * (self.vy[i] + self.vy[(i + 1) % 3]) - by
            two = []
            for t in (1, 2):
                k = (i + t) % 3
                det = nx[i] * ny[k] - ny[i] * nx[k]
                a, b = (mx * ny[k] - my * nx[k]) / det, (nx[i] * my - ny[i] * mx) / det
                two.append((a, b, (det != 0) & (a >= 0) & (b >= 0)))
            first = two[0][2]
            self.lim.append((torch.where(first, two[0][0], two[1][0]), torch.where(first, two[0][1], two[1][1]), first))
            ok = ok & (first | two[1][2])
        self.lim_ok = ok

    def limit(self, w):
        act, out = self.lim_ok & ~self.dry, w.clone()
        for v in range(3):
            m0 = w[v, 0] * math.sqrt(0.5)
            dm = [m0[self.nb[j]] - m0 for j in range(3)]
            d = [w[v, 1] * self.mphi[1][i] + w[v, 2] * self.mphi[2][i] for i in range(3)]
            l = []
            for i, (a, b, first) in enumerate(self.lim):
                e = 1.5 * (a * dm[i] + b * torch.where(first, dm[(i + 1) % 3], dm[(i + 2) % 3]))
                l.append(torch.where((d[i] > 0) & (e > 0), torch.minimum(d[i], e),
                                     torch.where((d[i] < 0) & (e < 0), torch.maximum(d[i], e), 0.0)))
                l[i] = torch.where(d[i] == 0, d[i], l[i])
            l, d = torch.stack(l), torch.stack(d)
            ch = act & (l != d).any(0)
            pos, neg = l.clamp(min=0).sum(0), (-l).clamp(min=0).sum(0)
            tp, tn = (neg / pos).nan_to_num(0.0).clamp(max=1.0), (pos / neg).nan_to_num(0.0).clamp(max=1.0)
            bal = tp * l.clamp(min=0) - tn * (-l).clamp(min=0)
            l = torch.where(l.sum(0) != 0, bal, l)
            f = m0 + l + torch.roll(l, 1, 0) - torch.roll(l, -1, 0)
            z = out[v].clone()
            self.linear(z, f)
            out[v] = torch.where(ch, z, out[v])
        return out

    def rain_at(self, t):
        q = self.q
        if q["nodal"] is not None:
            return self.T(q["nodal"])[self.tri].mean(1)
        if q["storm"] is not None:
            s = q["storm"]
            r = torch.hypot(self.vx - (s.x0 + s.speed * (t - s.t0) * math.cos(s.heading)),
                            self.vy - (s.y0 + s.speed * (t - s.t0) * math.sin(s.heading)))
            return torch.where(r < s.rm, s.rpeak * (0.5 + 0.5 * r / s.rm), s.rpeak * torch.exp(-(r - s.rm) / s.re)).mean(0)
        if q["grid"] is not None:
            g = q["grid"]
            gx, gy = ((self.vx - g.x0) / g.dx).clamp(0, g.nx - 1), ((self.vy - g.y0) / g.dy).clamp(0, g.ny - 1)
            gt = min(max((t - g.t0) / g.dt_rec, 0.0), g.nt - 1.0)
            ix, iy, it = gx.floor().clamp(max=g.nx - 2), gy.floor().clamp(max=g.ny - 2), min(int(gt), g.nt - 2)
            fx, fy, ft = gx - ix, gy - iy, gt - it
            ix, iy = ix.long(), iy.long()
            val = 0.0
            for k, wt in ((it, 1 - ft), (it + 1, ft)):
                f = self.T(g.mm_per_h[k])
                val = val + wt * ((1 - fy) * ((1 - fx) * f[iy, ix] + fx * f[iy, ix + 1])
                                  + fy * ((1 - fx) * f[iy + 1, ix] + fx * f[iy + 1, ix + 1]))
            return val.mean(0) / 3.6e6
        return torch.zeros_like(self.area)

    def flux(self, L, R, nx, ny):
        """Numerical flux (zeta, qx, qy) between traces (zeta, qx, qy, hb) along n."""
        def side(s):
            H = (s[0] + s[3]).clamp(min=self.H0)
            P = 0.5 * G * s[0] * (s[0] + 2 * s[3])
            un = (s[1] * nx + s[2] * ny) / H
            return H, un, (s[1] * nx + s[2] * ny, s[1] * un + P * nx, s[2] * un + P * ny)
        HL, uL, FL = side(L)
        HR, uR, FR = side(R)
        d = [R[k] - L[k] for k in range(3)]
        if self.c["flux"] == "llf":
            lam = torch.maximum(uL.abs() + (G * HL).sqrt(), uR.abs() + (G * HR).sqrt())
            return [0.5 * (FL[k] + FR[k] - lam * d[k]) for k in range(3)]
        sL, sR = HL.sqrt(), HR.sqrt()
        u, v = (L[1] / sL + R[1] / sR) / (sL + sR), (L[2] / sL + R[2] / sR) / (sL + sR)
        cc = (0.5 * G * (HL + HR)).sqrt()
        un, ut = u * nx + v * ny, v * nx - u * ny
        dn, dt = d[1] * nx + d[2] * ny, d[2] * nx - d[1] * ny
        w = (dn - un * d[0]) / cc
        a1, a2, a3 = (un - cc).abs() * 0.5 * (d[0] - w), un.abs() * (dt - ut * d[0]), (un + cc).abs() * 0.5 * (d[0] + w)
        D3 = (a1 + a3, a1 * (u - cc * nx) - a2 * ny + a3 * (u + cc * nx), a1 * (v - cc * ny) + a2 * nx + a3 * (v + cc * ny))
        return [0.5 * (FL[k] + FR[k] - D3[k]) for k in range(3)]

    def rate(self, w, t):
        """L_h(w) of every element, the rain volume rate and the boundary inflow rate."""
        npm, q = w.shape[1], self.q
        R = torch.zeros_like(w)
        bdry = 0.0
        tabs = self.T(self.ephi)
        for j in range(3):
            ax, ay = self.vx[j], self.vy[j]
            bx, by = self.vx[(j + 1) % 3], self.vy[(j + 1) % 3]
            ln = torch.hypot(bx - ax, by - ay)
            nx, ny = (by - ay) / ln, (ax - bx) / ln
            kind = torch.where(self.inner[j] & (self.kind[j] == 0), -1, self.kind[j])
            nb = self.nb[j]
            pts, ec = [], 0.0
            for k in range(self.ng):
                hb = sum(self.el[j, k, i] * self.hv[i] for i in range(3))
                L = [sum(self.ephi[j][m][k] * w[v, m] for m in range(npm)) for v in range(3)]
                ph = tabs[:, :, self.ng - 1 - k][self.nj[j]]
                N = [sum(ph[:, m] * w[v, m][nb] for m in range(npm)) for v in range(3)]
                qn = L[1] * nx + L[2] * ny
                M = [L[0], L[1] - 2 * qn * nx, L[2] - 2 * qn * ny]  # mirror image: a wall
                O, mass = list(L), None
                if q["tide"] is not None:
                    td = q["tide"]
                    z = self.T(td.amp * np.sin(2 * np.pi * t / td.period + td.phase))[self.seg[j].clamp(max=len(td.amp) - 1)]
                    O[0] = torch.where(kind == W.OCEAN, z, O[0])
                if q["river"] is not None:
                    r = q["river"]
                    f = min(max((t - r.t0) / r.dt, 0.0), len(r.q) - 1.0)
                    i0 = min(int(f), len(r.q) - 2)
                    mass = self.T((1 - f + i0) * r.q[i0] + (f - i0) * r.q[i0 + 1])[self.seg[j].clamp(max=r.q.shape[1] - 1)]
                    riv = kind == W.RIVER
                    O[1], O[2] = torch.where(riv, -mass * nx, O[1]), torch.where(riv, -mass * ny, O[2])
                S = [torch.where(kind == -1, N[v], torch.where(kind == W.LAND, M[v], O[v])) for v in range(3)]
                F = self.flux(L + [hb], S + [hb], nx, ny)
                F[0] = torch.where(kind == W.LAND, 0.0, F[0])
                if mass is not None:
                    F[0] = torch.where(kind == W.RIVER, -mass, F[0])
                Wl = self.flux(L + [hb], M + [hb], nx, ny)
                Wl[0] = torch.zeros_like(ln)
                wk = 0.5 * ln * self.gw[k]
                ec = ec + wk * F[0]
                pts.append((F, Wl, wk))
            shut = (self.dry & (ec > 0)) | ((kind == -1) & self.dry[nb] & (ec < 0))
            for k, (F, Wl, wk) in enumerate(pts):
                for v in range(3):
                    f = wk * torch.where(shut, Wl[v], F[v])
                    for m in range(npm):
                        R[v, m] -= self.ephi[j][m][k] * f
            bdry -= float(torch.where((kind > 0) & ~shut, ec, 0.0).sum())
        rain = self.rain_at(t)
        for k in range(len(self.qw)):
            z, qx, qy = (sum(self.qphi[m][k] * w[v, m] for m in range(npm)) for v in range(3))
            hb = sum(self.ql[k][i] * self.hv[i] for i in range(3))
            H = z + hb
            Hs = H.clamp(min=self.H0)
            u, v = qx / Hs, qy / Hs
            P = 0.5 * G * z * (z + 2 * hb)
            sp = torch.hypot(u, v)
            tau = G * self.man**2 * sp / Hs ** (4.0 / 3.0) if self.c["friction"] == "manning" else q["cf"] * sp / Hs
            sx, sy = G * z * self.hbx - tau * qx, G * z * self.hby - tau * qy
            if q["press"] is not None:
                x0, y0, sg, pk = q["press"]
                dx = sum(self.ql[k][i] * self.vx[i] for i in range(3)) - x0
                dy = sum(self.ql[k][i] * self.vy[i] for i in range(3)) - y0
                eta = pk * torch.exp(-(dx * dx + dy * dy) / (2 * sg * sg))
                sx, sy = sx - G * H * eta * dx / sg**2, sy - G * H * eta * dy / sg**2
            wq = self.qw[k] * self.det
            for m in range(npm):
                gx, gy = self.qr[m][k] * self.rx + self.qs[m][k] * self.sx, self.qr[m][k] * self.ry + self.qs[m][k] * self.sy
                R[0, m] += wq * (gx * qx + gy * qy + self.qphi[m][k] * rain)
                R[1, m] += wq * (gx * (qx * u + P) + gy * qx * v + self.qphi[m][k] * sx)
                R[2, m] += wq * (gx * qy * u + gy * (qy * v + P) + self.qphi[m][k] * sy)
        R[1:] = torch.where(self.dry, 0.0, R[1:])
        return R / self.det, float((self.area * rain).sum()), bdry

    def step(self):
        tab = {2: [(0, 1, 1, 0), (.5, .5, .5, 1)], 3: [(0, 1, 1, 0), (.75, .25, .25, 1), (1 / 3, 2 / 3, 2 / 3, .5)],
               5: [(0, 1, .25, 0), (0, 1, .25, .25), (0, 1, .25, .5), (0, 1, .25, .75), (.2, .8, .2, 1)]}[self.c["ssp"]]
        dt, w0 = self.q["dt"], self.w
        w, vol = w0, (0.0, 0.0)
        for an, ai, b, cs in tab:
            L, rain, bdry = self.rate(w, self.q["t0"] + (self.n + cs) * dt)
            w = self.positive(an * w0 + ai * w + b * dt * L)
            vol = (ai * vol[0] + b * dt * rain, ai * vol[1] + b * dt * bdry)
            if self.c["limiter"]:
                w = self.positive(self.limit(w))
        self.w, self.n = w, self.n + 1
        self.rain, self.bdry = self.rain + vol[0], self.bdry + vol[1]


def exact(case, seed):
    c = case
    if sum(_mesh(c["domain"], n).n_tri for n in _sizes(c)) * c["steps"] * c["ssp"] > 4e7:
        return None  # too long for a check
    out = []
    for i, n in enumerate(_sizes(c)):
        m = _Model(c, _inputs(c, n, seed + 1000 * i))
        for _ in range(c["steps"]):
            m.step()
        out.append(m)
    if c["use"] == "ensemble":
        return [m.w.cpu() for m in out]
    m = out[0]
    if c["use"] == "monitor":
        return {"state": m.w, "dry": None, "volume": m.volume(),
                "ledger": {"t": c["steps"] * m.q["dt"] + m.q["t0"], "steps": None, "V0": m.V0, "V": m.volume(),
                           "rain_in": m.rain, "bdry_in": m.bdry, "VH0": m.VH0, "wet_frac": float((~m.dry).double().mean())}}
    return m.w.cpu() if c["use"] == "exchange" else m.w
