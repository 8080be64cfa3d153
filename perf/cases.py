"""The calls whose speed matters to a user of this library, from one pixel cell to a pixel matrix.

listed() names the cases, draw() gives more of the same ranges, prepare() builds what a program
holds before the call (a sensor at the stage the call needs, output buffers, tracks), run() is the
call through the public entry points, work() the bytes and operations it cannot do without, and
exact() the same outputs in 64 bits by plain torch (dense sums over modes, Householder QR, dense
eigensolver, gathers), without the library.

A sensor is n_pix x n_pix pixels of 55 um (single cells of a batch: 40-110 um): a readout column
at each pixel centre, a bias column at each pixel corner, resistivities drawn per column.  Radii
lie where the band-limited fit is definite, near an odd half multiple of the lateral spacing.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2605_13987_gb300 as wt

UM = 1e-6
OHM_CM = 1e-2
EPS0 = 8.8541878128e-12
EPS_R = 5.7
E_CHARGE = 1.602176634e-19
SPEED = 1e5                       # carrier speed [m/s]
N_AZ, N_H = 4, 2                  # collocation azimuths and heights per source (the fit's defaults)
BATCH_NX = (96, 64, 128, 80, 112)
# grid sizes of a fit, and those of them that the field's transforms take
FIT_SIZES = (16, 20, 24, 28, 30, 32, 36, 40, 42, 48, 50, 54, 56, 60, 64, 70, 72, 80, 84, 90, 96, 100, 108, 112, 120,
             126, 128, 140, 144, 150, 160)
FIELD_SIZES = (16, 20, 24, 28, 30, 32, 36, 40, 48, 56, 60, 64, 72, 80, 96, 112, 120, 128, 144, 160, 192, 224, 240, 256)


def listed():
    return [
        # one pixel cell from geometry to charges: the inner step of a design study over many cells
        {"name": "setup_cell", "kind": "setup", "n_pix": 1, "nx": 32, "nz": 64, "m": 64, "n_t": 64},
        # a 3x3 matrix from geometry to charges, paid for every new geometry
        {"name": "setup_matrix", "kind": "setup", "n_pix": 3, "nx": 64, "nz": 128, "m": 128, "n_t": 256},
        # new resistivities (a depth profile on every column) on a fitted matrix: relaxation only
        {"name": "relax_profile", "kind": "relax", "n_pix": 3, "nx": 48, "nz": 100, "m": 96, "n_t": 512},
        # the field of one small cell: latency and launches
        {"name": "extend_cell", "kind": "extend", "n_pix": 1, "nx": 32, "nz": 64, "m": 64, "n_t": 64},
        # the field of the 3x3 matrix at full grid and 512 time samples: the headline workload
        {"name": "extend_matrix", "kind": "extend", "n_pix": 3, "nx": 128, "nz": 256, "m": 64, "n_t": 512},
        # the FP64 field on a grid that is no power of two, for those who need more than FP32
        {"name": "extend_fp64", "kind": "extend64", "n_pix": 3, "nx": 60, "nz": 120, "m": 48, "n_t": 64},
        # several single cells on uneven grids in one batched call
        {"name": "batch_cells", "kind": "batch", "n_sensors": 6, "first": 0, "scale": 1.0, "n_t": 256},
        # minimum-ionising tracks through a stored field (Eq. 1)
        {"name": "eq1_field", "kind": "eq1", "n_pix": 3, "nx": 96, "nz": 192, "m": 48, "n_t": 128,
         "n_tracks": 10000, "n_steps": 100},
        # 1e5 drifting carriers straight from the rank-r form (Eq. 1 without a stored field)
        {"name": "eq1_direct", "kind": "eq1_direct", "n_pix": 3, "nx": 96, "nz": 192, "m": 48, "n_t": 256,
         "n_tracks": 100000, "n_steps": 200},
        # one variant of a geometry scan with sensitivities: currents, their tangents, loss and gradient
        {"name": "tangents_scan", "kind": "tangents", "n_pix": 3, "nx": 20, "nz": 64, "m": 64, "n_t": 256,
         "n_tracks": 1000, "n_steps": 100},
        # front-end shaping and signal features (with sensitivities) of a run's currents
        {"name": "waveforms", "kind": "waveforms", "n_tracks": 20000, "n": 200, "n_dir": 4},
        # exact FP64 field at scattered points (checks, field maps along a line)
        {"name": "point_values", "kind": "points", "n_pix": 3, "nx": 64, "nz": 128, "m": 64, "n_t": 64,
         "n_points": 500, "n_at": 16},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _size(rng, lo, hi, sizes=FIELD_SIZES):
    return rng.choice([n for n in sizes if lo <= n <= hi])


def _grid(rng, nx_lo, nx_hi, nz_hi):
    """Lateral and vertical size of a field's grid: 1.2 to 2.2 times as many planes as rows."""
    nx = _size(rng, nx_lo, nx_hi)
    return {"nx": nx, "nz": _size(rng, 1.2 * nx, min(2.2 * nx, nz_hi))}


def draw(rng):
    kind = rng.choice(["setup", "relax", "extend", "extend", "extend64", "batch", "eq1", "eq1_direct", "tangents",
                       "waveforms", "points"])
    if kind == "waveforms":
        return {"kind": kind, "n_tracks": _log(rng, 50, 20000), "n": rng.randint(50, 400), "n_dir": rng.randint(0, 4)}
    if kind == "batch":
        return {"kind": kind, "n_sensors": rng.randint(2, 6), "first": rng.randint(0, 4),
                "scale": rng.choice([0.5, 1.0]), "n_t": rng.randint(48, 256)}
    n_pix = rng.choice([1, 2, 3])
    if kind in ("setup", "relax"):
        m = _log(rng, 24, 128 if kind == "setup" else 96)
        return {"kind": kind, "n_pix": n_pix, "nx": _size(rng, 10 * n_pix, 64, FIT_SIZES),
                "nz": _size(rng, m, 160, FIT_SIZES), "m": m, "n_t": rng.randint(32, 256)}
    if kind == "tangents":
        return {"kind": kind, "n_pix": n_pix, "nx": _size(rng, 7 * n_pix, 12 * n_pix + 6), "nz": _size(rng, 40, 64),
                "m": rng.randint(24, 64), "n_t": rng.randint(48, 256), "n_tracks": _log(rng, 50, 1000),
                "n_steps": rng.randint(40, 100)}
    case = {"kind": kind, "n_pix": n_pix, "m": rng.randint(32, 64)}
    if kind == "extend":
        return {**case, **_grid(rng, 32, 128, 256), "n_t": _log(rng, 40, 512)}
    if kind == "extend64":
        return {**case, **_grid(rng, 32, 60, 120), "n_t": _log(rng, 16, 64)}
    if kind == "points":
        return {**case, **_grid(rng, 32, 64, 128), "n_t": 64, "n_points": _log(rng, 20, 500), "n_at": rng.randint(1, 16)}
    if kind == "eq1":
        return {**case, **_grid(rng, 32, 96, 192), "n_t": rng.randint(48, 128), "n_tracks": _log(rng, 100, 10000),
                "n_steps": rng.randint(50, 100)}
    return {**case, **_grid(rng, 32, 96, 192), "n_t": rng.randint(64, 256), "n_tracks": _log(rng, 1000, 100000),
            "n_steps": rng.randint(50, 200)}


# ------------------------------------------------------------------ inputs
def _column(grid, x, y, r, rho, top, driven, m):
    return SimpleNamespace(x=x, y=y, z0=0.0, z1=grid.Lz, radius=r, resistivity=rho, terminal_top=top, driven=driven,
                           n_sources=m, rho_profile=None)


def _radius_steps(target, h):
    """The radius in lateral spacings, less a draw within 0.1: an even multiple (up to 6) plus a half, near `target`."""
    return 2 * min(3, max(0, round((target / h - 0.5) / 2))) + 0.5


def _times(n_t):
    return 10.0 ** np.linspace(-12.0, -8.0, n_t)


def _matrix(n_pix, nx, nz, m, seed, pitch=55 * UM, thick=None, target=6 * UM):
    rng = np.random.default_rng([seed, 1])
    thick = thick or (100 * UM if n_pix == 1 else 500 * UM)
    L = n_pix * pitch
    grid = SimpleNamespace(Lx=L, Ly=L, Lz=thick, Nx=nx, Ny=nx, Nz=nz, eps_r=EPS_R, zbc="mirror")
    steps = _radius_steps(target, L / nx)
    r = L / nx * (steps + rng.uniform(-0.1, 0.1))
    m = max(1, min(m, nz, int(3.25 * thick / (L / nx * (steps + 0.1)))))       # the same for every seed
    rho = rng.uniform(0.1, 1.0, 2 * n_pix * n_pix) * OHM_CM
    mid = n_pix // 2
    cols = [_column(grid, (i + 0.5) * pitch, (j + 0.5) * pitch, r, rho[i * n_pix + j], 1, int(i == mid and j == mid), m)
            for i in range(n_pix) for j in range(n_pix)]
    cols += [_column(grid, i * pitch, j * pitch, r, rho[(n_pix + i) * n_pix + j], 0, 0, m)
             for i in range(n_pix) for j in range(n_pix)]
    return grid, cols


def _geometry(case, seed):
    return _matrix(case["n_pix"], case["nx"], case["nz"], case["m"], seed)


def _batch_geometries(case, seed):
    rng = np.random.default_rng([seed, 2])
    out = []
    for k in range(case["n_sensors"]):
        nx = int(BATCH_NX[(case["first"] + k) % len(BATCH_NX)] * case["scale"]) // 2 * 2
        out.append(_matrix(1, nx, 2 * nx, 2 * nx, int(rng.integers(1 << 30)), rng.uniform(40, 110) * UM,
                           rng.uniform(300, 500) * UM, rng.uniform(4, 10) * UM))
    return out


def _profiles(cols, seed):
    """Resistivity of every node, a smooth depth profile of a few tens of per cent per column."""
    rng = np.random.default_rng([seed, 3])
    out = []
    for c in cols:
        z = (np.arange(c.n_sources) + 0.5) / c.n_sources
        out.append(c.resistivity * (1.0 + rng.uniform(-0.4, 0.4) * np.cos(math.pi * z) + rng.uniform(-0.2, 0.2) * z))
    return out


def _dev(a):
    return torch.as_tensor(a, dtype=torch.float64, device="cuda")


def _track_dict(p, v, dt, n_out, charge):
    f = lambda a: a.to(torch.float32).contiguous()  # noqa: E731
    return {"n_tracks": p[0].shape[0], "n_steps": p[0].shape[1], "n_out": n_out, "dt": dt, "charge": 1.0,
            "x": f(p[0]), "y": f(p[1]), "z": f(p[2]), "vx": f(v[0]), "vy": f(v[1]), "vz": f(v[2]), "q": f(charge)}


def _mip_tracks(grid, n, n_steps, seed):
    """Straight tracks from the top face, isotropic within 30 degrees of -z."""
    rng = np.random.default_rng([seed, 4])
    dt = grid.Lz / (n_steps * SPEED)
    ct = _dev(rng.uniform(math.cos(math.radians(30.0)), 1.0, n))[:, None]
    ph = _dev(rng.uniform(0, 2 * math.pi, n))[:, None]
    x0, y0 = _dev(rng.uniform(0, grid.Lx, n))[:, None], _dev(rng.uniform(0, grid.Ly, n))[:, None]
    st = torch.sqrt(1 - ct * ct)
    v = [SPEED * st * torch.cos(ph), SPEED * st * torch.sin(ph), -SPEED * ct]
    s = torch.arange(n_steps, device="cuda", dtype=torch.float64)[None, :] * dt
    p = [torch.remainder(x0 + v[0] * s, grid.Lx), torch.remainder(y0 + v[1] * s, grid.Ly), grid.Lz + v[2] * s]
    inside = (p[2] >= 0) & (p[2] <= grid.Lz)
    v = [torch.where(inside, a, 0.0) for a in v]
    p[2] = p[2].clamp(0, grid.Lz)
    return _track_dict(p, v, dt, 2 * n_steps, torch.ones(n, device="cuda"))


def _drift_tracks(grid, cols, n, n_steps, seed, dt=1.5e-12):
    """Electrons toward the nearest readout axis, holes toward the nearest bias axis, stopping at its surface."""
    rng = np.random.default_rng([seed, 5])
    p0 = [_dev(rng.uniform(0, L, n)) for L in (grid.Lx, grid.Ly, grid.Lz)]
    elec = torch.as_tensor(rng.random(n) < 0.5, device="cuda")
    best = torch.full((n,), math.inf, device="cuda", dtype=torch.float64)
    ux, uy = torch.zeros_like(best), torch.zeros_like(best)
    travel = torch.zeros_like(best)
    for c in cols:
        dx, dy = c.x - p0[0], c.y - p0[1]
        dx = dx - grid.Lx * torch.round(dx / grid.Lx)
        dy = dy - grid.Ly * torch.round(dy / grid.Ly)
        d = torch.hypot(dx, dy)
        take = (elec == bool(c.terminal_top)) & (d < best)
        best = torch.where(take, d, best)
        dn = d.clamp_min(1e-30)
        ux, uy = torch.where(take, dx / dn, ux), torch.where(take, dy / dn, uy)
        travel = torch.where(take, (d - c.radius).clamp_min(0), travel)
    t = torch.arange(n_steps, device="cuda", dtype=torch.float64)[None, :] * (dt * SPEED)
    moving = t < travel[:, None]
    s = torch.minimum(t, travel[:, None])
    p = [torch.remainder(p0[0][:, None] + ux[:, None] * s, grid.Lx),
         torch.remainder(p0[1][:, None] + uy[:, None] * s, grid.Ly), p0[2][:, None].expand(n, n_steps)]
    v = [torch.where(moving, SPEED * ux[:, None], 0.0), torch.where(moving, SPEED * uy[:, None], 0.0),
         torch.zeros((n, n_steps), device="cuda")]
    return _track_dict(p, v, dt, 2 * n_steps, torch.where(elec, -E_CHARGE, E_CHARGE))


def _tracks(case, seed, grid, cols):
    if case["kind"] == "eq1_direct":
        return _drift_tracks(grid, cols, case["n_tracks"], case["n_steps"], seed)
    return _mip_tracks(grid, case["n_tracks"], case["n_steps"], seed)


def _waveforms(case, seed):
    """Current-like pulses (rise, fall, tail; either sign), their tangents, unit noise."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    n, m, d = case["n_tracks"], case["n"], case["n_dir"]
    u = lambda *s: torch.rand(*s, generator=g, device="cuda", dtype=torch.float64)  # noqa: E731
    t = torch.linspace(0, 1, m, device="cuda", dtype=torch.float64)
    pulse = lambda a, t0, tr, tf: a * (torch.sigmoid((t - t0) / tr) * torch.exp(-(t - t0).clamp_min(0) / tf))  # noqa: E731
    sign = torch.where(u(n, 1) < 0.5, -1.0, 1.0)
    i = pulse(1e-6 * sign * (0.2 + u(n, 1)), 0.1 + 0.4 * u(n, 1), 0.01 + 0.03 * u(n, 1), 0.05 + 0.3 * u(n, 1))
    di = None
    if d:
        di = pulse(1e-6 * (u(d, n, 1) - 0.5), 0.1 + 0.4 * u(d, n, 1), 0.02 + 0.03 * u(d, n, 1), 0.1 + 0.2 * u(d, n, 1))
        di = di.to(torch.float32).contiguous()
    noise = torch.randn(n, m, generator=g, device="cuda")
    return i.to(torch.float32).contiguous(), di, noise


SHAPER = {"dt": 1e-11, "tau": 8e-11, "order": 2, "gain": 3.0, "noise_rms": 2e-8}


def _points(case, seed, grid):
    rng = np.random.default_rng([seed, 6])
    xyz = rng.uniform(0, 1, (case["n_points"], 3)) * [grid.Lx, grid.Ly, grid.Lz]
    return xyz, 10.0 ** rng.uniform(-12.0, -8.0, case["n_at"])


# ------------------------------------------------------------- the library
def prepare(case, seed):
    kind = case["kind"]
    if kind == "waveforms":
        grid, cols = _matrix(1, 16, 16, 8, seed)
        i, di, noise = _waveforms(case, seed)
        return {"kind": kind, "sensor": wt.Sensor(grid, cols), "i": i, "di": di, "noise": noise}
    if kind == "batch":
        sensors = []
        for grid, cols in _batch_geometries(case, seed):
            s = wt.Sensor(grid, cols)
            s.fit()
            s.relax(_times(case["n_t"]))
            sensors.append(s)
        H = [torch.empty(s.h_shape(), dtype=torch.float32, device="cuda") for s in sensors]
        return {"kind": kind, "sensors": sensors, "H": H}
    grid, cols = _geometry(case, seed)
    state = {"kind": kind, "grid": grid, "cols": cols, "times": _times(case["n_t"])}
    if kind == "setup":
        return state
    s = wt.Sensor(grid, cols)
    s.fit()
    state["sensor"] = s
    if kind == "relax":
        state["rho"] = _profiles(cols, seed)
        return state
    s.relax(state["times"])
    if kind == "extend":
        state["H"] = torch.empty(s.h_shape(), dtype=torch.float32, device="cuda")
    elif kind == "extend64":
        state["H"] = torch.empty(s.h_shape(), dtype=torch.float64, device="cuda")
    elif kind == "points":
        state["xyz"], state["at"] = _points(case, seed, grid)
    else:
        state["tracks"] = _tracks(case, seed, grid, cols)
        if kind != "tangents":
            state["i"] = torch.empty((case["n_tracks"], 2 * case["n_steps"]), dtype=torch.float32, device="cuda")
        if kind == "eq1":
            state["H"] = s.extend("fp32")
    return state


def run(state):
    kind = state["kind"]
    if kind == "setup":
        s = wt.Sensor(state["grid"], state["cols"])
        s.fit()
        s.relax(state["times"])
        out = {"charges": s.charges(), "modes": s.modes()}
        if s.n_sources <= 256:
            out["capacitance"] = s.capacitance()
        s.close()
        return out
    if kind == "batch":
        return wt.extend_batch(state["sensors"], "fp32", outs=state["H"])
    s = state["sensor"]
    if kind == "relax":
        for k, rho in enumerate(state["rho"]):
            s.set_resistivity_profile(k, rho)
        s.relax(state["times"])
        return {"charges": s.charges(), "modes": s.modes()}
    if kind == "extend":
        return s.extend("fp32", out=state["H"])
    if kind == "extend64":
        return s.extend("fp64", out=state["H"])
    if kind == "points":
        return s.sample_H(state["xyz"], state["at"])
    if kind == "eq1":
        return s.eq1(state["H"], state["tracks"], out=state["i"])
    if kind == "eq1_direct":
        return s.eq1_direct(state["tracks"], out=state["i"])
    if kind == "tangents":
        i, di, loss, grad = s.tangents(state["tracks"])
        # loss and gradient are sums over FP32 currents
        return {"i": i, "di": di, "loss": np.float32(loss), "grad": np.asarray(grad, dtype=np.float32)}
    k = SHAPER
    v = s.shape(state["i"], k["dt"], k["tau"], k["order"], k["gain"], noise=state["noise"], noise_rms=k["noise_rms"])
    f, df = s.features(state["i"], k["dt"], dx=state["di"])
    return {"shaped": v, "features": f, "sensitivities": df}


# -------------------------------------------------------------------- work
def work(case):
    kind = case["kind"]
    if kind == "waveforms":
        n, m, d = case["n_tracks"], case["n"], case["n_dir"]
        taps = min(m, int((SHAPER["order"] + 60) * SHAPER["tau"] / SHAPER["dt"]) + 1)
        return {"bytes": 4.0 * n * m * (3 + d) + 8.0 * n * 6 * (1 + d),
                "flops": 2.0 * n * (taps * (taps + 1) / 2 + taps * (m - taps)) + n * m * (4.0 + d)}
    if kind == "batch":
        b = f = 0.0
        for grid, cols in _batch_geometries(case, 0):
            npts, n = grid.Nx * grid.Ny * grid.Nz, sum(c.n_sources for c in cols)
            b += 12.0 * npts * case["n_t"] + 8.0 * n * 32
            f += 3.0 * npts * (2.0 * 32 * case["n_t"] + 32 * 2.5 * math.log2(npts))
        return {"bytes": b, "flops": f}
    grid, cols = _geometry(case, 0)
    n = float(sum(c.n_sources for c in cols))
    nc, n_t, npts = N_AZ * N_H * n, case["n_t"], float(grid.Nx * grid.Ny * grid.Nz)
    # normal matrix (half of it), its factor, two solves with n right-hand sides; the columns' tables
    fit = n * n * nc + n ** 3 / 3 + 2 * n ** 3 + 2.0 * nc * n * grid.Nz / len(cols)
    # factor, two-sided reduction, tridiagonal form, divide and conquer, back-transformation, charges
    relax = n ** 3 * (1 / 3 + 1 + 4 / 3 + 4 / 3 + 2 + 1) + 4.0 * n * n * n_t
    fields = 3.0 * npts * 32 * 2.5 * math.log2(npts)
    if kind == "setup":
        return {"bytes": 8.0 * (n * n_t + n + n_t + (n * n if n <= 256 else 0)), "flops": fit + relax}
    if kind == "relax":
        return {"bytes": 8.0 * (n * n + n * n_t + 2 * n + n_t), "flops": relax}
    if kind == "extend":
        return {"bytes": 12.0 * npts * n_t + 8.0 * n * 32, "flops": fields + 3.0 * npts * 2.0 * 32 * n_t}
    if kind == "extend64":
        return {"bytes": 24.0 * npts * n_t + 8.0 * n * n_t, "flops": 3.0 * npts * n_t * 2.5 * math.log2(npts)}
    if kind == "points":
        k = float(case["n_points"]) * len(cols) * grid.Nx * grid.Ny / 4.0 * grid.Nz
        return {"bytes": 24.0 * case["n_points"] * (1 + case["n_at"]) + 16.0 * n * n + 8.0 * npts / 4,
                "flops": 6.0 * k + 6.0 * case["n_points"] * case["n_at"] * len(cols) * grid.Nz}
    steps = float(case["n_tracks"]) * case["n_steps"]
    io = steps * 24.0 + case["n_tracks"] * (4.0 + 8.0 * case["n_steps"])
    lags = 4.0 * case["n_tracks"] * case["n_steps"] * (1.5 * case["n_steps"])
    used = float(n_t)
    if kind == "eq1":          # a point of the field is read once however many tracks pass
        return {"bytes": io + 4.0 * min(steps * 24, 3 * npts) * used, "flops": steps * used * 54 + lags}
    per = steps * (32 * 54.0 + 2 * 32 * used) + lags
    if kind == "eq1_direct":
        return {"bytes": io + 4.0 * min(steps * 24, 3 * npts) * 32, "flops": per}
    # fit and modal tangents of four parameters, five fields and currents
    tangent = 2 * (6.0 * nc * n * n + 4 * n ** 3) + 4 * 6.0 * n ** 3 + 8.0 * nc * n * grid.Nz / len(cols)
    return {"bytes": io + 4 * 8.0 * case["n_tracks"] * case["n_steps"] + 8.0 * (nc * n + 4 * n * n),
            "flops": tangent + 5 * (per + fields)}


# ----------------------------------------------- the same in 64 bits, plain
def _modes_xy(grid):
    kx = 2 * math.pi / grid.Lx * torch.arange(-(grid.Nx // 2 - 1), grid.Nx // 2, device="cuda", dtype=torch.float64)
    ky = 2 * math.pi / grid.Ly * torch.arange(-(grid.Ny // 2 - 1), grid.Ny // 2, device="cuda", dtype=torch.float64)
    kz = math.pi / grid.Lz * torch.arange(grid.Nz, device="cuda", dtype=torch.float64)
    return kx, ky, kz


def _inv_k2(kx, ky, kz):
    k2 = kx[:, None, None] ** 2 + ky[None, :, None] ** 2 + kz[None, None, :] ** 2
    return torch.where(k2 > 0, 1 / torch.where(k2 > 0, k2, 1.0), 0.0)


def _lateral(fx, fy, ik2):
    """sum over lateral modes of fx[n, kx] fy[n, ky] ik2[kx, ky, kz] -> [n, kz]"""
    out = []
    for a, b in zip(fx.split(256), fy.split(256)):
        t = (a @ ik2.reshape(ik2.shape[0], -1)).reshape(len(a), ik2.shape[1], -1)
        out.append(torch.einsum("nyk,ny->nk", t, b))
    return torch.cat(out)


def _pref(grid):
    return 1.0 / (EPS0 * grid.eps_r * grid.Lx * grid.Ly * 2 * grid.Lz)


def _zcos(grid, z, kz):
    return torch.cos(_dev(z)[:, None] * kz[None, :])


class _Solved:
    """Fit and relaxation of one sensor (every column has the same source count)."""

    def __init__(self, grid, cols, profiles=None):
        self.grid, self.cols = grid, cols
        kx, ky, kz = self.k = _modes_xy(grid)
        ncol, m = len(cols), cols[0].n_sources
        n, nh = ncol * m, N_H * m
        self.z = (np.arange(m) + 0.5) * grid.Lz / m
        zc = (np.arange(nh) + 0.5) * grid.Lz / nh
        ik2 = _inv_k2(kx, ky, kz)
        d = np.array([[c.x + c.radius * math.cos(2 * math.pi * a / N_AZ) - b.x,
                       c.y + c.radius * math.sin(2 * math.pi * a / N_AZ) - b.y]
                      for c in cols for a in range(N_AZ) for b in cols])
        L = _lateral(torch.cos(_dev(d[:, :1]) * kx), torch.cos(_dev(d[:, 1:]) * ky), ik2)
        w = torch.full_like(kz, 4.0)       # image charge, and +-k_z
        w[0] = 2.0
        L = (L * w * _pref(grid)).reshape(ncol * N_AZ, ncol, 1, -1)
        P = (_zcos(grid, zc, kz) * L) @ _zcos(grid, self.z, kz).T            # [group, column, height, source]
        P = P.permute(0, 2, 1, 3).reshape(ncol * N_AZ * nh, n)
        # target: node potentials interpolated to the collocation heights
        u = np.clip(zc / (grid.Lz / m) - 0.5, 0, m - 1)
        j = np.minimum(np.floor(u).astype(int), max(m - 2, 0))
        S1 = np.zeros((nh, m))
        S1[np.arange(nh), j] += 1 - (u - j)
        if m > 1:
            S1[np.arange(nh), j + 1] += u - j
        S = torch.block_diag(*[_dev(np.tile(S1, (N_AZ, 1)))] * ncol)
        # q = B y with 1.q = 0, one free offset; columns scaled; Householder QR
        v = torch.ones(n, device="cuda", dtype=torch.float64)
        v[0] += math.sqrt(n)
        self.v, self.beta = v, 2.0 / float(v @ v)
        A = P - self.beta * torch.outer(P @ v, v)
        A[:, 0] = 1.0
        scale = A.norm(dim=0)
        Q, R = torch.linalg.qr(A / scale)
        X = torch.linalg.solve_triangular(R, Q.T @ S, upper=True) / scale[:, None]
        del P, A, Q, S
        X[0] = 0
        F = X - self.beta * torch.outer(v, v @ X)
        self.C = 0.5 * (F + F.T)
        # resistive lines
        K = torch.zeros((n, n), dtype=torch.float64)
        dz = grid.Lz / m
        for k, c in enumerate(cols):
            rho = np.full(m, c.resistivity) if profiles is None else profiles[k]
            area, o = math.pi * c.radius ** 2, k * m
            for a in range(m - 1):
                g = area / (0.5 * (rho[a] + rho[a + 1]) * dz)
                p, q = o + a, o + a + 1
                K[p, p] -= g
                K[q, q] -= g
                K[p, q] += g
                K[q, p] += g
            t = m - 1 if c.terminal_top else 0
            K[o + t, o + t] -= area / (0.5 * rho[t] * dz)
        K = K.cuda()
        K1 = K.sum(1)
        K = K - torch.outer(K1, K1) / K1.sum()
        Am, Sm = self._reduce(self.C), -self._reduce(K)
        Lc = torch.linalg.cholesky(0.5 * (Am + Am.T))
        Y = torch.linalg.solve_triangular(Lc, Sm, upper=False)
        Y = torch.linalg.solve_triangular(Lc, Y.T.contiguous(), upper=False)
        self.mu, U = torch.linalg.eigh(0.5 * (Y + Y.T))
        V = torch.linalg.solve_triangular(Lc.T, U, upper=True)
        phi = torch.cat([torch.full((m,), float(c.driven), dtype=torch.float64) for c in cols]).cuda()
        self.q_inf = self.C @ phi
        g = -(self.q_inf - self.beta * v * (v @ self.q_inf))[1:]
        self.V, self.amp = V, V.T @ g

    def _reduce(self, M):
        M = M - self.beta * torch.outer(self.v, self.v @ M)
        M = M - self.beta * torch.outer(M @ self.v, self.v)
        return M[1:, 1:]

    def charges(self, t):
        """[n_t, n_sources]"""
        z = self.V @ (self.amp[:, None] * torch.exp(-torch.outer(self.mu, _dev(t))))
        z = torch.cat([torch.zeros_like(z[:1]), z])
        z = z - self.beta * torch.outer(self.v, self.v @ z)
        return (self.q_inf[:, None] + self.C @ z).T.contiguous()

    def _column_spectra(self, t):
        """Z[t, column, k_z], the weights of +-k_z in it"""
        m, kz = len(self.z), self.k[2]
        Z = self.charges(t).reshape(len(t), len(self.cols), m) @ (2 * _zcos(self.grid, self.z, kz))
        w = torch.full_like(kz, 2.0)
        w[0] = 1.0
        return Z * (w * _pref(self.grid))

    def points(self, xyz, t):
        """W[t, point, component]"""
        kx, ky, kz = self.k
        Z = self._column_spectra(t)
        ik2 = _inv_k2(kx, ky, kz)
        p = _dev(xyz)
        X = (p[:, None, 0] - _dev([c.x for c in self.cols])).reshape(-1, 1) * kx
        Y = (p[:, None, 1] - _dev([c.y for c in self.cols])).reshape(-1, 1) * ky
        cz, sz = torch.cos(p[:, 2:] * kz), torch.sin(p[:, 2:] * kz)
        shape = (len(xyz), len(self.cols), len(kz))
        T = [_lateral(kx * torch.sin(X), torch.cos(Y), ik2).reshape(shape) * cz[:, None],
             _lateral(torch.cos(X), ky * torch.sin(Y), ik2).reshape(shape) * cz[:, None],
             _lateral(torch.cos(X), torch.cos(Y), ik2).reshape(shape) * (kz * sz)[:, None]]
        return torch.stack([torch.einsum("tck,pck->tp", Z, a) for a in T], dim=-1)

    def field(self, t):
        """W[t, component, x, y, z]"""
        g, (kx, ky, kz) = self.grid, self.k
        Z = self._column_spectra(t).permute(2, 0, 1).contiguous()            # [k_z, t, column]
        ik2 = _inv_k2(kx, ky, kz)
        x = torch.arange(g.Nx, device="cuda", dtype=torch.float64) * (g.Lx / g.Nx)
        y = torch.arange(g.Ny, device="cuda", dtype=torch.float64) * (g.Ly / g.Ny)
        z = (torch.arange(g.Nz, device="cuda", dtype=torch.float64) + 0.5) * (g.Lz / g.Nz)
        cz, sz = torch.cos(torch.outer(kz, z)), kz[:, None] * torch.sin(torch.outer(kz, z))
        H = torch.empty((len(t), 3, g.Nx, g.Ny, g.Nz), dtype=torch.float64, device="cuda")
        step = max(1, int(3e8 / (g.Nx * g.Ny * g.Nz)))
        for comp in range(3):
            T = []
            for c in self.cols:
                X, Y = torch.outer(x - c.x, kx), torch.outer(y - c.y, ky)
                fx = kx * torch.sin(X) if comp == 0 else torch.cos(X)
                fy = ky * torch.sin(Y) if comp == 1 else torch.cos(Y)
                a = (fx @ ik2.reshape(len(kx), -1)).reshape(g.Nx, len(ky), g.Nz)
                T.append(torch.einsum("xqk,yq->kxy", a, fy).reshape(g.Nz, -1))
            T = torch.stack(T, dim=1)                                         # [k_z, column, xy]
            for t0 in range(0, len(t), step):
                R = torch.bmm(Z[:, t0:t0 + step], T)                           # [k_z, t, xy]
                n = R.shape[1]
                W = R.reshape(g.Nz, -1).T @ (sz if comp == 2 else cz)
                H[t0:t0 + n, comp] = W.reshape(n, g.Nx, g.Ny, g.Nz)
        return H

    def currents(self, times, tr):
        """Eq. 1: trilinear in space, linear in time (0 at t = 0, held after the last sample)."""
        g = self.grid
        H = self.field(times).reshape(len(times), 3, -1).permute(2, 1, 0).contiguous()       # [point, component, t]
        n_out, n_steps, dt = tr["n_out"], tr["n_steps"], tr["dt"]
        lag = (np.arange(n_out) + 0.5) * dt
        T = np.zeros((n_out, len(times)))
        for k, s in enumerate(lag):
            if s <= times[0]:
                T[k, 0] = s / times[0]
            elif s >= times[-1]:
                T[k, -1] = 1.0
            else:
                a = int(np.searchsorted(times, s, side="right")) - 1
                f = (s - times[a]) / (times[a + 1] - times[a])
                T[k, a], T[k, a + 1] = 1 - f, f
        T = _dev(T)
        out = torch.empty((tr["n_tracks"], n_out), dtype=torch.float64, device="cuda")
        chunk = max(1, int(5e8 / (n_steps * 3 * len(times))))
        for a in range(0, tr["n_tracks"], chunk):
            p = [tr[k][a:a + chunk].double() for k in "xyz"]
            v = torch.stack([tr[k][a:a + chunk].double() for k in ("vx", "vy", "vz")], dim=-1)
            fx, fy = p[0] / (g.Lx / g.Nx), p[1] / (g.Ly / g.Ny)
            fz = (p[2] / (g.Lz / g.Nz) - 0.5).clamp(0, g.Nz - 1)
            i0, j0, k0 = fx.floor(), fy.floor(), fz.floor().clamp_max(g.Nz - 2)
            wx, wy, wz = fx - i0, fy - j0, fz - k0
            s = torch.zeros(p[0].shape + (len(times),), dtype=torch.float64, device="cuda")
            for c in range(8):
                di, dj, dk = c >> 2, (c >> 1) & 1, c & 1
                w = (wx if di else 1 - wx) * (wy if dj else 1 - wy) * (wz if dk else 1 - wz)
                at = (((i0 + di).long() % g.Nx) * g.Ny + (j0 + dj).long() % g.Ny) * g.Nz + k0.long() + dk
                s += torch.einsum("nsct,nsc->nst", H[at], w[..., None] * v)
            s = s @ T.T                                                         # [track, step, lag]
            Q = torch.zeros((len(s), n_out), dtype=torch.float64, device="cuda")
            for step in range(n_steps):
                Q[:, step:] += s[:, step, : n_out - step] * dt
            Q = torch.diff(Q, prepend=torch.zeros_like(Q[:, :1]), dim=1)
            out[a:a + chunk] = -tr["q"][a:a + chunk].double()[:, None] * Q / dt
        return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "waveforms":
        i, _, noise = _waveforms(case, seed)
        k, n = SHAPER, case["n"]
        t = torch.arange(n, device="cuda", dtype=torch.float64) * (k["dt"] / k["tau"])
        h = k["gain"] * k["dt"] * t ** k["order"] * torch.exp(-t) / (math.factorial(k["order"]) * k["tau"])
        lag = torch.arange(n, device="cuda")[None, :] - torch.arange(n, device="cuda")[:, None]
        T = torch.where(lag >= 0, h[lag.clamp_min(0)], 0.0)
        # features turn on single-precision comparisons: no 64-bit value
        return {"shaped": i.double() @ T + k["noise_rms"] * noise.double(), "features": None, "sensitivities": None}
    if kind == "batch":
        return [_Solved(*g).field(_times(case["n_t"])) for g in _batch_geometries(case, seed)]
    grid, cols = _geometry(case, seed)
    times = _times(case["n_t"])
    s = _Solved(grid, cols, _profiles(cols, seed) if kind == "relax" else None)
    if kind in ("setup", "relax"):
        out = {"charges": s.charges(times), "modes": s.mu}
        if kind == "setup" and len(s.q_inf) <= 256:
            out["capacitance"] = s.C
        return out
    if kind in ("extend", "extend64"):
        return s.field(times)
    if kind == "points":
        return s.points(*_points(case, seed, grid))
    i = s.currents(times, _tracks(case, seed, grid, cols))
    if kind == "tangents":
        return {"i": i, "di": None, "loss": float((i * i).mean()), "grad": None}
    return i
