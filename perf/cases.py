"""Timed workloads of the particle-in-cell library, through its Python binding.

A pass of a stepping case is what a simulation does between two of its outputs:
advance the run by `steps` steps and read the whole state (fields and particles,
FP64) back into page-locked host buffers that the program keeps.  A pass of a
loading case fills a run with a new Maxwell-Juttner plasma and reads it back.

Case fields: kind ("step", "ensemble", "load"), precision ("mixed", "fp64"),
the grid (ndim, nx, ny, nz), ppc (particles per cell and species), theta
(temperature), mass (of the second species, in electron masses), walls
(conductors in x with a Harris sheet between them), smooth (current smoothing
passes), tile and sort (context options; "" and 0 are the library's defaults),
steps, and from_loader (initial state by the library's own loader, for the runs
whose state would be large to upload).
"""
import math

import numpy as np
import torch

import paper_1308_5892_gb300 as pic

DT = 0.5
GRID = 16777216.0            # offsets of the mixed path lie on a grid of 2^-24 cells
EXACT_PARTICLE_STEPS = 1.2e9   # the FP64 restatement below takes a few seconds up to here


def _case(name, kind="step", precision="mixed", ndim=2, nx=64, ny=64, nz=1, ppc=16, theta=0.1, mass=1.0, walls=False,
          smooth=0, tile="", sort=0, steps=16, from_loader=False, runs=1, method="exact"):
    c = dict(kind=kind, precision=precision, ndim=ndim, nx=nx, ny=ny, nz=nz, ppc=ppc, theta=theta, mass=mass,
             walls=walls, smooth=smooth, tile=tile, sort=sort, steps=steps, from_loader=from_loader, runs=runs,
             method=method)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest run of the tests, one step per output (debugging, step-by-step comparison):
        # launches, synchronisations and host calls are all there is
        _case("mixed2d_40x24_1step", nx=40, ny=24, ppc=8, theta=0.3, steps=1),
        # the benchmark's small 2D plasma: tens of short steps per output
        _case("mixed2d_64", nx=64, ny=64, ppc=16, theta=0.1, steps=16),
        # an ordinary 2D plasma, cold (particles drift little between re-sorts)
        _case("mixed2d_512", nx=512, ny=512, ppc=50, theta=0.01, steps=32, sort=16),
        # the largest 2D workload of the benchmark, with the tuner's choice of tile and sort interval
        _case("mixed2d_1024", nx=1024, ny=1024, ppc=50, theta=0.01, tile="16x16x1", sort=16, steps=32,
              from_loader=True),
        # reconnection set-up: Harris sheet between conducting walls, ragged grid, reflections at the walls
        _case("mixed2d_walls_harris", nx=251, ny=130, ppc=64, theta=0.1, walls=True, steps=16),
        # 3D ion-electron plasma on a ragged grid with current smoothing
        _case("mixed3d_ragged_ions", ndim=3, nx=45, ny=37, nz=51, ppc=20, theta=0.1, mass=25.0, smooth=1, steps=12),
        # the benchmark's hot 3D plasma at profiling size, library defaults
        _case("mixed3d_64", ndim=3, nx=64, ny=64, nz=64, ppc=32, theta=1.0, steps=24),
        # the headline workload, with the tuner's choice
        _case("mixed3d_128", ndim=3, nx=128, ny=128, nz=128, ppc=32, theta=1.0, tile="16x8x4", sort=3, steps=24,
              from_loader=True),
        # double precision, for runs that need it and for checking the mixed path: 3D and a ragged 2D grid
        _case("fp64_3d_64", precision="fp64", ndim=3, nx=64, ny=64, nz=64, ppc=32, theta=1.0, steps=6),
        _case("fp64_2d_ragged", precision="fp64", nx=300, ny=211, ppc=24, theta=0.1, steps=8),
        # a batch of independent uneven runs advanced together (parameter studies)
        _case("ensemble_16", kind="ensemble", runs=16, tile="32x16x1", sort=8, steps=32, from_loader=True),
        # start of a run: both species of a drifting pair plasma from the exact sampler, read back for a dump
        _case("load_3d_64", kind="load", ndim=3, nx=64, ny=64, nz=64, ppc=16, theta=0.5),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step"] * 7 + ["ensemble", "load"])
    if kind == "ensemble":
        return _case("", kind=kind, runs=rng.randint(2, 14), nx=rng.randint(1, 10000), tile=rng.choice(["", "32x16x1"]),
                     sort=rng.choice([0, 4, 8]), steps=rng.randint(4, 32), smooth=rng.choice([0, 0, 1]),
                     from_loader=True)
    ndim = rng.choice([2, 3])
    theta = round(math.exp(rng.uniform(math.log(0.01), 0.0)), 4)
    if ndim == 2:
        g = dict(nx=_log(rng, 24, 700), ny=_log(rng, 24, 700), nz=1)
    else:
        g = dict(nx=_log(rng, 12, 80), ny=_log(rng, 12, 80), nz=_log(rng, 12, 80))
    ppc = _log(rng, 4, 64)
    if kind == "load":
        return _case("", kind=kind, precision=rng.choice(["mixed", "fp64"]), ndim=ndim, ppc=ppc, theta=theta, **g)
    precision = rng.choice(["mixed", "mixed", "mixed", "fp64"])
    walls = ndim == 2 and rng.random() < 0.2
    particles = 2 * ppc * g["nx"] * g["ny"] * g["nz"]
    steps = min(rng.choice([1, 4, 8, 16, 24, 32]), max(1, int((2e8 if precision == "fp64" else 1e9) // particles)))
    tile, sort = "", 0
    if precision == "mixed":
        tile = rng.choice([""] * 3 + (["32x16x1", "16x8x1", "32x32x1"] if ndim == 2 else ["8x8x4", "16x8x4"]))
        sort = rng.choice([0, 0, 4, 8] if ndim == 2 else [0, 0, 1, 2, 4])
    return _case("", precision=precision, ndim=ndim, ppc=ppc, theta=theta, walls=walls,
                 mass=rng.choice([1.0, 1.0, 25.0]), smooth=0 if walls else rng.choice([0, 0, 0, 1, 2]),
                 tile=tile, sort=sort, steps=steps, **g)


# ------------------------------------------------------------------ sizes

def _members(c):
    """The runs of a case: dicts of nx, ny, nz, ppc, theta."""
    if c["kind"] != "ensemble":
        return [dict(nx=c["nx"], ny=c["ny"], nz=c["nz"], ppc=c["ppc"], theta=c["theta"])]
    rng = np.random.default_rng(4 if c["nx"] == 64 else c["nx"])   # the benchmark's members, or a drawn set
    out = []
    for _ in range(c["runs"]):
        nx, ny = (int(v) for v in rng.integers(32, 257, 2))
        ppc = int(rng.choice([4, 8, 16, 32, 64, 128, 256]))
        out.append(dict(nx=nx, ny=ny, nz=1, ppc=ppc, theta=float(np.exp(rng.uniform(np.log(0.01), 0.0)))))
    return out


def _sheet(c):
    """Half width L, centre x0 and particles per species of the Harris sheet."""
    L, x0 = c["nx"] / 12.0, c["nx"] / 2.0
    return L, x0, int(round(c["ppc"] * c["ny"] * L * 2.0 * math.tanh(x0 / L)))


def _count(c, m):
    return _sheet(c)[2] if c["walls"] else int(round(m["ppc"] * m["nx"] * m["ny"] * m["nz"]))


def _units(c, m):
    """n_x (cells per skin depth: the Debye length is a cell, 4 cells for a sheet) and rho_sp0."""
    return (4.0 if c["walls"] else m["theta"] ** -0.5), 2.0 * m["ppc"]


# ------------------------------------------------------------------ initial states

def _momenta(g, n, theta, mass):
    """Maxwell-Juttner momenta of temperature theta / mass: Gaussian when cold,
    the method of Sobol (products of uniforms, rejection) when hot."""
    th = theta / mass
    dev = g.device
    if th < 0.1:
        return torch.randn(3, n, generator=g, device=dev, dtype=torch.float64) * math.sqrt(th)
    got, have = [], 0
    while have < n:
        x = torch.rand(4, 2 * (n - have) + 1024, generator=g, device=dev, dtype=torch.float64).clamp_min(1e-300).log()
        u = -th * (x[0] + x[1] + x[2])
        u = u[(u - th * x[3]) ** 2 - u * u > 1.0]
        got.append(u)
        have += u.numel()
    u = torch.cat(got)[:n]
    r = torch.rand(2, n, generator=g, device=dev, dtype=torch.float64)
    cz = 2.0 * r[0] - 1.0
    s = (1.0 - cz * cz).sqrt()
    ph = 2.0 * math.pi * r[1]
    return torch.stack([u * s * ph.cos(), u * s * ph.sin(), u * cz])


def _initial(c, seed):
    """Fields (6, nz, ny, nx) and particles per species (6, n), FP64 on the device;
    momenta and fields are FP32 values and offsets lie on the mixed path's grid, so
    that both precisions start from the same state."""
    g = torch.Generator("cuda")
    g.manual_seed(int(seed))
    dev = g.device
    m = _members(c)[0]
    n, shape = _count(c, m), (c["nz"], c["ny"], c["nx"])
    size = (c["nx"], c["ny"], c["nz"])
    f = 0.01 * torch.randn(6, *shape, generator=g, device=dev, dtype=torch.float64)
    r = torch.rand(3, n, generator=g, device=dev, dtype=torch.float64)
    drift = 0.0
    if c["walls"]:
        L, x0, _ = _sheet(c)
        n_x = _units(c, m)[0]
        b0 = 2.0 * math.sqrt(c["theta"]) / n_x            # pressure balance across the sheet
        drift = b0 * n_x * n_x / (2.0 * L)                # and its current
        xs = torch.arange(c["nx"], device=dev, dtype=torch.float64) + 0.5
        f[4] += b0 * torch.tanh((xs - x0) / L)
        f[3][..., 0] = 0.0
        f[1][..., 0] = 0.0
        f[2][..., 0] = 0.0
        ta = math.tanh(x0 / L)
        r[0] = ((x0 + L * torch.atanh((2.0 * r[0] - 1.0) * ta)) / c["nx"]).clamp(0.0, 1.0)
    f = f.float().double()
    pos = torch.zeros(3, n, device=dev, dtype=torch.float64)
    for a in range(c["ndim"]):
        x = r[a] * size[a]
        x = x.floor() + ((x - x.floor()) * GRID).round() / GRID
        pos[a] = torch.where(x >= size[a], 0.0, x)
    parts = []
    for q, mass in ((-1.0, 1.0), (1.0, c["mass"])):
        u = _momenta(g, n, c["theta"], mass)
        u[2] += q * drift
        parts.append(torch.cat([pos, u.float().double()]))   # pairs on top of each other: no charge density
    return f, parts


def _pinned(m, n, species):
    f = torch.empty(6, m["nz"], m["ny"], m["nx"], dtype=torch.float64, pin_memory=True)
    return f, [torch.empty(6, n, dtype=torch.float64, pin_memory=True) for _ in range(species)]


def prepare(case, seed):
    c = case
    members = _members(c)
    descs, outs = [], []
    for m in members:
        n = _count(c, m)
        n_x, rho0 = _units(c, m)
        descs.append(pic.run_desc(c["ndim"], m["nx"], m["ny"], m["nz"], n_x, rho0, DT,
                                  [(-1.0, 1.0, n), (1.0, c["mass"], n)], bc=(1 if c["walls"] else 0, 0, 0),
                                  smooth_passes=c["smooth"]))
        outs.append(_pinned(m, n, 2))
    tile = tuple(int(v) for v in c["tile"].split("x")) if c["tile"] else (0, 0, 0)
    ctx = pic.Context(descs, precision=pic.PIC_FP64 if c["precision"] == "fp64" else pic.PIC_MIXED, tile=tile,
                      sort_interval=c["sort"])
    if c["kind"] != "load":
        if c["from_loader"]:
            for r, m in enumerate(members):
                _load(ctx, r, m["ppc"], m["theta"], (0.0, 0.0, 0.0), 1000 * seed + 2 * r)
        else:
            f, parts = _initial(c, seed)
            ctx.set_state(0, f.cpu().numpy(), [p.cpu().numpy() for p in parts])
    return dict(case=c, ctx=ctx, outs=outs, seed=seed, views=[(f.numpy(), [p.numpy() for p in ps]) for f, ps in outs])


def _load(ctx, run, ppc, theta, beta, seed, method=pic.PIC_MJ_EXACT):
    ctx.load_maxwell_juttner(run, 0, ppc, theta, beta, method=method, seed=seed)
    ctx.load_maxwell_juttner(run, 1, ppc, theta, beta, method=method, colocate_with=0, seed=seed + 1)


def run(state):
    c, ctx = state["case"], state["ctx"]
    if c["kind"] == "load":
        _load(ctx, 0, c["ppc"], c["theta"], (0.0, 0.0, 0.5), 1000 * state["seed"])
    else:
        ctx.step(c["steps"])
    for r, view in enumerate(state["views"]):
        ctx.get_state(r, out=view)
    outs = []
    for f, parts in state["outs"]:
        outs.append({"fields": f, "particles": [p for p in parts]})
    return outs


def work(case):
    c = case
    fp64 = c["precision"] == "fp64"
    per_p = {2: 40.0, 3: 48.0}[c["ndim"]] if fp64 else {2: 24.0, 3: 28.0}[c["ndim"]]
    per_c = 8.0 if fp64 else 4.0
    flops_p = {2: 232.0, 3: 332.0}[c["ndim"]]
    b = fl = 0.0
    for m in _members(c):
        n, cells = 2.0 * _count(c, m), float(m["nx"] * m["ny"] * m["nz"])
        out = 48.0 * (n + cells)
        if c["kind"] == "load":
            b += per_p * n + out
            fl += 200.0 * n
            continue
        # every step reads and writes the particles and the six field planes; the state is written out once
        b += c["steps"] * (2.0 * per_p * n + 12.0 * per_c * cells) + out
        fl += c["steps"] * (flops_p * n + 60.0 * cells)
    return {"bytes": b, "flops": fl}


# ------------------------------------------------------------------ the same step in FP64 tensors

def _roll(a, s, axis):
    """a at index + s along x (0), y (1) or z (2) of a (nz, ny, nx) block, periodic."""
    return torch.roll(a, -s, 2 - axis)


def _curl_e(e):
    return ((_roll(e[2], 1, 1) - e[2]) - (_roll(e[1], 1, 2) - e[1]), (_roll(e[0], 1, 2) - e[0]) - (_roll(e[2], 1, 0) - e[2]),
            (_roll(e[1], 1, 0) - e[1]) - (_roll(e[0], 1, 1) - e[0]))


def _curl_b(b):
    return ((b[2] - _roll(b[2], -1, 1)) - (b[1] - _roll(b[1], -1, 2)), (b[0] - _roll(b[0], -1, 2)) - (b[2] - _roll(b[2], -1, 0)),
            (b[1] - _roll(b[1], -1, 0)) - (b[0] - _roll(b[0], -1, 1)))


def _nodes(e, b, walls):
    """Node averages of e and b; with walls the x nodes are 0 .. nx and what lies
    inside the conductor, or vanishes on it, counts as zero."""
    e, b = list(e), list(b)
    if walls:
        def wide(a, staggered):
            z = torch.zeros_like(a[..., :1])
            a = torch.cat([z, a, z], 2)                   # x index -1 .. nx
            if not staggered:
                a[..., 1] = 0.0                           # on the low wall
            return a
        e = [wide(e[0], True), wide(e[1], False), wide(e[2], False)]
        b = [wide(b[0], False), wide(b[1], True), wide(b[2], True)]
    mean = lambda a, ax: 0.5 * (a + _roll(a, -1, ax))  # noqa: E731
    out = [mean(e[0], 0), mean(e[1], 1), mean(e[2], 2), mean(mean(b[0], 1), 2), mean(mean(b[1], 0), 2),
           mean(mean(b[2], 0), 1)]
    return [a[..., 1:].contiguous() for a in out] if walls else out


def _index(i, j, k, shape):
    return (k.remainder(shape[0]) * shape[1] + j.remainder(shape[1])) * shape[2] + i.remainder(shape[2])


def _gather(nodes, cell, d, ndim):
    shape = nodes[0].shape
    out = [torch.zeros_like(d[0]) for _ in range(6)]
    for xi in range(2 if ndim == 3 else 1):
        for eta in range(2):
            for eps in range(2):
                w = (d[0] if eps else 1.0 - d[0]) * (d[1] if eta else 1.0 - d[1])
                if ndim == 3:
                    w = w * (d[2] if xi else 1.0 - d[2])
                q = _index(cell[0] + eps, cell[1] + eta, cell[2] + xi, shape)
                for v in range(6):
                    out[v] += w * nodes[v].reshape(-1)[q]
    return out[:3], out[3:]


def _flux(J, x, D, alpha, ndim):
    """Adds the current of straight paths from x by D: cut at the planes they
    cross, each piece's exact flux through the faces of its cell."""
    shape = J[0].shape
    flat = [a.view(-1) for a in J]
    ts = []
    for a in range(ndim):
        lo, hi = x[a], x[a] + D[a]
        plane = torch.where(D[a] > 0, torch.floor(lo) + 1.0, torch.ceil(lo) - 1.0)
        cross = torch.where(D[a] > 0, plane < hi, plane > hi)
        ts.append(torch.where(cross, ((plane - lo) / torch.where(cross, D[a], 1.0)).clamp(0.0, 1.0), 1.0))
    t = torch.stack(ts + [torch.ones_like(ts[0])]).sort(0).values
    t0 = torch.zeros_like(ts[0])
    for k in range(ndim + 1):
        live = torch.nonzero(t[k] > t0).view(-1) if k else torch.arange(t0.numel(), device=t0.device)
        ta, tb = t0[live], t[k][live]
        t0 = t[k]
        if not live.numel():
            continue
        w, Dp, cell = [], [], []
        for a in range(3):
            Da = D[a][live]
            Dp.append(Da * (tb - ta))
            if a < ndim:
                mid = x[a][live] + Da * (0.5 * (ta + tb))
                ca = torch.floor(mid)
                cell.append(ca.long())
                w.append((1.0 - (mid - ca), mid - ca))
            else:
                cell.append(torch.zeros_like(live))
                w.append(None)
        for comp in range(3):
            p, q = ((1, 2), (2, 0), (0, 1))[comp]
            base = -alpha * Dp[comp]
            if ndim == 2 and comp < 2:
                o = 1 - comp                              # in-plane flux: the other axis alone weighs
                for s in range(2):
                    at = _index(cell[0] + (s if o == 0 else 0), cell[1] + (s if o == 1 else 0), cell[2], shape)
                    flat[comp].index_add_(0, at, base * w[o][s])
                continue
            twist = Dp[p] * Dp[q] / 12.0
            for sp in range(2):
                for sq in range(2):
                    off = [0, 0, 0]
                    off[p], off[q] = sp, sq
                    at = _index(cell[0] + off[0], cell[1] + off[1], cell[2] + off[2], shape)
                    sign = 1.0 if sp == sq else -1.0
                    flat[comp].index_add_(0, at, base * (w[p][sp] * w[q][sq] + sign * twist))


def _smooth(a, ndim):
    for ax in range(ndim):
        a = 0.25 * (_roll(a, -1, ax) + _roll(a, 1, ax)) + 0.5 * a
    return a


def _exact_step(c, m, f, parts):
    ndim, size = c["ndim"], (m["nx"], m["ny"], m["nz"])
    n_x, rho0 = _units(c, m)
    e, b = [f[k].clone() for k in range(3)], [f[3 + k].clone() for k in range(3)]

    def b_half():
        for a, cu in zip(b, _curl_e(e)):
            a -= 0.5 * DT * cu
        if c["walls"]:
            b[0][..., 0] = 0.0

    b_half()
    nodes = _nodes(e, b, c["walls"])
    J = [torch.zeros_like(e[0]) for _ in range(3)]
    for P, (q, mass) in zip(parts, ((-1.0, 1.0), (1.0, c["mass"]))):
        alpha, h = 2.0 * q / (n_x * n_x * rho0), q / mass
        for s0 in range(0, P.shape[1], 1 << 22):
            X = P[:, s0:s0 + (1 << 22)]
            cell, d = [], []
            for a in range(3):
                fl = X[a].floor()
                if c["walls"] and a == 0:
                    fl = fl.clamp_max(size[0] - 1)
                cell.append(fl.long() if a < ndim else torch.zeros_like(fl, dtype=torch.long))
                d.append(X[a] - fl if a < ndim else torch.zeros_like(fl))
            E, B = _gather(nodes, cell, d, ndim)
            u = [X[3 + a] + 0.5 * h * DT * E[a] for a in range(3)]
            gam = (1.0 + u[0] ** 2 + u[1] ** 2 + u[2] ** 2).sqrt()
            t = [0.5 * h * DT * B[a] / gam for a in range(3)]
            s = [2.0 * t[a] / (1.0 + t[0] ** 2 + t[1] ** 2 + t[2] ** 2) for a in range(3)]
            cross = lambda v, w: [v[1] * w[2] - v[2] * w[1], v[2] * w[0] - v[0] * w[2], v[0] * w[1] - v[1] * w[0]]  # noqa: E731
            up = [v + r for v, r in zip(u, cross(u, t))]
            u = [v + r + 0.5 * h * DT * E[a] for a, (v, r) in enumerate(zip(u, cross(up, s)))]
            gam = (1.0 + u[0] ** 2 + u[1] ** 2 + u[2] ** 2).sqrt()
            D = [DT * v / gam for v in u]
            x = [X[0].clone(), X[1].clone(), X[2].clone()]
            end = [x[a] + D[a] if a < ndim else x[a] for a in range(3)]
            if c["walls"]:
                hit = torch.nonzero((end[0] < 0.0) | (end[0] > size[0])).view(-1)
                if hit.numel():
                    wall = torch.where(end[0][hit] < 0.0, 0.0, float(size[0]))
                    th = (wall - x[0][hit]) / D[0][hit]
                    first = [wall - x[0][hit], D[1][hit] * th, D[2][hit] * th]
                    back = [-(D[0][hit] - first[0]), D[1][hit] - first[1], D[2][hit] - first[2]]
                    _flux(J, [v[hit] for v in x], first, alpha, ndim)
                    _flux(J, [wall, x[1][hit] + first[1], x[2][hit]], back, alpha, ndim)
                    end[0][hit] = wall + back[0]
                    u[0][hit] = -u[0][hit]
                    rest = torch.ones_like(x[0], dtype=torch.bool)
                    rest[hit] = False
                    rest = torch.nonzero(rest).view(-1)
                    _flux(J, [v[rest] for v in x], [v[rest] for v in D], alpha, ndim)
                else:
                    _flux(J, x, D, alpha, ndim)
            else:
                _flux(J, x, D, alpha, ndim)
            for a in range(3):
                if a < ndim:
                    xe = end[a]
                    if not (c["walls"] and a == 0):
                        xe = torch.where(xe < 0.0, xe + size[a], xe)
                        xe = torch.where(xe >= size[a], xe - size[a], xe)
                    X[a] = xe
                X[3 + a] = u[a]
    if c["smooth"]:
        for _ in range(c["smooth"]):
            J = [_smooth(a, ndim) for a in J]
    b_half()
    for a, cu, j in zip(e, _curl_b(b), J):
        a += DT * cu + j
    if c["walls"]:
        e[1][..., 0] = 0.0
        e[2][..., 0] = 0.0
    return torch.stack(e + b), parts


def exact(case, seed):
    c = case
    if c["kind"] != "step" or c["from_loader"]:
        return None                                       # the state comes from the library's own sampler
    m = _members(c)[0]
    if 2.0 * _count(c, m) * c["steps"] > EXACT_PARTICLE_STEPS:
        return None
    f, parts = _initial(c, seed)
    for _ in range(c["steps"]):
        f, parts = _exact_step(c, m, f, parts)
    return [{"fields": f, "particles": parts}]
