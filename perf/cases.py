"""Performance cases of the APM solver: what a user has it do, through its public entry points.

Every case is one call sequence of `Solver` on a grid hierarchy: a whole solve
(`step`), or one of its layers on its own (`deposit_all`, `solve_level`,
`accel`, `interp_all` + `kick_drift`).  The hierarchies are the repository's own
benchmark configurations and ordinary ones around them: isolated and periodic
roots, nested levels, levels of many equal or many uneven subgrids, gas or
particles only, lattice, random and clustered particles, both precisions and
the three gradient operators.  Launch shapes are the library's defaults.
"""
import math

import numpy as np
import torch

from paper_1410_0010_gb300.solver import PARTICLE_KEYS, Particles, Solver

FRAC = 52            # fraction bits of the mass fields (the library's default)
A_DX = 3.4           # smoothing diameter in cells (the library's default)
BORDER = 5           # mass-field border cells per side that follow from it
MARGIN = 3           # parent cells between a child and the edge of its parent
DEV = "cuda"

# fields of a case and their defaults
DEFAULTS = dict(kind="step", precision="fp32", gradient="fd2", root=64, periodic=True, per_axis=0, depth=1, child=64,
                child_lo=0, particles=0, dist="uniform", gas=False, order=False, tiles=False, graph=False)


def listed():
    return [
        # the smallest whole solve: a test-particle study on an isolated 32^3 root, one eager call
        dict(name="step-iso32-4k", root=32, periodic=False, particles=4096),
        # two levels with gas and few particles, replayed as a CUDA graph inside a time loop
        dict(name="step-two-level64-gas-graph", root=64, periodic=False, per_axis=1, child=64, particles=1024, gas=True,
             graph=True),
        # a clustered halo through three nested levels: every particle in a few cells, ordered with tiles
        dict(name="step-plummer128-1M", root=128, per_axis=1, depth=3, child=64, particles=1 << 20, dist="plummer",
             order=True, tiles=True),
        # the whole cosmological solve: 512^3 root, 2 x 64 subgrids of 128^3, 16.8 M lattice particles
        dict(name="step-cosmo512-16M", root=512, per_axis=4, depth=2, child=128, particles=1 << 24, dist="lattice"),
        # the mass deposit of randomly placed particles on a root with refined levels
        dict(name="deposit-uniform256-4M", kind="deposit", root=256, per_axis=2, depth=2, child=64, particles=1 << 22),
        # the second half of a timestep of random particles: order, interpolation, kick-drift
        dict(name="interp-kick-uniform256-4M", kind="interp", root=256, per_axis=2, depth=2, child=64,
             particles=1 << 22, order=True),
        # the potential solve of one level of many equal subgrids (transforms of length 150)
        dict(name="solve-32x128", kind="solve", root=384, per_axis=4, depth=1, child=128, child_lo=-32),
        # ... of one level of many small uneven subgrids, the shape that adaptive refinement gives
        dict(name="solve-uneven-343", kind="solve", root=256, per_axis=7, depth=1, child=64, child_lo=16),
        # ... of an isolated root of an ordinary size (transforms of length 192)
        dict(name="solve-iso96", kind="solve", root=96, periodic=False),
        # ... in FP64, as the accuracy studies run it
        dict(name="solve-fp64-8x128", kind="solve", precision="fp64", root=192, per_axis=2, depth=1, child=128),
        # the spectral gradient: four inverse transforms, then the accelerations, on subgrids of length 120
        dict(name="field-spectral-8x100", kind="field", gradient="spectral", root=160, per_axis=2, depth=1, child=100),
        # accelerations and parent carry of one level of equal subgrids
        dict(name="accel-32x128", kind="accel", root=384, per_axis=4, depth=1, child=128, child_lo=-32),
    ]


def _log_int(rng, lo, hi, even=False):
    v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return v - v % 2 if even else v


def _smooth(n):
    """The smallest {2, 3, 5, 7}-smooth integer at or above n."""
    while True:
        r = n
        for p in (2, 3, 5, 7):
            while r % p == 0:
                r //= p
        if r == 1:
            return n
        n += 1


def draw(rng):
    kind = rng.choice(["step", "step", "deposit", "interp", "solve", "solve", "solve", "field", "accel"])
    c = dict(kind=kind, precision="fp32" if rng.random() < 0.75 else "fp64",
             gradient=rng.choice(["fd2", "fd2", "fd2", "fd4", "spectral"]))
    periodic = rng.random() < 0.6
    if kind == "solve" and rng.random() < 0.4:          # the root level alone
        n = _log_int(rng, 24, 320 if periodic else 112)
        return dict(c, root=_smooth(n), periodic=periodic)
    heavy = c["precision"] == "fp64" or c["gradient"] == "spectral"   # several times the cost of an FP32 cell
    per = rng.choice([1, 1, 2, 2] if heavy else [1, 1, 2, 2, 3, 4])
    child = _log_int(rng, 16, 96 if heavy else 128, even=True)
    room = max(child // 2 + rng.randint(2, 8), 16) * per + 2 * MARGIN
    root = _smooth(room)
    if not periodic:
        root = min(root, 96 if heavy else 192)
        per = max(1, min(per, (root - 2 * MARGIN) // (child // 2 + 2)))
    c.update(root=root, periodic=periodic, per_axis=per, child=child,
             depth=rng.choice([1, 1, 2]) if not heavy and kind not in ("solve", "field", "accel") else 1)
    if kind in ("solve", "field", "accel") and rng.random() < 0.3 and child >= 32:
        c["child_lo"] = child // 4                       # uneven sizes in [child / 4, child]
    if kind in ("step", "deposit", "interp"):
        c["particles"] = _log_int(rng, 2000, 4_000_000)
        c["dist"] = rng.choice(["uniform", "uniform", "lattice", "plummer"])
        c["order"] = rng.random() < 0.4
        c["tiles"] = c["order"] and rng.random() < 0.5
        c["gas"] = rng.random() < 0.4 and kind != "interp"
        c["graph"] = kind == "step" and rng.random() < 0.5
    return c


# ---------------------------------------------------------------- hierarchy
def _grids(c, seed):
    """(level, parent, start, dims) of every grid: subgrids in per_axis^3 slots
    of the root, and below each a chain of equal, centred ones."""
    rng = np.random.default_rng([seed, 1])
    sizes = np.random.default_rng([c["root"], c["child"]])   # the sizes are the case's, the places the seed's
    out = [(0, -1, (0, 0, 0), (c["root"],) * 3)]
    per = c["per_axis"]
    if not per:
        return out
    usable = c["root"] - 2 * MARGIN
    edge = [MARGIN + usable * k // per for k in range(per + 1)]
    slots = [(i, j, k) for k in range(per) for j in range(per) for i in range(per)]
    if c["child_lo"] < 0:                                # only the first -child_lo slots
        slots = slots[:-c["child_lo"]]
    level = []
    for slot in slots:
        start, dims = [], []
        for s in slot:
            d = c["child"]
            if c["child_lo"] > 0:
                d = int(round(math.exp(sizes.uniform(math.log(c["child_lo"]), math.log(c["child"])))))
            span = (d + 1) // 2
            free = edge[s + 1] - edge[s] - span
            start.append(2 * (edge[s] + (free // 2 if per == 1 else int(rng.integers(0, free + 1)))))
            dims.append(d)
        level.append(len(out))
        out.append((1, 0, tuple(start), tuple(dims)))
    for lev in range(2, c["depth"] + 1):
        below = []
        for gi in level:
            _, _, s, d = out[gi]
            below.append(len(out))
            out.append((lev, gi, tuple(2 * (s[j] + (d[j] - (d[j] + 1) // 2) // 2) for j in range(3)), d))
        level = below
    return out


def _plan(c, g):
    """Sizes of one grid: mass-field box, transform lengths, window, its first cell, cell size."""
    lev, _, start, dims = g
    h = 3 if c["gradient"] == "fd4" else 2
    p = dict(h=h, W=[n + 2 * h for n in dims], E=[n + 2 for n in dims], delta=1.0 / (c["root"] * 2 ** lev),
             comps=4 if c["gradient"] == "spectral" else 1)
    if lev:
        p.update(G=[n + 2 * BORDER for n in dims], M=[_smooth(n + 4 * BORDER) for n in dims],
                 lo=[s - BORDER for s in start], s0=BORDER - h, kind="refined")
        return p
    M = list(dims)
    if not c["periodic"]:
        M = [2 * n for n in dims]
        if c["gradient"] == "fd4":
            M = [_smooth(2 * n + 2) for n in dims]
            while M[0] % 2:
                M = [_smooth(m + 1) for m in M]
    p.update(G=list(dims), M=M, lo=[0, 0, 0], s0=-h, kind="periodic" if c["periodic"] else "isolated")
    return p


def _shapes(c, g):
    p = _plan(c, g)
    W = tuple(p["W"][::-1])
    return dict(gmf=tuple(p["G"][::-1]), phis=(p["comps"],) + W if p["comps"] > 1 else W, phi=tuple(p["E"][::-1]),
                acc=(3,) + tuple(p["E"][::-1]))


def _level_buffers(c, grids, lev, key, dtype):
    """One allocation per level and field, and every grid's array as a view of it
    (each starting on a 512-byte boundary)."""
    shapes = [_shapes(c, g)[key] for g in grids if g[0] == lev]
    offs, n = [], 0
    for s in shapes:
        offs.append(n)
        n += (math.prod(s) + 127) // 128 * 128
    flat = torch.zeros(n, dtype=dtype, device=DEV)
    return flat, [flat[o:o + math.prod(s)].view(s) for o, s in zip(offs, shapes)]


# ------------------------------------------------------------------- inputs
def _gen(seed, what):
    return torch.Generator(device=DEV).manual_seed(1000003 * seed + what)


def _randn(shape, seed, what):
    return torch.randn(shape, dtype=torch.float64, device=DEV, generator=_gen(seed, what))


def _zeldovich(n_side, seed):
    """Positions and displacements of an n_side^3 lattice displaced by a P(k) ~ k^-2 field."""
    k1 = torch.fft.fftfreq(n_side, d=1.0 / n_side, dtype=torch.float64, device=DEV)
    kr = torch.fft.rfftfreq(n_side, d=1.0 / n_side, dtype=torch.float64, device=DEV)
    k2 = k1.view(-1, 1, 1) ** 2 + k1.view(1, -1, 1) ** 2 + kr.view(1, 1, -1) ** 2
    k2[0, 0, 0] = 1.0
    dk = torch.complex(_randn(tuple(k2.shape), seed, 11), _randn(tuple(k2.shape), seed, 12)) / k2.sqrt() / k2
    dk[0, 0, 0] = 0
    disp = torch.stack([torch.fft.irfftn(1j * k * dk, s=(n_side,) * 3).reshape(-1)
                        for k in (kr.view(1, 1, -1), k1.view(1, -1, 1), k1.view(-1, 1, 1))])
    disp *= 0.5 / n_side / disp.square().sum(0).mean().sqrt()
    q = (torch.arange(n_side, dtype=torch.float64, device=DEV) + 0.5) / n_side
    pos = torch.stack([q.view(1, 1, -1).expand((n_side,) * 3).reshape(-1), q.view(1, -1, 1).expand((n_side,) * 3).reshape(-1),
                       q.view(-1, 1, 1).expand((n_side,) * 3).reshape(-1)])
    return (pos + disp) % 1.0, disp


def _particles(c, seed):
    n = c["particles"]
    if c["dist"] == "lattice":
        side = max(4, round(n ** (1 / 3)))
        pos, disp = _zeldovich(side, seed)
        vel = 10.0 * disp
        n = side ** 3
    else:
        u = torch.rand((3, n), dtype=torch.float64, device=DEV, generator=_gen(seed, 21))
        vel = 0.1 * _randn((3, n), seed, 22)
        pos = 0.002 + 0.996 * u
        if c["dist"] == "plummer":
            r = (4.0 / c["root"]) / (u[0].clamp(1e-12, 1 - 1e-12) ** (-2.0 / 3.0) - 1.0).sqrt()
            d = _randn((3, n), seed, 23)
            pos = 0.5 + r * d / d.square().sum(0).sqrt()
            pos = pos % 1.0
            pos = pos.clamp(0.002, 0.998)
    m = torch.full((n,), 1.0 / n, dtype=torch.float64, device=DEV)
    return {k: t.contiguous() for k, t in zip(PARTICLE_KEYS, [*pos, *vel, m])}


def _gas(c, grids, seed):
    """Lognormal densities of mean 1 over every grid's interior."""
    return [torch.exp(_randn(tuple(g[3][::-1]), seed, 100 + i) - 0.5) for i, g in enumerate(grids)]


HALF_DT = 5e-4


def _case(case):
    c = dict(DEFAULTS)
    c.update(case)
    return c


def _top(grids):
    return max(g[0] for g in grids)


def _gmf_inputs(c, grids, lev, seed):
    """Lognormal cell masses in fixed point, as a deposit of gas and particles leaves them."""
    flat, views = _level_buffers(c, grids, lev, "gmf", torch.int64)
    d3 = (1.0 / (c["root"] * 2 ** lev)) ** 3
    for i, v in enumerate(views):
        v.copy_((torch.exp(_randn(tuple(v.shape), seed, 500 + i) - 0.5) * (d3 * 2.0 ** FRAC)).round().to(torch.int64))
    return views


def _field_inputs(c, grids, lev, key, dtype, seed):
    """Potential-like or acceleration-like fields of a level."""
    flat, views = _level_buffers(c, grids, lev, key, dtype)
    what = {"phis": 700, "phi": 3000, "acc": 5000}[key]
    for i, v in enumerate(views):
        v.copy_(_randn(tuple(v.shape), seed, what + i) - (3.0 if key != "acc" else 0.0))
    return views


def prepare(case, seed):
    c = _case(case)
    grids = _grids(c, seed)
    solver = Solver(grids, periodic=c["periodic"], precision=c["precision"], mass_frac_bits=FRAC, gradient=c["gradient"])
    st = dict(c=c, solver=solver)
    dt = solver.dtype
    nlev = _top(grids) + 1
    if c["kind"] in ("step", "deposit", "interp"):
        st["P"] = Particles(_particles(c, seed))
        st["gas"] = _gas(c, grids, seed) if c["gas"] else None
        if c["order"]:
            solver.reserve_order(st["P"].n)
            solver.set_deposit_tiles(c["tiles"])
    if c["kind"] == "step":
        flat = {(k, l): _level_buffers(c, grids, l, k, torch.int64 if k == "gmf" else dt)
                for k in ("gmf", "phis", "phi", "acc") for l in range(nlev)}
        st["bufs"] = [{k: flat[k, l][1] for k in ("gmf", "phis", "phi", "acc")} for l in range(nlev)]
        st["pacc"] = torch.zeros((3, st["P"].n), dtype=dt, device=DEV)
        st["out"] = {**{"%s%d" % (k, l): f for (k, l), (f, _) in flat.items()}, "pacc": st["pacc"]}
        if c["graph"]:
            solver.step(st["P"], HALF_DT, st["bufs"], st["pacc"], gas=st["gas"])
            st["graph"] = solver.capture(lambda: solver.step(st["P"], HALF_DT, st["bufs"], st["pacc"], gas=st["gas"]))
    elif c["kind"] == "deposit":
        flat = [_level_buffers(c, grids, l, "gmf", torch.int64) for l in range(nlev)]
        views = [iter(v) for _, v in flat]
        st["gmf"] = [next(views[g[0]]) for g in grids]
        st["out"] = {"gmf%d" % l: flat[l][0] for l in range(nlev)}
    elif c["kind"] == "interp":
        fields = [iter(_field_inputs(c, grids, l, "acc", dt, seed + 31 * l)) for l in range(nlev)]
        st["acc"] = [next(fields[g[0]]) for g in grids]
        st["pacc"] = torch.zeros((3, st["P"].n), dtype=dt, device=DEV)
        st["out"] = {"pacc": st["pacc"], **{k: st["P"].t[k] for k in ("x", "y", "z", "vx", "vy", "vz")}}
    else:
        lev = nlev - 1
        st["lev"], st["out"] = lev, {}
        if c["kind"] in ("solve", "field"):
            st["gmf"] = _gmf_inputs(c, grids, lev, seed)
            st["out"]["phis"], st["phis"] = _level_buffers(c, grids, lev, "phis", dt)
        if c["kind"] in ("field", "accel"):
            if c["kind"] == "accel":
                st["phis"] = _field_inputs(c, grids, lev, "phis", dt, seed)
            st["pphi"] = _field_inputs(c, grids, lev - 1, "phi", dt, seed)
            st["pacc"] = _field_inputs(c, grids, lev - 1, "acc", dt, seed)
            for k in ("phi", "acc"):
                st["out"][k], st[k] = _level_buffers(c, grids, lev, k, dt)
    return st


def run(st):
    c, s = st["c"], st["solver"]
    kind = c["kind"]
    if kind == "step":
        if "graph" in st:
            st["graph"].replay()
        else:
            s.step(st["P"], HALF_DT, st["bufs"], st["pacc"], gas=st["gas"])
    elif kind == "deposit":
        if c["order"]:
            s.order_particles(st["P"], HALF_DT)
        s.deposit_all(st["P"], HALF_DT, st["gmf"], st["gas"])
    elif kind == "interp":
        if c["order"]:
            s.order_particles(st["P"], HALF_DT)
        s.interp_all(st["acc"], st["P"], HALF_DT, st["pacc"])
        s.kick_drift(st["P"], st["pacc"], KICK_DT)
    else:
        if kind != "accel":
            s.solve_level(st["lev"], st["gmf"], st["phis"])
        if kind != "solve":
            s.accel(st["lev"], st["phis"], st["phi"], st["acc"], st["pphi"], st["pacc"])
    return st["out"]


# a timestep far below the crossing time of a cell: repeated passes leave the particles where they are
KICK_DT = 1e-9


# --------------------------------------------------------------------- work
def work(case):
    c = _case(case)
    grids = _grids(c, 0)
    r = 8 if c["precision"] == "fp64" else 4
    top = _top(grids)
    b = f = 0.0
    kind = c["kind"]
    n = c["particles"]
    if c["dist"] == "lattice":
        n = max(4, round(n ** (1 / 3))) ** 3
    if kind in ("step", "deposit"):
        b += 56.0 * n
        f += 27.0 * 4 * n
    if kind in ("step", "interp"):
        b += 3.0 * r * n
        f += 27.0 * 6 * n
    if kind == "interp":                       # six arrays read and written
        b += 96.0 * n
    for g in grids:
        p = _plan(c, g)
        cells, gm, M = math.prod(g[3]), math.prod(p["G"]), math.prod(p["M"])
        W, E = math.prod(p["W"]) * p["comps"], math.prod(p["E"])
        on = g[0] == top
        if kind in ("step", "deposit"):
            b += 8.0 * gm + (8.0 * cells if c["gas"] else 0.0)
        if kind == "interp":
            b += 3.0 * r * E if g[0] == 0 else 0.0
        if kind in ("solve", "field") and on:
            b += 8.0 * gm
        if kind == "step" or (kind in ("solve", "field") and on):
            b += r * W
            f += 2.5 * M * math.log2(M) * (1 + p["comps"])
        if kind == "accel" and on:
            b += r * W
        if kind == "step" or (kind in ("field", "accel") and on):
            b += 4.0 * r * E
            f += 40.0 * E
            if kind != "step" and g[1] >= 0:   # the parent cells under the subgrid
                b += 4.0 * r * math.prod(v // 2 + 2 for v in g[3])
    return {"bytes": b, "flops": f}


# -------------------------------------------------------------------- exact
def _shat(e):
    """S-hat(eta) = 12 / eta^4 (2 - 2 cos eta - eta sin eta), its Taylor series below 1."""
    s = torch.zeros_like(e)
    e2 = e.clamp(max=1.0) ** 2
    for m in range(13, 1, -1):
        s = s * e2 + (-1) ** m * (2 * m - 2) / math.factorial(2 * m)
    big = e.clamp(min=1.0)
    return torch.where(e < 1.0, 12.0 * s, 12.0 / big ** 4 * (2.0 - 2.0 * torch.cos(big) - big * torch.sin(big)))


def _optimal(M, delta, a, a_par, gradient, H):
    """The optimal influence function over the octant H = M // 2 + 1 (z, y, x), 0 where the gradient vanishes."""
    f, k, D, al = [], [], [], []
    for j in range(3):
        shape = [1, 1, 1]
        shape[2 - j] = H[j]
        kap = torch.arange(H[j], dtype=torch.float64, device=DEV).view(shape)
        fj = kap / M[j]
        kj = 2 * math.pi * fj / delta
        s2 = torch.sin(math.pi * fj) ** 2
        if gradient == "spectral":
            d = torch.where(2 * kap == M[j], torch.zeros_like(kj), kj)
        else:
            d = torch.sin(2 * math.pi * fj)
            d = torch.where((kap == 0) | (2 * kap == M[j]), torch.zeros_like(d), d)
            d = d * (4 - torch.cos(2 * math.pi * fj)) / 3 / delta if gradient == "fd4" else d / delta
        f.append(fj)
        k.append(kj)
        D.append(d)
        al.append(1 - s2 + 2.0 / 15.0 * s2 * s2)
    num = 0.0
    for n2 in (-1, 0, 1):
        for n1 in (-1, 0, 1):
            for n0 in (-1, 0, 1):
                q = [k[j] + 2 * math.pi * n / delta for j, n in enumerate((n0, n1, n2))]
                u = [torch.sinc(f[j] + n) ** 6 for j, n in enumerate((n0, n1, n2))]
                qq = q[0] ** 2 + q[1] ** 2 + q[2] ** 2
                qq = torch.where(qq == 0, torch.ones_like(qq), qq)
                r = qq.sqrt()
                F = _shat(r * a / 2) ** 2
                if a_par:
                    F = F - _shat(r * a_par / 2) ** 2
                num = num + u[0] * u[1] * u[2] * (D[0] * q[0] + D[1] * q[1] + D[2] * q[2]) * F / qq
    d2 = D[0] ** 2 + D[1] ** 2 + D[2] ** 2
    # modes with every kappa in {0, M/2} carry nothing
    deg = [torch.isclose(2 * f[j] % 1, torch.zeros_like(f[j])) for j in range(3)]
    dead = deg[0] & deg[1] & deg[2]
    out = -4 * math.pi * num / (torch.where(dead, torch.ones_like(d2), d2) * (al[0] * al[1] * al[2]) ** 2)
    return torch.where(dead, torch.zeros_like(out), out), dead


def _pair(xi):
    """Pair potential of two unit S spheres of diameter a at distance xi a, times a."""
    x = xi.clamp(max=0.5)
    near = (-104 / 35 + 32 / 5 * x ** 2 - 64 / 5 * x ** 4 + 32 / 5 * x ** 5 + 256 / 35 * x ** 6 - 192 / 35 * x ** 7)
    x = xi.clamp(min=0.5, max=1.0)
    mid = (-3 / (35 * x) - 64 / 35 - 32 / 5 * x + 128 / 5 * x ** 2 - 32 * x ** 3 + 64 / 5 * x ** 4 + 32 / 5 * x ** 5
           - 256 / 35 * x ** 6 + 64 / 35 * x ** 7)
    return torch.where(xi <= 0.5, near, torch.where(xi <= 1.0, mid, -1.0 / xi.clamp(min=1.0)))


def _half_table(c, p):
    """The Green's table on the half spectrum (z, y, x <= M0 / 2), in DFT units."""
    M, delta = p["M"], p["delta"]
    H = [m // 2 + 1 for m in M]
    a = A_DX * delta
    a_par = 2 * a if p["kind"] == "refined" else 0.0
    T, dead = _optimal(M, delta, a, a_par, c["gradient"], H)
    vol = delta ** 3
    if p["kind"] == "refined":
        T[0, 0, 0] = -4 * math.pi * (a_par ** 2 - a ** 2) / 30
        T = T / vol
    elif p["kind"] == "periodic":
        T = T / vol
    else:
        kk = 0.0
        r2 = 0.0
        for j in range(3):
            shape = [1, 1, 1]
            shape[2 - j] = H[j]
            kk = kk + (2 * math.pi * torch.arange(H[j], dtype=torch.float64, device=DEV) / (M[j] * delta)).view(shape) ** 2
            shape[2 - j] = M[j]
            i = torch.arange(M[j], device=DEV)
            r2 = r2 + (torch.minimum(i, M[j] - i).to(torch.float64) * delta).view(shape) ** 2
        cont = -4 * math.pi * _shat(kk.sqrt() * a / 2) ** 2 / torch.where(kk == 0, torch.ones_like(kk), kk)
        corr = torch.where(dead, torch.zeros_like(T), (T - cont) / vol)
        T = torch.fft.rfftn(_pair(r2.sqrt() / a) / a).real[:H[2], :H[1]] + corr
    fold = [torch.minimum(torch.arange(m, device=DEV), m - torch.arange(m, device=DEV)) for m in M]
    return T[fold[2]][:, fold[1]]


def _solve_exact(c, p, rho, table):
    """The window of the potential (and of the spectral accelerations) of one grid; rho: cell masses."""
    M = p["M"]
    spec = torch.fft.rfftn(rho, s=M[::-1]) * table
    idx = [(torch.arange(p["W"][j], device=DEV) + p["s0"]) % M[j] for j in range(3)]

    def back(s):
        return torch.fft.irfftn(s, s=M[::-1])[idx[2]][:, idx[1]][:, :, idx[0]]

    out = [back(spec)]
    if p["comps"] > 1:
        for j in range(3):
            i = torch.arange(M[j], dtype=torch.float64, device=DEV)
            k = 2 * math.pi / (M[j] * p["delta"]) * torch.where(2 * i < M[j], i, i - M[j])
            k = torch.where(2 * i == M[j], torch.zeros_like(k), k)
            if j == 0:
                k = k[:M[0] // 2 + 1]
            shape = [1, 1, 1]
            shape[2 - j] = -1
            out.append(back(spec * (-1j * k.view(shape))))
        return torch.stack(out)
    return out[0]


def _carry(g, parent, f):
    """Trilinear interpolation of a parent field (cells [-1, N + 1), last three axes) onto cells [-1, N + 1) of g."""
    for ax, j in ((-3, 2), (-2, 1), (-1, 0)):
        x = (torch.arange(g[3][j] + 2, dtype=torch.float64, device=DEV) + g[2][j] - 0.5) / 2 - 0.5 - parent[2][j] + 1
        k = x.floor().long()
        shape = [1, 1, 1]
        shape[ax] = -1
        w = (x - k).view(shape)
        f = (1 - w) * f.index_select(f.dim() + ax, k) + w * f.index_select(f.dim() + ax, k + 1)
    return f


def _accel_exact(c, p, g, parent, phis, pphi, pacc):
    E, h = p["E"], p["h"]
    first = phis[0] if p["comps"] > 1 else phis

    def at(j, o):
        s = [h - 1, h - 1, h - 1]
        s[j] += o
        return first[s[2]:s[2] + E[2], s[1]:s[1] + E[1], s[0]:s[0] + E[0]]

    phi = at(0, 0)
    if c["gradient"] == "spectral":
        acc = phis[1:, 1:1 + E[2], 1:1 + E[1], 1:1 + E[0]]
    elif c["gradient"] == "fd4":
        acc = torch.stack([-(8 * (at(j, 1) - at(j, -1)) - (at(j, 2) - at(j, -2))) / (12 * p["delta"]) for j in range(3)])
    else:
        acc = torch.stack([-(at(j, 1) - at(j, -1)) / (2 * p["delta"]) for j in range(3)])
    if parent is not None:
        phi = phi + _carry(g, parent, pphi)
        acc = acc + _carry(g, parent, pacc)
    return phi, acc


def _tsc(pos, delta):
    """Cells and the three weights per axis of drifted positions (3, n)."""
    u = pos / delta
    i = u.floor()
    t = u - i
    return i.long(), torch.stack([(1 - t) ** 2 / 2, 0.75 - (t - 0.5) ** 2, t * t / 2], 1)


def _deposit_exact(c, p, g, pos, m):
    G = p["G"]
    out = torch.zeros(math.prod(G), dtype=torch.float64, device=DEV)
    step = 1 << 22
    for o in range(0, pos.shape[1], step):
        i, w = _tsc(pos[:, o:o + step], p["delta"])
        i = i - torch.tensor(p["lo"], device=DEV).view(3, 1)
        mm = m[o:o + step]
        if g[0]:
            near = torch.ones_like(i[0], dtype=torch.bool)
            for j in range(3):
                near &= (i[j] >= -1) & (i[j] <= G[j])
            i, w, mm = i[:, near], w[:, :, near], mm[near]
        for dz in range(3):
            for dy in range(3):
                for dx in range(3):
                    cell, ok = [], torch.ones_like(i[0], dtype=torch.bool)
                    for j, d in enumerate((dx, dy, dz)):
                        v = i[j] + d - 1
                        if g[0]:
                            ok &= (v >= 0) & (v < G[j])
                            v = v.clamp(0, G[j] - 1)
                        elif c["periodic"]:
                            v = v % G[j]
                        else:
                            v = v.clamp(0, G[j] - 1)
                        cell.append(v)
                    q = mm * w[0, dx] * w[1, dy] * w[2, dz] * ok
                    out.index_add_(0, cell[0] + G[0] * (cell[1] + G[1] * cell[2]), q)
    return out.view(tuple(G[::-1]))


def _interp_exact(c, grids, acc, pos):
    n = pos.shape[1]
    out = torch.zeros((3, n), dtype=torch.float64, device=DEV)
    for g, a in zip(grids, acc):                    # coarse to fine: the finest owner writes last
        i, w = _tsc(pos, 1.0 / (c["root"] * 2 ** g[0]))
        i = i - torch.tensor(g[2], device=DEV).view(3, 1)
        inside = torch.ones(n, dtype=torch.bool, device=DEV)
        for j in range(3):
            inside &= (i[j] >= 0) & (i[j] < g[3][j])
        at = inside.nonzero().view(-1)
        i, w = i[:, at], w[:, :, at]
        E = [v + 2 for v in g[3]]
        flat = a.reshape(3, -1)
        got = torch.zeros((3, at.numel()), dtype=torch.float64, device=DEV)
        for dz in range(3):
            for dy in range(3):
                for dx in range(3):
                    cell = []
                    for j, d in enumerate((dx, dy, dz)):
                        v = i[j] + d
                        if g[0] == 0 and not c["periodic"]:
                            v = v.clamp(1, g[3][j])
                        cell.append(v)
                    got += w[0, dx] * w[1, dy] * w[2, dz] * flat[:, cell[0] + E[0] * (cell[1] + E[1] * cell[2])]
        out[:, at] = got
    return out


def _packed(c, grids, lev, key, values):
    flat, views = _level_buffers(c, grids, lev, key, torch.float64)
    for v, x in zip(views, values):
        v.copy_(x)
    return flat


def _gas_exact(c, grids, gi, gas, p):
    """Baryon masses of grid gi's mass-field box: its own gas inside, its parent's on the border."""
    g = grids[gi]
    if not g[0]:
        return gas[0] * p["delta"] ** 3
    par = grids[g[1]]
    idx, ok = [], []
    for j in range(3):
        v = (torch.arange(p["G"][j], device=DEV) + p["lo"][j]) // 2 - par[2][j]
        ok.append((v >= 0) & (v < par[3][j]))
        idx.append(v.clamp(0, par[3][j] - 1))
    rho = gas[g[1]][idx[2]][:, idx[1]][:, :, idx[0]]
    rho = rho * (ok[2].view(-1, 1, 1) & ok[1].view(1, -1, 1) & ok[0].view(1, 1, -1))
    B = BORDER
    rho[B:-B, B:-B, B:-B] = gas[gi]
    return rho * p["delta"] ** 3


def exact(case, seed):
    c = _case(case)
    kind = c["kind"]
    grids = _grids(c, seed)
    dt = torch.float64 if c["precision"] == "fp64" else torch.float32
    top = _top(grids)
    if kind == "deposit":
        return None                                  # whole numbers
    if kind in ("step", "interp"):
        P = _particles(c, seed)
        pos = torch.stack([P[k] + P["v" + k] * HALF_DT for k in "xyz"])
        if c["periodic"]:
            pos = pos % 1.0
    if kind == "interp":
        acc = [iter(_field_inputs(c, grids, l, "acc", dt, seed + 31 * l)) for l in range(top + 1)]
        a = _interp_exact(c, grids, [next(acc[g[0]]).double() for g in grids], pos)
        out = {"pacc": a}
        for j, k in enumerate("xyz"):
            v = P["v" + k] + a[j] * KICK_DT
            out["v" + k] = v
            out[k] = P[k] + (P["v" + k] + v) * 0.5 * KICK_DT
        return out
    tables = {}

    def table(p):
        key = (p["kind"], tuple(p["M"]), p["delta"])
        if key not in tables:
            if len(tables) > 8:
                tables.clear()
            tables[key] = _half_table(c, p)
        return tables[key]

    if kind != "step":
        mine = [g for g in grids if g[0] == top]
        plans = [_plan(c, g) for g in mine]
        out = {}
        if kind == "accel":
            phis = [v.double() for v in _field_inputs(c, grids, top, "phis", dt, seed)]
        else:
            gmf = _gmf_inputs(c, grids, top, seed)
            phis = [_solve_exact(c, p, m.double() * 2.0 ** -FRAC, table(p)) for p, m in zip(plans, gmf)]
            out["phis"] = _packed(c, grids, top, "phis", phis)
        if kind != "solve":
            pphi = _field_inputs(c, grids, top - 1, "phi", dt, seed)
            pacc = _field_inputs(c, grids, top - 1, "acc", dt, seed)
            first = [i for i, g in enumerate(grids) if g[0] == top - 1]
            got = [_accel_exact(c, p, g, grids[g[1]], f, pphi[first.index(g[1])].double(), pacc[first.index(g[1])].double())
                   for p, g, f in zip(plans, mine, phis)]
            out["phi"] = _packed(c, grids, top, "phi", [a for a, _ in got])
            out["acc"] = _packed(c, grids, top, "acc", [b for _, b in got])
        return out
    gas = _gas(c, grids, seed) if c["gas"] else None
    phis, phi, acc = [], [], []
    for gi, g in enumerate(grids):
        p = _plan(c, g)
        rho = _deposit_exact(c, p, g, pos, P["m"])
        if gas:
            rho = rho + _gas_exact(c, grids, gi, gas, p)
        phis.append(_solve_exact(c, p, rho, table(p)))
        par = g[1]
        a, b = _accel_exact(c, p, g, grids[par] if par >= 0 else None, phis[gi], phi[par] if par >= 0 else None,
                            acc[par] if par >= 0 else None)
        phi.append(a)
        acc.append(b)
    out = {}
    for l in range(top + 1):
        at = [i for i, g in enumerate(grids) if g[0] == l]
        out["gmf%d" % l] = None
        for key, v in (("phis", phis), ("phi", phi), ("acc", acc)):
            out["%s%d" % (key, l)] = _packed(c, grids, l, key, [v[i] for i in at])
    out["pacc"] = _interp_exact(c, grids, acc, pos)
    return out
