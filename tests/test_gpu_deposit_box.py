"""In bin order a CTA whose particles lie close together gathers their charges in a
box in shared memory: bit-exact against the oracle for clusters on the corner of a
periodic box (the clouds wrap) and of an isolated one (they fold, some particles
outside), inside a refined grid, across its outer border (cells drop) and in the
overlapping borders of two grids, with 32- and 64-bit charges, masses of zero,
negative ones and ones of a few units, for every level at once and one by one."""
import numpy as np
import pytest

import oracle
from apm_inputs import GridDesc

pytestmark = pytest.mark.gpu

GRIDS = [GridDesc(0, -1, (0, 0, 0), (24, 24, 24)), GridDesc(1, 0, (8, 10, 8), (12, 15, 12)),
         GridDesc(1, 0, (24, 10, 8), (13, 14, 16)), GridDesc(2, 1, (22, 26, 22), (10, 11, 12))]
# corner of the box, inside level 2, outer border of level 1, between the level-1 grids
CENTRES = [(0.0, 0.0, 0.0), (0.28, 0.33, 0.29), (0.07, 0.2, 0.2), (0.46, 0.35, 0.3)]


@pytest.mark.parametrize("periodic", [False, True])
@pytest.mark.parametrize("masses", ["narrow", "wide", "mixed"])
@pytest.mark.parametrize("n", [1, 40, 129, 3000])
def test_clusters_bit_exact(n, masses, periodic):
    import torch

    from paper_1410_0010_gb300.solver import Particles, Solver
    rng = np.random.default_rng(n)
    pos = np.array(CENTRES)[np.arange(n) * len(CENTRES) // n].T + rng.normal(scale=0.4 / 24, size=(3, n))
    if periodic:
        pos = pos % 1.0
    m = (1 + rng.random(n)) * 2.0 ** (-24 if masses == "narrow" else -4)
    if masses == "mixed":
        m = np.where(rng.random(n) < 0.5, m, rng.integers(0, 50, size=n) * 2.0 ** -52)
        m[rng.random(n) < 0.2] *= -1.0
    m[rng.random(n) < 0.05] = 0.0
    v = 0.02 * rng.normal(size=(3, n))
    parts = dict(x=pos[0], y=pos[1], z=pos[2], vx=v[0], vy=v[1], vz=v[2], m=m)
    cfg = oracle.Config(periodic=periodic)
    og = [oracle.Grid(*g) for g in GRIDS]
    want = [oracle.deposit(cfg, og, gi, parts, 1e-3) for gi in range(len(GRIDS))]

    s = Solver(GRIDS, periodic=periodic, device=0)
    P = Particles({k: torch.tensor(np.ascontiguousarray(a), device="cuda") for k, a in parts.items()})
    s.reserve_order(n)
    s.set_deposit_tiles(True)
    s.order_particles(P, 1e-3)
    for whole in (True, False):
        bufs = s.alloc_all()
        for b in bufs:
            for t in b["gmf"]:
                t.fill_(-1)
        if whole:
            s.deposit_all(P, 1e-3, s._per_grid(bufs, "gmf"))
        else:
            for lev in range(s.n_levels):
                s.deposit(lev, P, 1e-3, bufs[lev]["gmf"])
        for gi, got in enumerate(s._per_grid(bufs, "gmf")):
            assert np.array_equal(got.cpu().numpy(), want[gi][0]), (whole, gi)
    s.close()
