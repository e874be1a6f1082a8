"""The deposit's arrangements by the number of particles: straight up to 16384 (65536
where grids' borders overlap), in rows above, the candidate grids after the first
straight, and with two or more particles to a root cell every fourth one of a warp's
32 to an instruction (any order gives the same field).  Bit-exact against the oracle on
both sides of each line, for particles stored in x order, of 32- and 64-bit charges,
some of zero mass, with a ragged last warp, on the root, a refined level and in the
overlapping borders of two and of four grids, in the caller's order and the bins'."""
import numpy as np
import pytest

import oracle
from apm_inputs import GridDesc

pytestmark = pytest.mark.gpu

OVERLAP = [GridDesc(0, -1, (0, 0, 0), (24, 24, 24)), GridDesc(1, 0, (12, 12, 12), (12, 12, 12)),
           GridDesc(1, 0, (24, 12, 12), (8, 12, 13)), GridDesc(1, 0, (12, 24, 12), (12, 9, 12)),
           GridDesc(1, 0, (24, 24, 14), (9, 10, 8))]
ONE = OVERLAP[:2]


@pytest.mark.parametrize("periodic", [False, True])
@pytest.mark.parametrize("masses", ["narrow", "wide", "mixed"])
@pytest.mark.parametrize("GRIDS,n", [(g, n) for g in (ONE, OVERLAP) for n in
                                     (1, 33, 16384, 16385, 27647, 27648)] + [(OVERLAP, 65536), (OVERLAP, 65537)])
def test_arrangements_bit_exact(GRIDS, n, masses, periodic):   # 2 * 24^3 = 27648
    import torch

    from paper_1410_0010_gb300.solver import Particles, Solver
    rng = np.random.default_rng(n)
    x = (np.arange(n) + rng.random(n)) / 96 % 1.0       # rows along x, four to a cell
    row = np.arange(n) // 96
    pos = np.array([x, (row * 0.618 + 0.3) % 1.0, (row * 0.381 + 0.25) % 1.0])
    m = (1 + rng.random(n)) * 2.0 ** (-24 if masses == "narrow" else -6)
    if masses == "mixed":
        m = np.where(rng.random(n) < 0.9, m * 2.0 ** -20, -m)
        m[rng.random(n) < 0.05] = 3 * 2.0 ** -52
    m[rng.random(n) < 0.03] = 0.0
    zero = np.zeros(n)
    parts = dict(x=pos[0], y=pos[1], z=pos[2], vx=zero, vy=zero, vz=zero, m=m)
    cfg = oracle.Config(periodic=periodic)
    og = [oracle.Grid(*g) for g in GRIDS]
    want = [oracle.deposit(cfg, og, gi, parts, 0.0)[0] for gi in range(len(GRIDS))]
    s = Solver(GRIDS, periodic=periodic, device=0)
    P = Particles({k: torch.tensor(np.ascontiguousarray(a), device="cuda") for k, a in parts.items()})
    s.reserve_order(n)
    s.set_deposit_tiles(True)
    for ordered in (False, True):
        if ordered:
            s.order_particles(P, 0.0)
        for whole in (True, False):
            bufs = s.alloc_all()
            if whole:
                s.deposit_all(P, 0.0, s._per_grid(bufs, "gmf"))
            else:
                for lev in range(s.n_levels):
                    s.deposit(lev, P, 0.0, bufs[lev]["gmf"])
            for gi, got in enumerate(s._per_grid(bufs, "gmf")):
                assert np.array_equal(got.cpu().numpy(), want[gi]), (ordered, whole, gi)
    s.close()
