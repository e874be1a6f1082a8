"""The deposit sends each cloud row by row from shared memory, a warp at a time,
with 32- or 64-bit charges: bit-exact against the oracle at the sizes and masses
where that can go wrong -- ragged last warps, warps that mix narrow and wide,
zero and negative masses, particles outside an isolated box, on its faces and
in several overlapping borders of one level -- in the caller's and in bin order,
for every level at once and level by level."""
import numpy as np
import pytest

import oracle
from apm_inputs import GridDesc

pytestmark = pytest.mark.gpu

# two level-1 grids 4 cells apart (their borders overlap) and a level-2 grid
GRIDS = [GridDesc(0, -1, (0, 0, 0), (24, 24, 24)), GridDesc(1, 0, (8, 10, 8), (12, 15, 12)),
         GridDesc(1, 0, (24, 10, 8), (13, 14, 16)), GridDesc(2, 1, (22, 26, 22), (10, 11, 12))]


@pytest.mark.parametrize("periodic", [False, True])
@pytest.mark.parametrize("n", [1, 31, 33, 129, 3000])
def test_rows_bit_exact(n, periodic):
    import torch

    from paper_1410_0010_gb300.solver import Particles, Solver
    rng = np.random.default_rng(n)
    pos = rng.random((3, n))
    pos[:, : n // 3] = 0.25 + 0.35 * rng.random((3, n // 3))      # in the refined grids and their borders
    if n > 40:
        pos[0, 5:9] = [0.0, 1.0 - 2.0 ** -40, 0.5, 11.5 / 24]     # faces and cell edges
        if not periodic:
            pos[1, 9:12] = [-0.3, 1.2, 7.0]                       # outside: folded, flagged
    m = np.where(rng.random(n) < 0.5, 2.0 ** -24, 1.0 / 3.0) * rng.random(n)
    m[rng.random(n) < 0.1] = 0.0
    m[rng.random(n) < 0.1] *= -1.0
    v = 0.02 * rng.normal(size=(3, n))
    parts = dict(x=pos[0], y=pos[1], z=pos[2], vx=v[0], vy=v[1], vz=v[2], m=m)
    cfg = oracle.Config(periodic=periodic)
    og = [oracle.Grid(*g) for g in GRIDS]
    want = [oracle.deposit(cfg, og, gi, parts, 1e-3)[0] for gi in range(len(GRIDS))]

    s = Solver(GRIDS, periodic=periodic, device=0)
    P = Particles({k: torch.tensor(a, dtype=torch.float64, device="cuda") for k, a in parts.items()})
    s.reserve_order(n)
    s.set_deposit_tiles(True)
    for ordered in (False, True):
        if ordered:
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
            got = s._per_grid(bufs, "gmf")
            for gi in range(len(GRIDS)):
                assert np.array_equal(got[gi].cpu().numpy(), want[gi]), (ordered, whole, gi)
    s.close()
