"""Masses of a few fixed-point units: every one of the 26 outer charges is rounded
half up, so on cell corners, edges and faces they may sum to more than the mass,
and the centre cell's charge is then negative.  Bit-exact against the oracle for
M = 1 .. 64 and around 2^9 and 2^32 (where the charges' width changes), alone and
beside heavier and negative masses, on the root and a refined level, in the
caller's and in bin order."""
import numpy as np
import pytest

import oracle
from apm_inputs import GridDesc

pytestmark = pytest.mark.gpu

GRIDS = [GridDesc(0, -1, (0, 0, 0), (16, 16, 16)), GridDesc(1, 0, (8, 10, 8), (14, 12, 16))]


def _run(units, pos, frac, periodic):
    import torch

    from paper_1410_0010_gb300.solver import Particles, Solver
    n = len(units)
    parts = dict(x=pos[0], y=pos[1], z=pos[2], vx=np.zeros(n), vy=np.zeros(n), vz=np.zeros(n), m=units * 2.0 ** -frac)
    cfg = oracle.Config(periodic=periodic, mass_frac_bits=frac)
    og = [oracle.Grid(*g) for g in GRIDS]
    want = [oracle.deposit(cfg, og, gi, parts, 0.0)[0] for gi in range(len(GRIDS))]
    assert int(want[0].sum()) == int(units.sum())   # no cloud reaches an isolated face here
    s = Solver(GRIDS, periodic=periodic, mass_frac_bits=frac, device=0)
    P = Particles({k: torch.tensor(a, dtype=torch.float64, device="cuda") for k, a in parts.items()})
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


def _points(n, rng):
    """n positions in the refined grid and around it: on corners, edges and faces
    of its cells (and of the root's), and between them."""
    pos = 0.25 + 0.5 * rng.random((3, n))
    on = np.arange(n) % 8                       # bit j: axis j on a cell face
    for j in range(3):
        f = (on >> j) & 1 == 1
        pos[j, f] = np.floor(pos[j, f] * 32) / 32
    return pos


@pytest.mark.parametrize("periodic", [False, True])
@pytest.mark.parametrize("company", ["light", "heavy"])
@pytest.mark.parametrize("frac", [52, 8])
@pytest.mark.parametrize("times", [32, 256])   # 2304 and 18432 particles: straight and in rows
def test_small_masses_bit_exact(times, frac, company, periodic):
    rng = np.random.default_rng(frac + periodic)
    edges = [255, 256, 511, 512, 513, 2 ** 32 - 1, 2 ** 32, 2 ** 32 + 1]
    units = np.repeat(np.concatenate([np.arange(1, 65), edges]), times)
    pos = _points(len(units), rng)
    order = np.arange(len(units))               # whole warps of one mass
    if company == "heavy":                      # each warp a mixture, with wide and negative masses
        order = rng.permutation(len(units))
        units[order[::32]] = 2 ** 40 + 12345
        units[order[7::64]] *= -1
    _run(units[order].astype(np.int64), pos[:, order], frac, periodic)


@pytest.mark.parametrize("units", [1, 6, 25, 41])
def test_one_small_mass_on_a_corner(units):
    _run(np.array([units], dtype=np.int64), np.array([[0.5], [0.5], [0.5]]), 52, True)
