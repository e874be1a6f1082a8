"""Baryons of every size on cells of a power-of-two width (integer conversion from
2^50 units up, FP64 products beyond 2^62) and of another width: bit-exact against
the oracle."""
import numpy as np
import pytest

import oracle
from apm_inputs import GridDesc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [16, 18])
def test_gas_bit_exact_over_the_range(n):
    import torch

    from paper_1410_0010_gb300.solver import Particles, Solver
    grids = [GridDesc(0, -1, (0, 0, 0), (n, n, n)), GridDesc(1, 0, (8, 10, 8), (14, 12, 16))]
    rng = np.random.default_rng(n)
    gas = []
    for lev, _, _, d in grids:
        cell = (n * 2.0 ** lev) ** 3           # density of a unit mass in a cell
        q = np.exp2(rng.uniform(-60.0, 10.9, size=d[::-1]))
        q.flat[:12] = np.exp2([-3.0, -2.0, -1.0, 0.0, 9.0, 9.9, -52.0, -53.0, -54.0, -1074.0, -2.0, -1.5])
        q.flat[10] *= 1 + 2.0 ** -51            # around 2^50 units, odd significands
        gas.append(q * rng.choice([-1.0, 1.0], size=q.shape) * cell)
    none = {k: np.zeros(0) for k in ("x", "y", "z", "vx", "vy", "vz", "m")}
    cfg = oracle.Config(periodic=True)
    og = [oracle.Grid(*g) for g in grids]
    s = Solver(grids, periodic=True, device=0)
    bufs = s.alloc_all()
    tp = {k: torch.zeros(1, dtype=torch.float64, device="cuda") for k in none}   # one particle without mass
    tp["x"] += 0.5
    s.deposit_all(Particles(tp), 0.0, s._per_grid(bufs, "gmf"), gas=[torch.tensor(g, device="cuda") for g in gas])
    for gi, got in enumerate(s._per_grid(bufs, "gmf")):
        want = oracle.deposit(cfg, og, gi, none, 0.0, gas=gas[gi], parent_gas=gas[0] if gi else None)[0]
        assert np.array_equal(got.cpu().numpy(), want), gi
    s.close()

