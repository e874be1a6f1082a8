"""The two-point and spectral acceleration kernels march each thread through a
column of blocks where a level is large enough: every cell of levels that march
1, 2 and 8 blocks, with ragged last segments and odd sizes and starts, against
the difference (the window's components) and the trilinear carry in plain FP64
torch (FP64 1e-12, FP32 2e-5 / 1e-4, the suite's tolerances)."""
import itertools

import pytest

from apm_inputs import GridDesc
from gpu_helpers import TOL

pytestmark = pytest.mark.gpu


def _carry(f, start, dims, pstart):
    import torch
    for ax, j in ((-3, 2), (-2, 1), (-1, 0)):
        x = (torch.arange(dims[j] + 2, dtype=torch.float64, device="cuda") + start[j] - 0.5) / 2 + 0.5 - pstart[j]
        k = x.floor().long()
        shape = [1, 1, 1]
        shape[ax] = -1
        w = (x - k).view(shape)
        f = (1 - w) * f.index_select(f.dim() + ax, k) + w * f.index_select(f.dim() + ax, k + 1)
    return f


@pytest.mark.parametrize("gradient", ["fd2", "spectral"])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("per_axis,dims", [(1, (40, 33, 47)), (2, (52, 53, 50)), (3, (50, 45, 59)), (4, (52, 57, 60))])
def test_march_matches_plain_formula(per_axis, dims, precision, gradient):
    import torch

    from paper_1410_0010_gb300.solver import Solver
    step = 36
    root = step * per_axis + 8
    while not _smooth(root):
        root += 1
    grids = [GridDesc(0, -1, (0, 0, 0), (root,) * 3)]
    for i, o in enumerate(itertools.product(range(per_axis), repeat=3)):
        grids.append(GridDesc(1, 0, tuple(2 * (4 + step * v) + i % 2 for v in o), dims))
    s = Solver(grids, periodic=True, precision=precision, device=0, gradient=gradient)
    gen = torch.Generator(device="cuda").manual_seed(3)

    def field(shape):
        return torch.randn(shape, generator=gen, device="cuda", dtype=torch.float64).to(s.dtype)
    b = s.alloc_level(1)
    for t in b["phis"]:
        t.copy_(field(t.shape))
    E0 = (root + 2,) * 3
    pphi, pacc = field(E0), field((3,) + E0)
    for t in b["phi"] + b["acc"]:
        t.fill_(float("nan"))
    s.accel(1, b["phis"], b["phi"], b["acc"], [pphi], [pacc])
    d = s.info[1]["delta"]
    e = [n + 2 for n in dims]
    for g, phis, phi, acc in zip(grids[1:], b["phis"], b["phi"], b["acc"]):
        p = phis.double()
        comps = p[1:] if gradient == "spectral" else None
        p = p[0] if gradient == "spectral" else p

        def at(j, o):
            c = [1, 1, 1]
            c[j] += o
            return p[c[2]:c[2] + e[2], c[1]:c[1] + e[1], c[0]:c[0] + e[0]]
        if gradient == "spectral":
            want = comps[:, 1:1 + e[2], 1:1 + e[1], 1:1 + e[0]]
        else:
            want = torch.stack([-(at(j, 1) - at(j, -1)) / (2 * d) for j in range(3)])
        want = want + _carry(pacc.double(), g.start, dims, (0, 0, 0))
        wphi = at(0, 0) + _carry(pphi.double(), g.start, dims, (0, 0, 0))
        assert ((acc.double() - want).norm() / want.norm()).item() <= TOL[precision]["acc"]
        assert ((phi.double() - wphi).norm() / wphi.norm()).item() <= TOL[precision]["phi"]
    s.close()


def _smooth(n):
    for p in (2, 3, 5, 7):
        while n % p == 0:
            n //= p
    return n == 1
