"""The compile-time FFT plans of the lengths from 70 to 250, in both precisions,
and the fused planes that plan 0 runs for M0 = M1 from 70 to 192, against the
runtime-planned kernels: FP64 within the suite's 1e-12 (both sides round each
butterfly once; a few 1e-16 apart), FP32 within its 2e-5 of FP64."""
import itertools

import pytest

from apm_inputs import GridDesc

pytestmark = pytest.mark.gpu

# one grid of dims M - 20 per slot of a 512^3 level (transform lengths M)
MIXED = [(70, 72, 75), (80, 81, 84), (90, 96, 98), (100, 105, 108), (112, 120, 125), (126, 128, 135),
         (140, 144, 147), (160, 168, 250)]
MORE = [(180, 75, 192), (200, 84, 216), (224, 70, 240), (240, 98, 180), (75, 200, 90), (98, 224, 72),
        (81, 250, 168), (250, 160, 81)]
PLANES = [(70, 70, 36), (192, 192, 40), (200, 200, 36), (147, 147, 42), (125, 125, 45), (84, 84, 48), (160, 160, 36),
          (108, 108, 50)]


def _solver(lengths, precision):
    from paper_1410_0010_gb300.solver import Solver
    grids = [GridDesc(0, -1, (0, 0, 0), (256, 256, 256))]
    for m, slot in zip(lengths, itertools.product((6, 258), repeat=3)):
        grids.append(GridDesc(1, 0, slot, tuple(v - 20 for v in m)))
    s = Solver(grids, periodic=True, precision=precision, device=0)
    assert [tuple(s.info[i]["fft"]) for i in s.level_grids[1]] == list(lengths)
    return s


def _solve(s, plan):
    import torch
    bufs = s.alloc_level(1)
    gen = torch.Generator(device="cuda").manual_seed(7)
    for g in bufs["gmf"]:
        g.copy_((torch.randn(g.shape, generator=gen, device="cuda", dtype=torch.float64).exp() * 2.0 ** 40).long())
    sh = s.fft_shapes(1)
    sh["plan"] = [plan] * 5
    s.set_fft_shapes(1, sh)
    for t in bufs["phis"]:
        t.fill_(float("nan"))
    s.solve_level(1, bufs["gmf"], bufs["phis"])
    s.sync_status()
    return [t.double() for t in bufs["phis"]], s.pass_kernels(1)


@pytest.mark.parametrize("lengths", [MIXED, MORE, PLANES], ids=["mixed", "more", "planes"])
def test_compile_time_plans_match_runtime_plans(lengths):
    out = {}
    for precision in ("fp64", "fp32"):
        s = _solver(lengths, precision)
        out[precision, 1], kinds = _solve(s, 1)
        assert all(k == 0 for row in kinds for k in row)
        out[precision, 0], kinds = _solve(s, 0)
        s.close()
        for g, m in enumerate(lengths):
            fused = precision == "fp32" and m[0] == m[1] and 70 <= m[0] <= 192
            fast = [int(v >= 70 or precision == "fp32") for v in m]
            assert [row[g] for row in kinds] == ([2, 3, fast[2], 3, 2] if fused else
                                                 [fast[0], fast[1], fast[2], fast[1], fast[0]])
    for g in range(len(lengths)):
        ref = out["fp64", 1][g]
        norm = ref.norm()
        assert ((out["fp64", 0][g] - ref).norm() / norm).item() <= 1e-12
        for plan in (0, 1):
            assert ((out["fp32", plan][g] - ref).norm() / norm).item() <= 2e-5
