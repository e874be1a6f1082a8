"""The plan of each FFT pass: plan 3 keeps the x and y passes of the lengths that plan
0 runs as fused planes apart, a y pass with the runtime plan keeps them apart too,
and the tuner compares only different kernels: it leaves the launch shapes of passes
without a runtime-planned kernel alone and reports numbers that give the same
kernels again."""
import pytest

pytestmark = pytest.mark.gpu

GRIDS = [(0, -1, (0, 0, 0), (96, 96, 96)), (1, 0, (8, 8, 8), (64, 64, 64)), (1, 0, (100, 8, 8), (55, 55, 28))]


def _solver(precision):
    import torch

    from paper_1410_0010_gb300.solver import Solver
    s = Solver(GRIDS, periodic=True, precision=precision, device=0)
    b = s.alloc_level(1)
    gen = torch.Generator(device="cuda").manual_seed(3)
    for g in b["gmf"]:
        g.copy_((torch.randn(g.shape, generator=gen, device="cuda", dtype=torch.float64) * 2.0 ** 40).long())
    return s, b


def _solve(s, b, plan):
    s.set_fft_shapes(1, dict(s.fft_shapes(1), plan=plan))
    s.solve_level(1, b["gmf"], b["phis"])
    s.sync_status()
    return [t.clone() for t in b["phis"]], s.pass_kernels(1)


def test_unfused_compile_time_passes_can_be_asked_for():
    s, b = _solver("fp32")
    assert [tuple(s.info[i]["fft"]) for i in (1, 2)] == [(84, 84, 84), (75, 75, 48)]
    runtime, kinds = _solve(s, b, [1] * 5)
    assert kinds == [[0, 0]] * 5
    for plan, want in (([0] * 5, [2, 3, 1, 3, 2]), ([3, 0, 0, 0, 3], [1] * 5), ([3, 0, 0, 0, 0], [1, 1, 1, 3, 2]),
                       ([0, 1, 0, 1, 0], [1, 0, 1, 0, 1]), ([2, 1, 0, 1, 2], [2, 3, 1, 3, 2])):
        out, kinds = _solve(s, b, plan)
        assert [row[0] for row in kinds] == want and [row[1] for row in kinds] == want, plan
        for x, r in zip(out, runtime):      # the runtime plans round differently: the suite's FP32 tolerance
            assert ((x - r).double().norm() / r.double().norm()).item() <= 2e-5
    s.close()


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_tuner_compares_different_kernels_only(precision):
    from paper_1410_0010_gb300.solver import Solver
    # FP64 has compile-time plans from 70 up: every pass of these grids
    grids = GRIDS[:2] + [(1, 0, (100, 8, 8), (55, 55, 55))] if precision == "fp64" else GRIDS
    s = Solver(grids, periodic=True, precision=precision, device=0)
    b = s.alloc_level(1)
    for g in b["gmf"]:
        g.random_(-2 ** 40, 2 ** 40)
    default = s.fft_shapes(1)
    for _ in range(3):
        s.autotune_level(1, b["gmf"], b["phis"])
        tuned = s.fft_shapes(1)
        if precision == "fp64":
            assert dict(tuned, packing=0) == default
    kinds = s.pass_kernels(1)
    s.set_fft_shapes(1, tuned)
    assert s.pass_kernels(1) == kinds and s.fft_shapes(1) == tuned
    s.close()
