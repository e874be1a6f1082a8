"""Compile-time FFT plans: the FP64 ones of 75, 256 and 512, and in both precisions
192 and those of 288 to 480, on periodic roots (whose window wraps), against the
runtime-planned kernels: FP64 within the suite's 1e-12, FP32 within its 2e-5 of
FP64."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [75, 192, 256, 288, 300, 320, 360, 384, 400, 480, 512])
def test_long_plans_match_runtime_plans(n):
    import torch

    from paper_1410_0010_gb300.solver import Solver
    gen = torch.Generator(device="cuda").manual_seed(n)
    out = {}
    for precision in ("fp64", "fp32"):
        s = Solver([(0, -1, (0, 0, 0), (n, n, n))], periodic=True, precision=precision, device=0)
        b = s.alloc_level(0)
        if not out:
            gmf = b["gmf"][0].random_(-2 ** 45, 2 ** 45, generator=gen)
        for plan in (1, 0, 3):
            x = 0 if plan == 3 else plan        # plan 3: the x passes apart from the y passes
            s.set_fft_shapes(0, dict(s.fft_shapes(0), plan=[plan, x, x, x, plan]))
            kinds = {k for row in s.pass_kernels(0) for k in row}
            assert kinds == {0} if plan == 1 else 0 not in kinds
            s.solve_level(0, [gmf], b["phis"])
            s.sync_status()
            out[precision, plan] = b["phis"][0].double().clone()
        s.close()
        del b
    ref = out["fp64", 1]
    norm = ref.norm()
    for (precision, _), phi in out.items():
        assert ((phi - ref).norm() / norm).item() <= (1e-12 if precision == "fp64" else 2e-5)
