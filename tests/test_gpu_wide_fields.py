"""Mass fields with cells beyond 2^47 units, which the FP32 x-forward passes convert
by rounding to odd first: the fused planes, the compile-time-planned pass and the
runtime-planned one (odd rows: plain loads; even ones: the bulk copy), with a few
large cells among small ones and with nothing else, up to the ends of int64,
within the suite's 2e-5 of the FP64 solve."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [45, 64, 84, 105, 162, 189, 216])
@pytest.mark.parametrize("cells", ["few", "all"])
def test_wide_fields_match_fp64(n, cells):
    import torch

    from paper_1410_0010_gb300.solver import Solver
    gen = torch.Generator(device="cuda").manual_seed(n)
    out = {}
    for precision in ("fp64", "fp32"):
        s = Solver([(0, -1, (0, 0, 0), (n, n, n))], periodic=True, precision=precision, device=0)
        b = s.alloc_level(0)
        q = b["gmf"][0]
        gen.manual_seed(n)
        q.random_(-2 ** 62, 2 ** 62, generator=gen)
        if cells == "few":
            q[:] = q >> 20
            q.view(-1)[3::997] = q.view(-1)[3::997] << 16
        else:                                   # every size from 2^47 up, both signs
            q[:] = q >> (torch.arange(n, device="cuda") % 16)
            q.view(-1)[:4] = torch.tensor([2 ** 63 - 1, -2 ** 63, 2 ** 47, -2 ** 47 - 1], device="cuda")
        s.solve_level(0, b["gmf"], b["phis"])
        s.sync_status()
        out[precision] = b["phis"][0].double()
        s.close()
    ref = out["fp64"]
    assert ((out["fp32"] - ref).norm() / ref.norm()).item() <= 2e-5
