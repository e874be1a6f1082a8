"""The kick-drift on values of every kind -- zeros, subnormals, sums whose half loses
a bit, infinities, NaN, any exponent -- beside ordinary ones in the same warps, in
both precisions: the bits of the plain IEEE evaluation."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("dt", [3e-3, -0.7, 0.0, 3e-308, 5e-324, 1e300])
def test_kick_drift_bits_over_the_range(precision, dt):
    import torch

    from paper_1410_0010_gb300.solver import Particles, Solver
    rng = np.random.default_rng(5)
    n = 20001
    bits = lambda k: rng.integers(0, 2 ** 64, size=k, dtype=np.uint64).view(np.float64)   # noqa: E731
    tiny = lambda k: rng.integers(0, 2 ** 54, size=k, dtype=np.uint64).view(np.float64)   # noqa: E731
    x, v = bits((3, n)), rng.normal(size=(3, n))
    kind = np.arange(n) % 97                    # most warps hold ordinary values as well
    x[:, kind > 40] = rng.random((3, int((kind > 40).sum())))
    v[:, kind == 1], v[:, kind == 2], v[:, kind == 3] = (f((3, int((kind == q).sum())))
                                                         for q, f in ((1, bits), (2, tiny), (3, np.zeros)))
    a = rng.normal(size=(3, n))
    a[:, (kind >= 2) & (kind <= 4)] = 0.0
    a[:, kind == 5] = bits((3, int((kind == 5).sum())))
    a[:, kind == 6] = np.inf
    x[:, kind == 2] = 0.0                       # the position shows the halved sum itself
    with np.errstate(all="ignore"):
        acc = torch.tensor(a, device="cuda").to(torch.float64 if precision == "fp64" else torch.float32)
        a = acc.double().cpu().numpy()
        vn = v + a * dt
        xn = x + ((v + vn) * 0.5) * dt
    names = ("x", "y", "z"), ("vx", "vy", "vz")
    t = {k: torch.tensor(d[j], device="cuda") for ks, d in zip(names, (x, v)) for j, k in enumerate(ks)}
    P = Particles(dict(t, m=torch.zeros(n, dtype=torch.float64, device="cuda")))
    s = Solver([(0, -1, (0, 0, 0), (8, 8, 8))], precision=precision, device=0)
    s.kick_drift(P, acc, dt)
    torch.cuda.synchronize()
    for ks, want in zip(names, (xn, vn)):
        for j, k in enumerate(ks):
            got = P.t[k].cpu().numpy()
            both = np.isnan(got) & np.isnan(want[j])
            assert np.array_equal(got.view(np.int64)[~both], want[j].view(np.int64)[~both]), k
    s.close()
