"""The complex64 GMRES smoothing's inner products are sums of squares in FP32: inputs far
from one in magnitude give the scaled results of the same inputs near one.  The factors
are powers of two, so that every rounding is the same and the results agree exactly while
no value of a vector leaves FP32's normal range; a few roundings are allowed."""

import numpy as np
import pytest

from paper_1211_4752_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TOL = 4 * 2.0 ** -24
EXPONENTS = [-90, -60, -50, 50, 60]


@pytest.mark.parametrize("n,dim,batch", [(8, 2, 1), (64, 2, 1), (256, 2, 5), (512, 2, 1), (32, 3, 2), (128, 3, 1)])
def test_cycles_of_scaled_inputs(n, dim, batch):
    from paper_1211_4752_gb300 import HelmholtzMG
    mg = HelmholtzMG(n, dim=dim, k2=(0.5 * n) ** 2, layers=max(1, n // 16), precision="mixed",
                     smoother="gmres", max_batch=batch)
    f = torch.from_numpy(W.random_field((batch,) + (n - 1,) * dim, 81)).cuda()
    u = torch.from_numpy(W.random_field(f.shape, 82, scale=1.0 / n ** 2)).cuda()
    zero = torch.zeros_like(f)
    for a, b in ((f, u), (f, zero), (zero, u)):
        ref = mg.cycles(a, b, 3)
        for e in EXPONENTS:
            got = mg.cycles(a * 2.0 ** e, b * 2.0 ** e, 3) * 2.0 ** -e
            assert (got - ref).norm().item() <= TOL * ref.norm().item(), e
    # right-hand sides of one call far apart
    if batch > 1:
        s = torch.tensor([2.0 ** e for e in np.linspace(-60, 60, batch).astype(int)], device="cuda")
        s = s.reshape((batch,) + (1,) * dim)
        got = mg.cycles(f * s, u * s, 3) / s
        ref = mg.cycles(f, u, 3)
        assert (got - ref).norm().item() <= TOL * ref.norm().item()
    mg.close()


@pytest.mark.parametrize("how", ["solve", "adjoint", "fgmres"])
@pytest.mark.parametrize("exponent", [-60, -40, 40, 60])
def test_solves_of_scaled_sources(how, exponent):
    from paper_1211_4752_gb300 import HelmholtzMG
    n = 64
    mg = HelmholtzMG(n, k2=(0.5 * n) ** 2, layers=4, precision="mixed", smoother="gmres", max_batch=2)
    f = torch.zeros((2, n - 1, n - 1), dtype=torch.complex128, device="cuda")
    f[0, 31, 31] = 1.0
    f[1, 20, 40] = 1.0
    ref, info = getattr(mg, how)(f, tol=1e-8)
    got, scaled = getattr(mg, how)(f * 2.0 ** exponent, tol=1e-8)
    assert [i["status"] for i in scaled] == ["OK", "OK"]
    assert [i["cycles"] for i in scaled] == [i["cycles"] for i in info]
    assert (got * 2.0 ** -exponent - ref).norm().item() <= TOL * ref.norm().item()
    # from a guess, whose residual and not the source sets the scale
    if how != "fgmres":
        u0 = torch.from_numpy(W.random_field(f.shape, 83)).cuda()
        ref, info = getattr(mg, how)(f, 1e-8, u0)
        got, scaled = getattr(mg, how)(f * 2.0 ** exponent, 1e-8, u0 * 2.0 ** exponent)
        assert [(i["status"], i["cycles"]) for i in scaled] == [(i["status"], i["cycles"]) for i in info]
        assert (got * 2.0 ** -exponent - ref).norm().item() <= TOL * ref.norm().item()
    mg.close()
