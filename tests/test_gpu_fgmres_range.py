"""FGMRES in complex64 of sources far from one in magnitude: a restart's residual norm is
the sum of squares of FP32 values, taken in FP64.  Powers of two: the iterations are those
of the unscaled source, rounding by rounding."""

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("exponent", [-80, -60, 60])
def test_fgmres_of_scaled_sources(exponent):
    from paper_1211_4752_gb300 import HelmholtzMG
    n = 64
    mg = HelmholtzMG(n, k2=(0.5 * n) ** 2, layers=4, precision="mixed", max_batch=2)
    f = torch.zeros((2, n - 1, n - 1), dtype=torch.complex128, device="cuda")
    f[0, 31, 31] = 1.0
    f[1, 20, 40] = 1.0
    ref, info = mg.fgmres(f, tol=1e-6, restart=10)
    got, scaled = mg.fgmres(f * 2.0 ** exponent, tol=1e-6, restart=10)
    assert [(i["status"], i["cycles"]) for i in scaled] == [(i["status"], i["cycles"]) for i in info]
    assert (got * 2.0 ** -exponent - ref).norm().item() <= 4 * 2.0 ** -24 * ref.norm().item()
    mg.close()
