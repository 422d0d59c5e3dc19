"""GMRES-smoothed cycles of fewer right-hand sides than the handle holds: the work is
split for the call, so results and times are those of a handle made for that many."""

import ctypes as ct

import pytest

from paper_1211_4752_gb300 import _binding as B
from paper_1211_4752_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def make(n, dim, precision, batch):
    from paper_1211_4752_gb300 import HelmholtzMG
    return HelmholtzMG(n, dim=dim, k2=(0.5 * n) ** 2, layers=max(1, n // 16), precision=precision,
                       smoother="gmres", max_batch=batch)


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("n,dim,batch", [(64, 2, 1), (256, 2, 1), (256, 2, 3), (512, 2, 1), (32, 3, 2)])
def test_results_do_not_depend_on_capacity(n, dim, batch, precision):
    large, own = make(n, dim, precision, 20), make(n, dim, precision, batch)
    f = torch.from_numpy(W.random_field((batch,) + (n - 1,) * dim, 91)).cuda()
    u = torch.from_numpy(W.random_field(f.shape, 92, scale=1.0 / n ** 2)).cuda()
    assert torch.equal(large.cycles(f, u, 2), own.cycles(f, u, 2))
    # the stop test's sums follow the call as well
    tol = 1e-3
    (a, ia), (b, ib) = large.solve(f, tol=tol), own.solve(f, tol=tol)
    assert torch.equal(a, b) and [i["cycles"] for i in ia] == [i["cycles"] for i in ib]
    large.close(), own.close()


def cycle_ms(mg, batch):
    ms = ct.c_double()
    stream = ct.c_void_p(torch.cuda.current_stream().cuda_stream)
    best = 1e30
    for _ in range(3):
        B.check(B.lib().hh_time_kernel(mg._h, 5, 0, batch, 20, ct.byref(ms), stream))
        best = min(best, ms.value)
    return best


@pytest.mark.parametrize("n,dim,precision", [(1024, 2, "fp64"), (512, 2, "mixed"), (128, 3, "mixed"), (64, 3, "fp64")])
def test_time_does_not_depend_on_capacity(n, dim, precision):
    large, own = make(n, dim, precision, 16), make(n, dim, precision, 1)
    assert cycle_ms(large, 1) <= 1.25 * cycle_ms(own, 1)
    large.close(), own.close()
