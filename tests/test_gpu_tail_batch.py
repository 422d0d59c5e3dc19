"""The complex128 tail levels of a Jacobi cycle: up to which batch the dense operator serves
depends on the tail's size.  On neither side of the limit does a smaller batch take longer
than a large one, and the results are those of one right-hand side at a time."""

import ctypes as ct

import pytest

from paper_1211_4752_gb300 import _binding as B
from paper_1211_4752_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [16, 32, 64])
def test_tail_time_and_results(n):
    from paper_1211_4752_gb300 import HelmholtzMG
    mg = HelmholtzMG(n, k2=(0.5 * n) ** 2, layers=2, precision="fp64", max_batch=12)
    stream = ct.c_void_p(torch.cuda.current_stream().cuda_stream)

    def tail_ms(batch):
        ms, best = ct.c_double(), 1e30
        for _ in range(3):
            B.check(B.lib().hh_time_kernel(mg._h, 4, 0, batch, 50, ct.byref(ms), stream))
            best = min(best, ms.value)
        return best

    most = tail_ms(12)
    for b in range(1, 8):
        assert tail_ms(b) <= 1.2 * most, b
    f = torch.from_numpy(W.random_field((7, n - 1, n - 1), 95)).cuda()
    u = torch.from_numpy(W.random_field(f.shape, 96, scale=1.0 / n ** 2)).cuda()
    one = torch.cat([mg.cycles(f[b:b + 1].contiguous(), u[b:b + 1].contiguous(), 2) for b in range(7)])
    for b in range(2, 8):
        got = mg.cycles(f[:b].contiguous(), u[:b].contiguous(), 2)
        assert (got - one[:b]).norm().item() <= 1e-12 * one[:b].norm().item(), b
    mg.close()
