"""complex64 GMRES smoothing above 256 points per axis: the plain FP32 part of the inner
products.  On smooth right-hand sides, whose Krylov vectors are nearly parallel, the sums'
errors show: 16 of them on 511^2 (long runs of rows per thread), one cycle from zero against
the oracle.  With exact sums the vectors' own rounding leaves 1.1e-6 of the result; sums as
far off as FP64 sums of FP32 warp sums (6.7e-10) add 1.8e-6: together 2.1e-6, and 2.5e-6 are
allowed.  (Sums over runs of 32 rows, 1.4e-9, left 3.7e-6.)"""

import math

import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_smooth_right_hand_sides_of_a_batch():
    from paper_1211_4752_gb300 import HelmholtzMG
    n, batch = 512, 16
    rng = np.random.default_rng(5)
    x = np.arange(1, n) / n
    f = np.zeros((batch, n - 1, n - 1), dtype=np.complex128)
    for b in range(batch):
        for _ in range(6):
            i, j = rng.integers(1, 5, size=2)
            f[b] += rng.normal() * np.outer(np.sin(i * math.pi * x), np.sin(j * math.pi * x))
    k2, layers = (0.625 * n) ** 2, 16
    H = O.build_hierarchy(n, 2, k2, layers=layers, smoother="gmres")
    mg = HelmholtzMG(n, k2=k2, layers=layers, precision="mixed", smoother="gmres", max_batch=batch)
    g = torch.from_numpy(f).cuda()
    got = mg.cycles(g, torch.zeros_like(g), 1).cpu().numpy()
    num = den = 0.0
    for b in range(0, batch, 2):
        ref = O.vcycle(H, 0, np.zeros_like(f[b]), f[b])
        num += np.linalg.norm(got[b] - ref) ** 2
        den += np.linalg.norm(ref) ** 2
    assert math.sqrt(num / den) <= 2.5e-6
    mg.close()
