"""The one-reduction GMRES step (Chebyshev basis, Gram matrix) on the GPU against
the oracle's Arnoldi step, over the kernels and tile edges it is built of: tiles
with a thread per point and marches / large tiles (chosen by size and number of
right-hand sides), the uniform body up to the domain's edge and the layers' general
one, one to three products, several smoothing steps, complex scales, the paired
and the plain FP32 sums, and a Krylov space that ends early."""

import math

import numpy as np
import pytest

import oracle as O
from paper_1211_4752_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

CASES = [
    # n, batch, layers, k2, form, m, nu1, nu2
    (8, 1, 0, 30.0, "csl", 3, 1, 1),            # smallest grid: the one-block tail below one level
    (16, 3, (1, 2), 60.0, "csl", 2, 1, 1),
    (64, 1, 0, 400.0, "csl", 3, 1, 1),          # no layers: uniform up to the edge
    (128, 17, (5, 9), ("field", 30.0, 60.0), "csl", 3, 1, 1),  # too many tiles: marches, paired sums
    (128, 2, 8, 6400.0, "csg", 3, 1, 1),        # complex Laplacian scale: no uniform body
    (256, 1, (0, 21), ("field", 60.0, 120.0), "csl", 1, 2, 1),
    (256, 5, 7, 160.0 ** 2, "csl", 2, 1, 2),
    (512, 1, 0, 1e4, "csl", 3, 1, 1),           # marches, plain sums, uniform to the edge
    (512, 2, (13, 40), ("field", 90.0, 250.0), "csl", 3, 2, 2),
    (1024, 1, 33, 640.0 ** 2, "csl", 3, 1, 1),
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: f"n{c[0]}-b{c[1]}-m{c[5]}-nu{c[6]}{c[7]}")
def test_step_matches_oracle(case):
    from paper_1211_4752_gb300 import HelmholtzMG
    n, batch, layers, k2, form, m, nu1, nu2 = case
    if isinstance(k2, tuple):
        k2 = W.smooth_k2(n, 2, 4, k2[1], k2[2])
    P = int(round(math.log2(n)))
    c = [np.exp(-1j * (math.pi / 6) / P)] * (P - 2) if form == "csg" else None
    H = O.build_hierarchy(n, 2, k2, layers=layers, form=form, c=c, smoother="gmres", m=m, nu1=nu1, nu2=nu2)
    kt = torch.from_numpy(k2).cuda() if isinstance(k2, np.ndarray) else k2
    f = W.random_field((batch, n - 1, n - 1), 51)
    u0 = W.random_field((batch, n - 1, n - 1), 52, scale=1.0 / n ** 2)
    ref = {b: O.vcycle(H, 0, u0[b], f[b]) for b in {0, batch - 1}}
    for precision, tol in (("fp64", 1e-9), ("mixed", 1e-4)):
        mg = HelmholtzMG(n, k2=kt, layers=layers, form=form, c=c, smoother="gmres", gmres_m=m, nu1=nu1,
                         nu2=nu2, precision=precision, max_batch=batch)
        got = mg.cycles(torch.from_numpy(f).cuda(), torch.from_numpy(u0).cuda(), 1).cpu().numpy()
        for b, r in ref.items():
            assert np.linalg.norm(got[b] - r) <= tol * np.linalg.norm(r), (precision, b)
        mg.close()


@pytest.mark.parametrize("n", [64, 512])
def test_krylov_space_of_one_dimension(n):
    """f is an eigenvector of the Dirichlet Laplacian: one product spans the
    Krylov space, the others are rounding, and the first step is already the
    solution f / lambda."""
    from paper_1211_4752_gb300 import HelmholtzMG
    x = np.arange(1, n) / n
    f = np.outer(np.sin(3 * math.pi * x), np.sin(2 * math.pi * x)).astype(np.complex128)[None]
    lam = 4.0 * n * n * (math.sin(3 * math.pi / (2 * n)) ** 2 + math.sin(2 * math.pi / (2 * n)) ** 2)
    for precision, tol in (("fp64", 1e-10), ("mixed", 1e-4)):
        mg = HelmholtzMG(n, k2=0.0, smoother="gmres", precision=precision)
        g = torch.from_numpy(f).cuda()
        got = mg.cycles(g, torch.zeros_like(g), 1).cpu().numpy()
        assert np.linalg.norm(got - f / lam) <= tol * np.linalg.norm(f / lam), precision
        z = mg.cycles(torch.zeros_like(g), torch.zeros_like(g), 1)   # zero residual: no correction
        assert not z.abs().max().item()
        mg.close()


CASES_3D = [
    # n, batch, layers, k2, form, m, nu1, nu2
    (8, 2, 0, 20.0, "csl", 3, 1, 1),
    (16, 1, (1, 3), ("field", 5.0, 9.0), "csl", 1, 1, 1),
    (32, 3, (4, 2), 300.0, "csg", 2, 1, 2),
    (64, 1, 5, ("field", 18.0, 36.0), "csl", 3, 2, 1),
    (128, 1, 9, 60.0 ** 2, "csl", 3, 1, 1),          # plain sums
]


@pytest.mark.parametrize("case", CASES_3D, ids=lambda c: f"n{c[0]}-b{c[1]}-m{c[5]}-nu{c[6]}{c[7]}")
def test_step_matches_oracle_3d(case):
    from paper_1211_4752_gb300 import HelmholtzMG
    n, batch, layers, k2, form, m, nu1, nu2 = case
    if isinstance(k2, tuple):
        k2 = W.smooth_k2(n, 3, 4, k2[1], k2[2])
    P = int(round(math.log2(n)))
    c = [np.exp(-1j * (math.pi / 6) / P)] * (P - 2) if form == "csg" else None
    H = O.build_hierarchy(n, 3, k2, layers=layers, form=form, c=c, smoother="gmres", m=m, nu1=nu1, nu2=nu2)
    kt = torch.from_numpy(k2).cuda() if isinstance(k2, np.ndarray) else k2
    f = W.random_field((batch,) + (n - 1,) * 3, 53)
    u0 = W.random_field(f.shape, 54, scale=1.0 / n ** 2)
    ref = {b: O.vcycle(H, 0, u0[b], f[b]) for b in {0, batch - 1}}
    for precision, tol in (("fp64", 1e-9), ("mixed", 1e-4)):
        mg = HelmholtzMG(n, dim=3, k2=kt, layers=layers, form=form, c=c, smoother="gmres", gmres_m=m,
                         nu1=nu1, nu2=nu2, precision=precision, max_batch=batch)
        got = mg.cycles(torch.from_numpy(f).cuda(), torch.from_numpy(u0).cuda(), 1).cpu().numpy()
        for b, r in ref.items():
            assert np.linalg.norm(got[b] - r) <= tol * np.linalg.norm(r), (precision, b)
        mg.close()
