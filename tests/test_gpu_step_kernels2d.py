"""The 2-D single-step kernels (strips walking down a run of rows) and the complex128
passes and tail of the cycle against the oracle, at the sizes where their work is
split: strips and runs cut by the domain's edge, uniform to the edge, thin and thick
layers, constant and varying k^2, real and complex scales and weights, one to several
right-hand sides, and both sides of the tail operator's limit on the batch."""

import numpy as np
import pytest

import oracle as O
from paper_1211_4752_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

CASES = [
    # n, batch, layers, k2, form, omega
    (8, 1, 0, 30.0, "csl", 0.8),
    (16, 2, (1, 2), 60.0, "csl", 0.8),
    (64, 3, 0, 400.0, "csl", 0.8),                                # uniform to the edge
    (128, 2, (5, 9), ("field", 30.0, 60.0), "csl", 0.8),
    (128, 7, 8, 6400.0, "csg", 0.8),                              # complex Laplacian scale
    (256, 2, 7, 160.0 ** 2, "csl", 0.8 + 0.05j),                  # complex weight
    (512, 1, (0, 21), ("field", 90.0, 250.0), "csl", 0.8 + 0.05j),
    (1024, 1, 33, 640.0 ** 2, "csl", 0.8),
]


def make(case, **kw):
    from paper_1211_4752_gb300 import HelmholtzMG
    n, batch, layers, k2, form, omega = case
    if isinstance(k2, tuple):
        k2 = W.smooth_k2(n, 2, 4, k2[1], k2[2])
    c = None
    if form == "csg":
        P = int(round(np.log2(n)))
        c = [np.exp(-1j * (np.pi / 6) / P)] * (P - 2)
    H = O.build_hierarchy(n, 2, k2, layers=layers, form=form, c=c, omega=omega)
    kt = torch.from_numpy(k2).cuda() if isinstance(k2, np.ndarray) else k2
    mg = HelmholtzMG(n, k2=kt, layers=layers, form=form, c=c, omega=omega, max_batch=batch, **kw)
    return H, mg


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def close(got, ref, tol):
    return np.abs(got.cpu().numpy() - ref).max() <= tol * np.abs(ref).max()


@pytest.mark.parametrize("case", CASES, ids=lambda c: f"n{c[0]}-b{c[1]}-{c[4]}")
def test_steps_match_oracle(case):
    H, mg = make(case)
    Ha = O.adjoint_hierarchy(H)
    B = case[1]
    for l in range(min(3, len(H.levels) - 1)):
        lv, lc = H.levels[l], H.levels[l + 1]
        u, f = (W.random_field((B,) + lv.shape, 61 + i) for i in range(2))
        e = W.random_field((B,) + lc.shape, 63)
        for adj, hier in ((False, H), (True, Ha)):
            ref = np.stack([O.apply_operator(hier.levels[l], x) for x in u])
            assert close(mg.apply(dev(u), level=l, adjoint=adj), ref, 1e-13), (l, adj)
        ref = np.stack([O.jacobi(lv, u[b], f[b], H.omega) for b in range(B)])
        assert close(mg.smooth(l, dev(u), dev(f)), ref, 1e-13), l
        ref = np.stack([H.c[l] * O.restrict_fw(f[b] - O.apply_operator(lv, u[b])) for b in range(B)])
        assert close(mg.residual_restrict(l, dev(u), dev(f)), ref, 1e-12), l
        ref = np.stack([O.jacobi(lv, u[b] + O.prolong(e[b]), f[b], H.omega) for b in range(B)])
        assert close(mg.correct_smooth(l, dev(u), dev(e), dev(f)), ref, 1e-13), l
    mg.close()


@pytest.mark.parametrize("case", CASES, ids=lambda c: f"n{c[0]}-b{c[1]}-{c[4]}")
def test_complex128_cycles_match_oracle(case):
    """Two cycles from zero (the passes' zero branch) and from an iterate; the batch
    of 7 runs the tail levels' own kernel, the others the dense operator."""
    H, mg = make(case)
    B, shape = case[1], H.levels[0].shape
    f = W.random_field((B,) + shape, 71)
    for u0 in (np.zeros_like(f), W.random_field((B,) + shape, 72, scale=1.0 / case[0] ** 2)):
        got = mg.cycles(dev(f), dev(u0), 2).cpu().numpy()
        for b in {0, B - 1}:
            u = u0[b].copy()
            for _ in range(2):
                u = O.vcycle(H, 0, u, f[b])
            assert np.linalg.norm(got[b] - u) <= 1e-12 * np.linalg.norm(u), b
    mg.close()
