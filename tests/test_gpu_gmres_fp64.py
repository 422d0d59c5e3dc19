"""The complex128 GMRES smoothing is as accurate as an orthogonalised basis: one cycle of a
rough iterate under a point source against the same cycle in extended precision, on the
tiles, the large tiles, the one-block tail and in 3-D.  A cycle with an orthogonalised basis
in complex128 is 0.65e-15 to 1.4e-15 away; eight roundings (1.8e-15) are allowed."""

import numpy as np
import pytest

import oracle as O
from paper_1211_4752_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
EXT = np.clongdouble


def solve(A, b):
    """A x = b by Gauss-Jordan elimination with row interchanges."""
    M = np.concatenate([A, b[:, None]], axis=1).astype(EXT)
    m = len(b)
    for k in range(m):
        p = k + int(np.argmax(np.abs(M[k:, k])))
        M[[k, p]] = M[[p, k]]
        M[k] = M[k] / M[k, k]
        for i in range(m):
            if i != k:
                M[i] = M[i] - M[i, k] * M[k]
    return M[:, m]


def step(lv, u, f, m):
    """u + z with |f - A (u + z)| least over the Krylov space of dimension m."""
    V = [f - O.apply_operator(lv, u)]
    for _ in range(m):
        w = O.apply_operator(lv, V[-1])
        V.append(w / np.sqrt((w.conj() * w).sum().real))
    a = [O.apply_operator(lv, v) for v in V[:m]]
    dot = lambda x, y: (x.conj() * y).sum()  # noqa: E731
    y = solve(np.array([[dot(p, q) for q in a] for p in a]), np.array([dot(p, V[0]) for p in a]))
    return u + sum(y[j] * V[j] for j in range(m))


def vcycle(H, l, u, f, m):
    lv = H.levels[l]
    if l == len(H.levels) - 1:
        return solve(O.dense_matrix(lv), f.ravel()).reshape(f.shape)
    u = step(lv, u, f, m)
    fc = O.restrict_fw(f - O.apply_operator(lv, u))
    return step(lv, u + O.prolong(vcycle(H, l + 1, np.zeros_like(fc), fc, m)), f, m)


@pytest.mark.parametrize("n,dim,m", [(16, 2, 3), (32, 2, 3), (32, 2, 2), (64, 2, 3), (64, 2, 1), (128, 2, 3),
                                     (256, 2, 3), (256, 2, 2), (16, 3, 3), (32, 3, 3), (32, 3, 2)])
def test_cycle_is_accurate(n, dim, m):
    from paper_1211_4752_gb300 import HelmholtzMG
    k2, layers = (0.625 * n) ** 2, max(1, n // 32)
    H = O.build_hierarchy(n, dim, k2, layers=layers, smoother="gmres", m=m)
    mg = HelmholtzMG(n, dim=dim, k2=k2, layers=layers, precision="fp64", smoother="gmres", gmres_m=m)
    shape = (1,) + (n - 1,) * dim
    f = np.zeros(shape, dtype=np.complex128)
    f[(0,) + (n // 3,) * dim] = 1.0
    for seed in range(2):
        u0 = W.random_field(shape, 101 + seed, scale=1.0 / n ** 2)
        ref = vcycle(H, 0, u0[0].astype(EXT), f[0].astype(EXT), m)
        got = mg.cycles(torch.from_numpy(f).cuda(), torch.from_numpy(u0).cuda(), 1).cpu().numpy()[0]
        err = np.abs(got - ref).astype(np.float64)
        assert np.linalg.norm(err) <= 8 * 2.0 ** -52 * np.linalg.norm(got), seed
    mg.close()
