"""The complex64 marches of the 2-D GMRES steps with one and two products, where the levels
are too large for the tiles: plain sums above 256 points per axis, paired ones at 255^2 with
several right-hand sides, twelve and sixteen warps per block.  A k^2 field and odd layers, so
that general and uniform runs, the correction and the restriction all run."""

import numpy as np
import pytest

import oracle as O
from paper_1211_4752_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,batch,m", [(512, 1, 1), (512, 2, 2), (256, 5, 1), (256, 6, 2)])
def test_marches_match_oracle(n, batch, m):
    from paper_1211_4752_gb300 import HelmholtzMG
    k2, layers = W.smooth_k2(n, 2, 4, 0.25 * n, 0.5 * n), (13, 22)
    H = O.build_hierarchy(n, 2, k2, layers=layers, smoother="gmres", m=m)
    mg = HelmholtzMG(n, k2=torch.from_numpy(k2).cuda(), layers=layers, precision="mixed", smoother="gmres",
                     gmres_m=m, max_batch=batch)
    f = W.random_field((batch, n - 1, n - 1), 55)
    u0 = W.random_field(f.shape, 56, scale=1.0 / n ** 2)
    got = mg.cycles(torch.from_numpy(f).cuda(), torch.from_numpy(u0).cuda(), 1).cpu().numpy()
    for b in {0, batch - 1}:
        ref = O.vcycle(H, 0, u0[b], f[b])
        assert np.linalg.norm(got[b] - ref) <= 1e-4 * np.linalg.norm(ref), b
    mg.close()


@pytest.mark.parametrize("m", [1, 2, 3])
def test_large_grid_matches_complex128(m):
    """2047^2: more runs than blocks, several per warp."""
    from paper_1211_4752_gb300 import HelmholtzMG
    n = 2048
    g = torch.Generator(device="cuda").manual_seed(3)
    f, u = (torch.view_as_complex(torch.randn((1, n - 1, n - 1, 2), generator=g, device="cuda", dtype=torch.float64))
            for _ in range(2))
    u /= n ** 2
    out = []
    for precision in ("fp64", "mixed"):
        mg = HelmholtzMG(n, k2=(0.4 * n) ** 2, layers=(31, 64), precision=precision, smoother="gmres", gmres_m=m)
        out.append(mg.cycles(f, u, 1))
        mg.close()
    assert (out[1] - out[0]).norm().item() <= 1e-4 * out[0].norm().item()
