"""The work that users of this library have it do, as measurable cases.

listed() names twelve cases, draw(rng) gives more of the same ranges,
prepare(case, seed) makes what a user's program holds before the call (a
handle, right-hand sides, an iterate), run(state) is one pass through the
public entry points, work(case) what a pass cannot do without, and
exact(case, seed) the same outputs from plain torch in complex128.

Kinds of work:

* ``steps``     a user's own cycle or two-grid analysis from the step entry
                points, complex128: sweep, residual + restriction, a coarse
                sweep, correction + sweep, and the operator and its adjoint.
* ``cycles``    a fixed number of V-cycles from the current iterate (the cycle
                as a smoother or preconditioner inside a user's iteration).
* ``solve``     a whole solve to a relative residual.
* ``fgmres``    a whole solve by flexible GMRES around the cycle.
* ``gradient``  one step of an inversion: the medium is new, so the handle is
                set up, then forward solve, adjoint solve, gradients
                (autograd, complex128).

Mixed-precision handles run complex64 cycles; their results carry single
precision (a solve stops at 1e-6), so the program here keeps the wavefield in
complex64, as one does that stores the fields of many sources.  complex128
handles return complex128.

Media: ``const`` k h = 0.625 (the benchmark's), ``bump`` k h = 0.5 with a 10 %
Gaussian bump, ``layers`` three speeds with tilted interfaces, ``smooth`` a
smooth field with k h from 0.3 to 0.6.  Absorbing layers of ``lo`` / ``hi``
cells at the ends of every axis.
"""

import math

import torch

from paper_1211_4752_gb300 import HelmholtzMG, helmholtz_solve

ECS_ANGLE = math.pi / 6
THETA_MAX = math.pi / 6
OMEGA = 0.8


def _case(name, kind, n, dim=2, batch=1, precision="mixed", smoother="jacobi", medium="const",
          lo=None, hi=None, cycles=0, adjoint=False):
    c = dict(kind=kind, n=n, dim=dim, batch=batch, precision=precision, smoother=smoother,
             medium=medium, lo=n // 32 if lo is None else lo, hi=n // 32 if hi is None else hi,
             cycles=cycles, adjoint=adjoint)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest calls: step entry points on the 63^2 model problem's grid,
        # where launches and the host path count
        _case("steps_63", "steps", 64, precision="fp64", lo=4, hi=4),
        # the same on the benchmark's grid, three right-hand sides, variable k
        _case("steps_1023_b3", "steps", 1024, precision="fp64", batch=3, medium="smooth"),
        # a few cycles on a small grid: a chain of short dependent launches
        _case("jacobi_255", "cycles", 256, cycles=16),
        # many sources at once (one handle of the many-source workload)
        _case("jacobi_511_b21", "cycles", 512, batch=21, cycles=8),
        # a grid whose arrays exceed the L2 cache
        _case("jacobi_4095", "cycles", 4096, cycles=4),
        # the plain complex128 cycle on the benchmark's grid
        _case("jacobi_fp64_1023", "cycles", 1024, precision="fp64", cycles=4),
        # the benchmark: 1023^2, k = 640, one source, to 1e-6
        _case("solve_1023", "solve", 1024),
        # the paper's GMRES(3) smoother on the bump medium, to 1e-6
        _case("solve_gmres_bump_511", "solve", 512, smoother="gmres", medium="bump", lo=16, hi=16),
        # GMRES(3)-smoothed cycles on the benchmark's grid
        _case("gmres_1023", "cycles", 1024, smoother="gmres", cycles=4),
        # the 127^3 cube, GMRES(3) smoothing
        _case("gmres_cube_127", "cycles", 128, dim=3, smoother="gmres", lo=16, hi=16, cycles=2),
        # the three-layer medium, which needs FGMRES around the GMRES(3) cycle
        _case("fgmres_layers_511", "fgmres", 512, smoother="gmres", medium="layers", lo=12, hi=12),
        # one inversion step: 255^2, four sources on a row, receivers on another
        _case("gradient_255_b4", "gradient", 256, precision="fp64", smoother="gmres", medium="bump",
              lo=8, hi=8, batch=4),
    ]


def draw(rng):
    def width(n):
        """Layer widths from n/64 to n/8, odd ones among them; the ends differ at times."""
        a = rng.randint(max(2, n // 64), n // 8)
        return a, (a if rng.random() < 0.6 else rng.randint(max(2, n // 64), n // 8))

    def many(most):
        return max(1, min(64, int(math.exp(rng.uniform(0.0, math.log(max(1.0, most)))))))

    kind = rng.choice(["steps", "cycles", "cycles", "cycles", "cycles", "solve", "fgmres", "gradient"])
    if kind == "steps":
        dim = rng.choice([2, 2, 3])
        n = 2 ** (rng.randint(6, 11) if dim == 2 else rng.randint(4, 7))
        lo, hi = width(n)
        return _case(None, kind, n, dim=dim, batch=many(2 ** 23 / n ** dim), precision="fp64",
                     medium=rng.choice(["const", "smooth"]), lo=lo, hi=hi)
    if kind == "cycles":
        smoother = rng.choice(["jacobi", "jacobi", "gmres"])
        precision = rng.choice(["mixed", "mixed", "fp64"])
        dim = rng.choice([2, 2, 2, 3])
        top = 12 if smoother == "jacobi" and precision == "mixed" else 10
        n = 2 ** (rng.randint(6, top) if dim == 2 else rng.randint(4, 7))
        lo, hi = width(n)
        most = 2.0 ** (24 if precision == "mixed" else 22) / n ** dim
        return _case(None, kind, n, dim=dim, batch=many(most), precision=precision, smoother=smoother,
                     medium=rng.choice(["const", "const", "smooth"]), lo=lo, hi=hi,
                     cycles=rng.randint(1, 8))
    if kind == "solve":
        # Jacobi cycles converge on the constant medium at k h = 0.625 with thin
        # layers; GMRES(3) smoothing also on the bump
        if rng.random() < 0.5:
            n = 2 ** rng.randint(6, 9)
            return _case(None, kind, n, batch=many(4), lo=n // 32, hi=n // 32,
                         precision=rng.choice(["mixed", "mixed", "fp64"]) if n <= 256 else "mixed",
                         adjoint=rng.random() < 0.3)
        n = 2 ** rng.randint(7, 9)
        return _case(None, kind, n, batch=many(4), smoother="gmres", lo=n // 32, hi=n // 32,
                     medium=rng.choice(["const", "bump"]), adjoint=rng.random() < 0.3)
    if kind == "fgmres":
        n = 2 ** rng.randint(7, 9)
        return _case(None, kind, n, smoother="gmres", medium="layers", lo=n // 42, hi=n // 42,
                     batch=many(2))
    n = 2 ** rng.randint(6, 8)
    return _case(None, kind, n, precision="fp64", smoother="gmres", medium="bump", lo=n // 32,
                 hi=n // 32, batch=many(6))


# ---- inputs -------------------------------------------------------------------

def _gen(seed, device):
    g = torch.Generator(device=device)
    g.manual_seed(int(seed))
    return g


def _randn(shape, g, device):
    x = torch.randn((*shape, 2), generator=g, device=device, dtype=torch.float64)
    return torch.view_as_complex(x)


def _medium(c, g):
    """k^2: a number, or a field on the interior points."""
    n, dim = c["n"], c["dim"]
    dev = torch.device("cuda")
    u = torch.rand(8, generator=g, device=dev, dtype=torch.float64).tolist()
    if c["medium"] == "const":
        return (0.625 * n) ** 2
    x = torch.arange(1, n, device=dev, dtype=torch.float64) / n
    grids = torch.meshgrid(*([x] * dim), indexing="ij")
    if c["medium"] == "bump":
        r2 = sum((q - (0.3 + 0.4 * u[i])) ** 2 for i, q in enumerate(grids))
        return (0.5 * n) ** 2 * (1.0 + 0.1 * torch.exp(-r2 / (2 * 0.05 ** 2)))
    if c["medium"] == "layers":
        y, xx = grids
        speeds = [1.5 + 3.0 * u[i] for i in range(3)]
        tilt = [math.tan(math.radians(-20.0 + 40.0 * u[3 + i])) for i in range(2)]
        a, b = c["lo"] / n, 1.0 - c["hi"] / n
        d = [a + (b - a) / 3.0, a + 2.0 * (b - a) / 3.0]
        cc = torch.where(y < d[0] + tilt[0] * (xx - 0.5), speeds[0],
                         torch.where(y < d[1] + tilt[1] * (xx - 0.5), speeds[1], speeds[2]))
        return (0.625 * n * min(speeds) / cc) ** 2
    s = sum(torch.sin(2 * math.pi * (j + 1) * q + 6.0 * u[j]) for j, q in enumerate(grids))
    s = (s - s.min()) / (s.max() - s.min())
    return (n * (0.3 + 0.3 * s)) ** 2


def _inputs(c, seed):
    """(k2, f, u): medium, right-hand sides, current iterate."""
    dev = torch.device("cuda")
    g = _gen(seed, dev)
    n, dim, B = c["n"], c["dim"], c["batch"]
    N = n - 1
    k2 = _medium(c, g)
    shape = (B,) + (N,) * dim
    f = torch.zeros(shape, dtype=torch.complex128, device=dev)
    lo, hi = c["lo"], n - 2 - c["hi"]
    pos = lo + (torch.rand((B, dim), generator=g, device=dev, dtype=torch.float64) * (hi - lo + 1)).long()
    pos = pos.clamp(lo, hi).tolist()
    if c["kind"] == "gradient":          # sources on the first physical row
        for b in range(B):
            pos[b][0] = lo
    for b, p in enumerate(pos):
        f[(b, *p)] = 1.0
    u = None
    if c["kind"] in ("steps", "cycles"):
        # an iterate on the way: its residual is of the order of the source everywhere
        u = _randn(shape, g, dev) / n ** 2
    return k2, f, u


def _kwargs(c):
    kw = dict(dim=c["dim"], layers=(c["lo"], c["hi"]), precision=c["precision"],
              smoother=c["smoother"], max_batch=c["batch"])
    if c["kind"] == "fgmres":
        kw["max_cycles"] = 4000
    return kw


def prepare(case, seed):
    k2, f, u = _inputs(case, seed)
    st = dict(case=case, f=f, u=u, k2=k2)
    n = case["n"]
    if case["kind"] == "gradient":
        g = _gen(seed + 77, f.device)
        st["k2"] = k2.requires_grad_(True)
        st["f"] = f.requires_grad_(True)
        st["row"] = n - case["hi"] - 2
        st["data"] = _randn((case["batch"], n - 1), g, f.device) / n ** 2
        return st
    st["mg"] = HelmholtzMG(n, k2=k2, **_kwargs(case))
    if case["kind"] == "steps":
        g = _gen(seed + 77, f.device)
        Nc = st["mg"].level_points(1)
        st["e"] = _randn((case["batch"],) + (Nc,) * case["dim"], g, f.device) / n ** 2
    return st


def run(state):
    c = state["case"]
    if c["kind"] == "gradient":
        k2, f = state["k2"], state["f"]
        u = helmholtz_solve(k2, f, n=c["n"], **_kwargs(c))
        r = u[:, state["row"], :] - state["data"]
        loss = 0.5 * (r.real ** 2 + r.imag ** 2).sum()
        gk2, gf = torch.autograd.grad(loss, (k2, f))
        return u.detach(), gk2, gf
    mg, f = state["mg"], state["f"]
    if c["kind"] == "steps":
        v = mg.smooth(0, state["u"], f)
        fc = mg.residual_restrict(0, v, f)
        ec = mg.smooth(1, state["e"], fc)
        w = mg.correct_smooth(0, v, ec, f)
        return v, fc, ec, w, mg.apply(w), mg.apply(w, adjoint=True)
    if c["kind"] == "cycles":
        u = mg.cycles(f, state["u"], c["cycles"])
    elif c["kind"] == "solve":
        u, _ = (mg.adjoint if c["adjoint"] else mg.solve)(f, tol=1e-6)
    else:
        u, _ = mg.fgmres(f, tol=1e-6, restart=32)
    return u.to(torch.complex64) if c["precision"] == "mixed" else u


def work(case):
    """Bytes: every cycle has to read the iterate and the right-hand side of the
    finest level once and write the iterate once (the coarser levels are left
    out; a variable k^2 is read once more), in the cycle's precision.  A solve
    counts its cycles (about 9.4 n Jacobi cycles, 0.33 n GMRES-smoothed ones,
    0.45 n FGMRES iterations).  Flops: the stencil, the update and the
    transfers of one cycle, about 60 per point; a GMRES(3) step, about 130
    more, twice per cycle."""
    n, dim, B = case["n"], case["dim"], case["batch"]
    pts = float(n - 1) ** dim * B
    cb = 8 if case["precision"] == "mixed" else 16
    kb = 0 if case["medium"] == "const" else (4 if cb == 8 else 8)
    kpts = float(n - 1) ** dim
    if case["kind"] == "steps":
        # u, f and the coarse e in; v, fc, ec, w, A w, A^H w out
        return {"bytes": 16.0 * pts * (6 + 3 / 2.0 ** dim) + kb * kpts, "flops": 150.0 * pts}
    if case["kind"] == "cycles":
        cyc = case["cycles"]
    elif case["kind"] == "solve":
        cyc = 9.4 * n if case["smoother"] == "jacobi" else 0.35 * n
    elif case["kind"] == "fgmres":
        cyc = 0.45 * n
    else:
        cyc = 2 * 0.35 * n
    per = 60.0 if case["smoother"] == "jacobi" else 320.0
    return {"bytes": cyc * (3 * cb * pts + kb * kpts), "flops": cyc * per * pts}


# ---- the same in plain torch, complex128 -----------------------------------------

def _axis(n_l, a, b):
    """lo, dg, up of -D2 (three-point formula) on the scaled grid of n_l intervals."""
    x = torch.arange(n_l + 1, dtype=torch.float64, device="cuda") / n_l
    rot = complex(math.cos(ECS_ANGLE), math.sin(ECS_ANGLE))
    z = x.to(torch.complex128)
    z = torch.where(x < a, a + (x - a) * rot, z)
    z = torch.where(x > b, b + (x - b) * rot, z)
    h = z[1:] - z[:-1]
    hm, hp = h[:-1], h[1:]
    lo, up = 2.0 / ((hm + hp) * hm), 2.0 / ((hm + hp) * hp)
    return lo, lo + up, up


def _adjoint_axis(t):
    lo, dg, up = t
    l2, u2 = torch.zeros_like(lo), torch.zeros_like(up)
    l2[1:] = up[:-1].conj()
    u2[:-1] = lo[1:].conj()
    return l2, dg.conj(), u2


class _Level:
    def __init__(self, c, k2, l, adjoint=False):
        n_l = c["n"] >> l
        self.dim, self.N = c["dim"], n_l - 1
        t = _axis(n_l, c["lo"] / c["n"], 1.0 - c["hi"] / c["n"])
        self.t = _adjoint_axis(t) if adjoint else t
        th = l * THETA_MAX / math.log2(c["n"])
        self.beta = complex(math.cos(th), -math.sin(th) if adjoint else math.sin(th))
        self.k2 = k2
        d = -self.beta * (k2 if isinstance(k2, torch.Tensor) else
                          torch.full((self.N,) * self.dim, float(k2), dtype=torch.float64, device="cuda"))
        for ax in range(self.dim):
            d = d + self._along(self.t[1], ax)
        self.D = d

    def _along(self, v, ax):
        s = [1] * self.dim
        s[ax] = -1
        return v.reshape(s)

    def apply(self, u):
        y = self.D * u
        for ax in range(self.dim):
            d, N = ax + 1, self.N
            y.narrow(d, 1, N - 1).sub_(self._along(self.t[0], ax).narrow(ax, 1, N - 1) * u.narrow(d, 0, N - 1))
            y.narrow(d, 0, N - 1).sub_(self._along(self.t[2], ax).narrow(ax, 0, N - 1) * u.narrow(d, 1, N - 1))
        return y

    def jacobi(self, u, f):
        return u + OMEGA * (f - self.apply(u)) / self.D

    def gmres(self, u, f, m=3):
        B = u.shape[0]
        dot = lambda a, b: (a.conj() * b).reshape(B, -1).sum(1)  # noqa: E731
        at = lambda s: s.reshape((B,) + (1,) * self.dim)         # noqa: E731
        r = f - self.apply(u)
        beta = dot(r, r).real.sqrt()
        V = [r / at(beta)]
        H = torch.zeros((B, m + 1, m), dtype=torch.complex128, device=u.device)
        for j in range(m):
            w = self.apply(V[j])
            for i in range(j + 1):
                H[:, i, j] = dot(V[i], w)
                w = w - at(H[:, i, j]) * V[i]
            nw = dot(w, w).real.sqrt()
            H[:, j + 1, j] = nw
            V.append(w / at(nw))
        q, R = torch.linalg.qr(H)
        y = torch.linalg.solve_triangular(R, (q[:, :1, :].conj().transpose(1, 2)) * beta.reshape(B, 1, 1), upper=True)
        return u + sum(at(y[:, j, 0]) * V[j] for j in range(m))


def _restrict(r):
    for d in range(1, r.dim()):
        nc = (r.shape[d] + 1) // 2 - 1
        i = 2 * torch.arange(nc, device=r.device)
        r = 0.25 * r.index_select(d, i) + 0.5 * r.index_select(d, i + 1) + 0.25 * r.index_select(d, i + 2)
    return r


def _prolong(e):
    for d in range(1, e.dim()):
        nc = e.shape[d]
        s = list(e.shape)
        s[d] = 2 * nc + 1
        out = torch.zeros(s, dtype=e.dtype, device=e.device)
        i = torch.arange(nc, device=e.device)
        out.index_add_(d, 2 * i + 1, e)
        out.index_add_(d, 2 * i, 0.5 * e)
        out.index_add_(d, 2 * i + 2, 0.5 * e)
        e = out
    return e


def _vcycle(levels, sm, l, u, f):
    L = levels[l]
    if l == len(levels) - 1:                  # 3 points per axis: dense solve
        m = L.N ** L.dim
        eye = torch.eye(m, dtype=torch.complex128, device=f.device).reshape((m,) + (L.N,) * L.dim)
        A = L.apply(eye).reshape(m, m).T
        return torch.linalg.solve(A, f.reshape(-1, m).T).T.reshape(f.shape)
    u = getattr(L, sm)(u, f)
    fc = _restrict(f - L.apply(u))
    u = u + _prolong(_vcycle(levels, sm, l + 1, torch.zeros_like(fc), fc))
    return getattr(L, sm)(u, f)


def _direct(c, k2, f, adjoint=False):
    """A_0^{-1} f (or A_0^{-H} f) in 2-D: block elimination over the grid rows."""
    L = _Level(c, k2, 0, adjoint)
    N, (lo, _, up) = L.N, L.t
    T = torch.diag_embed(-lo[1:], -1) + torch.diag_embed(-up[:-1], 1)
    inv, g, y = [], [], None
    for j in range(N):
        S = T + torch.diag_embed(L.D[j])
        fj = f[:, j, :].T
        if j:
            S = S - (lo[j] * up[j - 1]) * inv[-1]
            fj = fj + lo[j] * y
        inv.append(torch.linalg.inv(S))
        y = inv[-1] @ fj
        g.append(y)
    u = torch.empty_like(f)
    x = g[-1]
    u[:, N - 1, :] = x.T
    for j in range(N - 2, -1, -1):
        x = g[j] + up[j] * (inv[j] @ x)
        u[:, j, :] = x.T
    return u


def exact(case, seed):
    c = case
    k2, f, u = _inputs(c, seed)
    n, dim = c["n"], c["dim"]
    if c["kind"] in ("solve", "fgmres", "gradient"):
        if dim != 2 or n > 512:
            return None
        if c["kind"] != "gradient":
            return _direct(c, k2, f, c["adjoint"])
        g = _gen(seed + 77, f.device)
        data = _randn((c["batch"], n - 1), g, f.device) / n ** 2
        u = _direct(c, k2, f)
        row = n - c["hi"] - 2
        gu = torch.zeros_like(u)
        gu[:, row, :] = u[:, row, :] - data
        lam = _direct(c, k2, gu, True)
        return u, (lam.conj() * u).real.sum(0), lam
    if c["kind"] == "steps":
        g = _gen(seed + 77, f.device)
        e = _randn((c["batch"],) + (n // 2 - 1,) * dim, g, f.device) / n ** 2
        inj = (slice(1, None, 2),) * dim
        L0 = _Level(c, k2, 0)
        L1 = _Level(c, k2[inj] if isinstance(k2, torch.Tensor) else k2, 1)
        v = L0.jacobi(u, f)
        fc = _restrict(f - L0.apply(v))
        ec = L1.jacobi(e, fc)
        w = L0.jacobi(v + _prolong(ec), f)
        return v, fc, ec, w, L0.apply(w), _Level(c, k2, 0, True).apply(w)
    levels, l = [], 0
    while True:
        levels.append(_Level(c, k2, l))
        if n >> l <= 4:
            break
        if isinstance(k2, torch.Tensor):
            k2 = k2[(slice(1, None, 2),) * dim]
        l += 1
    for _ in range(c["cycles"]):
        u = _vcycle(levels, c["smoother"], 0, u, f)
    return u
