"""The measured cases: the calls that a stability analysis makes, from one J v on the smallest layer to whole
solves, each through the package's public entry points.

Kinds:
  jv      Stab.apply_J: the linearised operator of one problem, the call under every Krylov step.  Base flows that
          vary in y only (parallel shear layers) and general ones, 2-D and 3-D, the epsilon-quotient (default) and
          the exact tangent, viscous and inviscid, uniform and stretched y.
  ortho   Stab.orthogonalize: one Arnoldi orthogonalisation (CGS2) against k vectors, with its coefficients and norm.
  batch   JvBatch.apply: J v of many uneven layers at once.
  solve   Stab.solve: (J - sigma I) x = b by preconditioned flexible GMRES, run to 1e-12 so that x is determined.
  lock    JvBatch.solve: the same for several uneven layers in lockstep.
  eigs    Stab.eigs: the whole Cayley-transformed IRAM.

``exact`` restates the operator in plain torch (dense derivative matrices, difference numbers in 64 bits).
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_1502_03701_gb300 import JvBatch, Stab

GAMMA = 1.4
PR = 0.71
SUTHERLAND = 110.4 / 273.15
LX = 2.0 * math.pi / 0.4  # the layer's streamwise (and spanwise) length
LY = (-15.0, 15.0)
SHIFT = -1.0 + 0.2j       # a Cayley zero tau: J v - tau v is the right-hand side of every Cayley solve


def _layer(kind, name, nx, ny, nz=1, **kw):
    c = dict(kind=kind, name=name, nx=nx, ny=ny, nz=nz, Ma=0.3, Re=1000.0, stretch=0.0, base="layer", tangent=False,
             tune=True)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest production layer (8,192 unknowns): launch latency of the operator's phases
        _layer("jv", "jv_32x64", 32, 64),
        # the two-dimensional production layer (524,288 unknowns), the operator of its inner solves
        _layer("jv", "jv_256x512", 256, 512, tangent=True),
        # odd sizes, a y grid clustered at the layer, epsilon-quotient, launch shapes left at their defaults
        _layer("jv", "jv_190x301_stretched", 190, 301, Ma=0.6, Re=500.0, stretch=1.7, tune=False),
        # a base state that varies in x and y (non-parallel flow): base tables per grid point
        _layer("jv", "jv_128x256_nonparallel", 128, 256, Ma=0.5, base="general"),
        # odd three-dimensional sizes, exact tangent, default launch shapes
        _layer("jv", "jv_60x90x28", 60, 90, 28, Ma=0.5, Re=800.0, tangent=True, tune=False),
        # the largest layer (10,485,760 unknowns), epsilon-quotient: the headline operator
        _layer("jv", "jv_128x256x64", 128, 256, 64),
        # one Arnoldi step's orthogonalisation on the small layer: latency, and the coefficients read on the host
        _layer("ortho", "cgs2_32x64_k29", 32, 64, k=29),
        # the same on the two-dimensional production layer near the end of an ncv = 60 cycle
        _layer("ortho", "cgs2_256x512_k55", 256, 512, k=55),
        # a fleet of uneven layers (Nx 32..256, Ny 64..512), one launch per phase
        dict(kind="batch", name="jv_batch_32_uneven", count=32, pick=1234),
        # an inner solve of the Cayley operator with the reduced-operator block-Jacobi preconditioner
        _layer("solve", "solve_128x256_reduced", 128, 256, tangent=True, precond=2, tx=8, ty=64, m=50, lgmres=0,
               sigma=1.0),
        # a small solve with exact FP32 block inverses: many short launches per iteration
        _layer("solve", "solve_32x64_block_jacobi", 32, 64, tangent=True, precond=1, tx=16, ty=16, m=30, lgmres=0,
               sigma=1.0),
        # the leading eigenvalue pair of a small layer of a fleet: the whole method
        _layer("eigs", "eigs_16x32", 16, 32, tangent=True, precond=1, tx=16, ty=16, m=30, lgmres=0, sigma=0.25, nev=2,
               ncv=12),
    ]


def draw(rng):
    def log(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    ma, re = round(rng.uniform(0.2, 0.9), 3), round(math.exp(rng.uniform(math.log(500.0), math.log(5000.0))), 1)
    pick = rng.random()
    flow = dict(Ma=ma, Re=re, tune=rng.random() < 0.3, stretch=rng.choice([0.0, 0.0, 1.2, 1.7]))
    if pick < 0.35:
        base = "general" if rng.random() < 0.25 else "layer"
        nx, ny = log(24, 300), log(40, 600)
        if rng.random() < 0.2:
            flow["Re"] = 0.0  # inviscid
        return _layer("jv", "", nx, ny, base=base, tangent=rng.random() < 0.5, **flow)
    if pick < 0.6:
        return _layer("jv", "", log(16, 128), log(24, 256), log(8, 64), tangent=rng.random() < 0.5, **flow)
    if pick < 0.78:
        return _layer("ortho", "", log(32, 256), log(64, 512), k=log(1, 60), **flow)
    if pick < 0.88:
        return dict(kind="batch", count=log(4, 32), pick=rng.randrange(1 << 20))
    if pick < 0.95:
        return _layer("solve", "", 8 * rng.randint(4, 12), 32 * rng.randint(2, 5), tangent=True,
                      precond=rng.choice([1, 2]), tx=8, ty=32, m=rng.choice([30, 50]), lgmres=0, sigma=1.0, Ma=ma,
                      Re=re, tune=False)
    return dict(kind="lock", count=rng.randint(3, 8), pick=rng.randrange(1 << 20), sigma=1.0)


# ---------------------------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------------------------
def _grid(c):
    dim = 3 if c["nz"] > 1 else 2
    return SimpleNamespace(dim=dim, nx=c["nx"], ny=c["ny"], nz=c["nz"], lx=LX, ly0=LY[0], ly1=LY[1],
                           lz=LX if dim == 3 else 1.0, stretch=c["stretch"], nv=dim + 2,
                           npts=c["nx"] * c["ny"] * c["nz"])


def _y(g):
    eta = np.arange(g.ny) / (g.ny - 1)
    if g.stretch == 0.0:
        return g.ly0 + (g.ly1 - g.ly0) * eta
    return 0.5 * (g.ly0 + g.ly1) + 0.5 * (g.ly1 - g.ly0) * np.sinh(g.stretch * (2 * eta - 1)) / math.sinh(g.stretch)


def _base(c, g):
    """The tanh mixing layer; base = "general": with a wave in x that grows and turns the layer."""
    q = np.zeros((g.nv, g.nz, g.ny, g.nx))
    q[0] = 1.0 / (GAMMA * c["Ma"] ** 2)
    y = _y(g)
    q[1] = np.tanh(y)[None, :, None]
    if c["base"] == "general":
        x = np.arange(g.nx) * (g.lx / g.nx)
        wave = np.exp(-0.1 * y ** 2)[None, :, None]
        kx = 2.0 * math.pi / g.lx
        q[1] += 0.02 * np.sin(kx * x)[None, None, :] * wave
        q[2] += 0.03 * np.cos(kx * x)[None, None, :] * wave
        q[0] *= 1.0 + 0.01 * np.cos(2 * kx * x)[None, None, :] * wave
        q[-1] += 0.01 * np.sin(2 * kx * x)[None, None, :] * wave
    return q


def _krylov(g, gen):
    """A unit vector as a Krylov basis holds them: a rough part over the grid and a part that follows the layer."""
    rough = torch.randn(g.nv, g.nz, g.ny, g.nx, 2, dtype=torch.float64, device="cuda", generator=gen)
    y = torch.from_numpy(_y(g)).cuda()
    v = torch.view_as_complex(rough) * (0.3 + torch.exp(-0.4 * y.abs()))[None, None, :, None]
    v = v.reshape(-1)
    return v / torch.linalg.vector_norm(v)


def _opts(c):
    o = dict(eps_mode=2 if c["tangent"] else 0)
    if c["kind"] in ("solve", "eigs"):
        o.update(precond=c["precond"], tile=(c["tx"], c["ty"]), precond_prec=32, gmres_m=c["m"], lgmres_k=c["lgmres"],
                 gmres_tol=1e-12, gmres_max_restarts=400)
    return o


def _problem(c, **more):
    g = _grid(c)
    s = Stab(_base(c, g), g, c["Ma"], c["Re"], PR, **{**_opts(c), **more})
    if c["tune"]:
        s.autotune()
    return s, g


def _members(c):
    """The uneven layers of a fleet: sizes from the sets, Ma uniform in [0.1, 0.9], Re log-uniform in [500, 5000]."""
    r = np.random.RandomState(c["pick"])
    nxs, nys = ((32, 64, 128, 256), (64, 128, 256, 512)) if c["kind"] == "batch" else ((16, 32, 48), (32, 64))
    out = []
    for _ in range(c["count"]):
        out.append(_layer("jv", "", int(r.choice(nxs)), int(r.choice(nys)),
                          Ma=float(r.uniform(0.1 if c["kind"] == "batch" else 0.3, 0.9)),
                          Re=float(np.exp(r.uniform(np.log(500.0), np.log(5000.0)))), tangent=c["kind"] == "lock",
                          tune=False))
    return out


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    kind = case["kind"]
    if kind in ("batch", "lock"):
        members = _members(case)
        more = {} if kind == "batch" else dict(precond=1, tile=(16, 16), precond_prec=32, gmres_m=30, gmres_tol=1e-12,
                                               gmres_max_restarts=400)
        made = [_problem(m, **more) for m in members]
        vs = [_krylov(g, gen) for _, g in made]
        if kind == "lock":
            for s, _ in made:
                s.precond_build(case["sigma"])
        b = JvBatch([s for s, _ in made])
        return dict(kind=kind, batch=b, v=vs, out=[torch.empty_like(v) for v in vs],
                    arg=[SHIFT if kind == "batch" else case["sigma"]] * len(vs))
    s, g = _problem(case)
    v = _krylov(g, gen)
    st = dict(kind=kind, s=s, v=v, out=torch.zeros_like(v))
    if kind == "ortho":
        k = case["k"]
        a = torch.view_as_complex(torch.randn(v.numel(), k, 2, dtype=torch.float64, device="cuda", generator=gen))
        for _ in range(2):  # Cholesky QR twice: orthonormal to working precision
            low = torch.linalg.cholesky(a.mH @ a)
            a = torch.linalg.solve_triangular(low.mH, a, upper=True, left=False)
        st["V"] = a.T.contiguous()  # column j contiguous
    elif kind in ("solve", "eigs"):
        s.precond_build(case["sigma"])
        st["sigma"] = case["sigma"]
        if kind == "eigs":
            st.update(nev=case["nev"], ncv=case["ncv"])
    return st


def run(state):
    kind = state["kind"]
    if kind == "jv":
        return state["s"].apply_J(state["v"], state["out"], SHIFT)
    if kind == "ortho":
        w = state["out"]
        w.copy_(state["v"])  # the vector that the step orthogonalises in place
        h, norm = state["s"].orthogonalize(state["V"], state["V"].shape[0], w)
        return {"w": w, "h": h, "norm": norm}
    if kind == "batch":
        return state["batch"].apply(state["v"], state["out"], state["arg"])
    if kind == "solve":
        state["s"].solve(state["sigma"], state["v"], state["out"])
        return state["out"]
    if kind == "lock":
        state["batch"].solve(state["arg"], state["v"], state["out"])
        return state["out"]
    r = state["s"].eigs(state["sigma"], -1.0, state["nev"], state["ncv"], 1e-11, v0=state["v"])
    return r.lam


def work(case):
    """J v: each unknown read and written once (32 bytes; a general base state is read too), and per derivative value
    the 10 (first) or 14 (second) operations of its compact scheme plus two per term of the pointwise map.  CGS2:
    the basis read once, the vector read and written.  Solves: the operator and the basis once per Krylov vector of
    one cycle, the least that a Krylov solve does."""
    kind = case["kind"]
    if kind in ("batch", "lock"):
        ws = [work(m) for m in _members(case)]
        scale = 1 if kind == "batch" else 30
        return {k: scale * sum(w[k] for w in ws) for k in ("bytes", "flops")}
    g = _grid(case)
    d, n = g.dim, g.nv * g.npts
    visc = case["Re"] > 0
    first = d * (d + 3) + d * (d - 1) if visc else d * (d + 2)
    second = d * (d + 1) if visc else 0
    flops = 2.0 * g.npts * (10 * first + 14 * second + 2 * g.nv * (first + second))
    byts = 32.0 * n + (8.0 * n if case["base"] == "general" else 0.0)
    if kind == "ortho":
        return {"bytes": 16.0 * n * (case["k"] + 2), "flops": 32.0 * n * case["k"]}
    if kind in ("solve", "eigs"):
        m = case["m"] if kind == "solve" else case["ncv"]
        return {"bytes": m * (byts + 16.0 * n), "flops": m * flops}
    return {"bytes": byts, "flops": flops}


# ---------------------------------------------------------------------------------------------------------------
# 64-bit restatement of the operator
# ---------------------------------------------------------------------------------------------------------------
class _D:
    """A difference number: base value a and w = (perturbed - base) / e."""
    __slots__ = ("a", "w", "e")

    def __init__(self, a, w, e):
        self.a, self.w, self.e = a, w, e

    def _of(self, o):
        return o if isinstance(o, _D) else _D(o, 0.0, self.e)

    def __add__(self, o):
        o = self._of(o)
        return _D(self.a + o.a, self.w + o.w, self.e)

    __radd__ = __add__

    def __neg__(self):
        return _D(-self.a, -self.w, self.e)

    def __sub__(self, o):
        return self + (-self._of(o))

    def __mul__(self, o):
        if not isinstance(o, _D):
            return _D(self.a * o, self.w * o, self.e)
        return _D(self.a * o.a, self.a * o.w + self.w * (o.a + self.e * o.w), self.e)

    __rmul__ = __mul__

    def inv(self):
        return _D(1.0 / self.a, -self.w / (self.a * (self.a + self.e * self.w)), self.e)

    def sqrt(self):
        r = torch.sqrt(self.a)
        return _D(r, self.w / (r + torch.sqrt(self.a + self.e * self.w)), self.e)

    def log(self):
        q = self.w / self.a
        return _D(torch.log(self.a), torch.log1p(self.e * q) / self.e if self.e else q, self.e)

    def exp(self):
        r = torch.exp(self.a)
        return _D(r, r * (torch.expm1(self.e * self.w) / self.e if self.e else self.w), self.e)


def _matrices(n, h, periodic):
    """Dense first- and second-derivative matrices of the sixth-order compact schemes."""
    out = []
    for order in (1, 2):
        al = 1.0 / 3.0 if order == 1 else 2.0 / 11.0
        a, b = np.eye(n), np.zeros((n, n))
        for t in range(n):
            if periodic or 2 <= t <= n - 3:
                for s in (-1, 1):
                    a[t, (t + s) % n] += al
                    if order == 1:
                        b[t, (t + s) % n] += s * 14.0 / 9.0 / (2 * h)
                        b[t, (t + 2 * s) % n] += s / 9.0 / (4 * h)
                    else:
                        b[t, (t + s) % n] += 12.0 / 11.0 / h ** 2
                        b[t, (t + 2 * s) % n] += 3.0 / 11.0 / (4 * h ** 2)
                if order == 2:
                    b[t, t] -= 2 * (12.0 / 11.0 + 3.0 / 44.0) / h ** 2
            elif t in (0, n - 1):
                s = 1 if t == 0 else -1
                a[t, t + s] = 2.0 if order == 1 else 11.0
                w = (-2.5 * s, 2.0 * s, 0.5 * s) if order == 1 else (13.0, -27.0, 15.0, -1.0)
                for k, x in enumerate(w):
                    b[t, t + k * s] += x / h ** order
            else:
                for s in (-1, 1):
                    a[t, t + s] = 0.25 if order == 1 else 0.1
                    b[t, t + s] += s * 0.75 / h if order == 1 else 1.2 / h ** 2
                if order == 2:
                    b[t, t] -= 2.4 / h ** 2
        out.append(torch.from_numpy(np.linalg.solve(a, b)).cuda())
    return out


class _Operator:
    def __init__(self, c):
        self.c, self.g = c, _grid(c)
        g = self.g
        self.q0 = torch.from_numpy(_base(c, g)).cuda()
        self.m = [_matrices(g.nx, g.lx / g.nx, True), _matrices(g.ny, 1.0 / (g.ny - 1), False)]
        if g.dim == 3:
            self.m.append(_matrices(g.nz, g.lz / g.nz, True))
        eta, be = np.arange(g.ny) / (g.ny - 1), g.stretch
        if be == 0.0:
            yp, ypp = np.full(g.ny, g.ly1 - g.ly0), np.zeros(g.ny)
        else:
            f = 0.5 * (g.ly1 - g.ly0) / math.sinh(be)
            yp = f * 2 * be * np.cosh(be * (2 * eta - 1))
            ypp = f * 4 * be * be * np.sinh(be * (2 * eta - 1))
        self.ey = torch.from_numpy(1.0 / yp).cuda()[None, :, None]
        self.eyy = torch.from_numpy(-ypp / yp ** 3).cuda()[None, :, None]
        self.R = 1.0 / (GAMMA * c["Ma"] ** 2)
        self.cp = GAMMA * self.R / (GAMMA - 1.0)

    def _raw(self, f, ax, order):
        m = self.m[ax][order - 1]
        if ax == 0:
            return f @ m.T
        if ax == 1:
            return m @ f
        return (m @ f.reshape(f.shape[0], -1)).reshape(f.shape)

    def _d(self, f, ax):
        one = self._raw
        s = self.ey if ax == 1 else 1.0
        return _D(one(f.a, ax, 1) * s, one(f.w, ax, 1) * s, f.e)

    def _dd(self, f, ax):
        def two(x):
            y = self._raw(x, ax, 2)
            return y * self.ey ** 2 + self._raw(x, 1, 1) * self.eyy if ax == 1 else y
        return _D(two(f.a), two(f.w), f.e)

    def _mixed(self, f, i, k):
        a, b = (k, i) if k == 1 or (k == 2 and i == 0) else (i, k)  # y first, then z, then x
        return self._d(self._d(f, a), b)

    def quotient(self, w, e):
        """[N(q0 + e w) - N(q0)] / e for a real direction w, shape [var][z][y][x]."""
        c, g, D = self.c, self.g, self.g.dim
        q = [_D(self.q0[a], w[a], e) for a in range(g.nv)]
        p, u, s = q[0], q[1:1 + D], q[-1]
        lp = (p * (1.0 / self.R)).log()
        rho = (lp * (1.0 / GAMMA) - s * (1.0 / self.cp)).exp()
        irho = rho.inv()
        dp = [self._d(p, a) for a in range(D)]
        ds = [self._d(s, a) for a in range(D)]
        du = [[self._d(u[b], a) for a in range(D)] for b in range(D)]  # du[b][a] = d u_b / d x_a
        div = sum((du[a][a] for a in range(1, D)), du[0][0])
        vis = [None] * D
        src = None
        if c["Re"] > 0:
            T = p * irho * (1.0 / self.R)
            # T's difference without the rounding of the quotient: its own exponential form
            T = _D(T.a, ((lp * (1 - 1.0 / GAMMA) + s * (1.0 / self.cp)).exp()).w, e)
            dT = [self._d(T, a) for a in range(D)]
            mu = T * T.sqrt() * (T + SUTHERLAND).inv() * ((1.0 + SUTHERLAND) / c["Re"])
            dmu = mu * (T.inv() * 1.5 - (T + SUTHERLAND).inv())
            kl = self.cp / PR
            lap = sum((self._dd(T, a) for a in range(1, D)), self._dd(T, 0))
            g2 = sum((dT[a] * dT[a] for a in range(1, D)), dT[0] * dT[0])
            src = (mu * lap + dmu * g2) * kl
            ss = None
            for a in range(D):
                for b in range(D):
                    sij = (du[a][b] + du[b][a]) * 0.5
                    ss = sij * sij if ss is None else ss + sij * sij
            src = src + mu * (ss - div * div * (1.0 / 3.0)) * 2.0
            for a in range(D):
                lapu, grad, cross = None, None, None
                for b in range(D):
                    d2 = self._dd(u[a], b)
                    lapu = d2 if lapu is None else lapu + d2
                    m = d2 if a == b else self._mixed(u[b], a, b)
                    grad = m if grad is None else grad + m
                    x = dT[b] * (du[a][b] + du[b][a])
                    cross = x if cross is None else cross + x
                vis[a] = mu * (lapu + grad * (1.0 / 3.0)) + dmu * cross + dmu * dT[a] * div * (-2.0 / 3.0)
        Yp = -(u[1] * dp[1] + p * du[1][1] * GAMMA)
        Yv = -(u[1] * du[1][1] + dp[1] * irho)
        # non-reflective rows: incoming wave amplitudes of the base state removed
        cs = (p * irho * GAMMA).sqrt()
        rc = rho * cs
        rcv = rc * du[1][1]
        Xp, Xm = (u[1] + cs) * (dp[1] + rcv) * 0.5, (u[1] - cs) * (dp[1] - rcv) * 0.5
        v0, c0 = self.q0[2], cs.a
        sign = torch.zeros(1, g.ny, 1, device="cuda", dtype=torch.float64)
        sign[:, 0], sign[:, -1] = 1.0, -1.0
        row = sign != 0
        keep_p = (~((v0 + c0) * sign > 0)).double()
        keep_m = (~((v0 - c0) * sign > 0)).double()
        drop = (v0 * sign > 0)
        Xp, Xm = Xp * keep_p, Xm * keep_m
        Bp, Bv = -(Xp + Xm), -((Xp - Xm) * rc.inv())

        def pick(at, x, y):
            return _D(torch.where(at, x.a, y.a), torch.where(at, x.w, y.w), e)
        Yp, Yv = pick(row, Bp, Yp), pick(row, Bv, Yv)
        convy = (~drop).double()
        out = []
        pt = Yp
        for a in range(D):
            if a != 1:
                pt = pt - (u[a] * dp[a] + p * du[a][a] * GAMMA)
        out.append(pt + src * (GAMMA - 1.0) if src is not None else pt)
        for b in range(D):
            r = Yv if b == 1 else -(dp[b] * irho)
            for a in range(D):
                if a == 1 and b == 1:
                    continue
                t = u[a] * du[b][a]
                r = r - (t * convy if a == 1 else t)
            out.append(r + vis[b] * irho if vis[b] is not None else r)
        st = None
        for a in range(D):
            t = u[a] * ds[a]
            t = -(t * convy) if a == 1 else -t
            st = t if st is None else st + t
        out.append(st + p.inv() * self.R * src if src is not None else st)
        return torch.stack([o.w for o in out])

    def apply(self, v, shift):
        g = self.g
        e = 0.0
        if not self.c["tangent"]:
            nv = float(torch.linalg.vector_norm(v))
            e = 2.0 ** -26 * (1.0 + float(torch.linalg.vector_norm(self.q0))) / nv
        w = v.reshape(g.nv, g.nz, g.ny, g.nx)
        r = torch.complex(self.quotient(w.real.contiguous(), e), self.quotient(w.imag.contiguous(), e))
        return r.reshape(-1) - shift * v


def exact(case, seed):
    kind = case["kind"]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    if kind == "jv":
        return _Operator(case).apply(_krylov(_grid(case), gen), SHIFT)
    if kind == "batch":
        members = _members(case)
        vs = [_krylov(_grid(m), gen) for m in members]
        return [_Operator(m).apply(v, SHIFT) for m, v in zip(members, vs)]
    if kind == "ortho":
        st = prepare(case, seed)
        V, w = st["V"], st["v"].clone()
        h = torch.zeros(V.shape[0], dtype=torch.complex128, device="cuda")
        for _ in range(2):
            t = V.conj() @ w
            w = w - V.T @ t
            h = h + t
        return {"w": w, "h": h, "norm": torch.linalg.vector_norm(w)}
    if kind == "solve":
        g = _grid(case)
        n = g.nv * g.npts
        if n > 9000:
            return None  # a dense solve of this size takes too long
        op = _Operator(case)
        a = torch.empty(n, n, dtype=torch.float64, device="cuda")
        for i in range(n):
            e = torch.zeros(g.nv, g.nz, g.ny, g.nx, dtype=torch.float64, device="cuda")
            e.view(-1)[i] = 1.0
            a[:, i] = op.quotient(e, 0.0).reshape(-1)
        a.diagonal().sub_(case["sigma"])
        b = _krylov(g, gen)
        x = torch.linalg.solve(a, torch.stack([b.real, b.imag], 1))
        return torch.complex(x[:, 0].contiguous(), x[:, 1].contiguous())
    return None
