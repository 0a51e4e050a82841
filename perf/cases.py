"""Timed cases: the calls of one design iteration of a topology-optimisation run, through the
package's public entry points (``nc.Problem``).

A run of the optimisation loop (``optimize.py``) filters the design, solves the state by Newton,
evaluates the objective, solves the adjoint, forms the element sensitivities and updates the
design; inside the solves the work is residuals, Jacobian products (FP32 inside mixed solves,
FP64 from the linearisation store or an assembled Jacobian in FP64 solves) and the Krylov
orthogonalisation.  Each of these is a case of its own here; two cases are whole solves.

Grids are those of the package's workloads and tests: 12^3 (the smallest cavity), 100x40x30
(ragged), 64^3, 96^3, 128^3, the quarter cavity 80x80x160 and the benchmark's 192x192x384.
States are random with the Dirichlet values imposed (u ~ N(0, 0.5^2), p ~ N(0, 50^2), T ~ N(0, 1),
as in the parity tests); designs are smoothed random fields in the design column.

``exact`` restates the operators in plain FP64 torch (whole-element arrays, forward- and
reverse-mode differentiation of the element residual), the density filter by fast diagonalisation
of its tensor-product matrices, MMA by its defining formulas.
"""
import math

import torch

from paper_1508_04596_gb300 import nc

DEV = "cuda"
DT = {"f64": torch.float64, "f32": torch.float32}
CAVITY = dict(Pr=0.71, alpha_max=1e4, q_alpha=1.0, q_f=1.0, Ck=0.1)
QUARTER = dict(Pr=1.0, alpha_max=1e5, q_alpha=8.0, q_f=0.881, Ck=1e-2)
# flop per element of the operators (one +, -, x, / or reciprocal square root = 1 flop, FMA = 2)
FLOP = dict(residual=1794, jvp=3076, jtvp=3196, sens=1796, linearize=848, jvp_lin=2214,
            jtvp_lin=2382)


def listed():
    return [
        # Newton's residual on the smallest cavity: a call that launches and latency bound
        dict(name="residual f64 12^3", kind="residual", nx=12, ny=12, nz=12, dtype="f64",
             bcs="cavity"),
        # a multigrid-level product on a ragged mid-size grid
        dict(name="jvp f32 100x40x30", kind="jvp", nx=100, ny=40, nz=30, dtype="f32",
             bcs="cavity"),
        # the FGMRES product of a mixed state solve at the benchmark's size
        dict(name="jvp f32 192x192x384", kind="jvp", nx=192, ny=192, nz=384, dtype="f32",
             bcs="flux"),
        # the adjoint solve's product on the quarter cavity with its heat source
        dict(name="jtvp f32 80x80x160", kind="jtvp", nx=80, ny=80, nz=160, dtype="f32",
             bcs="quarter"),
        # an FP64 Krylov solve: one linearisation, 16 products from its store
        dict(name="jvp_lin f64 64^3 x16", kind="lin", nx=64, ny=64, nz=64, dtype="f64",
             bcs="cavity", products=16, transpose=False),
        # the same with an assembled Jacobian: build it, then 16 products
        dict(name="assembled f64 64^3 x16", kind="assembled", nx=64, ny=64, nz=64, dtype="f64",
             bcs="cavity", products=16, transpose=False),
        # objective and element sensitivities of the flux-heated cavity
        dict(name="sensitivity f64 96^3", kind="sens", nx=96, ny=96, nz=96, dtype="f64",
             bcs="flux"),
        # one orthogonalisation step of FGMRES on the 128^3 cavity's vectors, 10 columns in
        dict(name="arnoldi f64 10.7M k10", kind="arnoldi", n=5 * 129 ** 3, k=10, dtype="f64"),
        # the density filter of the quarter cavity, radius 2.5 h
        dict(name="filter 80x80x160", kind="filter", nx=80, ny=80, nz=160, radius=2.5),
        # volume constraint and MMA update of the quarter cavity's design
        dict(name="mma 80x80x160", kind="mma", nx=80, ny=80, nz=160, it=5),
        # the mixed Newton solve of the next design from the previous one's state
        dict(name="state mixed 64^3", kind="state", nx=64, ny=64, nz=64, Gr=1e4),
        # the gradient of a design: objective, mixed adjoint solve, sensitivities
        dict(name="gradient mixed 96^3", kind="gradient", nx=96, ny=96, nz=96, Gr=1e5),
    ]


def _odd(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _grid(rng, emin, emax):
    """A grid of emin..emax elements (log-uniform) with aspect ratios of up to about 2."""
    e = math.exp(rng.uniform(math.log(emin), math.log(emax)))
    a, b = rng.uniform(0.6, 1.6), rng.uniform(0.6, 1.6)
    nx = max(3, int((e / (a * b)) ** (1 / 3)))
    ny = max(3, int(nx * a))
    return nx, ny, max(3, min(int(nx * b), int(emax // (nx * ny))))


def draw(rng):
    kind = rng.choice(["residual", "jvp", "jtvp", "lin", "assembled", "sens", "arnoldi", "filter",
                       "mma", "gradient", "state"])
    if kind == "arnoldi":
        return dict(kind=kind, n=_odd(rng, 5e4, 10.7e6), k=rng.randint(1, 20),
                    dtype=rng.choice(["f64", "f32"]))
    if kind in ("gradient", "state"):  # grids that the multigrid hierarchy halves several times
        n = rng.choice([32, 48, 64, 80])
        return dict(kind=kind, nx=n, ny=n, nz=rng.choice([n, n + 16]),
                    Gr=round(10 ** rng.uniform(3, 5), 1))
    lim = dict(residual=2.0e6, jvp=14e6, jtvp=4e6, lin=2.5e5, assembled=2.5e5, sens=8e5,
               filter=1.0e6, mma=1.0e6)[kind]
    nx, ny, nz = _grid(rng, 5e2 if kind in ("residual", "jvp", "jtvp") else 1e4, lim)
    c = dict(kind=kind, nx=nx, ny=ny, nz=nz)
    if kind == "filter":
        return dict(c, radius=round(rng.uniform(1.5, 4.0), 2))
    if kind == "mma":
        return dict(c, it=rng.randint(0, 20))
    c["bcs"] = rng.choice(["cavity", "flux", "quarter"])
    c["dtype"] = "f64"
    if kind in ("jvp", "jtvp", "residual") and nx * ny * nz * (1 if kind != "residual" else 4) > 2e6:
        c["dtype"] = "f32"
    elif kind in ("jvp", "jtvp", "residual", "assembled"):
        c["dtype"] = rng.choice(["f32", "f64"])
    if kind in ("lin", "assembled"):
        c.update(products=rng.choice([4, 8, 16]), transpose=rng.random() < 0.4)
    if kind == "sens" and c["bcs"] == "cavity":
        c["bcs"] = "flux"
    return c


# ---------------------------------------------------------------- inputs
class _Spec:
    """Geometry, coefficients and boundary data of a case in plain torch."""

    def __init__(self, case):
        nx, ny, nz = self.n = case["nx"], case["ny"], case["nz"]
        self.bcs = case.get("bcs", "flux")
        quarter = self.bcs == "quarter"
        self.h = 1.0 / nz if quarter else 1.0 / nx
        self.Gr = case.get("Gr", 1e5)
        self.mat = QUARTER if quarter else CAVITY
        self.Nn, self.E = (nx + 1) * (ny + 1) * (nz + 1), nx * ny * nz
        self.pin = (nx + 1) * (ny + 1) * nz if quarter else -1
        self.px = self._range(nx)
        self.py = self._range(ny)

    def _range(self, m):
        """Patch node range [lo, hi] of one direction: the middle third, closed."""
        L, tol = m * self.h, 1e-12 * max(self.n) * self.h
        on = [i for i in range(m + 1) if L / 3 - tol <= i * self.h <= 2 * L / 3 + tol]
        return (on[0], on[-1]) if on else (0, -1)

    def has_patch(self):
        return self.px[1] >= self.px[0] and self.py[1] >= self.py[0]

    def problem(self):
        p = nc.make_params(*self.n, self.h, self.Gr, **self.mat)
        if self.bcs == "quarter":
            b = nc.quarter_bcs(*self.n)
        else:
            b = nc.cavity_bcs(nc.PATCH_FLUX if self.bcs == "flux" else nc.PATCH_DIRICHLET, 1.0)
        prob = nc.Problem(p, b)
        if self.bcs == "quarter":
            prob.set_source(self.source())
        return prob

    def centroids(self):
        ax = [(torch.arange(m, dtype=torch.float64, device=DEV) + 0.5) * self.h for m in self.n]
        return ax[0][None, None, :], ax[1][None, :, None], ax[2][:, None, None]

    def regions(self):
        """(source block, design elements) as [nz, ny, nx] masks."""
        x, y, z = self.centroids()
        nx, ny, nz = self.n
        Lx, Ly, Lz = nx * self.h, ny * self.h, nz * self.h
        if self.bcs == "quarter":
            src = (x >= Lx - 0.05) & (y >= Ly - 0.05) & (z <= 0.05)
            des = (x >= Lx - 0.375) & (y >= Ly - 0.375) & (z > 0.05) & (z <= 0.8)
        else:
            des = ((x >= 0.25 * Lx) & (x <= 0.75 * Lx) & (y >= 0.25 * Ly) & (y <= 0.75 * Ly)
                   & (z <= 0.75 * Lz))
            src = torch.zeros_like(des)
        return src, des

    def source(self):
        return (1e4 * self.regions()[0].double()).reshape(-1).contiguous()

    def dirichlet(self):
        """Mask [5, nz+1, ny+1, nx+1] and the temperature values."""
        nx, ny, nz = self.n
        m = torch.zeros((5, nz + 1, ny + 1, nx + 1), dtype=torch.bool, device=DEV)
        T = torch.zeros((nz + 1, ny + 1, nx + 1), dtype=torch.float64, device=DEV)
        if self.bcs == "quarter":
            for q in (m[0:3, :, :, 0], m[0:3, :, 0, :], m[0:3, 0], m[0:3, nz]):
                q[...] = True
            m[0, :, :, nx] = True
            m[1, :, ny, :] = True
            for q in (m[4, :, :, 0], m[4, :, 0, :], m[4, nz]):
                q[...] = True
            m[3].view(-1)[self.pin] = True
            return m, T
        for q in (m[0:3, :, :, 0], m[0:3, :, :, nx], m[0:3, :, 0, :], m[0:3, :, ny, :], m[0:3, 0]):
            q[...] = True
        if self.bcs == "cavity" and self.has_patch():
            box = (0, slice(self.py[0], self.py[1] + 1), slice(self.px[0], self.px[1] + 1))
            m[(4,) + box] = True
            T[box] = 1.0
        for q in ((slice(None), slice(None), 0), (slice(None), slice(None), nx),
                  (slice(None), 0), (slice(None), ny), (nz,)):
            m[(4,) + q] = True
            T[q] = 0.0
        return m, T

    def design(self, gen):
        nx, ny, nz = self.n
        src, des = self.regions()
        u = torch.rand((nz, ny, nx), dtype=torch.float64, device=DEV, generator=gen)
        u = torch.nn.functional.avg_pool3d(u[None, None], 3, 1, 1, count_include_pad=False)[0, 0]
        if self.bcs == "quarter":
            u = (0.95 + 0.04 * (u - 0.5)).clamp(0, 1)
        g = torch.where(des, u, torch.ones_like(u))
        return torch.where(src, torch.zeros_like(g), g).reshape(-1).contiguous()

    def state(self, gen):
        s = torch.tensor([0.5, 0.5, 0.5, 50.0, 1.0], dtype=torch.float64, device=DEV)
        x = torch.randn((5, self.Nn), dtype=torch.float64, device=DEV, generator=gen) * s[:, None]
        m, T = self.dirichlet()
        x = torch.where(m.view(5, -1), torch.zeros_like(x), x)
        x[4] += torch.where(m[4], T, torch.zeros_like(T)).view(-1)
        return x.reshape(-1)

    def vector(self, gen):
        """A Krylov direction: zero on the Dirichlet unknowns, as in the solvers."""
        v = torch.randn((5, self.Nn), dtype=torch.float64, device=DEV, generator=gen)
        return v.masked_fill_(self.dirichlet()[0].view(5, -1), 0.0).view(-1)


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _orthonormal(case, gen):
    """k orthonormal columns (stride: whole multiples of 64 elements) and a vector."""
    n, k, dt = case["n"], case["k"], DT[case["dtype"]]
    ld = nc.mv_ld(n)
    V = torch.zeros((k, ld), dtype=torch.float64, device=DEV)
    V[:, :n] = torch.randn((k, n), dtype=torch.float64, device=DEV, generator=gen)
    for _ in range(2):  # Cholesky QR, twice
        V = torch.linalg.solve_triangular(torch.linalg.cholesky(V @ V.T), V, upper=False)
    w = torch.randn(n, dtype=torch.float64, device=DEV, generator=gen)
    w += V[:, :n].T @ torch.randn(k, dtype=torch.float64, device=DEV, generator=gen) * math.sqrt(n)
    return V.to(dt).contiguous(), w.to(dt), ld


def _mma_inputs(case, gen):
    sp = _Spec(dict(case, bcs="quarter"))
    act = sp.regions()[1].reshape(-1)
    if not bool(act.any()):
        act = torch.ones_like(act)
    E = sp.E
    r = lambda: torch.randn(E, dtype=torch.float64, device=DEV, generator=gen)  # noqa: E731
    x = torch.where(act, (0.93 + 0.05 * r()).clamp(0, 1), torch.ones(E, dtype=torch.float64, device=DEV))
    xo1 = torch.where(act, (x + 0.03 * r()).clamp(0, 1), x)
    xo2 = torch.where(act, (xo1 + 0.03 * r()).clamp(0, 1), x)
    low, upp = xo1 - 0.3, xo1 + 0.3
    df0 = torch.where(act, r() * torch.exp(r()), torch.zeros_like(x)) / E
    return sp, act, [x, xo1, xo2, low, upp], df0


VF = 0.05


def prepare(case, seed):
    kind = case["kind"]
    gen = _gen(seed)
    s = {"case": case}
    if kind == "arnoldi":
        V, w, ld = _orthonormal(case, gen)
        p = nc.make_params(2, 2, 2, 0.5, 1e3, 0.71)
        return dict(s, prob=nc.Problem(p, nc.cavity_bcs()), V=V.view(-1), w=w, ld=ld)
    if kind == "mma":
        sp, act, bufs, df0 = _mma_inputs(case, gen)
        return dict(s, prob=sp.problem(), bufs=bufs, df0=df0, active=act.to(torch.uint8),
                    df1=torch.empty_like(df0))
    sp = _Spec(dict(case, bcs="flux") if kind in ("filter", "gradient", "state") else case)
    s["prob"] = prob = sp.problem()
    gam = sp.design(gen)
    if kind == "filter":
        return dict(s, rho=gam, radius=case["radius"] * sp.h)
    if kind in ("gradient", "state"):
        # the previous design's converged state: where the next design iteration starts
        x = torch.zeros(prob.ndof, dtype=torch.float64, device=DEV)
        prob.newton_solve_sequenced(gam, x, nc.default_opts(rtol_newton=1e-10, ramp_steps=3))
        s.update(x=x, gam=gam)
        if kind == "state":
            s["gam"] = (gam + 0.02 * (sp.design(gen) - gam)).contiguous()
        return s
    dt = DT[case["dtype"]]
    s.update(x=sp.state(gen).to(dt), gam=gam.to(dt))
    if kind in ("jvp", "jtvp"):
        s["v"] = sp.vector(gen).to(dt)
    elif kind == "sens":
        s["lam"] = sp.vector(gen)
    elif kind in ("lin", "assembled"):
        s["v"] = [sp.vector(gen).to(dt) for _ in range(case["products"])]
        s["out"] = [torch.empty_like(s["x"]) for _ in range(case["products"])]
        if kind == "assembled":
            s["S"] = torch.empty(prob.STENCIL_VALUES * prob.Nn, dtype=dt, device=DEV)
    return s


def run(s):
    case, p = s["case"], s["prob"]
    kind = case["kind"]
    if kind == "residual":
        return p.residual(s["x"], s["gam"])
    if kind == "jvp":
        return p.jvp(s["x"], s["gam"], s["v"])
    if kind == "jtvp":
        return p.jtvp(s["x"], s["gam"], s["v"])
    if kind == "lin":
        p.linearize(s["x"], s["gam"])
        f = p.jtvp_lin if case["transpose"] else p.jvp_lin
        return [f(v, out=o) for v, o in zip(s["v"], s["out"])]
    if kind == "assembled":
        p.assemble(s["x"], s["gam"], S=s["S"])
        return [s["S"]] + [p.stencil_apply(s["S"], v, out=o, transpose=case["transpose"])
                           for v, o in zip(s["v"], s["out"])]
    if kind == "sens":
        phi, g = p.objective(s["x"])
        return [phi, g, p.sensitivity(s["x"], s["gam"], s["lam"])]
    if kind == "arnoldi":  # w is overwritten by the new basis vector: each pass takes a fresh one
        w = s["w"].clone()
        return [w, p.arnoldi_orth(s["V"], w, case["k"], s["ld"])]
    if kind == "filter":
        return p.filter(s["rho"], s["radius"])
    if kind == "mma":  # the iterates and asymptotes are updated in place: each pass takes fresh ones
        b = [t.clone() for t in s["bufs"]]
        g = p.volume(b[0], s["active"], VF, grad=s["df1"])
        lam, change = p.mma_update(case["it"], *b, s["df0"], g, s["df1"], active=s["active"])
        return b + [s["df1"], g, lam, change]
    if kind == "state":  # the state is updated in place: each pass starts from the previous one's
        x = s["x"].clone()
        p.newton_solve(s["gam"], x, nc.default_opts(rtol_newton=1e-10))
        return x
    phi, dphi = p.objective(s["x"])
    lam, _ = p.adjoint_solve(s["x"], s["gam"], -dphi, opts=nc.default_opts(rtol_adjoint=1e-11))
    return [phi, lam, p.sensitivity(s["x"], s["gam"], lam)]


# ---------------------------------------------------------------- work
def work(case):
    kind = case["kind"]
    B = 4 if case.get("dtype") == "f32" else 8
    if kind == "arnoldi":  # two passes of dots and updates over k columns
        n, k = case["n"], case["k"]
        return {"bytes": B * n * (k + 2), "flops": 8.0 * n * k}
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    E, Nn = nx * ny * nz, (nx + 1) * (ny + 1) * (nz + 1)
    nd = 5 * Nn
    if kind == "residual":
        return {"bytes": B * (2 * nd + E) + Nn, "flops": FLOP["residual"] * E}
    if kind in ("jvp", "jtvp"):
        return {"bytes": B * (3 * nd + E) + Nn, "flops": FLOP[kind] * E}
    if kind == "lin":
        m = case["products"]
        f = FLOP["jtvp_lin" if case["transpose"] else "jvp_lin"]
        return {"bytes": B * ((1 + 2 * m) * nd + E) + Nn,
                "flops": (FLOP["linearize"] + m * f) * E}
    if kind == "assembled":  # the 40 x 40 element entries formed and added, 675 FMA per node
        m = case["products"]
        return {"bytes": B * (nd + E + (1 + m) * 675 * Nn + 2 * m * nd),
                "flops": 3200 * E + 1350 * m * Nn}
    if kind == "sens":
        return {"bytes": B * (3 * nd + 2 * E) + Nn, "flops": FLOP["sens"] * E}
    if kind == "filter":  # right-hand side, about 25 conjugate-gradient steps, element means
        return {"bytes": 16 * E, "flops": 25 * 40 * Nn}
    if kind == "mma":  # three vectors shifted, four read, the dual evaluated a few times
        return {"bytes": 8 * 13 * E, "flops": 8 * 60 * E}
    if kind == "state":  # 2 Newton steps, 14 FGMRES iterations of one V-cycle (14 products)
        return {"bytes": 16 * nd + 8 * E,
                "flops": (14 * 15 * 8 / 7 * FLOP["jvp"] + 5 * FLOP["residual"]) * E}
    return {"bytes": 16 * nd + 16 * E,
            "flops": (22 * 15 * 8 / 7 * FLOP["jtvp"] + 4 * FLOP["jtvp_lin"] + FLOP["sens"]) * E}


# ---------------------------------------------------------------- the operators in 64 bits
def _shape():
    """N [8, 8] and dN/dx h [3, 8, 8] (point, node) of the trilinear element on [0, 1]^3."""
    q = [0.5 - 0.5 / math.sqrt(3.0), 0.5 + 0.5 / math.sqrt(3.0)]
    w = lambda i, t: t if i else 1.0 - t      # noqa: E731
    d = lambda i: 1.0 if i else -1.0          # noqa: E731
    N, D = torch.zeros(8, 8, dtype=torch.float64), torch.zeros(3, 8, 8, dtype=torch.float64)
    for g in range(8):
        X = [q[g & 1], q[(g >> 1) & 1], q[g >> 2]]
        for a in range(8):
            b = [a & 1, (a >> 1) & 1, a >> 2]
            f = [w(b[i], X[i]) for i in range(3)]
            N[g, a] = f[0] * f[1] * f[2]
            for i in range(3):
                D[i, g, a] = d(b[i]) * f[(i + 1) % 3] * f[(i + 2) % 3]
    return N.to(DEV), D.to(DEV)


class _Exact:
    CHUNK = 1 << 17

    def __init__(self, sp):
        self.sp = sp
        self.N, self.D = _shape()
        self.D = self.D / sp.h
        m = sp.mat
        self.beg = -sp.Gr * m["Pr"] ** 2  # gravity along -z
        self.src = sp.source() if sp.bcs == "quarter" else None
        self.mask = sp.dirichlet()[0].view(5, -1)

    def element(self, xe, gam, s):
        """Element residual rows [B, 5, 8] of xe [B, 5, 8]."""
        sp, m = self.sp, self.sp.mat
        h, Pr = sp.h, m["Pr"]
        al = m["alpha_max"] * (1 - gam) / (1 + m["q_alpha"] * gam)
        K = (gam * (m["Ck"] * (1 + m["q_f"]) - 1) + 1) / (m["Ck"] * (1 + m["q_f"] * gam))
        S = (xe[:, 0:3] ** 2).sum((1, 2)) / (4 * h) ** 2
        tau = (S + (4 * Pr / h ** 2) ** 2 + al ** 2) ** -0.5
        tauT = (S + (4 * K / h ** 2) ** 2) ** -0.5
        val = torch.einsum("pa,bfa->bfp", self.N, xe)
        grd = torch.einsum("jpa,bfa->bfjp", self.D, xe)
        u, p, T = val[:, 0:3], val[:, 3], val[:, 4]
        G, gp, gT = grd[:, 0:3], grd[:, 3], grd[:, 4]
        body = torch.einsum("bjp,bijp->bip", u, G) + al[:, None, None] * u
        body = torch.cat([body[:, 0:2], (body[:, 2] + self.beg * T)[:, None]], 1)
        rM = body + gp
        rT = (u * gT).sum(1) - s[:, None]
        F = Pr * (G + G.transpose(1, 2)) + (tau[:, None, None] * rM)[:, :, None] * u[:, None]
        F = F - torch.eye(3, dtype=F.dtype, device=DEV)[None, :, :, None] * p[:, None, None]
        f0 = torch.cat([body, (G[:, 0, 0] + G[:, 1, 1] + G[:, 2, 2])[:, None], rT[:, None]], 1)
        F1 = torch.cat([F, (tau[:, None, None] * rM)[:, None],
                        (K[:, None, None] * gT + u * (tauT[:, None] * rT)[:, None])[:, None]], 1)
        w = (h / 2) ** 3
        return w * (torch.einsum("pa,bfp->bfa", self.N, f0)
                    + torch.einsum("jpa,bfjp->bfa", self.D, F1))

    def chunks(self):
        nx, ny, nz = self.sp.n
        sy, sz = nx + 1, (nx + 1) * (ny + 1)
        off = torch.tensor([(a & 1) + ((a >> 1) & 1) * sy + (a >> 2) * sz for a in range(8)],
                           device=DEV)
        for e0 in range(0, self.sp.E, self.CHUNK):
            e = torch.arange(e0, min(e0 + self.CHUNK, self.sp.E), device=DEV)
            n0 = e % nx + sy * ((e // nx) % ny) + sz * (e // (nx * ny))
            src = self.src[e] if self.src is not None else torch.zeros(len(e), dtype=torch.float64, device=DEV)
            yield e, n0[:, None] + off, src

    def gather(self, f):
        """Nodal sums [5, Nn] of the element rows f(e, conn, src) [B, 5, 8]."""
        r = torch.zeros((5, self.sp.Nn), dtype=torch.float64, device=DEV)
        for e, conn, src in self.chunks():
            rows = f(e, conn, src)
            for a in range(8):
                r.index_add_(1, conn[:, a], rows[:, :, a].T.contiguous())
        return r

    @staticmethod
    def rows(x, conn):
        return x[:, conn].transpose(0, 1)

    def residual(self, x, gam):
        sp = self.sp
        x = x.view(5, -1)
        r = self.gather(lambda e, c, s: self.element(self.rows(x, c), gam[e], s))
        if sp.bcs == "flux" and sp.has_patch():
            nx, ny, _ = sp.n
            face = torch.zeros((ny + 2, nx + 2), dtype=torch.float64, device=DEV)
            face[1 + sp.py[0]:1 + sp.py[1], 1 + sp.px[0]:1 + sp.px[1]] = 1.0
            cnt = face[1:, 1:] + face[:-1, 1:] + face[1:, :-1] + face[:-1, :-1]
            r[4, :(nx + 1) * (ny + 1)] -= sp.h ** 2 / 4 * cnt.reshape(-1)
        T = sp.dirichlet()[1].view(-1)
        xd = torch.zeros_like(x)
        xd[4] = T
        return torch.where(self.mask, x - xd, r).reshape(-1)

    def product(self, x, gam, v, transpose):
        x, v = x.view(5, -1), v.view(5, -1)
        vi = torch.where(self.mask, torch.zeros_like(v), v)

        def f(e, c, s):
            fn = lambda y: self.element(y, gam[e], s)  # noqa: E731
            xe, ve = self.rows(x, c), self.rows(vi, c)
            if transpose:
                return torch.func.vjp(fn, xe)[1](ve)[0]
            return torch.func.jvp(fn, (xe,), (ve,))[1]
        return torch.where(self.mask, v, self.gather(f)).reshape(-1)

    def sensitivity(self, x, gam, lam):
        x, lam = x.view(5, -1), lam.view(5, -1)
        lam = torch.where(self.mask, torch.zeros_like(lam), lam)
        out = torch.empty_like(gam)
        for e, c, s in self.chunks():
            xe = self.rows(x, c)
            g = gam[e]
            d = torch.func.jvp(lambda t: self.element(xe, t, s), (g,), (torch.ones_like(g),))[1]
            out[e] = (self.rows(lam, c) * d).sum((1, 2))
        return out

    def stencil(self, x, gam):
        x = x.view(5, -1)
        S = torch.zeros((27, 5, 5, self.sp.Nn), dtype=torch.float64, device=DEV)
        for e, c, s in self.chunks():
            xe = self.rows(x, c)
            fn = lambda y: self.element(y, gam[e], s)  # noqa: E731
            for b in range(8):
                for g in range(5):
                    v = torch.zeros_like(xe)
                    v[:, g, b] = (~self.mask[g, c[:, b]]).double()
                    col = torch.func.jvp(fn, (xe,), (v,))[1]
                    for a in range(8):
                        o = sum(((b >> i & 1) - (a >> i & 1) + 1) * 3 ** i for i in range(3))
                        S[o, :, g].index_add_(1, c[:, a], col[:, :, a].T.contiguous())
        for f in range(5):
            S[:, f, :, self.mask[f]] = 0.0
            S[13, f, f, self.mask[f]] = 1.0
        return S.reshape(-1)


def _exact_filter(sp, rho, R):
    """Filtered element values by fast diagonalisation: (r^2 K + M)^-1 with K, M sums and
    products of the 1-D stiffness and mass matrices, r = R / (2 sqrt 3)."""
    r2 = R * R / 12.0
    lam, Phi = [], []
    for m in sp.n:
        A = torch.zeros((m + 1, m + 1), dtype=torch.float64)
        K = torch.zeros_like(A)
        i = torch.arange(m)
        for t, d, o in ((A, 2.0, 1.0), (K, 1.0, -1.0)):
            t[i, i] += d
            t[i + 1, i + 1] += d
            t[i, i + 1] += o
            t[i + 1, i] += o
        A, K = A * sp.h / 6.0, K / sp.h
        L = torch.linalg.cholesky(A)
        Li = torch.linalg.inv(L)
        w, Q = torch.linalg.eigh(Li @ K @ Li.T)
        lam.append(w.to(DEV))
        Phi.append((Li.T @ Q).to(DEV))
    nx, ny, nz = sp.n
    r = torch.nn.functional.pad(rho.view(nz, ny, nx), (1, 1, 1, 1, 1, 1))
    box = lambda t: sum(t[k:t.shape[0] - 1 + k, j:t.shape[1] - 1 + j, i:t.shape[2] - 1 + i]  # noqa: E731
                        for k in (0, 1) for j in (0, 1) for i in (0, 1))
    b = box(r) * sp.h ** 3 / 8.0
    y = torch.einsum("kji,ia,jb,kc->cba", b, Phi[0], Phi[1], Phi[2])
    y = y / (1.0 + r2 * (lam[0][None, None, :] + lam[1][None, :, None] + lam[2][:, None, None]))
    x = torch.einsum("cba,ia,jb,kc->kji", y, Phi[0], Phi[1], Phi[2])
    return (box(x) / 8.0).reshape(-1)


def _exact_mma(case, seed):
    sp, act, (x, xo1, xo2, low, upp), df0 = _mma_inputs(case, _gen(seed))
    n = int(act.sum())
    zero = torch.zeros_like(x)
    g1 = float(torch.where(act, 1.0 - x, zero).sum()) / (VF * n) - 1.0
    df1 = torch.where(act, torch.full_like(x, -1.0 / (VF * n)), zero)
    if case["it"] < 2:
        l, u = x - 0.5, x + 0.5
    else:
        s = (x - xo1) * (xo1 - xo2)
        f = lambda t: torch.tensor(t, dtype=torch.float64, device=DEV)  # noqa: E731
        fac = torch.where(s < 0, f(0.7), torch.where(s > 0, f(1.2), f(1.0)))
        l = torch.minimum(torch.maximum(x - fac * (xo1 - low), x - 10.0), x - 0.01)
        u = torch.minimum(torch.maximum(x + fac * (upp - xo1), x + 0.01), x + 10.0)
    l, u = torch.where(act, l, low), torch.where(act, u, upp)
    X, L, U, A0, A1 = (t[act] for t in (x, l, u, df0, df1))
    lo_, hi_ = (torch.maximum(torch.clamp(L + 0.1 * (X - L), min=0.0), X - 0.2),
                torch.minimum(torch.clamp(U - 0.1 * (U - X), max=1.0), X + 0.2))

    def pq(a):
        ap, am = a.clamp(min=0), (-a).clamp(min=0)
        return ((U - X) ** 2 * (1.001 * ap + 0.001 * am + 1e-5),
                (X - L) ** 2 * (0.001 * ap + 1.001 * am + 1e-5))
    p0, q0 = pq(A0)
    p1, q1 = pq(A1)

    def at(lam):
        P, Q = torch.sqrt(p0 + lam * p1), torch.sqrt(q0 + lam * q1)
        y = torch.minimum(torch.maximum((L * P + U * Q) / (P + Q), lo_), hi_)
        f = p1 * (1 / (U - y) - 1 / (U - X)) + q1 * (1 / (y - L) - 1 / (X - L))
        return g1 + float(f.sum()), y
    lam = 0.0
    if at(0.0)[0] > 0.0:
        hi, lo = 1.0, 0.0
        for _ in range(200):
            if at(hi)[0] <= 0.0:
                break
            hi *= 2.0
        while lo < 0.5 * (lo + hi) < hi:
            mid = 0.5 * (lo + hi)
            if at(mid)[0] > 0.0:
                lo = mid
            else:
                hi = mid
        lam = hi
    y = x.clone()
    y[act] = at(lam)[1]
    return [y, x, xo1, l, u, df1, g1, lam, float((y - x).abs().max())]


def exact(case, seed):
    kind = case["kind"]
    gen = _gen(seed)
    if kind in ("gradient", "state"):  # a nonlinear solve on 10^5 to 10^6 elements
        return None
    if kind == "arnoldi":
        V, w, _ = _orthonormal(case, gen)
        V, w = V[:, :case["n"]].double(), w.double()
        h = V @ w
        w = w - V.T @ h
        h2 = V @ w
        w = w - V.T @ h2
        nw = float(w.norm())
        return [w / nw, [float(t) for t in h + h2] + [nw]]
    if kind == "mma":
        return _exact_mma(case, seed)
    sp = _Spec(dict(case, bcs="flux") if kind == "filter" else case)
    gam = sp.design(gen)
    if kind == "filter":
        return _exact_filter(sp, gam, case["radius"] * sp.h)
    dt = DT[case["dtype"]]
    x, gam = sp.state(gen).to(dt).double(), gam.to(dt).double()
    ex = _Exact(sp)
    if kind == "residual":
        return ex.residual(x, gam)
    if kind in ("jvp", "jtvp"):
        return ex.product(x, gam, sp.vector(gen).to(dt).double(), kind == "jtvp")
    if kind == "sens":
        lam = sp.vector(gen)
        if sp.bcs == "quarter":  # thermal compliance: s_e h^3 / 8 to each element node's T row
            g = ex.gather(lambda e, c, s: torch.cat(
                [torch.zeros((len(e), 4, 8), dtype=torch.float64, device=DEV),
                 (s * sp.h ** 3 / 8)[:, None, None].expand(-1, 1, 8)], 1))
        else:  # mean temperature of the patch
            g = torch.zeros((5, sp.Nn), dtype=torch.float64, device=DEV)
            nx, ny, _ = sp.n
            face = torch.zeros((ny + 2, nx + 2), dtype=torch.float64, device=DEV)
            face[1 + sp.py[0]:1 + sp.py[1], 1 + sp.px[0]:1 + sp.px[1]] = 1.0
            cnt = face[1:, 1:] + face[:-1, 1:] + face[1:, :-1] + face[:-1, :-1]
            if float(cnt.sum()) > 0:
                g[4, :(nx + 1) * (ny + 1)] = cnt.reshape(-1) / cnt.sum()
        g = g.reshape(-1)
        return [float(g @ x), g, ex.sensitivity(x, gam, lam)]
    vs = [sp.vector(gen).to(dt).double() for _ in range(case["products"])]
    outs = [ex.product(x, gam, v, case["transpose"]) for v in vs]
    return [ex.stencil(x, gam)] + outs if kind == "assembled" else outs
