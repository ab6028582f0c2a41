"""The calls a user of the evaporation operators makes, as timed cases: operator applies of both precisions and degrees,
the adjoint and the autograd function, the level-set operators and their geometry solver, setting the fields, the
momentum solve and the coupled time step, each through the package's public entry points.

Domain [0, 1]^3, the interface thickness one cell width, the parameters of the paper's droplet case (rho_l = 1000,
density ratio 1e3 or 1e4, mu 1e-3 / 1e-5, dt = 1e-4).  Level set phi = tanh(d / (2 eps)) of a signed distance d;
velocities are random Fourier sums of unit RMS, applied vectors uniform in [-1, 1].  Inputs are drawn on the GPU from
the seed alone.  exact() evaluates the same operators plainly in FP64 (full Gauss quadrature, cell by cell, gradients
by torch.autograd, constant-coefficient solves by diagonalization), without the package.
"""
import math

import numpy as np
import torch

import paper_2401_07805_gb300 as evap

RHO_L, MU_L, MU_G, DT = 1000.0, 1e-3, 1e-5, 1e-4
GEOMETRIES = ("sphere", "spheres", "slab", "deformed")


# ------------------------------------------------------------------------------------------------------- the cases
def _case(kind, n, p=2, **over):
    c = dict(kind=kind, n=n, p=p, geom="spheres", ratio=1e3, prec=64, divergence=True, newton=1, variant=2, n_sub=1,
             faces=63, steps=0, mixed=True)
    c.update(over)
    return c


def listed():
    def named(name, *a, **k):
        return dict(_case(*a, **k), name=name)

    return [
        # one operator apply on the smallest mesh of the test problems: launch latency
        named("apply-q2-8", "apply", 8, geom="sphere"),
        # the usual apply: the residual of a solve on the four-drop problem
        named("apply-q2-64", "apply", 64),
        # cubic velocity on an odd mesh, the larger density ratio
        named("apply-q3-45", "apply", 45, p=3, geom="deformed", ratio=1e4),
        # the largest apply (51 M velocity unknowns), without the continuity row
        named("apply-q2-128", "apply", 128, geom="deformed", ratio=1e4, divergence=False),
        # the FP32 operator of mixed-precision solvers, on a mesh that is no multiple of 32 cells
        named("apply32-q2-75", "apply", 75, prec=32, geom="slab", divergence=False),
        # all gradients of the momentum operator (sensitivities of a loss, the 48^3 drop)
        named("adjoint-q2-48", "adjoint", 48, geom="sphere"),
        # one training step through the autograd function: new fields, apply, backward
        named("autograd-q2-33", "autograd", 33, geom="sphere"),
        # new coefficient fields with the extrapolated transport velocity, and the first apply on them
        named("fields-q2-64", "fields", 64),
        # the three level-set operators
        named("levelset-64", "levelset", 64),
        # the level-set geometry of one time step: normal, curvature, surface force, reinitialization
        named("geometry-64", "geometry", 64, steps=2),
        # the mixed-precision momentum solve on the slab problem
        named("solve-q2-96", "solve", 96, geom="slab"),
        # one coupled time step, the top face open
        named("step-q2-64", "step", 64, newton=0, faces=31, steps=2),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(("apply", "apply", "apply", "adjoint", "autograd", "fields", "levelset", "geometry", "solve", "step"))
    p = 3 if kind != "levelset" and kind != "geometry" and rng.random() < 0.3 else 2
    top = {"apply": (120, 70), "adjoint": (72, 40), "autograd": (48, 30), "fields": (80, 40), "levelset": (120, 120),
           "geometry": (80, 80), "solve": (90, 50), "step": (56, 28)}[kind][p - 2]
    n = size(6, top)
    geom, ratio = rng.choice(GEOMETRIES), rng.choice((1e3, 1e4))
    over = dict(geom=geom, ratio=ratio, newton=rng.choice((0, 1)), divergence=rng.random() < 0.7)
    if kind == "apply":
        over["prec"] = rng.choice((64, 32))
        over["faces"] = rng.choice((63, 31, 0))
    if kind in ("apply", "adjoint", "fields", "levelset") and n <= 60:
        over["n_sub"] = rng.choice((1, 1, 2))
    if kind in ("fields", "step"):
        over["variant"] = rng.choice((1, 2, 3))
    if kind == "solve":  # the all-FP64 solver costs several mixed ones
        over["mixed"] = n > 48 or rng.random() < 0.7
    if kind in ("geometry", "step"):
        over["steps"] = rng.randint(1, 4)
    if kind == "step":
        over.update(faces=31, newton=0, ratio=1e3)
    return _case(kind, n, p, **over)


# ------------------------------------------------------------------------------------------------- inputs of a case
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _nodes(n, p):
    """1D node positions of the Q_p space on n cells (Gauss-Lobatto points in each cell)."""
    ref = {1: [0.0, 1.0], 2: [0.0, 0.5, 1.0], 3: [0.0, 0.5 - 0.5 / math.sqrt(5.0), 0.5 + 0.5 / math.sqrt(5.0), 1.0]}[p]
    x = np.empty(p * n + 1)
    for c in range(n):
        x[p * c:p * c + p + 1] = (c + np.array(ref)) / n
    return torch.from_numpy(x).cuda()


def _distance(geom, x, g):
    """Signed distance at the lattice x (x) x (x) x, [z, y, x], positive in the liquid."""
    X, Y, Z = x[None, None, :], x[None, :, None], x[:, None, None]

    def ball(c, r):
        return r - torch.sqrt((X - c[0]) ** 2 + (Y - c[1]) ** 2 + (Z - c[2]) ** 2)

    u = torch.rand(32, generator=g, device="cuda", dtype=torch.float64).tolist()
    if geom == "slab":
        return 0.45 + 0.1 * u[0] - Z.expand(len(x), len(x), len(x))
    if geom == "sphere":
        return ball([0.45 + 0.1 * u[k] for k in range(3)], 0.22 + 0.06 * u[3])
    if geom == "spheres":
        d = None
        for k in range(4):
            b = ball([0.2 + 0.6 * u[4 * k + a] for a in range(3)], 0.08 + 0.12 * u[4 * k + 3])
            d = b if d is None else torch.maximum(d, b)
        return d
    # a sphere whose radius varies with the direction
    dx, dy, dz = X - 0.5, Y - 0.5, Z - 0.5
    r = torch.sqrt(dx * dx + dy * dy + dz * dz)
    s = torch.clamp(r, min=1e-12)
    ct, ph = dz / s, torch.atan2(dy + 0 * r, dx + 0 * r)
    f = 0.0
    for l in range(1, 7):
        f = f + (u[2 * l] - 0.5) * torch.cos(l * torch.arccos(torch.clamp(ct, -1.0, 1.0))) + \
            (u[2 * l + 1] - 0.5) * torch.sqrt(torch.clamp(1.0 - ct * ct, min=0.0)) ** l * torch.cos(l * ph + 6.28 * u[20 + l])
    return 0.3 * (1.0 + 0.1 * f / f.abs().max()) - r


def _fourier(x, g, kmax=4):
    """Velocity at the lattice of x, three components, random Fourier modes, unit RMS of its length."""
    ks = torch.arange(-kmax, kmax + 1, device="cuda", dtype=torch.float64)
    E = torch.exp(2j * math.pi * ks[:, None] * x[None, :])
    K = len(ks)
    out = []
    for _ in range(3):
        a = torch.randn(2, K, K, K, generator=g, device="cuda", dtype=torch.float64)
        c = torch.complex(a[0], -a[1])
        c[kmax, kmax, kmax] = 0
        t = torch.einsum("abc,cx->abx", c, E)
        t = torch.einsum("abx,by->ayx", t, E)
        out.append(torch.einsum("ayx,az->zyx", t, E).real.contiguous())
    u = torch.stack(out)
    return (u / torch.sqrt((u * u).sum(0).mean())).reshape(-1)


def _uniform(g, k, dtype=torch.float64):
    return (2.0 * torch.rand(k, generator=g, device="cuda", dtype=torch.float64) - 1.0).to(dtype)


def _params(c):
    return dict(rho_l=RHO_L, rho_g=RHO_L / c["ratio"], mu_l=MU_L, mu_g=MU_G, dt=DT, newton=c["newton"],
                variant=c["variant"], n_sub=c["n_sub"], dirichlet_faces=c["faces"])


def _inputs(c, seed):
    """The tensors of a case, from the seed alone."""
    g = _gen(seed)
    n, p, ns = c["n"], c["p"], c["n_sub"]
    xl = _nodes(ns * n, 1)
    eps = 1.0 / n
    phi = torch.tanh(_distance(c["geom"], xl, g) / (2.0 * eps)).contiguous().reshape(-1)
    n_u, n_phi, n_p = (p * n + 1) ** 3, (ns * n + 1) ** 3, (n + 1) ** 3
    u0 = _fourier(_nodes(n, p), g)
    mdot = 0.5 + torch.rand(n_phi, generator=g, device="cuda", dtype=torch.float64)
    s = dict(phi=phi, u0=u0, mdot=mdot)
    if c["kind"] == "levelset":
        s["ug"] = _fourier(xl, g)
        s["psi"] = torch.clamp(phi + 0.02 * _uniform(g, n_phi), -1.0, 1.0)
    elif c["kind"] == "geometry":
        s["psi"] = phi.clone()
    elif c["kind"] == "step":
        s["p"] = torch.zeros(n_p, device="cuda", dtype=torch.float64)
        # no flow through the walls: the velocity fades out towards them
        x = _nodes(n, p)
        w = 16.0 * (x * (1.0 - x)) ** 2
        wz = torch.sin(0.5 * math.pi * x) ** 2
        s["u0"] = (u0.view(3, len(x), len(x), len(x)) * (wz[:, None, None] * w[None, :, None] * w[None, None, :])).reshape(-1).contiguous()
    else:
        s["x"] = _uniform(g, 3 * n_u, torch.float32 if c["prec"] == 32 else torch.float64)
        if c["kind"] in ("adjoint", "autograd"):
            s["w"] = _uniform(g, 3 * n_u)
            s["wp"] = _uniform(g, n_p)
    return s


def prepare(case, seed):
    """The inputs, and the operator of the mesh with its fields set where the timed call finds them set."""
    s = _inputs(case, seed)
    op = evap.Operator(case["n"], case["p"], 1.0, _params(case))
    if case["kind"] not in ("fields", "autograd", "step"):
        op.set_fields(s["phi"], s["u0"], s["mdot"])
    if case["kind"] == "levelset":
        op.set_transport_velocity(s["ug"])
    if case["kind"] == "autograd":
        for k in ("x", "phi", "u0", "mdot"):
            s[k].requires_grad_(True)
    return dict(s, op=op, case=case)


# ----------------------------------------------------------------------------------------------------- the timed call
def run(s):
    c, op = s["case"], s["op"]
    kind = c["kind"]
    if kind == "apply":
        r = op.apply_momentum(s["x"], prec=c["prec"], with_divergence=c["divergence"])
        return list(r) if c["divergence"] else [r]
    if kind == "adjoint":
        return op.apply_adjoint(s["w"], s["x"], s["wp"])
    if kind == "autograd":
        y, yp = evap.MomentumFunction.apply(op, s["x"], s["phi"], s["u0"], s["mdot"])
        grads = torch.autograd.grad((y, yp), (s["x"], s["u0"], s["phi"], s["mdot"]), (s["w"], s["wp"]))
        return dict(y=y, yp=yp, x=grads[0], u0=grads[1], phi=grads[2], mdot=grads[3])
    if kind == "fields":
        op.set_fields(s["phi"], s["u0"], s["mdot"])
        y, yp = op.apply_momentum(s["x"], with_divergence=True)
        ug, flags, _ = op.transport_velocity()
        return dict(y=y, yp=yp, ug=ug, flags=flags)
    if kind == "levelset":
        return [op.apply_levelset(s["psi"], mode=m) for m in ("advect", "reinit", "reinit_rhs")]
    if kind == "geometry":
        nrm, _ = op.projected_normal()
        kappa, _ = op.curvature(nrm)
        f = op.surface_tension(nrm, kappa, 0.07)
        op.set_levelset_normal(nrm)
        psi, _ = op.reinitialize(s["psi"], c["steps"])
        op.set_levelset_normal(None)
        return dict(normal=nrm, kappa=kappa, force=f, psi=psi)
    if kind == "solve":
        return [op.solve(s["x"], mixed=c["mixed"])[0]]
    # one advection pass with the closest-point variants: a second one moves the creases of the discrete interface by
    # amounts that depend on rounding
    phi, u, p, _ = op.time_step(s["phi"], s["u0"], s["p"], s["mdot"], gravity=(0.0, 0.0, -9.81),
                                fp_iters=2 if c["variant"] == 1 else 1, reinit_steps=c["steps"])
    return dict(phi=phi, u=u, p=p)


# ------------------------------------------------------------------------------------------------ what a pass needs
def work(case):
    """Bytes: each input vector and coefficient field read once, each result written once.  Flops: sum factorization
    of the sweeps plus the point work; for the iterative calls one application per unknown vector as the least."""
    n, p, ns = case["n"], case["p"], case["n_sub"]
    q, nq, cells = p + 1, (p + 1) ** 3, n ** 3
    nu, nphi, npr = (p * n + 1) ** 3, (ns * n + 1) ** 3, (n + 1) ** 3
    apply = cells * (72 * q * nq + 100 * nq)
    adjoint = 2 * cells * (72 * q * nq + 80 * nq)
    fields = cells * nq * 100
    ls = (ns * n) ** 3 * 800
    kind = case["kind"]
    b = case["prec"] // 8
    if kind == "apply":
        return dict(bytes=b * (9 * nu + 2 * nphi + (npr if case["divergence"] else 0)), flops=apply)
    if kind == "adjoint":
        return dict(bytes=8 * (15 * nu + 4 * nphi + npr), flops=adjoint)
    if kind == "autograd":
        return dict(bytes=8 * (18 * nu + 4 * nphi + 2 * npr), flops=apply + adjoint + fields)
    if kind == "fields":
        return dict(bytes=8 * (9 * nu + 5 * nphi + npr) + 4 * nphi, flops=apply + fields)
    if kind == "levelset":
        return dict(bytes=8 * 8 * nphi, flops=3 * ls)
    if kind == "geometry":  # four Helmholtz solves and the pseudo-time steps, about 40 iterations of 27 terms each
        return dict(bytes=8 * (6 * nphi + 3 * nu), flops=(4 + case["steps"]) * 40 * 27 * 2 * nphi)
    if kind == "solve":
        return dict(bytes=8 * (9 * nu + 2 * nphi), flops=15 * apply)
    return dict(bytes=8 * (6 * nu + 3 * nphi + 2 * npr), flops=40 * apply + fields)


# -------------------------------------------------------------------------------------- plain FP64 evaluation (exact)
class _Plain:
    """Full Gauss quadrature on every cell in FP64; a field at the points is [cells, points]."""

    def __init__(self, c):
        self.c, self.n, self.p, self.ns = c, c["n"], c["p"], c["n_sub"]
        n, p, ns = self.n, self.p, self.ns
        self.h = 1.0 / n
        t, w = np.polynomial.legendre.leggauss(p + 1)
        t, w = 0.5 * (t + 1.0), 0.5 * w
        ref = _nodes(1, p).cpu().numpy()
        self.S, self.D = self.lagrange(ref, t)
        # the level set: Q1 on the ns sub-intervals; a point on a sub-interval's end takes the upper one's slope
        N, DN = np.zeros((p + 1, ns + 1)), np.zeros((p + 1, ns + 1))
        for q in range(p + 1):
            k = min(int(math.floor(ns * t[q] + 1e-12)), ns - 1)
            xi = ns * t[q] - k
            N[q, k], N[q, k + 1], DN[q, k], DN[q, k + 1] = 1 - xi, xi, -ns, ns
        self.NL, self.DL = N, DN
        self.N1 = np.stack([1 - t, t], 1)
        self.W = torch.from_numpy(np.einsum("a,b,c->abc", w, w, w).reshape(-1) * self.h ** 3).cuda()
        self.iu, self.il, self.ip = self.cells(n, p), self.cells(n, ns), self.cells(n, 1)

    @staticmethod
    def lagrange(nodes, t):
        m = len(nodes)
        V = np.vander(nodes, m, increasing=True)
        A = np.vander(t, m, increasing=True)
        B = np.zeros_like(A)
        for k in range(1, m):
            B[:, k] = k * t ** (k - 1)
        C = np.linalg.inv(V)
        return A @ C, B @ C

    @staticmethod
    def cells(n, s):
        """Node numbers of every cell, [n^3, (s + 1)^3], of a lattice with s intervals a cell."""
        M = s * n + 1
        c = torch.arange(n, device="cuda") * s
        a = torch.arange(s + 1, device="cuda")
        base = (c[None, None, :] + M * (c[None, :, None] + M * c[:, None, None])).reshape(-1)
        loc = (a[None, None, :] + M * (a[None, :, None] + M * a[:, None, None])).reshape(-1)
        return base[:, None] + loc[None, :]

    def matrices(self, V, DV):
        """[points, nodes] of the value and the three physical gradients from 1D values and derivatives."""
        k = lambda z, y, x: torch.from_numpy(np.kron(z, np.kron(y, x))).cuda()  # noqa: E731
        return k(V, V, V), [k(V, V, DV) / self.h, k(V, DV, V) / self.h, k(DV, V, V) / self.h]

    def scatter(self, size, idx, v):
        return torch.zeros(size, dtype=torch.float64, device="cuda").index_add(0, idx.reshape(-1), v.reshape(-1))

    def material(self, phi):
        c, h = self.c, self.h
        eps, rl, rg = h, RHO_L, RHO_L / c["ratio"]
        B, G = self.matrices(self.NL, self.DL)
        pv = phi[self.il]
        f, g = pv @ B.T, [pv @ x.T for x in G]
        band = math.tanh(1.5)
        zone = f.abs() < band
        fs = torch.where(zone, f, torch.zeros_like(f))
        d = eps * torch.log((1.0 + fs) / (1.0 - fs))
        H = 0.5 + d / (6.0 * eps) + torch.sin(math.pi * d / (3.0 * eps)) / (2.0 * math.pi)
        dH = (1.0 + torch.cos(math.pi * d / (3.0 * eps))) / (6.0 * eps)
        H = torch.where(zone, H, (f >= band).double())
        rho, mu = 1.0 / (H / rl + (1.0 - H) / rg), H * MU_L + (1.0 - H) * MU_G
        gg = g[0] ** 2 + g[1] ** 2 + g[2] ** 2
        ok = gg * h * h > 1e-8
        gn = torch.sqrt(torch.where(ok, gg, torch.ones_like(gg)))
        nv = [torch.where(ok, x / gn, torch.zeros_like(x)) for x in g]
        tiny = torch.sqrt(torch.where(gg > 0, gg, torch.ones_like(gg))) * (gg > 0)
        delta = torch.where(zone, dH * 2.0 * eps / (1.0 - fs * fs) * tiny, torch.zeros_like(f))
        return zone, rho, mu, nv, delta, B

    def dirichlet(self):
        M = self.p * self.n + 1
        m = torch.zeros(M, M, M, dtype=torch.bool, device="cuda")
        for axis in range(3):
            for side in range(2):
                if self.c["faces"] >> (2 * axis + side) & 1:
                    m.select(2 - axis, -side if side else 0).fill_(True)
        return m.reshape(-1).repeat(3)

    def momentum(self, x, phi, u0, mdot, divergence=True):
        c, nu = self.c, (self.p * self.n + 1) ** 3
        zone, rho, mu, nv, delta, B = self.material(phi)
        cons = self.dirichlet()
        xf = torch.where(cons, torch.zeros_like(x), x)
        V, G = self.matrices(self.S, self.D)
        X, dX, U, dU = [], [], [], []
        for k in range(3):
            xc, uc = xf[k * nu:(k + 1) * nu][self.iu], u0[k * nu:(k + 1) * nu][self.iu]
            X.append(xc @ V.T)
            dX.append([xc @ g.T for g in G])
            U.append(uc @ V.T)
            dU.append([uc @ g.T for g in G] if c["newton"] else None)
        tr = dX[0][0] + dX[1][1] + dX[2][2]
        y = []
        for k in range(3):
            F = X[k] / DT + U[0] * dX[k][0] + U[1] * dX[k][1] + U[2] * dX[k][2]
            if c["newton"]:
                F = F + dU[k][0] * X[0] + dU[k][1] * X[1] + dU[k][2] * X[2]
            r = (self.W * rho * F) @ V
            for b in range(3):
                T = 0.5 * (dX[k][b] + dX[b][k]) - torch.where(zone, tr * nv[k] * nv[b], torch.zeros_like(tr))
                r = r + (2.0 * self.W * mu * T) @ G[b]
            y.append(self.scatter(nu, self.iu, r))
        y = torch.where(cons, x, torch.cat(y))
        if not divergence:
            return y, None
        c1 = c["ratio"] / RHO_L - 1.0 / RHO_L
        src = c1 * (mdot[self.il] @ B.T) * delta
        Np, _ = self.matrices(self.N1, self.N1)
        return y, self.scatter((self.n + 1) ** 3, self.ip, (self.W * (tr - src)) @ Np)


class _PlainLevelSet:
    """Q1 operators on the level-set mesh with the 2-point Gauss rule."""

    def __init__(self, n, h, dtau, eps):
        self.n, self.h, self.dtau, self.eps = n, h, dtau, eps
        r = 1.0 / math.sqrt(3.0)
        t = np.array([0.5 * (1 - r), 0.5 * (1 + r)])
        N, D = np.stack([1 - t, t], 1), np.array([[-1.0, 1.0], [-1.0, 1.0]])
        k = lambda z, y, x: torch.from_numpy(np.kron(z, np.kron(y, x))).cuda()  # noqa: E731
        self.B, self.G = k(N, N, N), [k(N, N, D) / h, k(N, D, N) / h, k(D, N, N) / h]
        self.idx, self.size, self.W = _Plain.cells(n, 1), (n + 1) ** 3, h ** 3 / 8

    def assemble(self, v):
        return torch.zeros(self.size, dtype=torch.float64, device="cuda").index_add(0, self.idx.reshape(-1), v.reshape(-1))

    def at(self, f):
        v = f[self.idx]
        return v @ self.B.T, [v @ g.T for g in self.G]

    def unit(self, g, least):
        gn = torch.sqrt(g[0] ** 2 + g[1] ** 2 + g[2] ** 2)
        ok = gn > least
        return [torch.where(ok, x / torch.where(ok, gn, torch.ones_like(gn)), torch.zeros_like(x)) for x in g]

    def advect(self, x, ug, theta=0.5):
        X, gX = self.at(x)
        U = [self.at(ug[k * self.size:(k + 1) * self.size])[0] for k in range(3)]
        return self.assemble((self.W * (X + theta * DT * (U[0] * gX[0] + U[1] * gX[1] + U[2] * gX[2]))) @ self.B)

    def reinit(self, x, nv):
        X, gX = self.at(x)
        s = self.eps * (gX[0] * nv[0] + gX[1] * nv[1] + gX[2] * nv[2])
        return self.assemble(self.W * ((X / self.dtau) @ self.B + sum((s * nv[d]) @ self.G[d] for d in range(3))))

    def reinit_rhs(self, x, nv):
        X, _ = self.at(x)
        s = 0.5 * (1.0 - X * X)
        return self.assemble(self.W * ((X / self.dtau) @ self.B + sum((s * nv[d]) @ self.G[d] for d in range(3))))

    def helmholtz_inverse(self, c, b):
        """(M + c K)^-1 b by diagonalizing the 1D pair (K, M)."""
        n, h = self.n, self.h
        M, K = np.zeros((n + 1, n + 1)), np.zeros((n + 1, n + 1))
        for e in range(n):
            M[e:e + 2, e:e + 2] += h / 6 * np.array([[2.0, 1.0], [1.0, 2.0]])
            K[e:e + 2, e:e + 2] += 1 / h * np.array([[1.0, -1.0], [-1.0, 1.0]])
        Li = np.linalg.inv(np.linalg.cholesky(M))
        lam, Q = np.linalg.eigh(Li @ K @ Li.T)
        V = torch.from_numpy(Li.T @ Q).cuda()
        lam = torch.from_numpy(lam).cuda()
        m = n + 1
        t = torch.einsum("zyx,zc,yb,xa->cba", b.view(m, m, m), V, V, V)
        t = t / (1.0 + c * (lam[:, None, None] + lam[None, :, None] + lam[None, None, :]))
        return torch.einsum("cba,zc,yb,xa->zyx", t, V, V, V).reshape(-1)

    def solve_reinit(self, nv, b):
        x = torch.zeros_like(b)
        r = b.clone()
        p, rr = r.clone(), float(r @ r)
        stop = 1e-28 * rr
        for _ in range(2000):
            if rr <= stop:
                break
            q = self.reinit(p, nv)
            a = rr / float(p @ q)
            x += a * p
            r -= a * q
            rn = float(r @ r)
            p = r + (rn / rr) * p
            rr = rn
        return x


def _unit_normal(A, g):
    """A nodal normal field at the points, normalized (zero where it nearly vanishes)."""
    return A.unit(g, 1e-4)


def exact(case, seed):
    kind, n = case["kind"], case["n"]
    if kind in ("solve", "step"):
        return None
    s = _inputs(case, seed)
    if kind in ("apply", "fields", "adjoint", "autograd"):
        P = _Plain(case)
        x = s["x"].double()
        if kind in ("apply", "fields"):
            with torch.no_grad():
                y, yp = P.momentum(x, s["phi"], s["u0"], s["mdot"], kind == "fields" or case["divergence"])
            if kind == "fields":
                return dict(y=y, yp=yp, ug=None, flags=None)
            return [y, yp] if case["divergence"] else [y]
        v = {k: t.detach().requires_grad_(True) for k, t in dict(x=x, u0=s["u0"], phi=s["phi"], mdot=s["mdot"]).items()}
        y, yp = P.momentum(v["x"], v["phi"], v["u0"], v["mdot"])
        g = torch.autograd.grad((y, yp), list(v.values()), (s["w"], s["wp"]), allow_unused=True)
        out = {k: (t if t is not None else torch.zeros_like(v[k])) for k, t in zip(v, g)}
        return out if kind == "adjoint" else dict(out, y=y.detach(), yp=yp.detach())
    hl = 1.0 / (n * case["n_sub"])
    A = _PlainLevelSet(n * case["n_sub"], hl, min(1.0 / n, DT), 1.0 / n)
    _, g = A.at(s["phi"])
    nv = A.unit(g, 1e-4 / hl)
    if kind == "levelset":
        return [A.advect(s["psi"], s["ug"]), A.reinit(s["psi"], nv), A.reinit_rhs(s["psi"], nv)]
    c = 2.0 * hl * hl
    nrm = [A.helmholtz_inverse(c, A.assemble((A.W * nv[d]) @ A.B)) for d in range(3)]
    div = sum(A.at(nrm[d])[1][d] for d in range(3))
    kappa = A.helmholtz_inverse(c, -A.assemble((A.W * div) @ A.B))
    # surface force at the velocity quadrature points
    P = _Plain(case)
    zone, rho, mu, _, delta, B = P.material(s["phi"])
    rl, rg = RHO_L, RHO_L / case["ratio"]
    crho = (rg - rl) / (rl * rg * math.log(rg / rl))
    nq = _unit_normal(A, [f[P.il] @ B.T for f in nrm])
    V, _ = P.matrices(P.S, P.D)
    amp = P.W * 0.07 * crho * (kappa[P.il] @ B.T) * delta * rho
    f = torch.cat([P.scatter((P.p * n + 1) ** 3, P.iu, (amp * nq[d]) @ V) for d in range(3)])
    f = torch.where(P.dirichlet(), torch.zeros_like(f), f)
    frozen = _unit_normal(A, [A.at(v)[0] for v in nrm])
    psi = s["psi"]
    for _ in range(case["steps"]):
        psi = A.solve_reinit(frozen, A.reinit_rhs(psi, frozen))
    return dict(normal=torch.cat(nrm), kappa=kappa, force=f, psi=psi)

