"""The work that users of the JFNK library have it do, as cases that can be timed.

Every case goes through the public binding (`paper_1512_03662_gb300.Solver`)
on seeded synthetic states made on the GPU, and has a plain 64-bit restatement
in torch (`exact`) that shares no code with the library.  Kinds of case:

  step       one implicit time step: the step size from the CFL number, then
             the Newton-Krylov step, on a copy of the state (the call a
             simulation makes)
  residual   F(X; X^n) alone (a user's own nonlinear solver, or a check of a
             state)
  jv         one Jacobian-free product at a new linearisation point
  precond    one preconditioner apply with coefficients built at a new state
  vjp        (dG/dX)^T w, the reverse of the residual
  adjoint    gradients through one implicit step (the backward pass of the
             differentiable step)
"""
import math

import numpy as np
import torch

import paper_1512_03662_gb300 as jf

DEVICE = "cuda"
F64 = torch.float64
LAMBDA, ALPHA1, ALPHA2 = 1e-7, 1e-5, 1.0


def _case(name, kind, family, n, precision="fp64", precond=0, theta=0.5, cfl=100.0, energy=0, mach=1e-3, cycles=2, nu=2):
    n = tuple(n) + (1,) * (3 - len(n))
    return {"name": name, "kind": kind, "family": family, "nx": n[0], "ny": n[1], "nz": n[2], "precision": precision,
            "precond": precond, "theta": theta, "cfl": cfl, "energy": energy, "mach": mach, "cycles": cycles, "nu": nu}


def listed():
    return [
        # the steady Gresho vortex at 64^2, backward Euler, the default FP64 handle: the smallest step that
        # anyone takes, where launches and latency count
        _case("step_gresho_64_fp64", "step", "vortex", (64, 64), precond=1, theta=1.0, cfl=10.0, mach=1e-2),
        # the stratified atmosphere with conduction at 256^2, FP32 Krylov space: the ordinary 2D run
        _case("step_strat_256_mixed", "step", "strat", (256, 256), "mixed", precond=2, cfl=100.0, mach=0.0),
        # the Taylor-Green vortex at 64^3 on the FP64 handle: the ordinary 3D study
        _case("step_tgv_64_fp64", "step", "tgv", (64, 64, 64), precond=1, cfl=50.0, mach=1e-2),
        # the low-Mach vortex tube at 128^3, FP32 Krylov space, sound waves only
        _case("step_tube_128_mixed", "step", "vortex", (128, 128, 128), "mixed", precond=1, cfl=1000.0, mach=1e-4),
        # the convective box at 256^3 with one V(1,1) cycle per apply: the largest run, the benchmark's settings
        _case("step_convbox_256_mixed", "step", "strat", (256, 256, 256), "mixed", precond=2, cfl=200.0, mach=1e-3,
              cycles=1, nu=1),
        # the residual alone on a small ragged 2D grid, total energy (the smallest call that computes anything)
        _case("residual_100x60_etot", "residual", "vortex", (100, 60), energy=1, mach=1e-2),
        # the residual on an odd 3D grid with walls, gravity, conduction and the total energy
        _case("residual_150x131x117_etot", "residual", "strat", (150, 131, 117), energy=1),
        # a Jacobian-free product of the largest run, FP32 Krylov vectors
        _case("jv_convbox_256_mixed", "jv", "strat", (256, 256, 256), "mixed", cfl=200.0),
        # a preconditioner apply of the largest run: sound waves and conduction in FP32
        _case("precond_convbox_256_mixed", "precond", "strat", (256, 256, 256), "mixed", precond=2, cfl=200.0),
        # a preconditioner apply in 2D on the default FP64 handle, sound waves only
        _case("precond_gresho_256_fp64", "precond", "vortex", (256, 256), precond=1, theta=1.0, cfl=10.0, mach=1e-2),
        # the reverse of the residual in 3D (the adjoint runs in FP64 only)
        _case("vjp_convbox_128", "vjp", "strat", (128, 128, 128), cfl=100.0),
        # gradients through one step of the stratified atmosphere at 128^2
        _case("adjoint_strat_128", "adjoint", "strat", (128, 128), precond=2, cfl=50.0, mach=1e-4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "residual", "residual", "jv", "precond", "precond", "vjp", "adjoint"])
    precision = "fp64" if kind in ("vjp", "adjoint", "residual") else rng.choice(["fp64", "mixed", "mixed"])
    if kind == "jv":
        precision = "mixed"                    # the quotient's own rounding is 1e-8 of an FP64 product
    family = "strat" if kind == "adjoint" else rng.choice(["vortex", "strat", "strat"])
    ndim = 2 if kind == "adjoint" else rng.choice([2, 3])
    energy = rng.choice([0, 0, 1]) if kind in ("residual", "jv", "vjp", "precond") else 0
    mach = 10.0 ** rng.uniform(-4, -2) if family == "vortex" else 10.0 ** rng.uniform(-4, -2.5)
    if kind in ("residual", "jv", "vjp"):
        n = tuple(_log_int(rng, 17, 700) for _ in range(2)) if ndim == 2 else tuple(_log_int(rng, 9, 220) for _ in range(3))
        return _nameless(_case("", kind, family, n, precision, cfl=rng.choice([10.0, 50.0, 100.0]), energy=energy, mach=mach,
                               theta=rng.choice([0.5, 1.0])))
    # the preconditioner coarsens by two: powers of two, each extent of its own
    ex = {("step", 2): (5, 8), ("step", 3): (4, 7), ("precond", 2): (5, 10), ("precond", 3): (4, 7), ("adjoint", 2): (5, 7)}[kind, ndim]
    n = [2 ** rng.randint(*ex) for _ in range(ndim)]
    if kind != "precond":                      # cubic cells in the box: at most a factor of two between the extents
        n = [max(k, max(n) // 2) for k in n]
    precond = 2 if family == "strat" else 1
    cfl = min(10.0, 0.15 * max(n)) if family == "vortex" else 0.4 * min(n)
    nu = rng.choice([1, 2])
    return _nameless(_case("", kind, family, n, precision, precond, rng.choice([0.5, 1.0]), cfl * rng.uniform(0.5, 1.0), energy, mach,
                           cycles=2, nu=nu))


def _nameless(c):
    return {k: v for k, v in c.items() if k != "name"}


# ---------------------------------------------------------------------------
# physics and inputs
# ---------------------------------------------------------------------------

class Physics:
    """Grid, equation of state, gravity, conduction of one case."""

    def __init__(self, c):
        self.n = (c["nx"], c["ny"], c["nz"])
        self.ndim = 3 if c["nz"] > 1 else 2
        self.shape = self.n[::-1]
        self.nc = self.n[0] * self.n[1] * self.n[2]
        self.energy, self.theta = c["energy"], c["theta"]
        tgv = c["family"] == "tgv"
        self.gamma = 1.4 if tgv else 5.0 / 3.0
        self.gm1 = self.gamma - 1.0
        self.lo, self.hi = (0.0,) * 3, ((2.0 * math.pi,) * 3 if tgv else (1.0,) * 3)
        self.dx = [(self.hi[d] - self.lo[d]) / self.n[d] for d in range(self.ndim)]
        self.bc, self.g = [0, 0, 0], [0.0, 0.0, 0.0]
        self.K0 = 0.0
        if c["family"] == "strat":
            self.bc[self.ndim - 1], self.g[self.ndim - 1] = 1, -1.0

    def fields(self, X):
        return [X[k * self.nc:(k + 1) * self.nc].view(self.shape) for k in range(2 + self.ndim)]

    def coord(self, d, face=False):
        h = self.dx[d]
        x = self.lo[d] + (torch.arange(self.n[d], dtype=F64, device=DEVICE) + (0.0 if face else 0.5)) * h
        s = [1, 1, 1]
        s[2 - d] = self.n[d]
        return x.view(s)


def _gresho(r):
    u = torch.where(r < 0.2, 5.0 * r, torch.where(r < 0.4, 2.0 - 5.0 * r, torch.zeros_like(r)))
    r1 = r.clamp_min(1e-300)
    p = torch.where(r < 0.2, 12.5 * r * r, torch.where(r < 0.4, 12.5 * r * r - 20.0 * r + 4.0 + 4.0 * torch.log(5.0 * r1),
                                                       torch.full_like(r, -2.0 + 4.0 * math.log(2.0))))
    return u, p


def _state(c, P, gen, amp=1.0):
    """One seeded state of the case's family; `amp` scales its perturbations."""
    rand = lambda: 2.0 * torch.rand(P.shape, dtype=F64, device=DEVICE, generator=gen) - 1.0  # noqa: E731
    zero = torch.zeros(P.shape, dtype=F64, device=DEVICE)
    gm1 = P.gm1
    if c["family"] == "vortex":                # Gresho vortex in x-y, isobaric density noise of 1e-6
        xc, yc, xf, yf = (P.coord(d, f) - 0.5 for f in (False, True) for d in (0, 1))
        p = 1.0 / (P.gamma * c["mach"] ** 2) + _gresho(torch.sqrt(xc * xc + yc * yc) + zero)[1]
        rho = 1.0 + amp * 1e-6 * rand()
        rx, ry = torch.sqrt(xf * xf + yc * yc) + zero, torch.sqrt(xc * xc + yf * yf) + zero
        u = [-_gresho(rx)[0] * yc / rx.clamp_min(1e-300), _gresho(ry)[0] * xc / ry.clamp_min(1e-300)]
        u += [zero] * (P.ndim - 2)
        e = p / (gm1 * rho)
    elif c["family"] == "tgv":                 # Taylor-Green vortex, the same noise
        x, y, z, xf, yf = (P.coord(0), P.coord(1), P.coord(2), P.coord(0, True), P.coord(1, True))
        p = 1.0 / (P.gamma * c["mach"] ** 2) + (2.0 + torch.cos(2.0 * z)) * (torch.cos(2.0 * x) + torch.cos(2.0 * y)) / 16.0
        rho = 1.0 + amp * 1e-6 * rand()
        u = [torch.sin(xf) * torch.cos(y) * torch.cos(z), -torch.cos(x) * torch.sin(yf) * torch.cos(z), zero]
        e = p / (gm1 * rho)
    else:                                      # polytrope in discrete hydrostatic equilibrium, blobs, velocity noise
        gd = P.ndim - 1
        index, contrast = (1.5, 10.0) if P.ndim == 2 else (1.4, 20.0)
        nh, h = P.n[gd], P.dx[gd]
        dT, ratio = 1.0 / (index + 1.0), contrast ** (1.0 / index)
        Tb = dT / (ratio - 1.0) * ratio
        T = Tb - (np.arange(nh) + 0.5) * h / (index + 1.0)
        p = np.empty(nh)
        p[0] = T[0] * (T[0] / Tb) ** index
        for j in range(nh - 1):
            p[j + 1] = p[j] * (1.0 - h / (2.0 * T[j])) / (1.0 + h / (2.0 * T[j + 1]))
        s = [1, 1, 1]
        s[2 - gd] = nh
        T0 = torch.as_tensor(T, device=DEVICE).view(s)
        p = torch.as_tensor(p, device=DEVICE).view(s) + zero
        T = T0 + zero
        at = torch.rand((8, P.ndim), dtype=F64, device=DEVICE, generator=gen).tolist()
        for b in (at if P.ndim == 2 else at[:2]):
            r2 = zero
            for d in range(P.ndim):
                w = P.coord(d) - b[d]
                r2 = r2 + (w - torch.round(w) if P.bc[d] == 0 else w) ** 2
            T = T * (1.0 + amp * 1e-4 * torch.exp(-200.0 * r2))
        rho, e = p / T, T / gm1
        P.K0 = min(P.dx) * math.sqrt(P.gamma * float(T0.max())) / float((T0 ** 3 * gm1 / (p / T0)).max())
        u = [amp * math.sqrt(3.0) * c["mach"] * torch.sqrt(P.gamma * T0) * rand() for _ in range(P.ndim)]
        u[gd].select(2 - gd, 0).zero_()        # wall faces
    if P.energy:
        e = e + _kinetic(P, u)
    return torch.cat([f.reshape(-1) for f in [rho, e] + u])


def _inputs(c, seed):
    P = Physics(c)
    gen = torch.Generator(device=DEVICE).manual_seed(1000003 * int(seed) + 17)
    X = _state(c, P, gen)
    dt = _dt(P, X, c["cfl"])
    s = {"kind": c["kind"], "P": P, "X": X, "dt": dt, "cfl": c["cfl"]}
    if c["kind"] == "residual":                # an iterate near X^n
        s["Xn"], s["X"] = X, X * (1.0 + 1e-3 * (2.0 * torch.rand(X.shape, dtype=F64, device=DEVICE, generator=gen) - 1.0))
    if c["kind"] in ("jv", "precond", "vjp"):  # a Krylov vector: random, of unit norm, zero on wall faces
        v = _masked(P, torch.randn(X.shape, dtype=F64, device=DEVICE, generator=gen))
        s["v"] = (v / v.norm()).to(torch.float32 if c["precision"] == "mixed" else F64)
    if c["kind"] == "adjoint":                 # the step's output, a nearby state, and the gradient of its kinetic energy
        s["Xn"], s["X"] = X, X * (1.0 + 1e-4 * (2.0 * torch.rand(X.shape, dtype=F64, device=DEVICE, generator=gen) - 1.0))
        f = P.fields(s["X"])
        s["gbar"] = torch.cat([sum(0.5 * u * u for u in f[2:]).reshape(-1), torch.zeros(P.nc, dtype=F64, device=DEVICE)]
                              + [(f[0] * u).reshape(-1) for u in f[2:]])
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    P = s["P"]
    o = jf.default_options(theta=P.theta, precond=case["precond"], precision=jf.MIXED if case["precision"] == "mixed" else jf.FP64,
                           mg_cycles=case["cycles"], mg_nu1=case["nu"], mg_nu2=case["nu"],
                           eta=1e-8 if case["kind"] == "adjoint" else 1e-4)
    s["solver"] = jf.Solver(P.ndim, P.n, P.lo, P.hi, P.bc, P.gamma, P.energy, P.g, P.K0, 3.0, o, device=DEVICE)
    return s


def run(s):
    S, kind = s["solver"], s["kind"]
    if kind == "step":
        X = s["X"].clone()
        S.step(X, S.dt_from_cfl(X, s["cfl"]))
        return X
    if kind == "residual":
        return S.residual(s["X"], s["Xn"], s["dt"])
    if kind == "jv":
        return S.jv(s["X"], s["dt"], s["v"])
    if kind == "precond":
        return S.precond_apply(s["X"], s["dt"], s["v"])
    if kind == "vjp":
        return S.vjp_residual(s["X"], s["dt"], s["v"])
    return S.vjp(s["Xn"], s["X"], s["dt"], s["gbar"])[:2]


def work(case):
    """Bytes: vectors in and out, once each.  Operations: the fewest that the kind can do with.  A step evaluates
    R_U at X^n and, in each of at least two Newton iterations, once for the linearisation and once in a product."""
    P = Physics(case)
    nv, small = (2 + P.ndim) * P.nc, 4 if case["precision"] == "mixed" else 8
    vectors = {"step": 16, "residual": 24, "jv": 8 + 2 * small, "precond": 8 + 2 * small, "vjp": 24, "adjoint": 32}[case["kind"]]
    rhs = (330 if P.ndim == 3 else 170) * P.nc           # one evaluation of R_U
    evals = {"step": 5, "residual": 2, "jv": 2, "precond": 1, "vjp": 2, "adjoint": 4}[case["kind"]]
    return {"bytes": vectors * nv, "flops": evals * rhs}


# ---------------------------------------------------------------------------
# the same in plain 64-bit torch
# ---------------------------------------------------------------------------

def _at(P, q, d, k):
    """Cell quantity at i + k along d (periodic, or mirrored at walls)."""
    n = P.n[d]
    i = torch.arange(n, device=q.device) + k
    i = i % n if P.bc[d] == 0 else torch.where(i < 0, -i - 1, torch.where(i >= n, 2 * n - 1 - i, i))
    return q.index_select(2 - d, i)


def _along(P, u, d, k):
    """Velocity normal to d at face i + k (at walls zero, beyond them the odd mirror)."""
    n = P.n[d]
    i = torch.arange(n, device=u.device) + k
    if P.bc[d] == 0:
        return u.index_select(2 - d, i % n)
    sign = torch.where((i < 0) | (i > n), -1.0, torch.where((i == 0) | (i == n), 0.0, 1.0)).to(u.dtype)
    s = [1, 1, 1]
    s[2 - d] = n
    return u.index_select(2 - d, torch.where(i < 0, -i, torch.where(i > n, 2 * n - i, i % n))) * sign.view(s)


def _edge(P, d, upper):
    """0 on the wall slot of d (the lowest, or the uppermost cell), 1 elsewhere."""
    m = torch.ones(P.n[d], dtype=F64, device=DEVICE)
    if P.bc[d] == 1:
        m[-1 if upper else 0] = 0.0
    s = [1, 1, 1]
    s[2 - d] = P.n[d]
    return m.view(s)


def _upper(P, f, d):
    """Flux on the upper face of each cell (zero on a wall)."""
    return _at(P, f, d, 1) * _edge(P, d, True)


def _masked(P, X):
    f = P.fields(X)
    return torch.cat([q.reshape(-1) for q in f[:2] + [f[2 + d] * _edge(P, d, False) for d in range(P.ndim)]])


def _kinetic(P, u):
    return sum(0.25 * (u[d] ** 2 + _along(P, u[d], d, 1) ** 2) for d in range(P.ndim))


def _unpack(P, X):
    """rho, energy unknown, velocities (zero on walls), internal energy."""
    f = P.fields(X)
    u = [f[2 + d] * _edge(P, d, False) for d in range(P.ndim)]
    return f[0], f[1], u, f[1] - _kinetic(P, u) if P.energy else f[1]


def _dt(P, X, cfl):
    _, _, u, e = _unpack(P, X)
    u2 = sum((0.5 * (u[d] + _along(P, u[d], d, 1))) ** 2 for d in range(P.ndim))
    return cfl * min(P.dx) / float((torch.sqrt(u2) + torch.sqrt(P.gamma * P.gm1 * e)).max())


def _upwind(left, qm2, qm1, q0, qp1):
    """van Leer face value between qm1 and q0, from the left where `left`."""
    near, far, other = torch.where(left, qm1, q0), torch.where(left, qm2, qp1), torch.where(left, q0, qm1)
    a, b = near - far, other - near
    on = a * b > 0
    return near + torch.where(on, a * b / torch.where(on, a + b, torch.ones_like(a)), torch.zeros_like(a))


def _rhs(P, X, K0=None):
    """Conserved variables U(X) and the right-hand side R_U(X)."""
    rho, E, u, e = _unpack(P, X)
    K0 = P.K0 if K0 is None else K0
    p, T = P.gm1 * rho * e, P.gm1 * e
    chi = K0 * T ** 3
    nd, h = P.ndim, P.dx
    fm, fe = [], []
    for d in range(nd):
        left = u[d] >= 0
        st = lambda q: [_at(P, q, d, k) for k in (-2, -1)] + [q, _at(P, q, d, 1)]  # noqa: E731
        fm.append(u[d] * _upwind(left, *st(rho)))
        f = fm[d] * _upwind(left, *st(E))
        if P.energy:
            f = f + 0.5 * (_at(P, p, d, -1) + p) * u[d]
        fe.append(f - 0.5 * (_at(P, chi, d, -1) + chi) * (T - _at(P, T, d, -1)) / h[d])
    Rr = -sum((_upper(P, fm[d], d) - fm[d]) / h[d] for d in range(nd))
    RE = -sum((_upper(P, fe[d], d) - fe[d]) / h[d] for d in range(nd))
    if P.energy:
        RE = RE + sum(P.g[d] * 0.5 * (fm[d] + _upper(P, fm[d], d)) for d in range(nd) if P.g[d])
    else:
        RE = RE - p * sum((_along(P, u[d], d, 1) - u[d]) / h[d] for d in range(nd))
    U, R = [rho, rho * E], [Rr, RE]
    for c in range(nd):
        rf = 0.5 * (_at(P, rho, c, -1) + rho)
        r = (_at(P, p, c, -1) - p) / h[c] + rf * P.g[c]
        for d in range(nd):
            if c == d:
                m = 0.5 * (fm[c] + _upper(P, fm[c], c))
                psi = m * _upwind(m >= 0, *[_along(P, u[c], c, k) for k in (-1, 0, 1, 2)])
                r = r - (psi - _at(P, psi, c, -1)) / h[c]
            else:
                m = 0.5 * (_at(P, fm[d], c, -1) + fm[d])
                psi = m * _upwind(m >= 0, *[_at(P, u[c], d, k) for k in (-2, -1, 0, 1)])
                r = r - (_upper(P, psi, d) - psi) / h[d]
        U.append(rf * u[c])
        R.append(r * _edge(P, c, False))
    return torch.cat([q.reshape(-1) for q in U]), torch.cat([q.reshape(-1) for q in R])


def _G(P, X, dt):
    U, R = _rhs(P, X)
    return U / dt - P.theta * R


def _scaling(P, X):
    rho, E, u, e = _unpack(P, X)
    cs = torch.sqrt(P.gamma * P.gm1 * e)
    L, R = [rho, rho * E], [rho, E]
    for d in range(P.ndim):
        cf, rf, w = 0.5 * (_at(P, cs, d, -1) + cs), 0.5 * (_at(P, rho, d, -1) + rho), _edge(P, d, False) > 0
        one = torch.ones_like(cf)
        L.append(torch.where(w, rf * torch.maximum(u[d].abs(), ALPHA1 * cf), one))
        R.append(torch.where(w, torch.maximum(u[d].abs(), ALPHA2 * cf), one))
    return torch.cat([q.reshape(-1) for q in L]), torch.cat([q.reshape(-1) for q in R])


class Preconditioner:
    """M^-1 at a state: transform to (p, e, u), the semi-implicit system by V-cycles, back substitution."""

    def __init__(self, c, P, X, dt):
        self.P, self.dt, self.nf, self.cycles, self.nu = P, dt, c["precond"], c["cycles"], c["nu"]
        self.L, self.R = _scaling(P, X)
        self.rho, self.E, self.u, e = _unpack(P, X)
        th, rho, gm1 = P.theta, self.rho, P.gm1
        p = gm1 * rho * e
        self.dpr, self.dpe, self.cde = gm1 * e, gm1 * rho, 1.0 / (P.gamma * rho)
        self.rf = [0.5 * (_at(P, rho, d, -1) + rho) for d in range(P.ndim)]
        bpp = th * th * dt * P.gamma * p
        if self.nf == 1:
            self.B = [[1.0 / bpp]]
        else:
            bpe, bep, bee = th * gm1, th * th * dt * p / rho, th / rho
            det = bpp * bee - bpe * bep
            self.B = [[bee / det, -bpe / det], [-bep / det, bpp / det]]
        M = [[b / dt for b in row] for row in self.B]
        chi = P.K0 * (gm1 * e) ** 3
        K = [[_edge(P, d, False) / self.rf[d] for d in range(P.ndim)]]
        if self.nf == 2:
            K.append([_edge(P, d, False) * 0.5 * (_at(P, chi, d, -1) + chi) * gm1 for d in range(P.ndim)])
        self.levels = [self._level(M, K, list(P.n), list(P.dx))]
        while max(self.levels[-1]["n"]) > 1:
            self.levels.append(self._coarser(self.levels[-1]))

    def _level(self, M, K, n, h):
        nz, ny, nx = (torch.arange(k, device=DEVICE) for k in n[::-1])
        red = (nz.view(-1, 1, 1) + ny.view(1, -1, 1) + nx.view(1, 1, -1)) % 2 == 0
        dirs = [d for d in range(self.P.ndim) if n[d] > 1]
        A = [[M[i][j] for j in range(self.nf)] for i in range(self.nf)]
        for f in range(self.nf):
            A[f][f] = A[f][f] + sum((K[f][d] + torch.roll(K[f][d], -1, 2 - d)) / h[d] ** 2 for d in dirs)
        if self.nf == 1:
            inv = [[1.0 / A[0][0]]]
        else:
            det = A[0][0] * A[1][1] - A[0][1] * A[1][0]
            inv = [[A[1][1] / det, -A[0][1] / det], [-A[1][0] / det, A[0][0] / det]]
        return {"M": M, "K": K, "n": n, "h": h, "red": red, "dirs": dirs, "inv": inv}

    def _coarser(self, v):
        def halve(q, d, mean):
            a = q.unflatten(2 - d, (q.shape[2 - d] // 2, 2))
            return a.mean(3 - d) if mean else a.select(3 - d, 0)
        M = v["M"]
        K = [[k for k in row] for row in v["K"]]
        n, h = list(v["n"]), list(v["h"])
        for d in v["dirs"]:
            M = [[halve(q, d, True) for q in row] for row in M]
            K = [[halve(q, d, a != d) for a, q in enumerate(row)] for row in K]
            n[d], h[d] = n[d] // 2, 2.0 * h[d]
        for row in K:
            for d in range(self.P.ndim):
                if n[d] == 1:
                    row[d] = torch.zeros_like(row[d])
        return self._level(M, K, n, h)

    def _diffusion(self, v, x, f, diagonal):
        """Off-diagonal (diagonal False) or whole diffusion operator of field f, with the sign of M."""
        out = torch.zeros_like(x)
        for d in v["dirs"]:
            a = 2 - d
            K = v["K"][f][d]
            Ku, up, dn = torch.roll(K, -1, a), torch.roll(x, -1, a), torch.roll(x, 1, a)
            out = out - (Ku * (up - x) - K * (x - dn) if diagonal else Ku * up + K * dn) / v["h"][d] ** 2
        return out

    def _times(self, A, x):
        return [sum(A[i][j] * x[j] for j in range(self.nf)) for i in range(self.nf)]

    def _sweep(self, v, x, b, colour):
        r = [b[f] - self._diffusion(v, x[f], f, False) for f in range(self.nf)]
        at = v["red"] if colour == 0 else ~v["red"]
        return [torch.where(at, y, q) for y, q in zip(self._times(v["inv"], r), x)]

    def _prolong(self, x, fine, coarse):
        for d in fine["dirs"]:
            a, n = 2 - d, coarse["n"][d]
            i = torch.arange(n, device=DEVICE)
            lo, hi = ((i - 1) % n, (i + 1) % n) if self.P.bc[d] == 0 else ((i - 1).clamp_min(0), (i + 1).clamp_max(n - 1))
            x = torch.stack([0.75 * x + 0.25 * x.index_select(a, lo), 0.75 * x + 0.25 * x.index_select(a, hi)], a + 1).flatten(a, a + 1)
        return x

    def _vcycle(self, l, x, b):
        v = self.levels[l]
        if l + 1 == len(self.levels):
            return self._times(v["inv"], b)
        for _ in range(self.nu):
            x = self._sweep(v, self._sweep(v, x, b, 0), b, 1)
        w = self._times(v["M"], x)
        r = [b[f] - w[f] - self._diffusion(v, x[f], f, True) for f in range(self.nf)]
        for d in v["dirs"]:
            r = [q.unflatten(2 - d, (q.shape[2 - d] // 2, 2)).mean(3 - d) for q in r]
        y = self._vcycle(l + 1, [torch.zeros_like(q) for q in r], r)
        x = [q + self._prolong(z, v, self.levels[l + 1]) for q, z in zip(x, y)]
        for _ in range(self.nu):
            x = self._sweep(v, self._sweep(v, x, b, 1), b, 0)
        return x

    def apply(self, w):
        P, dt, th, nd = self.P, self.dt, self.P.theta, self.P.ndim
        v = P.fields(self.L * w)
        mean = lambda a: sum(0.5 * (self.u[d] * a[d] + _along(P, self.u[d], d, 1) * _upper(P, a[d], d)) for d in range(nd))  # noqa: E731
        ru = [(v[2 + d] - self.u[d] * 0.5 * (_at(P, v[0], d, -1) + v[0])) / self.rf[d] * _edge(P, d, False) for d in range(nd)]
        re = (v[1] - self.E * v[0]) / self.rho - (mean(ru) if P.energy else 0.0)
        rp = self.dpr * v[0] + self.dpe * re
        b = self._times(self.B, [rp, re][:self.nf])
        x = [torch.zeros_like(rp) for _ in range(self.nf)]
        for _ in range(self.cycles):
            x = self._vcycle(0, x, b)
        dp = x[0]
        de = x[1] if self.nf == 2 else dt * (re + (dp / dt - rp) * self.cde)
        du = [dt * (ru[d] - th * _edge(P, d, False) / (P.dx[d] * self.rf[d]) * (dp - _at(P, dp, d, -1))) for d in range(nd)]
        z = [(dp - self.dpe * de) / self.dpr, de + (mean(du) if P.energy else 0.0)] + du
        return torch.cat([q.reshape(-1) for q in z]) / self.R


def _gmres(A, b, tol, most=200):
    """Full GMRES with two Gram-Schmidt passes from a zero start."""
    beta = float(b.norm())
    V, H, y = [b / beta], [], None
    for j in range(most):
        w, h = A(V[j]), np.zeros(j + 2)
        for _ in range(2):
            for i, q in enumerate(V):
                a = float(torch.dot(q, w))
                h[i] += a
                w = w - a * q
        h[j + 1] = float(w.norm())
        H.append(h)
        V.append(w / h[j + 1])
        m = np.zeros((j + 2, j + 1))
        for k, col in enumerate(H):
            m[:len(col), k] = col
        rhs = np.zeros(j + 2)
        rhs[0] = beta
        y = np.linalg.lstsq(m, rhs, rcond=None)[0]
        if np.linalg.norm(m @ y - rhs) < tol * beta:
            break
    return sum(float(y[i]) * V[i] for i in range(len(y)))


def _step(c, P, X, dt):
    """X^{n+1} by Newton with the exact derivative."""
    U, R = _rhs(P, X)
    bn = U / dt + (1.0 - P.theta) * R
    for _ in range(12):
        M = Preconditioner(c, P, X, dt)
        product = lambda w: torch.func.jvp(lambda Y: _G(P, Y, dt), (X,), (_masked(P, M.R * w),))[1] / M.L  # noqa: E731, B023
        F = _masked(P, (_G(P, X, dt) - bn) / M.L)
        dx = M.apply(_gmres(lambda w: product(M.apply(w)), -F, 1e-6))  # noqa: B023
        X = X + M.R * dx
        if float(dx.abs().max()) < 1e-11:
            break
    return X


def exact(case, seed):
    kind = case["kind"]
    if kind == "step" and case["nx"] * case["ny"] * case["nz"] > 2 ** 21:
        return None
    s = _inputs(case, seed)
    P, X, dt = s["P"], s["X"], s["dt"]
    if kind == "step":
        return _step(case, P, X, dt)
    if kind == "residual":
        (U, R), (Un, Rn) = _rhs(P, X), _rhs(P, s["Xn"])
        return _masked(P, (U - Un) / dt - P.theta * R - (1.0 - P.theta) * Rn)
    if kind == "jv":
        v = s["v"].double()
        L, R = _scaling(P, X)
        delta = LAMBDA * (LAMBDA + float(_masked(P, X / R).norm()) / float(v.norm()))
        return _masked(P, (_G(P, X + delta * R * v, dt) - _G(P, X, dt)) / L / delta), delta
    if kind == "precond":
        return Preconditioner(case, P, X, dt).apply(s["v"].double())
    if kind == "vjp":
        return _reverse(lambda Y: _G(P, Y, dt), X, s["v"], P)
    M = Preconditioner(case, P, X, dt)
    apply_t = lambda w: torch.func.vjp(M.apply, w)[1](w)[0]  # noqa: E731
    jt = lambda w: _masked(P, M.R * _reverse(lambda Y: _G(P, Y, dt), X, w / M.L, P))  # noqa: E731
    lam = apply_t(_gmres(lambda w: jt(apply_t(w)), _masked(P, M.R * s["gbar"]), 1e-11)) / M.L

    def back(Y, share):                        # (dU/dX / dt + share dR/dX)^T lam, and lam . dR/dK0
        def f(Z, K0):
            U, R = _rhs(P, Z, K0)
            return U / dt + share * R
        g, k = torch.func.vjp(f, Y, torch.tensor(P.K0, dtype=F64, device=DEVICE))[1](lam)
        return _masked(P, g), float(k)
    g, kn = back(s["Xn"], 1.0 - P.theta)
    return g, kn + back(X, P.theta)[1]


def _reverse(f, X, w, P):
    return _masked(P, torch.func.vjp(f, X)[1](w)[0])
