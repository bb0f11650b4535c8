"""What this library is measured on: calls of its public entry points over the
range of meshes, degrees, systems and step kinds that its users step.

``listed`` gives the fixed cases, ``draw`` one more of the same ranges,
``prepare`` what a program holds before the call (context, coefficients,
state), ``run`` one call, ``exact`` the same result from a plain FP64 torch
restatement of the method (its own derivation of the reference element, no
code of this library), ``work`` the bytes and operations a call cannot do
without.

All fields are FP64 and periodic: bathymetry made of Gaussians, a free surface
near 1 with a small wave or bump (with the limiter a dam break, so that the
limiter acts), a weak current, and for advection a sine over a varying speed.
"""
import math

import numpy as np
import torch

GRAVITY = 9.81
LENGTH = 100.0
SAFETY = 0.5
CHEZY = 0.0025
DAMPING = 3.0
# CFL(N) of each node family (von Neumann limit of the scheme), without and
# with a source; given to the contexts so that both sides use the same number
CFL = {"gl": (1.0, 0.3333333333335, 0.17082039325001908, 0.10392896184871106,
              0.0698339246590344),
       "gll": (None, 1.0, 0.33333333333338905, 0.17082039324997397, 0.10393143536412303)}
CFL_SOURCE = {"gl": (1.0, 0.33333333333350007, 0.17082039325001908, 0.10392896184871109,
                     0.06983356899807755),
              "gll": (None, 1.0, 0.33333333333338905, 0.17325286209315088, 0.10592411182188002)}
VARIABLES = {"varadv1d": 1, "swe1d": 2, "swe1d_wb": 2, "swe2d": 3, "swe2d_wb": 3}


def _case(kind, system, degree, nx, ny=0, nodes="gl", steps=1, source="", limiter="", name=None):
    c = dict(kind=kind, system=system, degree=degree, nx=nx, ny=ny, nodes=nodes, steps=steps,
             source=source, limiter=limiter)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest runs: a 1D verification mesh, time step from the state,
        # a few kernel launches of little work
        _case("step", "varadv1d", 3, 100, steps=20, name="advection-100-N3"),
        # an ordinary 1D run: 1e5 elements at the highest degree
        _case("step", "swe1d", 4, 100000, steps=4, name="swe1d-100000-N4"),
        # 1D flood wave: well-balanced form, Lobatto points, limiter on, an odd size
        _case("step", "swe1d_wb", 3, 30011, nodes="gll", steps=4, limiter="blend",
              name="swe1d_wb-30011-N3-gll-limited"),
        # ragged ensemble of 1D meshes (parameter study), replayed graph
        _case("ensemble", "swe1d", 0, 256, steps=2, name="swe1d-ensemble-256"),
        # a small 2D run (coarse grid of a convergence study)
        _case("step", "swe2d", 2, 65, 47, nodes="gll", steps=8, name="swe2d-65x47-N2-gll"),
        # the headline workload: a large 2D mesh
        _case("step", "swe2d", 3, 1024, 1024, steps=2, name="swe2d-1024x1024-N3"),
        # bottom friction, treated implicitly
        _case("step", "swe2d", 3, 512, 512, steps=2, source="chezy",
              name="swe2d-512x512-N3-chezy"),
        # well-balanced form, highest degree, odd sizes
        _case("step", "swe2d_wb", 4, 401, 307, steps=2, name="swe2d_wb-401x307-N4"),
        # dam break with the subcell limiter
        _case("step", "swe2d", 3, 640, 384, steps=2, limiter="blend",
              name="swe2d-640x384-N3-limited"),
        # forward and backward pass: gradient with respect to the bathymetry
        _case("adjoint", "swe2d", 3, 256, 256, steps=6, name="adjoint-256x256-N3"),
        # coupling to a program that keeps its state on the host
        _case("host", "swe2d", 3, 768, 768, steps=1, name="host-swe2d-768x768-N3"),
        # the right-hand side alone, as an outer time integrator calls it
        _case("residual", "swe2d", 1, 719, 523, name="residual-swe2d-719x523-N1"),
    ]


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step"] * 9 + ["noalloc", "ensemble", "adjoint", "host", "residual"])
    nodes = rng.choice(["gl", "gl", "gll"])
    if kind == "ensemble":
        return _case(kind, rng.choice(["swe1d", "swe1d_wb", "varadv1d"]), 0, _spread(rng, 8, 200),
                     nodes=nodes, steps=rng.randint(1, 2), source=rng.choice(["", "", "source"]))
    if kind == "noalloc":
        return _case(kind, rng.choice(["swe1d", "swe1d_wb", "varadv1d"]), rng.randint(1, 4),
                     _spread(rng, 20, 100000), nodes=nodes, steps=rng.randint(1, 8))
    if kind == "step" and rng.random() < 0.4:
        system = rng.choice(["swe1d", "swe1d", "swe1d_wb", "varadv1d"])
        source = rng.choice(["", "", "linear" if system == "varadv1d" else "chezy"])
        return _case(kind, system, rng.randint(1, 4), _spread(rng, 20, 250000), nodes=nodes,
                     steps=rng.randint(1, 8), source=source,
                     limiter=rng.choice(["", "", "blend"]))
    degree = rng.randint(1, 4)
    nx, ny = _spread(rng, 9, 900), _spread(rng, 9, 900)
    steps = rng.randint(2, 6) if kind == "adjoint" else rng.randint(1, 4)
    if kind == "adjoint":
        nx, ny, nodes = min(nx, 300), min(ny, 300), "gl"
    if kind == "residual":
        steps = 1
    # at most about half the largest listed case's work
    budget = 16e6 / ((degree + 1) ** 2 * steps * (4 if kind == "adjoint" else 1))
    while nx * ny > budget:
        nx, ny = (nx * 3) // 4, (ny * 3) // 4
    plain = kind in ("adjoint", "residual")
    return _case(kind, "swe2d" if kind == "adjoint" else rng.choice(["swe2d", "swe2d", "swe2d_wb"]),
                 degree, nx, ny, nodes=nodes, steps=steps,
                 source="" if plain else rng.choice(["", "", "chezy"]),
                 limiter="" if plain else rng.choice(["", "", "blend"]))


# ---------------------------------------------------------------------------
# the reference element, in FP64 from the definitions
# ---------------------------------------------------------------------------
class _Element:
    def __init__(self, degree, family):
        n = degree + 1
        if family == "gl" or n == 1:
            x, w = np.polynomial.legendre.leggauss(n)
        else:
            P = np.polynomial.legendre.Legendre.basis(degree)
            x = np.concatenate([[-1.0], np.sort(P.deriv().roots().real), [1.0]])
            x = 0.5 * (x - x[::-1])
            w = 2.0 / (degree * n * P(x) ** 2)
        self.n, self.xi, self.w = n, 0.5 * (x + 1.0), 0.5 * w
        # barycentric weights; D by the negative sum trick
        d = x[:, None] - x[None, :] + np.eye(n)
        bw = 1.0 / np.prod(d, axis=1)
        D = 2.0 * (bw[None, :] / bw[:, None]) / d
        np.fill_diagonal(D, 0.0)
        np.fill_diagonal(D, -D.sum(axis=1))
        self.D = D
        end = lambda s: np.array([np.prod([(s - x[k]) / (x[j] - x[k]) for k in range(n) if k != j])
                                  for j in range(n)])
        self.l0, self.l1 = end(-1.0), end(1.0)
        # derivatives of the Radau (GL points) or g_2 (GLL points) corrections
        self.gL, self.gR = -self.l0 / self.w, self.l1 / self.w
        modes = np.stack([np.polynomial.legendre.Legendre.basis(j)(x) * math.sqrt((2 * j + 1) / 2)
                          for j in range(n)], axis=1)
        self.to_modes = np.linalg.inv(modes)


def _tableau(degree, source):
    """(explicit a, implicit a, b) of the stages."""
    if source:
        al, be, et = 0.241694260788, 0.0604235651970, 0.12915286960590
        A = [[0, 0, 0, 0], [0, 0, 0, 0], [0, 1, 0, 0], [0, 0.25, 0.25, 0]]
        Ai = [[al, 0, 0, 0], [-al, al, 0, 0], [0, 1 - al, al, 0], [be, et, 0.5 - be - et - al, al]]
        return A, Ai, [0, 1 / 6, 1 / 6, 2 / 3]
    A, b = {0: ([[0]], [1]),
            1: ([[0, 0], [1, 0]], [0.5, 0.5]),
            2: ([[0, 0, 0], [1, 0, 0], [0.25, 0.25, 0]], [1 / 6, 1 / 6, 2 / 3]),
            3: ([[0, 0, 0, 0], [0.5, 0, 0, 0], [0, 0.5, 0, 0], [0, 0, 1, 0]],
                [1 / 6, 1 / 3, 1 / 3, 1 / 6]),
            4: ([[0] * 6, [0.25, 0, 0, 0, 0, 0], [0.125, 0.125, 0, 0, 0, 0],
                 [0, -0.5, 1, 0, 0, 0], [3 / 16, 0, 0, 9 / 16, 0, 0],
                 [-3 / 7, 2 / 7, 12 / 7, -12 / 7, 8 / 7, 0]],
                [7 / 90, 0, 32 / 90, 12 / 90, 32 / 90, 7 / 90])}[degree]
    return A, None, b


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _source_of(case):
    """(source, coefficient) of a case ("source": that of its system)."""
    if not case["source"]:
        return None, 0.0
    return ("linear", DAMPING) if case["system"] == "varadv1d" else ("chezy", CHEZY)


def _cfl_number(case, degree):
    return (CFL_SOURCE if case["source"] else CFL)[case["nodes"]][degree]


def _gap(x, centre):
    d = (x - centre).abs()
    return torch.minimum(d, LENGTH - d)


def _positions(element, E, device):
    xi = torch.tensor(element.xi, device=device)
    return (torch.arange(E, device=device, dtype=torch.float64)[:, None] + xi) * (LENGTH / E)


def _fields(case, seed, degree, nx, ny, device):
    """(state, coefficient field) of a mesh in the library's layout."""
    rng = np.random.default_rng(seed)
    el = _Element(degree, case["nodes"])
    x = _positions(el, nx, device)
    if case["system"] == "varadv1d":
        k = 2 * math.pi / LENGTH
        a, v = rng.uniform(0.0, 2 * math.pi, 2)
        return torch.sin(k * x + v)[None].contiguous(), 1.0 + 0.5 * torch.sin(k * x + a)
    two = VARIABLES[case["system"]] == 3
    count = 32 if two else 8
    amp, width = rng.uniform(0.05, 0.3, count), rng.uniform(1.0, 5.0, count)
    cx, cy = rng.uniform(0.0, LENGTH, (2, count))
    phase, current = rng.uniform(0.0, 2 * math.pi, 4), rng.uniform(-0.3, 0.3, 2)
    bell = lambda t, c, s: torch.exp(-_gap(t, c) ** 2 / (2 * s * s))
    if two:
        y = _positions(el, ny, device)
        # sum of products of 1D bells: one matrix product over the Gaussians
        bx = torch.stack([A * bell(x, c, s).reshape(-1) for A, s, c in zip(amp, width, cx)])
        by = torch.stack([bell(y, c, s).reshape(-1) for s, c in zip(width, cy)])
        b = (by.T @ bx).reshape(ny, el.n, nx, el.n)
        gx, gy = _gap(x, cx[0]).reshape(-1), _gap(y, cy[0]).reshape(-1)
        r2 = (gy[:, None] ** 2 + gx[None, :] ** 2).reshape(ny, el.n, nx, el.n)
        b, r2 = (t.permute(0, 2, 1, 3).contiguous() for t in (b, r2))
        eta = 1.0 + (0.3 * (r2 < 400.0) if case["limiter"] else
                     0.01 * torch.exp(-r2 / (2 * width[0] ** 2)))
    else:
        b = sum(A * bell(x, c, s) for A, s, c in zip(amp, width, cx))
        k = 2 * math.pi / LENGTH
        eta = 1.0 + (0.3 * (_gap(x, cx[0]) < 20.0) if case["limiter"] else
                     0.01 * sum(torch.sin((j + 1) * k * x + p) for j, p in enumerate(phase)) / 4)
    b = b * min(1.0, 0.7 / float(b.max()))
    h = eta - b
    return torch.stack([h] + [float(c) * h for c in current[:1 + two]]), b


def _members(case):
    """(degree, elements) of each mesh of an ensemble: 2^10 to 2^16 elements."""
    rng = np.random.default_rng(case["nx"])
    E = np.floor(2.0 ** rng.uniform(10, 16, case["nx"])).astype(int)
    return [(int(d), int(e)) for d, e in zip(rng.choice([2, 3, 4], case["nx"]), E)]


def _fixed_dt(case):
    speed = 0.6 + math.sqrt(GRAVITY * 1.4)
    return (SAFETY * _cfl_number(case, case["degree"]) /
            (speed * (case["nx"] + case["ny"]) / LENGTH))


def _eta0(state, b):
    return state[0] + b


# ---------------------------------------------------------------------------
# the library
# ---------------------------------------------------------------------------
def prepare(case, seed):
    from paper_2512_08611_gb300 import crkfr
    source, coef = _source_of(case)
    if case["kind"] == "ensemble":
        members = _members(case)
        # CFL numbers per degree come from the library here
        batch = crkfr.Batch(case["system"], [(d, e, 0.0, LENGTH) for d, e in members],
                            nodes=case["nodes"], gravity=GRAVITY, cfl_safety=SAFETY, source=source,
                            source_coef=coef)
        u0 = torch.empty(batch.state_offsets[-1], dtype=torch.float64, device="cuda")
        c = torch.empty(batch.coef_offsets[-1], dtype=torch.float64, device="cuda")
        for i, (d, e) in enumerate(members):
            u, b = _fields(case, [seed, i], d, e, 0, "cuda")
            batch.state_view(u0, i).copy_(u)
            batch.coef_view(c, i).copy_(b)
        batch.set_coefficients(c)
        return dict(case=case, batch=batch, u0=u0, u=torch.empty_like(u0), c=c)
    u0, c = _fields(case, seed, case["degree"], case["nx"], case["ny"], "cuda")
    state = dict(case=case, u0=u0, c=c)
    cfl = _cfl_number(case, case["degree"])
    if case["kind"] == "noalloc":
        state["u"] = torch.empty_like(u0)
        return state
    s = crkfr.Solver(case["system"], case["degree"], nodes=case["nodes"], gravity=GRAVITY,
                     cfl_safety=SAFETY, cfl_number=cfl, source=source, source_coef=coef)
    if VARIABLES[case["system"]] == 3:
        s.set_mesh([case["nx"], case["ny"]], [0.0, 0.0], [LENGTH, LENGTH])
    else:
        s.set_mesh([case["nx"]], [0.0], [LENGTH])
    s.set_coefficients(c)
    if case["limiter"]:
        s.set_limiter(case["limiter"])
    state["solver"] = s
    if case["kind"] == "host":
        pinned = lambda: torch.empty(u0.shape, dtype=torch.float64, pin_memory=True)
        state["in"], state["out"] = pinned(), pinned()
        state["in"].copy_(u0)
        del state["u0"]
    elif case["kind"] == "adjoint":
        # an observed free surface to fit, and the first guess of the bathymetry
        state["b"] = c.clone().requires_grad_(True)
        state["eta0"] = _eta0(u0, c)
        state["target"] = 1.0 + 0.005 * torch.sin(torch.linspace(0, 40, c.numel(), device="cuda",
                                                                 dtype=torch.float64)).view_as(c)
        from paper_2512_08611_gb300.adjoint import quadrature_weights
        state["weights"] = quadrature_weights(s)
    else:
        state["u"] = torch.empty_like(u0)
    return state


def run(state):
    case = state["case"]
    kind, steps = case["kind"], case["steps"]
    if kind == "ensemble":
        state["u"].copy_(state["u0"])
        return state["batch"].step(state["u"], 0.0, steps)
    if kind == "noalloc":
        from paper_2512_08611_gb300 import crkfr
        return crkfr.step_1d_noalloc(case["system"], case["degree"], case["nx"], 0.0, LENGTH,
                                     state["c"], state["u0"], state["u"], 0.0, steps,
                                     nodes=case["nodes"], gravity=GRAVITY, cfl_safety=SAFETY,
                                     cfl_number=_cfl_number(case, case["degree"]))
    s = state["solver"]
    if kind == "host":
        return s.step_host(state["in"].numpy(), state["out"].numpy(), 0.0, steps)
    if kind == "residual":
        return s.residual(state["u0"], _fixed_dt(case), state["u"])
    if kind == "adjoint":
        from paper_2512_08611_gb300.adjoint import BathymetryToState, surface_misfit
        b = state["b"]
        b.grad = None
        u = BathymetryToState.apply(b, s, state["eta0"], _fixed_dt(case), steps, 3)
        surface_misfit(u, b, state["target"], state["weights"]).backward()
        return {"u": u.detach(), "gradient": b.grad}
    state["u"].copy_(state["u0"])
    return s.step(state["u"], 0.0, steps)


def work(case):
    """Per step: the state read and written and the coefficients read, once;
    operations of the stages, the traces and the face terms as the method
    states them (an FMA is two).  An adjoint pass steps forward, steps again
    from its checkpoint, and back: three times a step's bytes, four times its
    operations (the linearised stages forward and back)."""
    M = VARIABLES[case["system"]]
    dim = 2 if M == 3 else 1
    meshes = _members(case) if case["kind"] == "ensemble" else [
        (case["degree"], case["nx"] * max(1, case["ny"]))]
    nbytes = flops = 0
    for degree, elements in meshes:
        n = degree + 1
        A, _, b = _tableau(degree, case["source"])
        used = [any(row[j] for row in A) or bool(b[j]) for j in range(len(b))]
        per_node = 0
        for i in range(len(b)):
            per_node += 2 * M * sum(1 for a in A[i] if a) + 2 * (3 * M - 1) * bool(b[i])
            if case["source"]:
                per_node += 4 * M + 16 * (M > 1)
            if used[i]:
                per_node += 2 * dim * M * n + (2 if M == 1 else 6 * M)
        traces = 2 * (2 * M + 1) * dim
        nodes = elements * n ** dim
        flops += nodes * (per_node + 2 * traces + 6 * M * dim) + elements * dim * n ** (dim - 1) * 40
        if case["limiter"]:
            flops += nodes * dim * (14 * M)
        nbytes += nodes * (2 * M + 1) * 8
    times = case["steps"]
    adjoint = case["kind"] == "adjoint"
    return {"bytes": float(nbytes * times * (3 if adjoint else 1)),
            "flops": float(flops * times * (4 if adjoint else 1))}


# ---------------------------------------------------------------------------
# the method in plain torch
# ---------------------------------------------------------------------------
class _Method:
    """One mesh: states u[var, ey, ex, q, p] (1D: ey and q of length 1)."""

    def __init__(self, case, degree, nx, ny, device):
        self.case, self.el = case, _Element(degree, case["nodes"])
        self.system = case["system"]
        self.M = VARIABLES[self.system]
        self.dims = (0, 1) if self.M == 3 else (0,)
        self.wb = self.system.endswith("_wb")
        self.h = (LENGTH / nx, LENGTH / max(ny, 1))
        self.A, self.Ai, self.b = _tableau(degree, case["source"])
        self.cfl = SAFETY * _cfl_number(case, degree)
        t = lambda a: torch.tensor(a, dtype=torch.float64, device=device)
        el = self.el
        self.D, self.l0, self.l1, self.gL, self.gR, self.w = map(
            t, (el.D, el.l0, el.l1, el.gL, el.gR, el.w))
        self.modes = t(el.to_modes)

    # -- along one direction (0: x, the last axis; 1: y, the one before) --------
    def dloc(self, F, d):
        return (F @ self.D.T if d == 0 else self.D @ F) / self.h[d]

    def trace(self, F, row, d):
        return F @ row if d == 0 else row @ F

    def next(self, F, d, by=-1):
        """Value of the next element (trace arrays [.., ey, ex, node])."""
        return torch.roll(F, by, -2 if d == 0 else -3)

    def outer(self, T, g, d):
        return T[..., None] * g if d == 0 else T[..., None, :] * g[:, None]

    # -- the system ---------------------------------------------------------------
    def flux(self, u, d):
        if self.M == 1:
            return torch.zeros_like(u)
        h, m = u[0], u[1:]
        v = m[d] / h
        f = [m[d]] + [m[k] * v + (0.5 * GRAVITY * h * h if k == d and not self.wb else 0.0)
                      for k in range(self.M - 1)]
        return torch.stack(f)

    def product(self, u, c, du, dc, d):
        """B_d(u, c) (du, dc)."""
        if self.M == 1:
            return c * du
        out = [torch.zeros_like(u[0]) for _ in range(self.M)]
        out[1 + d] = GRAVITY * u[0] * (du[0] + dc if self.wb else dc + torch.zeros_like(u[0]))
        return torch.stack(out)

    def speed(self, u, c, d):
        return c.abs() if self.M == 1 else (u[1 + d] / u[0]).abs() + torch.sqrt(GRAVITY * u[0])

    def jump(self, up, um, cp, cm):
        j = up - um
        return torch.cat([j[:1] + (cp - cm), j[1:]]) if self.wb else j

    def implicit(self, r, gamma):
        """u with u - gamma s(u) = r."""
        if self.M == 1:
            return r / (1.0 + gamma * DAMPING)
        q = torch.sqrt((r[1:] ** 2).sum(0)) * (4.0 * gamma * CHEZY) / r[0] ** 2
        return torch.cat([r[:1], r[1:] * (2.0 / (1.0 + torch.sqrt(1.0 + q)))])

    def source(self, u):
        if self.M == 1:
            return -DAMPING * u
        speed = torch.sqrt((u[1:] ** 2).sum(0)) / u[0]
        return torch.cat([torch.zeros_like(u[:1]), -CHEZY * speed * u[1:] / u[0]])

    def time_step(self, u, c):
        w = self.w
        mean = lambda F: (F @ w if len(self.dims) == 1 else (F @ w) @ w)
        if len(self.dims) == 1:
            um, cm = mean(u), mean(c)
        else:
            um, cm = mean(u), mean(c)
        return self.cfl / sum(self.speed(um, cm, d) / self.h[d] for d in self.dims).max()

    # -- one step -------------------------------------------------------------------
    def update(self, u, c, dt):
        """(u^n - dt times the residual's local part, face data of each direction)."""
        dc = [self.dloc(c, d) for d in self.dims]
        Ls, Ss = [], []
        V = U = S = 0.0
        F = [0.0 for _ in self.dims]
        for i in range(len(self.b)):
            r = u
            for j in range(i):
                if self.A[i][j]:
                    r = r - (dt * self.A[i][j]) * Ls[j]
                if self.Ai and self.Ai[i][j]:
                    r = r + (dt * self.Ai[i][j]) * Ss[j]
            if self.Ai:
                r = self.implicit(r, dt * self.Ai[i][i])
                Ss.append(self.source(r))
                S = S + self.b[i] * Ss[i]
            f = [self.flux(r, d) for d in self.dims]
            Ls.append(sum(self.dloc(f[d], d) +
                          self.product(r, c, self.dloc(r, d), dc[d], d) for d in self.dims))
            if self.b[i]:
                V, U = V + self.b[i] * Ls[i], U + self.b[i] * r
                F = [F[d] + self.b[i] * f[d] for d in self.dims]
        return V, U, F, S

    def residual(self, u, c, dt):
        V, U, F, S = self.update(u, c, dt)
        R = V - S
        for d in self.dims:
            a, b = lambda X: self.trace(X, self.l1, d), lambda X: self.next(
                self.trace(X, self.l0, d), d)
            (um, cm), (up, cp) = (a(u), a(c)), (b(u), b(c))
            lam = torch.maximum(self.speed(um, cm, d), self.speed(up, cp, d))
            Um, Up = a(U), b(U)
            dF, dU, db = b(F[d]) - a(F[d]), Up - Um, cp - cm
            D = lam * self.jump(Up, Um, cp, cm)
            Tm = 0.5 * (dF - D + self.product(um, cm, dU, db, d))
            Tp = -0.5 * (dF + D + self.product(up, cp, dU, db, d))
            R = R + (self.outer(Tm, self.gR, d) +
                     self.outer(self.next(Tp, d, 1), self.gL, d)) / self.h[d]
        return R

    def step(self, u, c, dt):
        return self.limited(u, c, dt) if self.case["limiter"] else u - dt * self.residual(u, c, dt)

    # -- the limiter ------------------------------------------------------------------
    def alpha(self, u):
        n, N = self.el.n, self.el.n - 1
        m = u[0] @ self.modes.T
        if len(self.dims) == 2:
            m = self.modes @ m
        m2 = m * m
        part = lambda k: (m2[..., :k] if len(self.dims) == 1 else m2[..., :k, :k]).sum((-2, -1))
        share = lambda top, rest: torch.where(top > 0, (top - rest) / torch.where(top > 0, top, 1.0),
                                              0.0)
        if len(self.dims) == 1:      # the top mode itself, not a difference of sums
            share = lambda top, rest: rest / top
            energy = share(part(n), m2[..., 0, N])
            if N >= 2:
                energy = torch.maximum(energy, share(part(N), m2[..., 0, N - 1]))
        else:
            energy = share(part(n), part(N))
            if N >= 2:
                energy = torch.maximum(energy, share(part(N), part(N - 1)))
        T = 0.5 * 10.0 ** (-1.8 * n ** 0.25)
        al = 1.0 / (1.0 + torch.exp(-math.log((1 - 1e-4) / 1e-4) / T * (energy - T)))
        al = torch.where(al < 1e-3, 0.0, torch.where(al > 1 - 1e-3, 1.0, al))
        near = [torch.roll(al, s, -1 - d) for d in self.dims for s in (1, -1)]
        return torch.maximum(al, 0.5 * torch.stack(near).amax(0))

    def low_flux(self, um, up, cm, cp, d):
        lam = torch.maximum(self.speed(um, cm, d), self.speed(up, cp, d))
        f = 0.5 * (self.flux(um, d) + self.flux(up, d)) - 0.5 * lam * self.jump(up, um, cp, cm)
        mean, cmean = 0.5 * (um + up), 0.5 * (cm + cp)
        return (f + self.product(um, cm, mean, cmean, d), f + self.product(up, cp, mean, cmean, d))

    def theta(self, low, new):
        eps = 0.1 * low
        gap = torch.where(new != low, new - low, 1.0)
        return torch.where(new < eps, ((eps - low) / gap).abs().clamp(max=1.0), 1.0)

    def limited(self, u, c, dt):
        V, U, F, S = self.update(u, c, dt)
        al, w, N = self.alpha(u), self.w, self.el.n - 1
        RH, low = V - S, u
        for d in self.dims:
            axis = -1 - d
            at = lambda X, k: X.select(axis, k)
            a, b = lambda X: self.trace(X, self.l1, d), lambda X: self.next(
                self.trace(X, self.l0, d), d)
            (um, cm), (up, cp) = (a(u), a(c)), (b(u), b(c))
            lam = torch.maximum(self.speed(um, cm, d), self.speed(up, cp, d))
            Um, Up, Fm, Fp = a(U), b(U), a(F[d]), b(F[d])
            f = 0.5 * (Fm + Fp) - 0.5 * lam * self.jump(Up, Um, cp, cm)
            mean, cmean = 0.5 * (Um + Up), 0.5 * (cm + cp)
            Hm = f + self.product(um, cm, mean, cmean, d)
            Hp = f + self.product(up, cp, mean, cmean, d)
            totm = Fm + self.product(um, cm, Um, cm, d)
            totp = Fp + self.product(up, cp, Up, cp, d)
            # first-order fluxes: at the element faces and the inner subfaces
            n0, nc0 = self.next(at(u, 0), d), self.next(at(c, 0), d)
            om, op = self.low_flux(at(u, N), n0, at(c, N), nc0, d)
            left, right = (X.narrow(axis, 0, N) for X in (u, c)), (X.narrow(axis, 1, N)
                                                                   for X in (u, c))
            (ul, cl), (ur, cr) = left, right
            im, ip = self.low_flux(ul, ur, cl, cr, d)
            af = (0.5 * (al + torch.roll(al, -1, axis)))[..., None]
            Lm, Lp = (1 - af) * Hm + af * om, (1 - af) * Hp + af * op
            if self.M > 1:
                k0, kN = (len(self.dims) * dt / (w[k] * self.h[d]) for k in (0, N))
                f0, fN = self.next(at(im, 0), d)[0], at(ip, N - 1)[0]
                th = torch.minimum(
                    self.theta(n0[0] - k0 * (f0 - op[0]), n0[0] - k0 * (f0 - Lp[0])),
                    self.theta(at(u, N)[0] - kN * (om[0] - fN), at(u, N)[0] - kN * (Lm[0] - fN)))
                Lm, Lp = th * Lm + (1 - th) * om, th * Lp + (1 - th) * op
            RH = RH + (self.outer(Lm - totm, self.gR, d) +
                       self.outer(self.next(Lp - totp, d, 1), self.gL, d)) / self.h[d]
            hi = torch.cat([im, Lm.unsqueeze(axis)], axis)
            lo = torch.cat([self.next(Lp, d, 1).unsqueeze(axis), ip], axis)
            low = low - dt / self.h[d] * (hi - lo) / (w if d == 0 else w[:, None])
        if self.Ai:
            low = self.implicit(low, dt)
        out = u - dt * RH
        a4 = al[..., None, None]
        out = (1 - a4) * out + a4 * low
        if self.M > 1:
            eps = 0.1 * low[0].amin((-2, -1), keepdim=True)
            gap = torch.where(out[0] != low[0], out[0] - low[0], 1.0)
            th = torch.where(out[0] < eps, ((eps - low[0]) / gap).abs().clamp(max=1.0), 1.0)
            th = th.amin((-2, -1), keepdim=True)
            out = th * out + (1 - th) * low
        return out

    def steps(self, u, c, count):
        for _ in range(count):
            u = self.step(u, c, self.time_step(u, c))
        return u


def exact(case, seed):
    device = "cuda" if torch.cuda.is_available() else "cpu"
    if case["kind"] == "ensemble":
        out = []
        for i, (d, e) in enumerate(_members(case)):
            u, c = _fields(case, [seed, i], d, e, 0, device)
            m = _Method(case, d, e, 0, device)
            out.append(m.steps(u[:, None, :, None], c[None, :, None], case["steps"]).reshape(-1))
        return torch.cat(out)
    u, c = _fields(case, seed, case["degree"], case["nx"], case["ny"], device)
    shape = u.shape
    m = _Method(case, case["degree"], case["nx"], case["ny"], device)
    if m.M < 3:
        u, c = u[:, None, :, None], c[None, :, None]
    if case["kind"] == "residual":
        return -m.residual(u, c, _fixed_dt(case)).reshape(shape)
    if case["kind"] == "adjoint":
        dt = _fixed_dt(case)
        eta0 = _eta0(u, c)
        target = 1.0 + 0.005 * torch.sin(torch.linspace(0, 40, c.numel(), device=device,
                                                        dtype=torch.float64)).view_as(c)
        b = c.clone().requires_grad_(True)
        z = torch.zeros_like(b)
        v = torch.stack([eta0 - b, z, z])
        for _ in range(case["steps"]):
            v = v - dt * m.residual(v, b, dt)
        weights = m.w[:, None] * m.w[None, :] * (m.h[0] * m.h[1])
        (0.5 * (weights * (v[0] + b - target) ** 2).sum()).backward()
        return {"u": v.detach(), "gradient": b.grad}
    out = m.steps(u, c, case["steps"]).reshape(shape)
    return out.cpu().numpy() if case["kind"] == "host" else out
