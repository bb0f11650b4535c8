"""Components far below the others of their element: steps of zero size, a
momentum far below the other one, depths far below their neighbours', mesh
widths far apart, and the adjoint's small component.

The reference is the oracle in extended precision.  Tolerances: each value is
a sum of at most a few hundred products, each rounded to 2^-53 of itself in
FP64, so C = 256 times 2^-53 times the largest magnitudes of the terms of the
component's own equation bounds the error of an FP64 evaluation; terms whose
derivatives cancel exactly (equal values, entries of D that are powers of two)
count for nothing.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from gpu_common import G, golden_cfl, golden_cfl_imex, load, positions_2d, to_dev, to_host

pytestmark = pytest.mark.gpu
C = 256 * 2.0 ** -53
LD = np.longdouble


@pytest.fixture(scope="module")
def crk():
    return load()


def scheme(system, N, dx, dy, family):
    from oracle.crkfr import Scheme2D
    from oracle.systems import ShallowWater2D, ShallowWater2DWB
    return Scheme2D((ShallowWater2DWB if system == "swe2d_wb" else ShallowWater2D)(G), N, dx, dy,
                    family=family)


def solver(crk, system, N, family, Ex, Ey, Lx, Ly, b, source=None):
    cfl = golden_cfl_imex(N, family) if source else golden_cfl(N, family)
    s = crk.Solver(system, N, nodes=family, gravity=G, cfl_safety=0.5, cfl_number=cfl,
                   source=source, source_coef=0.01 if source else 0.0)
    s.set_mesh([Ex, Ey], [0.0, 0.0], [Lx, Ly])
    s.set_coefficients(to_dev(b))
    return s


def derivative_norm(bs):
    """Largest row sum of |D| plus the largest |g'| of both sides."""
    return float(np.abs(bs.D).sum(axis=1).max() + np.abs(bs.gRp).max() + np.abs(bs.gLp).max())


# ---- steps of zero size ------------------------------------------------------
@pytest.mark.parametrize("system,source", [("swe2d", None), ("swe2d_wb", None), ("swe2d", "chezy")])
@pytest.mark.parametrize("N,family", [(1, "gl"), (2, "gll"), (3, "gl"), (4, "gl")])
def test_steps_after_the_end_change_nothing(crk, system, source, N, family):
    # crkfr_advance queues steps in chunks; those past t_end have size zero
    from oracle.basis import Basis
    Ex, Ey, L = 33, 21, 8.0
    x, y, _, _ = positions_2d(Basis(N, family), Ex, Ey, L)
    k = 2 * np.pi / L
    b = 0.1 * np.sin(k * x) * np.cos(k * y)
    h = 1.0 + 0.2 * np.cos(k * x + 1.0) * np.sin(2 * k * y) - b
    u = np.stack([h, h * np.sin(k * x + 2 * k * y), 1e-3 * h * np.sin(3 * k * x - k * y)])
    s = solver(crk, system, N, family, Ex, Ey, L, L, b, source)
    t_end = 3.5 * s.compute_dt(to_dev(u))
    one, many = to_dev(u), to_dev(u)
    taken = s.advance(many, t_end)
    assert 3 <= taken < 16
    s.set_time(0.0)
    assert s.advance(one, t_end, max_steps=taken) == taken
    assert torch.equal(one, many)


@pytest.mark.parametrize("system,source", [("swe2d", None), ("swe2d_wb", None), ("swe2d", "chezy")])
@pytest.mark.parametrize("N,family", [(1, "gl"), (2, "gll"), (3, "gl"), (4, "gl")])
def test_a_step_below_the_last_bit_changes_nothing(crk, system, source, N, family):
    from oracle.basis import Basis
    Ex, Ey, L = 33, 21, 8.0
    x, y, _, _ = positions_2d(Basis(N, family), Ex, Ey, L)
    k = 2 * np.pi / L
    b = 0.1 * np.sin(k * x) * np.cos(k * y)
    h = 1.0 + 0.2 * np.cos(k * x + 1.0) * np.sin(2 * k * y) - b
    u = np.stack([h, h * np.sin(k * x + 2 * k * y + 0.1),
                  1e-3 * h * np.sin(3 * k * x - k * y + 0.1)])
    assert (np.abs(u) > 1e-100).all()
    s = solver(crk, system, N, family, Ex, Ey, L, L, b, source)
    d = to_dev(u)
    assert s.advance(d, 1e-200) == 1
    assert torch.equal(d, to_dev(u))


# ---- one momentum far below the other ---------------------------------------
def aligned_flow(N, family, froude, small, system):
    """h, b, hu and hv functions of x alone, hv `small` times hu."""
    Ex, Ey, L = 6, 3, 8.0 * 6 / 8
    Lx, Ly = float(Ex), float(Ey)   # unit elements: entries of D are those of the reference
    sch = scheme(system, N, 1.0, 1.0, family)
    x, y, _, _ = positions_2d(sch.basis, Ex, Ex, Lx)
    x = np.ascontiguousarray(x[:Ey])
    k = 2 * np.pi / Lx
    b = 0.05 * np.sin(k * x)
    h = 1.0 + 0.1 * np.cos(k * x + 1.0) - b
    hu = froude * np.sqrt(G) * h * (1.0 + 0.1 * np.sin(k * x + 0.3))
    return sch, np.stack([h, hu, small * hu * np.cos(k * x + 0.5)]), b, Ex, Ey, Lx, Ly


@pytest.mark.parametrize("system", ["swe2d", "swe2d_wb"])
@pytest.mark.parametrize("N,family,froude", [(1, "gll", 0.3), (1, "gll", 300.0), (1, "gl", 300.0),
                                             (2, "gll", 300.0), (3, "gl", 300.0), (4, "gl", 300.0)])
@pytest.mark.parametrize("small", [1e-6, 1e-10])
def test_small_transverse_momentum(crk, system, N, family, froude, small):
    sch, u, b, Ex, Ey, Lx, Ly = aligned_flow(N, family, froude, small, system)
    dt = 0.2 * float(sch.compute_dt(u, b, golden_cfl(N, family), 0.5))
    s = solver(crk, system, N, family, Ex, Ey, Lx, Ly, b)
    d = to_dev(u)
    s.step(d, dt, 1)
    want = sch.step(u.astype(LD), b.astype(LD), LD(dt))
    h, hu, hv = (float(np.abs(v).max()) for v in u)
    c = np.sqrt(G * h)
    terms = (hu * hv / u[0].min() + (hu / u[0].min() + c) * hv) + c * hv
    if not (N == 1 and family == "gll"):
        terms += G * h * (h + float(np.abs(b).max()))   # (equal values along y otherwise)
    tol = C * (hv + dt * derivative_norm(sch.basis) * terms)
    assert tol < 0.1 * hv
    assert float(np.abs(to_host(d)[2] - want[2]).max()) < tol


# ---- a depth far below the others, beside a steep bottom ----------------------
@pytest.mark.parametrize("dim", [1, 2])
@pytest.mark.parametrize("N", [2, 4])
def test_shallow_node_on_a_steep_bottom(crk, dim, N):
    # still water; the middle node of a GLL element takes nothing from the faces,
    # and at the first instants only -(h g b_x + d(g h^2/2)/dx)
    from oracle.crkfr import Scheme1D
    from oracle.systems import ShallowWater1D
    E, slope, low, dt = 4, 1e6, 1e-10 / 3, 1e-12
    sch = (Scheme1D(ShallowWater1D(G), N, 1.0, family="gll") if dim == 1
           else scheme("swe2d", N, 1.0, 1.0, "gll"))
    xi = sch.basis.xi
    b = np.stack([slope * (xi if e % 2 == 0 else 1.0 - xi) for e in range(E)])
    h = np.ones((E, N + 1))
    h[1, N // 2] = low
    if dim == 1:
        u = np.stack([h, np.zeros_like(h)])
        s = crk.Solver("swe1d", N, nodes="gll", gravity=G, cfl_safety=0.5,
                       cfl_number=golden_cfl(N, "gll"))
        s.set_mesh([E], [0.0], [float(E)])
    else:
        shape = (2, E, N + 1, N + 1)
        b, h = (np.ascontiguousarray(np.broadcast_to(v[None, :, None, :], shape)) for v in (b, h))
        u = np.stack([h, np.zeros_like(h), np.zeros_like(h)])
        s = crk.Solver("swe2d", N, nodes="gll", gravity=G, cfl_safety=0.5,
                       cfl_number=golden_cfl(N, "gll"))
        s.set_mesh([E, 2], [0.0, 0.0], [float(E), 2.0])
    s.set_coefficients(to_dev(b))
    d = to_dev(u)
    s.step(d, dt, 1)
    want = sch.step(u.astype(LD), b.astype(LD), LD(dt))[1][..., 1, :] if dim == 1 else \
        sch.step(u.astype(LD), b.astype(LD), LD(dt))[1][:, 1]
    got = to_host(d)[1][..., 1, :] if dim == 1 else to_host(d)[1][:, 1]
    err = np.abs(got - want)[..., N // 2].max()
    # (b_x itself is a derivative of b: its rounding is relative to `slope`)
    tol = C * dt * (low * G * slope * derivative_norm(sch.basis)
                    + derivative_norm(sch.basis) * 0.5 * G)
    assert tol < 1e-2 * dt * low * G * slope
    assert float(err) < tol


# ---- mesh widths far apart ----------------------------------------------------
def test_mesh_widths_far_apart(crk):
    # fields of y alone on elements 2^-34 wide in x: nothing comes from the x
    # derivatives, and those in y keep their precision
    N, Ex, Ey, dx = 1, 3, 6, 2.0 ** -34
    sch = scheme("swe2d", N, dx, 1.0, "gll")
    y, _, _, _ = positions_2d(sch.basis, Ey, Ey, float(Ey))
    y = np.ascontiguousarray(np.swapaxes(np.swapaxes(y, 0, 1), 2, 3)[:, :Ex])
    k = 2 * np.pi / Ey
    b = 0.1 * np.sin(k * y)
    h = 1.0 + 0.1 * np.cos(k * y + 1.0) - b
    u = np.stack([h, 0.3 * h, h * np.sin(k * y + 0.4)])
    dt = 0.2 * golden_cfl(N, "gll") / 5.0
    s = solver(crk, "swe2d", N, "gll", Ex, Ey, Ex * dx, float(Ey), b)
    d = to_dev(u)
    s.step(d, dt, 1)
    want = sch.step(u.astype(LD), b.astype(LD), LD(dt))
    terms = [float(np.abs(u[2]).max()) + 4.5, 2.0, 10.0]
    for v in range(3):
        tol = C * (float(np.abs(u[v]).max()) + dt * derivative_norm(sch.basis) * terms[v])
        assert float(np.abs(to_host(d)[v] - want[v]).max()) < tol, v


# ---- the adjoint's small component ----------------------------------------------
@pytest.mark.parametrize("N", [1, 2, 3, 4])
def test_small_component_of_the_adjoint(crk, N):
    # still water of constant depth: the adjoint of hv takes from that of h at
    # first order in the step, from that of hu at second order only
    Ex, Ey = 5, 4
    sch = scheme("swe2d", N, 1.0, 1.0, "gl")
    n = N + 1
    u = np.zeros((3, Ey, Ex, n, n))
    u[0] = 1.0
    b = np.zeros((Ey, Ex, n, n))
    w = np.random.default_rng(7).standard_normal(u.shape)
    w[0] *= 1e-14
    w[2] *= 1e-14
    dt = 1e-8
    ut = torch.tensor(u, requires_grad=True)
    (sch.step(ut, torch.tensor(b), dt) * torch.tensor(w)).sum().backward()
    s = solver(crk, "swe2d", N, "gl", Ex, Ey, float(Ex), float(Ey), b)
    got, _ = s.step_adjoint(to_dev(u), to_dev(w), dt)
    kappa = dt * np.sqrt(G) * derivative_norm(sch.basis)
    tol = C * (np.abs(w[2]).max() + kappa * np.abs(w[0]).max() + kappa ** 2 * np.abs(w[1]).max())
    assert float(np.abs(to_host(got)[2] - ut.grad.numpy()[2]).max()) < tol
