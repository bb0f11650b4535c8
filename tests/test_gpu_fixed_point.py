"""The block fixed-point contractions of the step kernels (fixed_point.cuh)
at the edges of their ranges: element counts around a block's, fields whose
magnitude grows between the stages of a step, scales far from one, and
non-finite values.

Tolerance of the parity cases: both sides round the stage values and the
update to FP64, u^{n+1} = u^n - dt R with |dt R| below |u| under the CFL
condition, and every operation before that is at most a few hundred roundings
of 2^-53 of the update's scale, so 1e-13 of the state's norm bounds the
difference; a lost operand bit or a wrong exponent shows at 1e-9 or more.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from gpu_common import G, golden_cfl, load, positions_2d, rel_l2, to_dev, to_host

pytestmark = pytest.mark.gpu
TOL = 1e-13


@pytest.fixture(scope="module")
def crk():
    return load()


def case_2d(N, family, Ex, Ey, scale=1.0, still=False, seed=0):
    """(scheme, state, bathymetry, dx): smooth random fields of size `scale`
    (lengths and, through gravity fixed, speeds of sqrt(scale))."""
    from oracle.crkfr import Scheme2D
    from oracle.systems import ShallowWater2D
    L = 10.0
    sch = Scheme2D(ShallowWater2D(G), N, L / Ex, L / Ey, family=family)
    x, y, _, _ = positions_2d(sch.basis, Ex, Ey, L)
    rng = np.random.default_rng(seed)
    a = rng.uniform(0, 2 * np.pi, 8)
    k = 2 * np.pi / L
    b = scale * 0.2 * np.sin(k * x + a[0]) * np.cos(k * y + a[1])
    h = scale * (1.0 + 0.1 * np.sin(k * x + a[2]) * np.sin(k * y + a[3])) - b
    c = np.sqrt(scale)
    m = [0.0 if still else 0.3 * c, 0.0 if still else -0.2 * c]
    u = np.stack([h, h * m[0] * np.cos(k * y + a[4]), h * m[1] * np.sin(k * x + a[5])])
    return sch, u, b, L


def run(crk, sch, N, family, u, b, L, Ex, Ey, dt, steps=1):
    s = crk.Solver("swe2d", N, nodes=family, gravity=G, cfl_safety=0.5,
                   cfl_number=golden_cfl(N, family))
    s.set_mesh([Ex, Ey], [0.0, 0.0], [L, L])
    s.set_coefficients(to_dev(b))
    d = to_dev(u)
    s.step(d, dt, steps)
    return s, to_host(d)


# elements of a block: 128, 32, 14, 8, 5 threads / n^2
@pytest.mark.parametrize("N,family,Ex,Ey", [
    (1, "gl", 31, 1), (1, "gll", 33, 3), (2, "gl", 13, 1), (2, "gll", 15, 1), (2, "gl", 7, 5),
    (3, "gl", 7, 1), (3, "gll", 3, 3), (3, "gl", 1, 1), (4, "gl", 5, 1), (4, "gll", 2, 3),
    (4, "gl", 11, 1)])
@pytest.mark.parametrize("still", [False, True])
def test_block_edges_and_growing_momentum(crk, N, family, Ex, Ey, still):
    # still: the momentum is zero at the first stage and grows from nothing
    sch, u, b, L = case_2d(N, family, Ex, Ey, still=still)
    dt = sch.compute_dt(u, b, golden_cfl(N, family), 0.5)
    _, got = run(crk, sch, N, family, u, b, L, Ex, Ey, dt)
    assert rel_l2(got, sch.step(u, b, dt)) < TOL


def case_1d(N, family, E, still=False, seed=0):
    from oracle.crkfr import Scheme1D
    from oracle.systems import ShallowWater1D
    L = 10.0
    sch = Scheme1D(ShallowWater1D(G), N, L / E, family=family)
    x = (np.arange(E)[:, None] + sch.basis.xi[None, :]) * (L / E)
    a = np.random.default_rng(seed).uniform(0, 2 * np.pi, 4)
    k = 2 * np.pi / L
    b = 0.2 * np.sin(k * x + a[0])
    h = 1.0 + 0.1 * np.sin(k * x + a[1]) - b
    return sch, np.stack([h, (0.0 if still else 0.3) * h * np.cos(k * x + a[2])]), b, L


# elements a block owns, threads / 32 * (32 / n) - 2: N = 1: 14 (32 threads) ..
# 126 (256), N = 2: 8 .. 78, N = 3: 6 .. 62, N = 4: 4 .. 46
@pytest.mark.parametrize("N,family,E", [
    (0, "gl", 1), (0, "gl", 31), (0, "gl", 255), (1, "gl", 1), (1, "gll", 15), (1, "gl", 127),
    (2, "gl", 2), (2, "gll", 9), (2, "gl", 79), (3, "gl", 1), (3, "gll", 7), (3, "gl", 63),
    (4, "gl", 1), (4, "gll", 5), (4, "gl", 47), (4, "gl", 20011)])
@pytest.mark.parametrize("still", [False, True])
def test_block_edges_1d(crk, N, family, E, still):
    sch, u, b, L = case_1d(N, family, E, still)
    dt = sch.compute_dt(u, b, golden_cfl(N, family), 0.5)
    want = sch.step(u, b, dt)
    s = crk.Solver("swe1d", N, nodes=family, gravity=G, cfl_safety=0.5,
                   cfl_number=golden_cfl(N, family))
    s.set_mesh([E], [0.0], [L])
    s.set_coefficients(to_dev(b))
    for threads in (0, 64, 96, 128):
        s.set_tile_1d(threads)
        d = to_dev(u)
        s.step(d, dt, 1)
        assert rel_l2(to_host(d), want) < TOL


@pytest.mark.parametrize("N", [1, 2, 3, 4])
@pytest.mark.parametrize("scale", [1e-12, 1e9])
def test_scales(crk, N, scale):
    sch, u, b, L = case_2d(N, "gl", 6, 5, scale=scale)
    dt = sch.compute_dt(u, b, golden_cfl(N, "gl"), 0.5)
    _, got = run(crk, sch, N, "gl", u, b, L, 6, 5, dt)
    want = sch.step(u, b, dt)
    for v in range(3):
        assert rel_l2(got[v], want[v]) < 10 * TOL   # (each variable by itself)


@pytest.mark.parametrize("N", [1, 2, 3, 4])
@pytest.mark.parametrize("value", [np.nan, np.inf])
def test_non_finite_stays_in_its_neighbourhood(crk, N, value):
    Ex, Ey = 9, 7
    sch, u, b, L = case_2d(N, "gl", Ex, Ey)
    dt = sch.compute_dt(u, b, golden_cfl(N, "gl"), 0.5)
    good = run(crk, sch, N, "gl", u, b, L, Ex, Ey, dt)[1]
    u[1, 3, 4, N // 2, 0] = value
    s, got = run(crk, sch, N, "gl", u, b, L, Ex, Ey, dt)
    with pytest.raises(crk.CrkfrError):
        s.status()
    assert not np.isfinite(got[:, 3, 4]).any()
    touched = np.zeros((Ey, Ex), dtype=bool)
    for e in ((3, 4), (2, 4), (4, 4), (3, 3), (3, 5)):
        touched[e] = True
    assert np.array_equal(got[:, ~touched], good[:, ~touched])


# The fluxes in the element's fixed point: momenta far below and far above
# sqrt(g h) h, either sign, and depths spread over a factor of e^4 inside the
# mesh, so that the bound of the flux exponent is met from both of its terms.
# Tolerance as for the scales above: |dt R| stays below the state's norm.
@pytest.mark.parametrize("system", ["swe2d", "swe2d_wb"])
@pytest.mark.parametrize("N", [1, 3, 4])
@pytest.mark.parametrize("froude", [1e-9, 1e-2, 1.0, 40.0])
def test_flux_ratios(crk, system, N, froude):
    from oracle.crkfr import Scheme2D
    from oracle.systems import ShallowWater2D, ShallowWater2DWB
    Ex, Ey = 27, 25   # (fine enough for positive depths at the faces)
    sch, u, b, L = case_2d(N, "gl", Ex, Ey)
    if system == "swe2d_wb":
        sch = Scheme2D(ShallowWater2DWB(G), N, L / Ex, L / Ey, family="gl")
    x, y, _, _ = positions_2d(sch.basis, Ex, Ey, L)
    k = 2 * np.pi / L
    h = np.exp(2 * np.sin(k * x) * np.sin(k * y + 1.0)) + 0 * b
    v = froude * np.sqrt(G * h)
    u = np.stack([h, h * v * np.cos(k * (x + y)), -h * v * np.sin(k * (x - y) + 0.5)])
    dt = 0.2 * sch.compute_dt(u, b, golden_cfl(N, "gl"), 0.5)
    s = crk.Solver(system, N, nodes="gl", gravity=G, cfl_safety=0.5,
                   cfl_number=golden_cfl(N, "gl"))
    s.set_mesh([Ex, Ey], [0.0, 0.0], [L, L])
    s.set_coefficients(to_dev(b))
    d = to_dev(u)
    s.step(d, dt, 1)
    got, want = to_host(d), sch.step(u, b, dt)
    assert np.isfinite(want).all()
    for w in range(3):
        assert rel_l2(got[w], want[w]) < 10 * TOL


# the same for the 1D step
@pytest.mark.parametrize("system", ["swe1d", "swe1d_wb"])
@pytest.mark.parametrize("N,E", [(0, 40), (2, 33), (4, 61)])
@pytest.mark.parametrize("froude", [1e-9, 1.0, 40.0])
def test_flux_ratios_1d(crk, system, N, E, froude):
    from oracle.crkfr import Scheme1D
    from oracle.systems import ShallowWater1D, ShallowWater1DWB
    L = 10.0
    sch = Scheme1D((ShallowWater1DWB if system == "swe1d_wb" else ShallowWater1D)(G), N, L / E)
    x = (np.arange(E)[:, None] + sch.basis.xi[None, :]) * (L / E)
    k = 2 * np.pi / L
    b = 0.2 * np.sin(k * x)
    h = np.exp(2 * np.sin(k * x + 1.0))
    u = np.stack([h, froude * h * np.sqrt(G * h) * np.cos(k * x)])
    dt = 0.2 * sch.compute_dt(u, b, golden_cfl(N, "gl"), 0.5)
    s = crk.Solver(system, N, nodes="gl", gravity=G, cfl_safety=0.5,
                   cfl_number=golden_cfl(N, "gl"))
    s.set_mesh([E], [0.0], [L])
    s.set_coefficients(to_dev(b))
    d = to_dev(u)
    s.step(d, dt, 1)
    got, want = to_host(d), sch.step(u, b, dt)
    assert np.isfinite(want).all()
    for w in range(2):
        assert rel_l2(got[w], want[w]) < 10 * TOL


# depths that have no finite reciprocal
@pytest.mark.parametrize("value", [0.0, np.nan, np.inf])
def test_non_finite_depth(crk, value):
    sch, u, b, L = case_2d(3, "gl", 5, 5)
    dt = sch.compute_dt(u, b, golden_cfl(3, "gl"), 0.5)
    u[0, 2, 2, 1, 1] = value
    s, got = run(crk, sch, 3, "gl", u, b, L, 5, 5, dt)
    with pytest.raises(crk.CrkfrError):
        s.status()
    assert np.isnan(got[1:, 2, 2]).all()
