"""A step's bits do not depend on where an element lies in its warp or block: a
rolled periodic mesh gives the rolled result.  Water at rest beside flowing
water, so that the exponents of some elements are raised in later stages while
the depths of others pass a power of two."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from gpu_common import G, golden_cfl, golden_cfl_imex, load, to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def crk():
    return load()


def step(crk, system, N, family, source, limiter, u, b, dt):
    shape = b.shape[:-2] if system.startswith("swe2d") else b.shape[:-1]
    cfl = golden_cfl_imex(N, family) if source else golden_cfl(N, family)
    s = crk.Solver(system, N, nodes=family, gravity=G, cfl_safety=0.5, cfl_number=cfl,
                   source=source, source_coef=0.01 if source else 0.0)
    s.set_mesh([int(e) for e in shape[::-1]], [0.0] * len(shape), [float(e) for e in shape[::-1]])
    s.set_coefficients(to_dev(b))
    if limiter:
        s.set_limiter("blend")
    d = to_dev(u)
    s.step(d, dt, 2)
    return to_host(d)


def fields(shape, moments, seed):
    """Depths just below one, momenta zero in half of the elements, so that stages
    of the others pass one while those at rest raise their momenta's exponents."""
    rng = np.random.default_rng(seed)
    h = 1.0 - 2e-3 * rng.random(shape)
    elements = shape[:len(shape) - moments]
    on = (rng.random(elements) < 0.5) * 10.0 ** rng.uniform(-2, 0, elements)
    m = [0.2 * rng.standard_normal(shape) * on[(...,) + (None,) * moments] for _ in range(moments)]
    return np.stack([h] + m), 1e-3 * rng.standard_normal(shape)


@pytest.mark.parametrize("N,family", [(1, "gl"), (2, "gll"), (3, "gl"), (3, "gll"), (4, "gl")])
@pytest.mark.parametrize("system,source,limiter", [
    ("swe2d", None, False), ("swe2d_wb", None, False), ("swe2d", "chezy", False),
    ("swe2d", None, True), ("swe2d_wb", None, True)])
def test_rolled_mesh_2d(crk, system, source, limiter, N, family):
    Ex, Ey, n = 37, 23, N + 1
    u, b = fields((Ey, Ex, n, n), 2, N)
    want = step(crk, system, N, family, source, limiter, u, b, 5e-3)
    assert np.isfinite(want).all()
    for dy, dx in ((0, 1), (1, 0), (3, 5), (11, 2)):
        ur, br = np.roll(u, (dy, dx), axis=(1, 2)), np.roll(b, (dy, dx), axis=(0, 1))
        got = step(crk, system, N, family, source, limiter, ur, br, 5e-3)
        assert np.array_equal(got, np.roll(want, (dy, dx), axis=(1, 2))), (dy, dx)


@pytest.mark.parametrize("N,family", [(1, "gl"), (2, "gll"), (3, "gl"), (4, "gl")])
@pytest.mark.parametrize("system,source,limiter", [
    ("swe1d", None, False), ("swe1d_wb", None, False), ("swe1d", "chezy", False),
    ("swe1d_wb", None, True)])
def test_rolled_mesh_1d(crk, system, source, limiter, N, family):
    E, n = 1001, N + 1
    u, b = fields((E, n), 1, N)
    want = step(crk, system, N, family, source, limiter, u, b, 5e-3)
    assert np.isfinite(want).all()
    for d in (1, 2, 7, 500):
        got = step(crk, system, N, family, source, limiter, np.roll(u, d, axis=1),
                   np.roll(b, d, axis=0), 5e-3)
        assert np.array_equal(got, np.roll(want, d, axis=1)), d
