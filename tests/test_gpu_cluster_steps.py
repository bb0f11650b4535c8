"""Several 1D steps in one launch (meshes of at most 8 blocks of 128 threads):
the same bits as a launch per step, at the edges of the block sizes and of the
cluster, for odd and even counts, fixed and CFL steps, and beyond the steps of
one launch.  A fixed tile size takes a launch per step."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from gpu_common import G, golden_cfl, golden_cfl_imex, load, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def crk():
    return load()


def solver(crk, system, N, family, E, source, tile):
    cfl = golden_cfl_imex(N, family) if source else golden_cfl(N, family)
    s = crk.Solver(system, N, nodes=family, gravity=G, cfl_safety=0.5, cfl_number=cfl,
                   source=source, source_coef=0.01 if source else 0.0)
    s.set_mesh([E], [0.0], [10.0])
    x = s.positions()
    k = 2 * np.pi / 10.0
    if system == "varadv1d":
        c, u = 1.0 + 0.2 * np.sin(k * x), np.sin(k * x + 0.3)[None]
    else:
        c = 0.2 * np.sin(k * x)
        h = 1.0 + 0.1 * np.cos(k * x) - c
        u = np.stack([h, 0.2 * h * np.sin(k * x + 0.5)])
    s.set_coefficients(to_dev(c))
    s.set_tile_1d(tile)
    return s, to_dev(u)


def edges(N):
    own = [t // 32 * (32 // (N + 1)) - 2 for t in (32, 64, 128)]
    return sorted({1, 2, own[0], own[0] + 1} | {8 * o for o in own} | {8 * o + 1 for o in own})


@pytest.mark.parametrize("system,N,family,source", [
    ("varadv1d", 3, "gl", None), ("varadv1d", 1, "gll", "linear"), ("swe1d", 0, "gl", None),
    ("swe1d", 4, "gl", None), ("swe1d", 2, "gll", "chezy"), ("swe1d_wb", 3, "gl", None)])
def test_same_bits_as_a_launch_per_step(crk, system, N, family, source):
    for E in edges(N):
        for dt, steps in ((0.0, 5), (1e-4, 2), (1e-4, 3)):
            one, u = solver(crk, system, N, family, E, source, 64)
            many, v = solver(crk, system, N, family, E, source, 0)
            n0 = many.launch_count()
            for _ in range(2):
                one.step(u, dt, steps)
                many.step(v, dt, steps)
            assert torch.equal(u, v) and bool(torch.isfinite(v).all()), (E, dt, steps)
            # (a rate kernel a call with CFL steps)
            joined = E <= 8 * (128 // 32 * (32 // (N + 1)) - 2)
            assert many.launch_count() - n0 == 2 * ((1 if joined else steps) + (dt == 0.0)), E


def test_advance_and_more_steps_than_a_launch_takes(crk):
    one, u = solver(crk, "swe1d", 1, "gl", 40, None, 64)
    many, v = solver(crk, "swe1d", 1, "gl", 40, None, 0)
    assert one.advance(u, 0.5) == many.advance(v, 0.5)
    assert torch.equal(u, v)
    one.step(u, 0.0, 2051)
    many.step(v, 0.0, 2051)
    assert torch.equal(u, v) and bool(torch.isfinite(v).all())
