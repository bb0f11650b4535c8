"""Components far below the others of their element: steps of zero size leave
every bit of them."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from gpu_common import G, golden_cfl, golden_cfl_imex, load, positions_2d, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def crk():
    return load()


def solver(crk, system, N, family, Ex, Ey, Lx, Ly, b, source=None):
    cfl = golden_cfl_imex(N, family) if source else golden_cfl(N, family)
    s = crk.Solver(system, N, nodes=family, gravity=G, cfl_safety=0.5, cfl_number=cfl,
                   source=source, source_coef=0.01 if source else 0.0)
    s.set_mesh([Ex, Ey], [0.0, 0.0], [Lx, Ly])
    s.set_coefficients(to_dev(b))
    return s


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
