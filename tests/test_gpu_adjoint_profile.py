"""The kernel timing of the adjoint step: CRKFR_KERNEL_ADJOINT_2D holds one
record a step, around the face and the local kernel together, so that its time
over its count is a step's."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from gpu_common import load, to_dev
from test_gpu_adjoint import adjoint_slab, case, solver

pytestmark = pytest.mark.gpu
N, EX, EY, STEPS = 2, 7, 6, 3


def counts(s):
    return {k: v[0] for k, v in s.profile_read().items()}


def test_one_record_a_step():
    crk = load()
    u, b, _, _ = case(N, EX, EY)
    w = np.random.default_rng(2).standard_normal(u.shape)
    s = solver(crk, N, EX, EY, b)
    x, y, dt = to_dev(u), to_dev(w), 1e-3
    rec = s.new_records(1)[0]
    s.step_record(x, dt, rec, advance=False)
    s.profile(True)
    for _ in range(STEPS):
        s.step_adjoint(x, y, dt)
    assert counts(s) == {"local_2d": STEPS, "adjoint_2d": STEPS}
    s.profile(True)
    for _ in range(STEPS):
        s.step_adjoint_recorded(x, rec, y, dt)
    assert counts(s) == {"adjoint_2d": STEPS}


def test_one_record_a_step_on_a_slab():
    crk = load()
    u, b, _, _ = case(N, EX, EY)
    w = np.random.default_rng(3).standard_normal(u.shape)
    s = adjoint_slab(crk, N, EX, EY, b, 0, EY)
    x, y, dt = to_dev(u), to_dev(w), 1e-3
    s.profile(True)
    for _ in range(STEPS):
        s.adjoint_local(x, y, dt)
        s.adjoint_faces(x, y, dt)
    assert counts(s) == {"local_2d": STEPS, "adjoint_2d": STEPS}
