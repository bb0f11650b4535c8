"""The adjoint step's buffer of recomputed stage values: without one of its own
(a first call in a stream capture, which may not allocate) the step works in
the context's work state, in row parts, with the same bits."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from gpu_common import load, to_dev
from test_gpu_adjoint import adjoint_slab, solver

pytestmark = pytest.mark.gpu


def fields(N, Ex, Ey):
    """A state and its bathymetry, random to some percent of the depth, and an
    adjoint state."""
    rng = np.random.default_rng(10 * N + Ey)
    shape = (Ey, Ex, N + 1, N + 1)
    u = np.stack([1.0 + 0.05 * rng.random(shape), *(0.1 * rng.standard_normal((2,) + shape))])
    return u, 0.02 * rng.random(shape), rng.standard_normal(u.shape)


def captured(call, *outs):
    """The outputs of `call` captured in a CUDA graph and replayed once."""
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call()
    for o in outs:
        o.zero_()
    graph.replay()
    torch.cuda.synchronize()
    return [o.clone() for o in outs]


# rows of the work state: one in S - 1 (N = 1: all; 2: half; 3: a third; 4: a
# fifth), and one on meshes of fewer rows
@pytest.mark.parametrize("N,Ey", [(1, 4), (2, 5), (3, 2), (3, 7), (4, 1), (4, 3), (4, 11)])
def test_adjoint_step_without_a_buffer(N, Ey):
    crk = load()
    Ex = 6
    u, b, w = fields(N, Ex, Ey)
    s = solver(crk, N, Ex, Ey, b)
    x, y, dt = to_dev(u), to_dev(w), 1e-2
    rec = s.new_records(1)[0]
    s.step_record(x, dt, rec, advance=False)
    s.step_adjoint_recorded(x, rec, y, dt)   # (allocates the trace buffers)
    ub, bb = torch.zeros_like(y), torch.zeros(s.coef_shape, dtype=torch.float64, device="cuda")
    got = captured(lambda: s.step_adjoint(x, y, dt, ubar0=ub, bbar=bb), ub, bb)
    want = s.step_adjoint(x, y, dt)          # (outside a capture: its own buffer)
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
    assert torch.equal(x, to_dev(u))


@pytest.mark.parametrize("N", [2, 4])
def test_slab_adjoint_without_a_buffer(N):
    crk = load()
    Ex, Ey = 6, 7
    u, b, w = fields(N, Ex, Ey)
    s = adjoint_slab(crk, N, Ex, Ey, b, 0, Ey)
    x, y, dt = to_dev(u), to_dev(w), 1e-2
    rec = s.new_records(1)[0]
    s.step_local_record(x, dt, rec, advance=False)
    s.adjoint_sums(y)
    s.adjoint_faces_recorded(x, rec, y, dt)   # (allocates the trace buffers)
    s.adjoint_local(x, y, dt)
    for bufs in (s.halo_buffers(), s.adjoint_halo_buffers()):
        bufs[2].copy_(bufs[1])
        bufs[3].copy_(bufs[0])
    ub, bb = torch.zeros_like(y), torch.zeros((Ey,) + tuple(b.shape[1:]), dtype=torch.float64,
                                              device="cuda")
    got = captured(lambda: s.adjoint_faces(x, y, dt, ubar0=ub, bbar=bb), ub, bb)
    want = s.adjoint_faces(x, y, dt)
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
