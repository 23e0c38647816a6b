"""Many steps of one call (one cooperative launch) give the bits of as many
calls of one step, on meshes around the tiles' edges, with walls, in batches with
paused and non-finite instances, and across the launches' longest run."""
import numpy as np
import pytest

from paper_1802_02868_gb300 import dugks
from paper_1802_02868_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _sim(nx, ny, prec, walls):
    prm = I.stationary_drop().params
    m = I.uniform_mesh(nx, ny)
    if walls:
        m = I.Mesh(1.0 + 0.2 * np.cos(np.arange(nx)), 1.0 + 0.2 * np.sin(np.arange(ny)), I.PERIODIC, I.WALL)
    phi = I.drop_field(m, 0.3 * min(nx, ny), (0.5 * nx, 0.4 * ny), 4.0)
    return dugks.Sim(m, prm, prec).init(phi)


# less than a tile; narrow last columns and rows (1 to 3 cells), so that a ring
# reaches past the neighbouring tile; one tile per block, and several
SIZES = [(3, 5, 17), (9, 33, 16), (33, 65, 18), (35, 97, 21), (64, 64, 40), (130, 250, 19), (200, 515, 17), (256, 1024, 33)]


@pytest.mark.parametrize("prec", [dugks.FP64, dugks.FP32])
@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("nx,ny,n", SIZES)
def test_many_steps_equal_single_steps(nx, ny, n, walls, prec):
    a, b = _sim(nx, ny, prec, walls), _sim(nx, ny, prec, walls)
    a.step(n)
    for _ in range(n):
        b.step(1)
    for x, y in zip(a.state(), b.state()):
        assert np.array_equal(x, y)
    # and again from there, after an odd number of steps
    a.step(n)
    for _ in range(n):
        b.step(1)
    for x, y in zip(a.state(), b.state()):
        assert np.array_equal(x, y)


def test_a_long_call_and_a_new_state_after_it():
    a, b = _sim(64, 64, dugks.FP32, False), _sim(64, 64, dugks.FP32, False)
    start = a.state()
    a.step(1050)
    for _ in range(70):
        b.step(15)
    for x, y in zip(a.state(), b.state()):
        assert np.array_equal(x, y)
    a.set_state(*start)
    b.set_state(*start)
    a.step(20)
    b.step(10).step(10)
    for x, y in zip(a.state(), b.state()):
        assert np.array_equal(x, y)


def test_batches_with_paused_and_nonfinite_instances():
    cs = [I.stationary_drop(n=n, radius=0.25 * n) for n in (24, 41, 64)]

    def sim():
        return dugks.Sim([c.mesh for c in cs], [c.params for c in cs], dugks.FP64).init([c.phi0 for c in cs])
    a, b = sim(), sim()
    for s, each in ((a, 20), (b, 1)):
        s.set_paused([False, True, False])
        for _ in range(20 // each):
            s.step(each)
    fa, fb = a.state(), b.state()
    assert all(np.array_equal(x, y) for x, y in zip(fa, fb))
    # instance 1 overflows: the others go on as if it were not there
    f, g = (v.copy() for v in sim().state())
    o, k = cs[0].mesh.ncells, cs[1].mesh.ncells
    f[:, o:o + k] *= 1e300
    a, b = sim(), sim()
    a.set_state(f, g)
    a.step(30)
    b.step(30)
    assert a.status() == [0, -3, 0] and b.status() == [0, 0, 0]
    fa, fb = a.state(), b.state()
    keep = np.r_[0:o, o + k:a.ncells]
    assert all(np.array_equal(x[:, keep], y[:, keep]) for x, y in zip(fa, fb))


def test_two_sims_on_two_streams_and_threads():
    """Many-step launches of two sims in flight at once, from two host threads."""
    import threading

    import torch
    cs = [I.stationary_drop(n=96, radius=24.0), I.rayleigh_taylor(nx=128, ny=256)]
    streams = [torch.cuda.Stream() for _ in cs]
    sims = [dugks.Sim(c.mesh, c.params, dugks.FP32, stream=st.cuda_stream).init(c.phi0) for c, st in zip(cs, streams)]
    ts = [threading.Thread(target=lambda s=s: [s.step(40) for _ in range(10)]) for s in sims]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    for c, s in zip(cs, sims):
        ref = dugks.Sim(c.mesh, c.params, dugks.FP32).init(c.phi0)
        for _ in range(40):
            ref.step(10)
        for x, y in zip(s.state(), ref.state()):
            assert np.array_equal(x, y)
