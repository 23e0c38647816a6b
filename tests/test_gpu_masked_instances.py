"""A batch whose one instance overflows while most of its thread blocks have still to
start: the blocks of that instance that see it masked and those that do not leave the
other instances alone, whatever the kernel (tiles, strips, many-step launches, the
adjoint's recomputation)."""
import numpy as np
import pytest

from paper_1802_02868_gb300 import dugks
from paper_1802_02868_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _batch(prec, shape, big):
    cs = [I.stationary_drop(n=n, radius=0.25 * n) for n in (96, big, 57)]
    s = dugks.Sim([c.mesh for c in cs], [c.params for c in cs], prec)
    if shape is not None:
        s.set_tile_shape(shape)
    s.init([c.phi0 for c in cs])
    o, k = cs[0].mesh.ncells, cs[1].mesh.ncells
    return s, cs, np.r_[0:o, o + k:s.ncells], (o, k)


@pytest.mark.parametrize("prec", [dugks.FP64, dugks.FP32])
@pytest.mark.parametrize("shape", range(dugks.NUM_TILE_SHAPES))
def test_an_instance_that_overflows_leaves_the_others_alone(shape, prec):
    a, cs, keep, (o, k) = _batch(prec, shape, 768)
    b = _batch(prec, shape, 768)[0]
    f, g = (v.copy() for v in a.state())
    f[:, o + 3] = 1e300 if prec == dugks.FP64 else 3e38     # one cell of its first tile
    for n in ((1, 1, 1), (20,)):                           # single launches; one call of many steps
        a.set_state(f, g)
        b.set_state(*(v.copy() for v in _batch(prec, shape, 768)[0].state()))
        for m in n:
            a.step(m)
            b.step(m)
        assert a.status() == [0, -3, 0] and b.status() == [0, 0, 0]
        for x, y in zip(a.state(), b.state()):
            assert np.array_equal(x[:, keep], y[:, keep])


@pytest.mark.parametrize("prec", [dugks.FP64, dugks.FP32])
def test_gradients_beside_an_instance_that_overflows(prec):
    a, cs, keep, (o, k) = _batch(prec, None, 384)
    b = _batch(prec, None, 384)[0]
    phi = [c.phi0.copy() for c in cs]
    phi[1][0, 3] = 1e300 if prec == dugks.FP64 else 1e30    # psi'(phi) overflows
    t = [np.full(c.phi0.shape, 0.4) for c in cs]
    try:
        a.init(phi)
    except dugks.NonFiniteError:
        pytest.fail("a finite phi is taken")
    ra, rb = (s.adjoint(6, t, ckpt_every=3) for s in (a, b))
    assert a.status() == [0, -3, 0]
    for m in (0, 2):
        assert np.array_equal(ra["dphi0"][m], rb["dphi0"][m])
        assert ra["dkappa"][m] == rb["dkappa"][m] and ra["dlambda"][m] == rb["dlambda"][m] and ra["loss"][m] == rb["loss"][m]
