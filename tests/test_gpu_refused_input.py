"""dugks_init and dugks_load refuse a non-finite input, checked on the device, and
leave the simulation as it was: state, status and further steps."""
import numpy as np
import pytest

from paper_1802_02868_gb300 import dugks
from paper_1802_02868_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [dugks.FP64, dugks.FP32])
@pytest.mark.parametrize("batch", [False, True])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_refused_inputs_change_nothing(prec, batch, bad):
    cs = [I.stationary_drop(n=n, radius=0.25 * n) for n in ((33, 20) if batch else (33,))]

    def sim():
        return dugks.Sim([c.mesh for c in cs] if batch else cs[0].mesh, [c.params for c in cs] if batch else cs[0].params, prec)
    phi = [c.phi0.copy() for c in cs]
    a, b = (sim().init(phi if batch else phi[0]) for _ in range(2))
    a.step(18)
    b.step(18)
    f, g = (v.copy() for v in a.state())
    phi[-1][-1, -1] = bad                      # the last cell
    with pytest.raises(dugks.NonFiniteError):
        a.init(phi if batch else phi[0])
    h = g.copy()
    h.reshape(9, -1)[8, -1] = bad              # the last value of the buffer
    with pytest.raises(dugks.NonFiniteError):
        a.set_state(f, h)
    h = f.copy()
    h.reshape(-1)[0] = bad
    with pytest.raises(dugks.NonFiniteError):
        a.set_state(h, g)
    assert a.status() == [0] * len(cs)
    for s in (a, b):
        s.step(17)
    for x, y in zip(a.state(), b.state()):
        assert np.array_equal(x, y)
    # the gradient still starts from the accepted inputs
    t = [np.full(c.phi0.shape, 0.5) for c in cs]
    ga, gb = (s.adjoint(3, t if batch else t[0]) for s in (a, b))
    assert np.array_equal(ga["loss"], gb["loss"])


def test_velocity_and_pressure_inputs_are_taken():
    """init with ux, uy, p given reproduces them at once (Eq. auxf's moments)."""
    c = I.stationary_drop(n=40, radius=10.0)
    rng = np.random.default_rng(3)
    ux, uy, p = (1e-3 * rng.standard_normal(c.phi0.shape) for _ in range(3))
    m = dugks.Sim(c.mesh, c.params, dugks.FP64).init(c.phi0, ux, uy, p).moments()
    for k, v in (("ux", ux), ("uy", uy), ("p", p), ("phi", c.phi0)):
        assert np.abs(m[k] - v).max() < 1e-12
