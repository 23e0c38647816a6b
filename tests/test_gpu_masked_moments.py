"""What dugks_moments reports of an instance that became non-finite: rho, u and p as
the last call found them while it was finite (before any call, rho zero and the u and p
of dugks_init), beside the present moments of the other instances."""
import numpy as np
import pytest

from paper_1802_02868_gb300 import dugks
from paper_1802_02868_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [dugks.FP64, dugks.FP32])
@pytest.mark.parametrize("called", [False, True])
def test_a_masked_instance_keeps_its_last_finite_moments(called, prec):
    cs = [I.stationary_drop(n=n, radius=0.25 * n) for n in (33, 20)]
    rng = np.random.default_rng(5)
    ux, uy, p = ([1e-3 * rng.standard_normal(c.phi0.shape) for c in cs] for _ in range(3))

    def sim():
        return dugks.Sim([c.mesh for c in cs], [c.params for c in cs], prec).init([c.phi0 for c in cs], ux, uy, p)
    a, b = sim(), sim()
    for s in (a, b):
        s.step(5)
    if called:
        last = {k: v[1].copy() for k, v in a.moments().items()}
    else:
        last = {"rho": np.zeros(cs[1].phi0.shape)}
        last.update({k: v[1].astype(np.float32 if prec == dugks.FP32 else np.float64) for k, v in (("ux", ux), ("uy", uy), ("p", p))})
    f, g = (v.copy() for v in a.state())
    b.set_state(f, g)
    f[:, cs[0].mesh.ncells:] *= 1e300 if prec == dugks.FP64 else 1e38
    a.set_state(f, g)
    for s in (a, b):
        s.step(3)
    assert a.status() == [0, -3]
    for _ in range(2):                              # a call leaves them as they are
        m, n = a.moments(), b.moments()
        for k in ("rho", "ux", "uy", "p"):
            assert np.array_equal(m[k][1], last[k]), k
        for k in m:
            assert np.array_equal(m[k][0], n[k][0]), k
