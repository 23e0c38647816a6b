"""A wait of a many-step launch that runs out: the launch ends, every synchronising call
reports it, and a new state is as good as that of a fresh simulation.  The limit is set
to no poll at all, so that a tile gives up on the first neighbour that is still at
work."""
import numpy as np
import pytest

from paper_1802_02868_gb300 import dugks
from paper_1802_02868_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [dugks.FP64, dugks.FP32])
@pytest.mark.parametrize("sizes", [(200,), (96, 130)])
def test_a_wait_that_runs_out_is_reported_until_a_new_state(sizes, prec, monkeypatch):
    cs = [I.stationary_drop(n=n, radius=0.25 * n) for n in sizes]

    def sim():
        return dugks.Sim([c.mesh for c in cs], [c.params for c in cs], prec)
    phi = [c.phi0 for c in cs]
    monkeypatch.setenv("DUGKS_WAIT_POLLS", "0")
    a = sim().init(phi)
    monkeypatch.delenv("DUGKS_WAIT_POLLS")
    b = sim().init(phi)
    start = [v.copy() for v in a.state()]
    for fresh in (lambda s: s.init(phi), lambda s: s.set_state(*start)):
        a.step(200)
        for call in (a.state, a.status, a.moments, a.conservation, lambda: a.step_each([1] * len(sizes))):
            with pytest.raises(dugks.DugksError) as e:
                call()
            assert e.value.rc == -5
        fresh(a)
        fresh(b)
        a.step(7)                      # one launch per step: no wait
        b.step(7)
        assert a.status() == [0] * len(sizes)
        for x, y in zip(a.state(), b.state()):
            assert np.array_equal(x, y)
