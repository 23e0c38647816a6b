"""FP32 gradients with respect to kappa over many steps of a flow: the rounding of a
reverse step must not shift the adjoint the same way every step.  Unbiased rounding of
n steps leaves about sqrt(n) units of FP32 rounding (6e-8); a bias of a tenth of a unit
per step leaves n / 10 of them, 10 to 50 times as much on these runs."""
import numpy as np
import pytest

from paper_1802_02868_gb300 import dugks
from paper_1802_02868_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,seed,n", [(64, 128, None, 200), (256, 512, 7, 500), (256, 512, 11, 500)])
def test_dkappa_of_rayleigh_taylor(nx, ny, seed, n):
    if seed is None:
        amps, tgt_amps = [0.1 * nx], [0.12 * nx]
    else:
        rng = np.random.default_rng(seed)
        amps = np.concatenate([[0.1 * nx], rng.normal(0.0, 0.01 * nx, 7)])
        tgt_amps = amps + rng.normal(0.0, 0.01 * nx, 8)
    c = I.rayleigh_taylor(nx=nx, ny=ny, amplitudes=list(amps))
    tgt = I.rt_field(c.mesh, float(nx), 0.5 * ny, list(tgt_amps), 4.0)
    k = {}
    for p in (dugks.FP32, dugks.FP64):
        with dugks.Sim(c.mesh, c.params, p).init(c.phi0) as s:
            k[p] = s.adjoint(n, tgt, ckpt_every=100)["dkappa"]
    assert abs(k[dugks.FP32] / k[dugks.FP64] - 1) < np.sqrt(n) * 6e-8
