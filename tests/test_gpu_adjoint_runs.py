"""The reverse sweep's runs of 32 cells and faces and its tiles, on meshes that leave
remainders of both, with walls and periodic, below and above the size at which a
cell's work is split over four warps: FP64 gradients against the oracle's
complex-step derivatives (the bounds of test_gpu_adjoint), FP32 ones the same twice."""
import numpy as np
import pytest

import oracle
from paper_1802_02868_gb300 import dugks
from paper_1802_02868_gb300 import inputs as I

pytestmark = pytest.mark.gpu

SIZES = [(5, 40, I.PERIODIC, I.WALL), (33, 18, I.WALL, I.PERIODIC), (31, 35, I.WALL, I.WALL), (65, 17, I.PERIODIC, I.PERIODIC),
         (40, 330, I.PERIODIC, I.WALL)]


def _case(nx, ny, bx, by):
    beta, kappa = I.params_from_sigma_width(1e-2, 3.0)
    m = I.Mesh(1.0 + 0.2 * np.sin(np.arange(nx)), 1.0 + 0.1 * np.cos(np.arange(ny)), bx, by)
    p = I.Params(rhoA=2.0, rhoB=1.0, nuA=0.1, nuB=0.2, mobility=0.3, beta=beta, kappa=kappa, gx=1e-5, gy=-1e-4, rho_ref=1.5)
    return m, p, I.drop_field(m, 0.3 * min(nx, ny), (0.45 * nx, 0.55 * ny), 3.0)


@pytest.mark.parametrize("nx,ny,bx,by", SIZES)
def test_gradients_against_the_oracle(nx, ny, bx, by):
    m, p, phi0 = _case(nx, ny, bx, by)
    rng = np.random.default_rng(7)
    target = 0.5 + 0.1 * rng.standard_normal(phi0.shape)
    v = rng.standard_normal(phi0.shape)
    got = dugks.Sim(m, p, dugks.FP64).init(phi0).adjoint(6, target, ckpt_every=4)
    ref = oracle.complex_step_gradient(m, p, phi0, 6, target, direction_phi0=v, which=("kappa", "mobility"))
    assert got["dkappa"] == pytest.approx(ref["kappa"], rel=1e-8)
    assert got["dlambda"] == pytest.approx(ref["mobility"], rel=1e-8)
    assert np.sum(got["dphi0"] * v) == pytest.approx(ref["phi0_dir"], rel=1e-8)


@pytest.mark.parametrize("prec", [dugks.FP64, dugks.FP32])
def test_gradients_are_reproducible_and_a_batch_gives_its_instances(prec):
    cs = [_case(*s) for s in SIZES[:4]]
    t = [np.full(c[2].shape, 0.4) for c in cs]
    b = dugks.Sim([c[0] for c in cs], [c[1] for c in cs], prec).init([c[2] for c in cs])
    r = [b.adjoint(6, t, ckpt_every=4) for _ in range(2)]
    for k in range(4):
        s = dugks.Sim(cs[k][0], cs[k][1], prec).init(cs[k][2]).adjoint(6, t[k], ckpt_every=3)
        assert np.array_equal(r[0]["dphi0"][k], r[1]["dphi0"][k])
        assert r[0]["dkappa"][k] == r[1]["dkappa"][k] and r[0]["dlambda"][k] == r[1]["dlambda"][k]
        # alone, the tiles and the split may be others: to rounding
        tol = 1e-11 if prec == dugks.FP64 else 1e-4
        assert np.abs(r[0]["dphi0"][k] - s["dphi0"]).max() < tol * np.abs(s["dphi0"]).max()
