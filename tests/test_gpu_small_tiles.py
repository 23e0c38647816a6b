"""The smaller tiles that shape 0 is cut into on meshes too small to occupy the
device give the results of the strips: the same bits on uniform periodic
meshes, to rounding with walls or uneven spacing."""
import numpy as np
import pytest

from paper_1802_02868_gb300 import dugks
from paper_1802_02868_gb300 import inputs as I

pytestmark = pytest.mark.gpu

# sizes around the tiles' edges and remainders, from less than one tile to the
# sizes at which the rule goes from 8x4 and 4x8 to 8x8, to 16x8 and to 32x8 in
# FP64, and from 8x8 to 16x8 and to 32x8 in FP32
SIZES = [(3, 70), (4, 256), (5, 9), (9, 33), (64, 64), (81, 90), (100, 100), (127, 128), (130, 250), (256, 260)]


def _states(meshes, prms, phis, prec, shape, steps):
    s = dugks.Sim(meshes, prms, prec)
    s.set_tile_shape(shape)
    s.init(phis).step(steps)
    out = s.state()
    s.close()
    return out


def _norm(a, b):
    return np.abs(a - b).max() / np.abs(b).max()


@pytest.mark.parametrize("prec", [dugks.FP64, dugks.FP32])
@pytest.mark.parametrize("nx,ny", SIZES)
def test_small_tiles_equal_the_strips(nx, ny, prec):
    prm = I.stationary_drop().params
    m = I.uniform_mesh(nx, ny)
    phi = I.drop_field(m, 0.3 * min(nx, ny), (0.5 * nx, 0.4 * ny), 4.0)
    a = _states(m, prm, phi, prec, 0, 7)
    b = _states(m, prm, phi, prec, 4, 7)
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
    # walls on both axes, stretched spacings; 1e-13 and 1e-6 are the bounds that
    # every pair of shapes is held to
    m = I.Mesh(1.0 + 0.2 * np.cos(np.arange(nx)), 1.0 + 0.2 * np.sin(np.arange(ny)), I.WALL, I.WALL)
    a = _states(m, prm, phi, prec, 0, 7)
    b = _states(m, prm, phi, prec, 4, 7)
    tol = 1e-13 if prec == dugks.FP64 else 1e-6
    assert _norm(a[0], b[0]) < tol and _norm(a[1], b[1]) < tol


def test_a_batch_of_small_meshes_pauses_and_steps_like_its_instances():
    cs = [I.stationary_drop(n=n, radius=0.25 * n) for n in (24, 41, 64)]
    b = dugks.Sim([c.mesh for c in cs], [c.params for c in cs], dugks.FP64).init([c.phi0 for c in cs])
    b.step_each([5, 2, 9])
    f, g = b.state()
    o = 0
    for c, n in zip(cs, (5, 2, 9)):
        s = dugks.Sim(c.mesh, c.params, dugks.FP64).init(c.phi0).step(n)
        fs, gs = s.state()
        k = c.mesh.ncells
        assert np.array_equal(f[:, o:o + k], fs.reshape(9, -1)) and np.array_equal(g[:, o:o + k], gs.reshape(9, -1))
        o += k
