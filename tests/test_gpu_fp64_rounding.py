"""Rounding of the FP64 step: against the oracle compiled in extended precision (its
source with every double and every literal made long double), the step is no further
off than the oracle in double, which rounds the paper's formulas operation by
operation.  Root mean square over the field: g after one step from the same state, and
f after ten (f is driven through mu by the rounding of phi = sum g)."""
import ctypes
import re
import subprocess

import numpy as np
import pytest

import oracle
from paper_1802_02868_gb300 import dugks
from paper_1802_02868_gb300 import inputs as I

pytestmark = pytest.mark.gpu
LD = np.longdouble


@pytest.fixture(scope="module")
def extended(tmp_path_factory):
    if np.finfo(LD).eps > 1e-18:
        pytest.skip("long double is double here")
    d = tmp_path_factory.mktemp("extended")
    src = open(oracle.SRC).read()
    src = re.sub(r"\bdouble\b", "long double", src)
    src = re.sub(r"\b(sqrt|fabs|pow)\(", r"\1l(", src)
    src = re.sub(r'(?<![\w."<])(\d+\.\d+(?:e-?\d+)?)', r"\1L", src)
    (d / "o.c").write_text(src)
    subprocess.run(["gcc", "-O2", "-std=c11", "-fPIC", "-shared", "-ffp-contract=off", "-fopenmp", str(d / "o.c"), "-o",
                    str(d / "o.so"), "-lm"], check=True, stdout=subprocess.PIPE, stderr=subprocess.PIPE)
    L = ctypes.CDLL(str(d / "o.so"))
    vp = ctypes.c_void_p
    L.oracle_create.restype = vp
    L.oracle_create.argtypes = [ctypes.c_int] * 4 + [vp] * 3
    L.oracle_init.argtypes = [vp] * 5
    L.oracle_step.argtypes = [vp, ctypes.c_long]
    L.oracle_set_state.argtypes = L.oracle_get_state.argtypes = [vp] * 3
    L.oracle_destroy.argtypes = [vp]
    return L


def _extended_run(L, c, f, g, marks):
    ld = [np.ascontiguousarray(a, dtype=LD) for a in (c.mesh.dx, c.mesh.dy, c.params.as_list(), c.phi0, f, g)]
    p = [a.ctypes.data for a in ld]
    h = L.oracle_create(c.mesh.nx, c.mesh.ny, int(c.mesh.bc_x), int(c.mesh.bc_y), *p[:3])
    assert L.oracle_init(h, p[3], None, None, None) == 0
    L.oracle_set_state(h, p[4], p[5])
    out, done = {}, 0
    for n in marks:
        assert L.oracle_step(h, n - done) == 0
        done = n
        F, G = np.zeros(f.shape, LD), np.zeros(g.shape, LD)
        L.oracle_get_state(h, F.ctypes.data, G.ctypes.data)
        out[n] = (F, G)
    L.oracle_destroy(h)
    return out


@pytest.mark.parametrize("name", ["drop", "rayleigh_taylor", "cfl"])
def test_no_further_off_than_the_plain_double_evaluation(extended, name):
    c = {"drop": I.stationary_drop, "rayleigh_taylor": lambda: I.rayleigh_taylor(nx=48, ny=96),
         "cfl": lambda: I.cfl_sweep()[1]}[name]()
    s = dugks.Sim(c.mesh, c.params, dugks.FP64).init(c.phi0)
    f0, g0 = s.state()
    o = oracle.Oracle(c.mesh, c.params).init(c.phi0)
    o.set_state(f0, g0)
    ref = _extended_run(extended, c, f0, g0, (1, 10))

    def rms(a, b):
        return float(np.sqrt(np.mean((a - b) ** 2)))
    s.step(1)
    o.step(1)
    assert rms(s.state()[1], ref[1][1]) <= rms(o.state()[1], ref[1][1])
    s.step(9)
    o.step(9)
    assert rms(s.state()[0], ref[10][0]) <= rms(o.state()[0], ref[10][0])
