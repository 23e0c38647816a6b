"""The reverse sweep's other routes give the gradient of the usual one to rounding (the
tolerances of test_gpu_adjoint_runs): without room for the recomputation's records,
where every reverse step forms them again, and on the four-kernel step, which recomputes
in place.  The state afterwards is that of the forward run."""
import numpy as np
import pytest

from paper_1802_02868_gb300 import dugks
from paper_1802_02868_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _cases():
    beta, kappa = I.params_from_sigma_width(1e-2, 3.0)
    p = I.Params(rhoA=2.0, rhoB=1.0, nuA=0.1, nuB=0.2, mobility=0.3, beta=beta, kappa=kappa, gx=1e-5, gy=-1e-4, rho_ref=1.5)
    out = []
    for nx, ny, by in ((40, 70, I.WALL), (48, 48, I.PERIODIC)):
        m = I.Mesh(1.0 + 0.2 * np.sin(np.arange(nx)), 1.0 + 0.1 * np.cos(np.arange(ny)), I.PERIODIC, by)
        out.append((m, p, I.drop_field(m, 0.3 * min(nx, ny), (0.45 * nx, 0.55 * ny), 3.0)))
    return out


def _run(prec, n=11, k=4):
    cs = _cases()
    with dugks.Sim([c[0] for c in cs], [c[1] for c in cs], prec).init([c[2] for c in cs]) as s:
        r = s.adjoint(n, [np.full(c[2].shape, 0.4) for c in cs], ckpt_every=k)
        after = [v.copy() for v in s.state()]
        t = dugks.Sim([c[0] for c in cs], [c[1] for c in cs], prec).init([c[2] for c in cs]).step(n).state()
    assert all(np.array_equal(x, y) for x, y in zip(after, t))
    return r


def _same(a, b, prec):
    tol = 1e-11 if prec == dugks.FP64 else 1e-4
    for k in range(2):
        assert np.abs(a["dphi0"][k] - b["dphi0"][k]).max() < tol * np.abs(b["dphi0"][k]).max()
        for v in ("dkappa", "dlambda", "loss"):
            assert a[v][k] == pytest.approx(b[v][k], rel=10 * tol)


@pytest.mark.parametrize("prec", [dugks.FP64, dugks.FP32])
def test_without_room_for_the_records(prec):
    import torch
    usual = _run(prec)
    sizes, limit = [], [1 << 62]

    def alloc(n, stream):
        if n > limit[0]:
            return 0
        sizes.append(n)
        return torch.cuda.caching_allocator_alloc(n, torch.cuda.current_device(), stream)
    dugks.set_allocator(alloc, lambda p, stream: torch.cuda.caching_allocator_delete(p))
    try:
        _same(_run(prec), usual, prec)
        limit[0] = max(sizes) - 1                  # refuses the one buffer with the records
        most = max(sizes)
        del sizes[:]
        _same(_run(prec), usual, prec)
        assert max(sizes) < most
    finally:
        dugks.set_allocator()


@pytest.mark.parametrize("prec", [dugks.FP64, dugks.FP32])
def test_on_the_four_kernel_step(prec, monkeypatch):
    usual = _run(prec)
    monkeypatch.setenv("DUGKS_UNFUSED", "1")
    _same(_run(prec), usual, prec)
