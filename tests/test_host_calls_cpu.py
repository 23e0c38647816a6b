"""The library's host code on a stand-in for the CUDA runtime that keeps "device"
memory on the host, runs no kernel and records what is ordered on which stream
(host_calls/recording_cudart.cpp): which stream every table goes to, and what the
calls report.  No GPU is needed."""
import ctypes
import glob
import importlib.util
import os
import shutil
import subprocess
import types

import numpy as np
import pytest

from paper_1802_02868_gb300 import build, dugks
from paper_1802_02868_gb300 import inputs as I

HERE = os.path.dirname(os.path.abspath(__file__))
STREAM = 0x5550   # what the calls get as the caller's stream: never dereferenced


class Recorder:
    def __init__(self, lib):
        self.lib = lib
        lib.rec_op.restype = ctypes.c_char_p
        for n in ("rec_count", "rec_coop_launches"):
            getattr(lib, n).restype = ctypes.c_long
        for n in ("rec_dst", "rec_bytes", "rec_stream", "rec_unreachable"):
            getattr(lib, n).restype = ctypes.c_ulonglong
        lib.rec_unreachable.argtypes = [ctypes.c_size_t]
        lib.rec_set_late.argtypes = [ctypes.c_ulonglong]

    def calls(self, fn):
        """What fn() put on the streams: (operation, destination, bytes, stream)."""
        L = self.lib
        L.rec_clear()
        fn()
        return [(L.rec_op(k).decode(), L.rec_dst(k), L.rec_bytes(k), L.rec_stream(k)) for k in map(ctypes.c_long, range(L.rec_count()))]


@pytest.fixture(scope="module")
def recording_library(tmp_path_factory):
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc")))
    if not shutil.which("g++") or not os.path.isdir(os.path.join(cuda, "include")):
        pytest.skip("no host compiler or CUDA headers")
    build.build()
    objs = sorted(glob.glob(os.path.join(build.BUILD_DIR, "dugks_*.o")))
    out = str(tmp_path_factory.mktemp("rec") / "libdugks_recording.so")
    r = subprocess.run(["g++", "-shared", "-fPIC", "-O1", "-std=c++17", "-I", os.path.join(cuda, "include"), "-Wl,-Bsymbolic",
                        "-Wl,--no-undefined", os.path.join(HERE, "host_calls", "recording_cudart.cpp")] + objs + ["-o", out],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return out


@pytest.fixture
def rec(recording_library):
    # a second copy of the binding, so that simulations of the real library, which may
    # be collected at any time, never meet this one
    spec = importlib.util.spec_from_file_location("paper_1802_02868_gb300.dugks_recording", dugks.__file__)
    binding = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(binding)
    binding._build = types.SimpleNamespace(LIB=recording_library)
    r = Recorder(binding.load())
    r.dugks = binding
    yield r
    r.lib.rec_set_capturing(0)
    r.lib.rec_set_late(0)


def _drops(rec, sizes, prec, stream=STREAM):
    cs = [I.stationary_drop(n=n, radius=0.25 * n) for n in sizes]
    s = rec.dugks.Sim([c.mesh for c in cs], [c.params for c in cs], prec, stream=stream)
    return s, [c.phi0 for c in cs]


@pytest.mark.parametrize("prec", [dugks.FP64, dugks.FP32])
@pytest.mark.parametrize("sizes", [(64,), (24, 41, 64)])
def test_tables_and_status_are_written_on_the_sims_stream(rec, sizes, prec):
    """A non-blocking stream has no order with the legacy stream of a plain copy:
    every write goes to the sim's stream, and the host waits on that stream for a
    copy out of its own memory before the call returns."""
    made = []
    log = [rec.calls(lambda: made.append(_drops(rec, sizes, prec)))]
    s, phi = made[0]
    with s:
        log.append(rec.calls(lambda: s.init(phi)))
        log.append(rec.calls(lambda: s.step(64)))          # the many-step launch's tables
        assert any(op.startswith("cooperative") for op, *_ in log[-1])
        log.append(rec.calls(lambda: s.step(3)))
        log.append(rec.calls(lambda: s.set_tile_shape(5)))
        log.append(rec.calls(s.diagnostics_array))
        log.append(rec.calls(lambda: s.set_paused([k == 0 for k in range(len(sizes))])))
        log.append(rec.calls(lambda: s.set_paused([False] * len(sizes))))
        log.append(rec.calls(lambda: s.step_each([20 + k for k in range(len(sizes))])))
        log.append(rec.calls(lambda: s.adjoint(3, phi)))
    for calls in log:
        writes = [k for k, c in enumerate(calls) if c[0] == "copy h2d" or c[0] == "memset"]
        assert all(calls[k][3] == STREAM for k in writes), [calls[k] for k in writes]
        up = [k for k in writes if calls[k][0] == "copy h2d"]
        if up:
            assert any(c[0] == "sync" and c[3] == STREAM for c in calls[up[-1] + 1:])
    assert sum(c[0] == "copy h2d" for c in sum(log, [])) >= 15


def test_a_table_made_while_the_caller_captures_stays_out_of_the_capture(rec):
    s, phi = _drops(rec, (64,), dugks.FP32)
    with s:
        s.init(phi)
        rec.lib.rec_set_capturing(1)
        calls = rec.calls(lambda: s.step(1))               # the first step makes the tile table
        up = [c for c in calls if c[0] == "copy h2d"]
        assert len(up) == 1 and up[0][3] not in (0, STREAM)
        assert ("sync", 0, 0, up[0][3]) in calls
        assert not any(c[0] == "sync" and c[3] == STREAM for c in calls)


@pytest.mark.parametrize("sizes", [(64,), (24, 41, 64)])
def test_every_synchronising_call_reports_a_wait_that_ran_out(rec, sizes):
    made = []
    n = len(sizes)
    calls = rec.calls(lambda: made.append(_drops(rec, sizes, dugks.FP32)))
    s, phi = made[0]
    with s:
        # the per-instance status, the error word, the refused word
        (at,) = {c[1] for c in calls if c[0] == "memset" and c[2] == 4 * (n + 2)}
        s.init(phi)
        start = s.state()
        rec.lib.rec_set_late(at + 4 * n)
        s.step(64)
        assert rec.lib.rec_coop_launches() > 0
        rec.lib.rec_set_late(0)
        for name, fn in (("save", s.state), ("status", s.status), ("set_paused", lambda: s.set_paused([False] * n)),
                         ("step_each", lambda: s.step_each([1] * n)), ("moments", s.moments), ("conservation", s.conservation),
                         ("diagnostics", s.diagnostics_array), ("laplace_pressure", s.laplace_pressure),
                         ("kernel_times", s.kernel_times), ("set_tile_shape", lambda: s.set_tile_shape(1)), ("autotune", s.autotune)):
            with pytest.raises(rec.dugks.DugksError) as e:
                fn()
            assert e.value.rc == -5, name
        s.init(phi)                                     # a new state: nothing to report
        s.step(64)
        assert s.status() == [0] * n
        rec.lib.rec_set_late(at + 4 * n)
        s.step(64)
        rec.lib.rec_set_late(0)
        s.set_state(*start)
        s.state()


def test_outputs_that_the_host_cannot_write_are_left_to_the_copy(rec):
    """Device memory as an output of a size whose pages are touched ahead of the copy:
    the runtime refuses the copy, and the process lives to see it."""
    s, phi = _drops(rec, (128,), dugks.FP64)              # 128 KB a field
    n = 8 * s.ncells
    with s:
        s.init(phi)

        def refused(name, *args):
            return getattr(rec.lib, name)(s.h, *args) == -2   # the runtime's error
        tgt = np.zeros(s.ncells)
        at = [ctypes.c_void_p(rec.lib.rec_unreachable(n)) for _ in range(5)]
        big = ctypes.c_void_p(rec.lib.rec_unreachable(18 * n))
        checks = [lambda: refused("dugks_moments", *[ctypes.cast(a, ctypes.POINTER(ctypes.c_double)) for a in at]),
                  lambda: refused("dugks_laplace_pressure", ctypes.cast(at[0], ctypes.POINTER(ctypes.c_double))),
                  lambda: refused("dugks_save", big, ctypes.byref(ctypes.c_size_t(18 * n))),
                  lambda: refused("dugks_adjoint", 2, 1, tgt.ctypes.data_as(ctypes.POINTER(ctypes.c_double)), None,
                                  ctypes.cast(at[0], ctypes.POINTER(ctypes.c_double)), None, None)]
        for k, ok in enumerate(checks):
            pid = os.fork()                                # a child: the fault would be a signal
            if pid == 0:
                os._exit(0 if ok() else 1)
            assert os.waitpid(pid, 0)[1] == 0, k


@pytest.mark.parametrize("nx,ny,prec,n,least,most", [(256, 1024, dugks.FP64, 512, 12, 20), (512, 1024, dugks.FP64, 512, 24, 40),
                                                     (64, 64, dugks.FP32, 512, 1, 1), (64, 64, dugks.FP64, 512, 1, 1),
                                                     (64, 64, dugks.FP32, 1050, 3, 3)])
def test_a_many_step_launch_holds_the_device_for_milliseconds(rec, nx, ny, prec, n, least, most):
    """512 steps of a small mesh, but about 20 ms of a large one: a step of
    256x1024 in FP64 takes 0.6 ms, one of 512x1024 twice that, one of 64x64 0.02 ms."""
    m = I.uniform_mesh(nx, ny)
    with rec.dugks.Sim(m, I.stationary_drop().params, prec, stream=STREAM) as s:
        s.init(I.drop_field(m, 0.3 * nx, (0.5 * nx, 0.5 * ny), 4.0))
        calls = rec.calls(lambda: s.step(n))
        assert least <= rec.lib.rec_coop_launches() <= most
        assert not any(c[0].startswith(("kernel", "graph")) for c in calls)   # they take every step of the call


@pytest.mark.parametrize("steps", [5, 20])
def test_autotune_sets_up_before_it_times(rec, steps):
    """Between the two events of a trial there are only launches, of kernels that ran
    before: no allocation, upload, capture or wait for one."""
    s, phi = _drops(rec, (64,), dugks.FP32)
    with s:
        s.init(phi)
        calls = rec.calls(lambda: s.autotune(steps))
        marks = [k for k, c in enumerate(calls) if c[0] == "event"]
        assert len(marks) == 2 * dugks.NUM_TILE_SHAPES
        for a, b in zip(marks[::2], marks[1::2]):
            timed = [c[0] for c in calls[a + 1:b]]
            assert timed and all(op.startswith(("kernel", "cooperative", "graph")) for op in timed), timed
            assert {op for op in timed if op != "graph"} <= {c[0] for c in calls[:a]}
        assert any(c[0].startswith("cooperative") for c in calls) == (steps >= 16)


def test_segments_on_another_tile_keep_the_usual_tiles_graph(rec):
    """Per-instance step counts may run a segment on another tile; the two-step graph of
    short calls is not captured again after each."""
    s, phi = _drops(rec, (100, 100, 100, 100), dugks.FP64)
    with s:
        s.init(phi)
        s.step(4)
        for _ in range(2):
            s.step_each([20, 20, 20, 60])               # the last segment: one instance, smaller tiles
            calls = rec.calls(lambda: s.step(4))
            assert any(c[0] == "graph" for c in calls)
            assert not any(c[0] == "begin capture" for c in calls)
