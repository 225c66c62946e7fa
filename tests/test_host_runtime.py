"""The host runtime on a CUDA runtime that runs nothing (host_runtime.cpp): which launches
a call issues, and what it leaves behind when one of them fails."""
import ctypes
import os
import shutil
import subprocess

import pytest

from paper_1406_6438_gb300 import build as B
from paper_1406_6438_gb300._binding import Params, _CLaunch

HERE = os.path.dirname(os.path.abspath(__file__))
ERR_ARG, ERR_CUDA, FAKE = -1, -2, ctypes.c_void_p(1 << 20)      # FAKE: never read or written


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("host") / "host_runtime.so")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(B._nvcc()))), "include")
    subprocess.run([shutil.which("g++"), "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", B.INCLUDE,
                    "-I", B.CSRC, "-isystem", cuda, "-include", "cstring", "-include", "cstdlib", "-x", "c++",
                    os.path.join(B.CSRC, "vans_api.cu"), os.path.join(HERE, "host_runtime.cpp"), "-o", so], check=True)
    so = ctypes.CDLL(so)
    so.fake_log.restype, so.fake_steps.restype = ctypes.c_char_p, ctypes.c_longlong
    so.vans_workspace_bytes.restype = so.vans_batch_workspace_bytes.restype = ctypes.c_size_t
    return so


class Handle:
    """A handle with its porosity set; log() is what has been launched since the last."""

    def __init__(self, lib, launch=None, **kw):
        self.lib, self.h = lib, ctypes.c_void_p()
        lib.fake_reset()
        p = Params(**dict(dict(q=9, nx=600, ny=400, tau=0.7), **kw)).c()
        n = lib.vans_workspace_bytes(ctypes.byref(p))
        assert lib.vans_create(ctypes.byref(p), FAKE, ctypes.c_size_t(n), None, ctypes.byref(self.h)) == 0
        assert self("set_eps", FAKE) == 0
        if launch:
            assert self("set_launch", ctypes.byref(_CLaunch(*launch))) == 0
        self.log()

    def __call__(self, name, *a):
        return getattr(self.lib, "vans_" + name)(self.h, *a)

    def log(self):
        lines = self.lib.fake_log().decode().split("\n")[:-1]
        self.lib.fake_reset()
        return lines

    def steps(self):
        n = self.lib.fake_steps()
        self.lib.fake_reset()
        return n


KINDS = [(4, 4, 1, 0, 0), (2, 4, 4, 9, 0), (2, 4, 3, 9, 0), (2, 4, 2, 9, 0)]


@pytest.mark.parametrize("launch", KINDS)
@pytest.mark.parametrize("what", ["capture", "instantiate"])
@pytest.mark.parametrize("nth", [1, 2])
def test_a_failed_capture_ends_no_run_half_done(lib, launch, what, nth):
    """Graphs of several sizes serve a run: where one of them cannot be made, the run takes
    its steps all the same, and the next one captures again."""
    for warm in (0, 1):
        h = Handle(lib, launch)
        h("step", warm)
        h.log()
        for n, call in ((63 * launch[2], ("step", 63 * launch[2])), (190, ("step_monitored", 190, 63, FAKE, FAKE, FAKE))):
            h.log()
            lib.fake_fail(what.encode(), nth)
            assert h(*call) == 0
            # (kind 9 emits between launches of several steps, which then are all of the steps)
            assert h.steps() == n
        assert h("step", 63 * launch[2]) == 0
        assert h.steps() == 63 * launch[2]


@pytest.mark.parametrize("launch", KINDS)
def test_a_captured_stream_takes_no_run_that_needs_graphs(lib, launch):
    """Refused with nothing recorded, whether its graphs exist, are made or cannot be."""
    for warm in (False, True):
        for fails in (False, True):
            h = Handle(lib, launch)
            if warm:
                h("step", 64 * launch[2])
                h.log()
            if fails:
                lib.fake_fail(b"capture", 1)
            lib.fake_user_capture(1)
            assert h("step", 64 * launch[2]) == ERR_CUDA
            assert h.steps() == 0


@pytest.mark.parametrize("launch", KINDS)
@pytest.mark.parametrize("n", [0, 1, 2, 3, 5, 9, 131, 2**31 - 1])
def test_a_run_takes_the_steps_it_was_asked_for(lib, launch, n):
    h = Handle(lib, launch)
    lib.fake_quiet()
    assert h("step", n) == 0
    assert h.steps() == n


@pytest.mark.parametrize("warm", [False, True])
def test_update_eps_is_refused_under_capture(lib, warm):
    """It has to wait for its range check.  The refusal leaves nothing in the capture: the
    caller's graph would update the state of a call that failed."""
    h = Handle(lib)
    if warm:
        assert h("update_eps", FAKE) == 0
        assert h.log()[-2:] == ["rebase", "pad"]
    lib.fake_user_capture(1)
    assert h("update_eps", FAKE) == ERR_CUDA
    assert h.log() == []
    assert h("update_eps", FAKE) == 0


def test_a_reverse_shape_that_does_not_fit_is_refused(lib):
    """Stages that exceed 227 KB were accepted here and failed at every launch."""
    h = Handle(lib, q=19, nx=40, ny=5, nz=3)
    most = {2: 8, 3: 8, 4: 8, 5: 7, 6: 5, 7: 5}
    for warps in range(2, 8):
        for stages in range(2, 9):
            rc = h("set_adjoint_launch", ctypes.byref(_CLaunch(1, warps, stages, 1, 0)))
            assert rc == (0 if stages <= most[warps] else ERR_ARG), (warps, stages)


@pytest.mark.parametrize("nx,warps", [(1, 2), (24, 2), (32, 2), (64, 2), (65, 3), (150, 5), (256, 8), (300, 5)])
def test_autotune_tries_the_tile_that_fits_the_rows(lib, nx, warps):
    """Of the D3Q19 tiles with one cell per thread and 2 stages: the narrowest of 64 to 256
    cells that takes a row in as few tiles as there can be."""
    h = Handle(lib, q=19, nx=nx, ny=40, nz=30)
    assert h("autotune", None) == 0
    tried = {tuple(s.split()[2:]) for s in h.log() if s.startswith("step 1 kind 6")}
    assert [t[3] for t in tried if t[5] == "2"] == [str(warps)], tried


def test_strips_are_chosen_when_the_shape_is_set(lib):
    """The search over strip counts is not part of a step, of whatever length."""
    h = Handle(lib)
    for k in (2, 3, 4):
        assert h("set_launch", ctypes.byref(_CLaunch(2, 4, k, 9, 0))) == 0
        assert h.log() == ["strips %d" % n for n in range(2, max(3, k) + 1)]
        for call in (("step", 131), ("step", 5), ("step", 2), ("step_monitored", 20, 10, FAKE, FAKE, FAKE)):
            assert h(*call) == 0
            lines = h.log()
            assert not [s for s in lines if s.startswith("strips")]
            assert all(s == "multi %d strips %d0" % (int(s[6]), int(s[6])) for s in lines if s.startswith("multi"))
    assert h("autotune", None) == 0
    h.log()
    assert h("step", 131) == 0
    assert not [s for s in h.log() if s.startswith("strips")]


@pytest.mark.parametrize("launch", KINDS[1:])
@pytest.mark.parametrize("n", [2, 3, 4, 5, 7, 9, 10, 11, 131])
def test_no_step_is_left_alone(lib, launch, n):
    """A run of two or more steps issues launches of several steps only: a single-step
    launch rounds otherwise, and the result would depend on how the run was split."""
    h = Handle(lib, launch)
    for call in (("step", n), ("step_monitored", 3 * n + 3, n + 1, FAKE, FAKE, FAKE)):
        assert h(*call) == 0
        lines = [s for s in h.log() if s.startswith(("step", "multi"))]
        if call[0] == "step_monitored":
            lines = lines[:-1]              # the last emission's step has none after it
        assert lines and all(s.startswith("multi") for s in lines)
