"""What the host keeps between calls (step state, tuned choices), on a fake
CUDA runtime (fake_cudart.cpp) that logs copies and launches: a call that was
only captured into the caller's graph, or whose launches failed, has left
nothing that a later call may rely on."""
import ctypes
import glob
import os
import shutil
import subprocess

import pytest

import paper_0710_5912_gb300 as shf
from paper_0710_5912_gb300 import _native

HERE = os.path.dirname(os.path.abspath(__file__))
INIT, OMEGA, STAGE1 = "k_step_state_init", "k_colpass_single", "k_stage1_rows"


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("no host compiler")
    _native.build(force=not glob.glob(os.path.join(_native.BUILD_DIR, "*.o")))
    out = str(tmp_path_factory.mktemp("fake") / "libshf_fake.so")
    cuda = os.path.join(os.path.dirname(os.path.dirname(_native.nvcc_path())), "include")
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", cuda, "-o", out,
                    os.path.join(HERE, "fake_cudart.cpp"), *glob.glob(os.path.join(_native.BUILD_DIR, "*.o"))],
                   check=True)
    lib = ctypes.CDLL(out)
    _native._declare(lib)
    lib.fake_log.restype = ctypes.c_char_p
    return lib


class Run:
    """A grid on the fake runtime; log() gives the lines since the last look."""

    def __init__(self, lib, rho=1.0):
        self.lib, self.h = lib, ctypes.c_void_p()
        assert lib.shf_create_grid(ctypes.byref(self.h), 64, 64, 1.0, shf.SHF_FP32, shf.SHF_REMAP_SHIFT,
                                   ctypes.c_void_p(0x10)) == 0
        assert lib.shf_set_params(self.h, 1.0, 1.0, 1.0, 1.0, 1.0, rho, 0.1, 0.01) == 0
        self.log()

    def log(self):
        lines = self.lib.fake_log().decode().splitlines()
        self.lib.fake_clear()
        return lines

    def step(self, n=1, rc=0):
        assert self.lib.shf_step(self.h, n) == rc
        return self.log()

    def captured_step(self):
        self.lib.fake_capture(1)
        try:
            return self.step()
        finally:
            self.lib.fake_capture(0)


@pytest.fixture
def run(fake):
    r = Run(fake)
    yield r
    fake.fake_capture(0)
    fake.fake_fail_launch(-1)
    fake.fake_fail_copy(-1)
    fake.shf_destroy_grid(r.h)


def has(log, kernel):
    return sum(kernel in line for line in log)


def test_state_is_formed_once_and_kept(run):
    first, second = run.step(), run.step()
    assert has(first, INIT) == 1 and has(first, STAGE1) == 1
    assert has(second, INIT) == 0 and has(second, STAGE1) == 1
    assert len(first) == len(second) + 3                # the state, omega's row and column transforms


def test_a_captured_call_leaves_nothing_behind(run):
    captured, eager = run.captured_step(), run.step()
    assert has(captured, INIT) == 1
    assert has(eager, INIT) == 1 and len(eager) == len(captured)


def test_a_captured_call_does_not_lean_on_the_state_of_the_moment(run):
    run.step()
    captured = run.captured_step()
    assert has(captured, INIT) == 1                     # it may be replayed after shf_set_step


@pytest.mark.parametrize("launch", [0, 1, 2, 5])
def test_a_failed_launch_is_not_taken_for_done(run, launch):
    run.lib.fake_fail_launch(launch)
    run.step(rc=shf.SHF_ECUDA)
    again = run.step()
    assert has(again, INIT) == 1 and has(again, OMEGA) == 3 and has(again, STAGE1) == 1


@pytest.mark.parametrize("copy", range(6))
def test_no_copy_outlives_a_failed_host_call(run, copy):
    """Host arrays belong to the caller once the call has returned, and the
    next call on the grid's stream must not meet this one's uploads."""
    f = [(ctypes.c_float * (64 * 64))() for _ in range(6)]
    run.lib.fake_fail_copy(copy)
    assert run.lib.shf_step_host_f32(run.h, 1, *f) == shf.SHF_ECUDA
    lines = [line.split() for line in run.log()]
    for stream in {line[1] for line in lines if line[0] == "copy"}:
        names = [line[0] for line in lines if line[1] == stream]
        assert "sync" in names[len(names) - names[::-1].index("copy"):]
    assert has(run.step(), INIT) == 1


def tune(run, path):
    out = (ctypes.c_int * 2)()
    assert run.lib.shf_autotune(run.h, str(path).encode(), out, 2) == 0
    return out[0], has(run.log(), STAGE1)               # the choice and the trial launches


def test_tuned_choices_are_taken_from_like_runs_only(run, tmp_path):
    """On this runtime every launch takes the same time, and 8 points are tried
    first: a trial ends with 8, a cached 16 is seen to be applied."""
    path = tmp_path / "tune.json"
    old = '"64x64:fp32:inertial": {"stage1_points": 16, "stage2_points": 16'
    path.write_text("{\n  %s, \"launch\": 2}\n}\n" % old)
    assert tune(run, path) == (16, 0)
    for line in (old + "}",                             # timed before thread groups
                 old.replace("16, ", "7, ") + ', "launch": 2}',     # no variant
                 old.replace('inertial"', 'inertial:96"') + ', "launch": 2}'):
        path.write_text("{\n  %s\n}\n" % line)
        choice, trials = tune(run, path)
        assert choice == 8 and trials > 0
        assert '"64x64:fp32:inertial": {"stage1_points": 8, ' in path.read_text()


def test_tuned_choices_of_many_members_have_their_own_entry(fake, tmp_path):
    path, n = tmp_path / "tune.json", 5
    ens, sizes = ctypes.c_void_p(), (ctypes.c_int * n)(*[64] * n)
    params = (ctypes.c_double * (8 * n))(*[1.0, 1.0, 1.0, 1.0, 1.0, 1.0, 0.1, 0.01] * n)
    assert fake.shf_create_ensemble(ctypes.byref(ens), n, sizes, sizes, None, params, None, 0.0, shf.SHF_FP32, None) == 0
    assert fake.shf_autotune(ens, str(path).encode(), None, 0) == 0
    assert '"64x64:fp32:inertial:5"' in path.read_text()
    fake.shf_destroy_grid(ens)
    fake.fake_clear()
