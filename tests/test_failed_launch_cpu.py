"""Calls whose kernel launches the runtime refuses, with the library's own host
objects linked against a fake runtime on host memory (tests/host_emulation/
fake_cudart.cpp; kernels do not run): the error is returned and not left behind as
the thread's last error, where the next launch, of this library or of another one,
would report it as its own. A step or a reset that fails after cells may have been
queued for the limiter leaves the queue's count at 0, for every launch that can
fail; if even that memset is refused, the next call that relies on the count starts
with it. A CFL reduction that was not launched leaves nothing behind."""
import ctypes as C
import os
import shutil
import subprocess

import pytest

import paper_1602_09079_gb300 as dg
from paper_1602_09079_gb300 import _build

EMU = os.path.join(os.path.dirname(os.path.abspath(__file__)), "host_emulation")
N_FLAG = 3  # 32-bit word of the control block at the start of the scratch


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    dg.load()  # builds the objects
    objs = [os.path.join(_build.OUT_DIR, u.replace(".cu", ".o")) for u in _build.UNITS]
    so = str(tmp_path_factory.mktemp("fake") / "libdg_fake.so")
    r = subprocess.run(["g++", "-shared", "-fPIC", "-O1", "-Wl,-Bsymbolic", os.path.join(EMU, "fake_cudart.cpp"), *objs,
                        "-o", so], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-4000:]
    lib = C.CDLL(so)
    for name, (res, args) in dg._SIGS.items():
        getattr(lib, name).restype, getattr(lib, name).argtypes = res, args
    return lib


class Bound:
    """A context on host buffers."""

    def __init__(self, lib, order, mixed, n=(6, 5, 4)):
        m = dg.dg_mesh()
        for a in range(3):
            m.n[a], m.length[a] = n[a], 1.0
        self.lib, self.ctx = lib, C.c_void_p()
        lib.fake_fail(-1, 0)
        assert lib.dg_init(C.byref(m), order, 5.0 / 3.0, C.byref(self.ctx)) == 0
        length, scratch = C.c_size_t(), C.c_size_t()
        assert lib.dg_sizes(self.ctx, 0, C.byref(length), C.byref(scratch)) == 0
        self.y = (C.c_double * length.value)()
        self.buf = C.create_string_buffer(scratch.value + 256)
        self.scratch = -(-C.addressof(self.buf) // 256) * 256
        assert lib.dg_bind(self.ctx, C.addressof(self.y), self.scratch, scratch.value, None) == 0
        self.words = (C.c_uint32 * 8).from_address(self.scratch)
        if mixed:
            assert lib.dg_set_precision(self.ctx, dg.DG_PREC_MIXED) == 0

    def __del__(self):
        self.lib.dg_destroy(self.ctx)


def calls(b):
    dt = C.c_double()
    return {"step": lambda: b.lib.dg_step(b.ctx, 1e-3), "limit": lambda: b.lib.dg_limit(b.ctx, None, None),
            "reset": lambda: b.lib.dg_energy_reset(b.ctx, 1.0, 1.0, None),
            "rhs": lambda: b.lib.dg_rhs(b.ctx, None, b.y), "cfl": lambda: b.lib.dg_cfl_dt(b.ctx, 0.3, C.byref(dt))}


@pytest.mark.parametrize("order", [1, 2, 3, 4])
@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("call", ["step", "limit", "reset", "rhs", "cfl"])
def test_error_is_not_left_behind(lib, order, mixed, call):
    b = Bound(lib, order, mixed)
    C.c_double.from_address(b.scratch).value = 2.0  # what dg_cfl_dt reads
    run = calls(b)[call]
    lib.fake_fail(-1, 0)
    assert run() == 0
    for j in range(lib.fake_launches()):
        b = Bound(lib, order, mixed)
        C.c_double.from_address(b.scratch).value = 2.0
        run = calls(b)[call]
        lib.fake_fail(j, 0)
        assert run() == dg.DG_ERR_CUDA
        assert lib.fake_pending_error() == 0
        assert calls(b)["limit"]() == 0


@pytest.mark.parametrize("order", [1, 2, 3, 4])
@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("call", ["step", "reset"])
def test_queue_is_empty_after_a_failed_call(lib, order, mixed, call):
    b = Bound(lib, order, mixed)
    run = calls(b)[call]
    assert run() == 0  # the first step limits its input
    lib.fake_fail(-1, 0)
    assert run() == 0
    n = lib.fake_launches()
    assert n >= (6 if call == "step" else 3)
    for j in range(n):
        b.words[N_FLAG] = 7  # what that launch would have queued
        lib.fake_fail(j, 0)
        assert run() == dg.DG_ERR_CUDA
        assert b.words[N_FLAG] == 0, j
        # the same where the memset is refused too: the next call begins with it
        b.words[N_FLAG] = 7
        lib.fake_fail(j, 1)
        assert run() == dg.DG_ERR_CUDA
        lib.fake_fail(-1, 0)
        assert b.lib.dg_energy_reset(b.ctx, 1.0, 1.0, None) == 0
        assert b.words[N_FLAG] == 0 and lib.fake_memsets() == 1


@pytest.mark.parametrize("order", [1, 3])
def test_cfl_reduction_that_was_not_launched(lib, order):
    """With kernels that do not run, dg_cfl_dt reads the result that the control
    block holds: the same word whatever calls failed before."""
    b = Bound(lib, order, False)
    result = C.c_double.from_address(b.scratch)
    dt = C.c_double()
    for fail in (-1, 0, -1, 0, 0, -1):
        result.value = 2.0
        lib.fake_fail(fail, 0)
        st = b.lib.dg_cfl_dt(b.ctx, 0.3, C.byref(dt))
        assert st == (0 if fail < 0 else dg.DG_ERR_CUDA)
        assert result.value == 2.0
