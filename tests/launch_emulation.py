"""The emulated kernels of tests/host_emulation/launch_driver.cpp (library
kernels on the CPU, with the routes and sizes of the library's launchers):
build and run helpers of the tests that use it."""
import concurrent.futures as cf
import os
import shutil
import subprocess
import tempfile

import numpy as np
import pytest

import test_kernels_host_sanitized_cpu as emu

_dir = None


def _build(k):
    exe = os.path.join(_dir.name, f"launch_k{k}")
    return subprocess.run(["g++", *emu.FLAGS, "-I", emu.EMU, "-I", _dir.name, "-include",
                           os.path.join(emu.EMU, "emu.h"), f"-DDG_K={k}", os.path.join(emu.EMU, "launch_driver.cpp"),
                           "-o", exe], capture_output=True, text=True)


def driver(k):
    """The driver of degree k (all are compiled on the first call, once per
    test process)."""
    global _dir
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    if _dir is None:
        _dir = tempfile.TemporaryDirectory(prefix="dg_launch_emu_")
        emu._generate(_dir.name)
        # the own transform's kernels (dg_spectrum.cu's second anonymous namespace)
        sp = open(os.path.join(emu.CSRC, "dg_spectrum.cu")).read()
        a = sp.index("struct Cx {")
        body = sp[a:sp.index("}  // namespace\n", a)]
        assert "fft_packed_bins_kernel" in body and "cufft" not in body
        open(os.path.join(_dir.name, "fft_kernels.inc"), "w").write(emu._host_smem(body))
        with cf.ThreadPoolExecutor(4) as ex:
            for r in ex.map(_build, range(4)):
                assert r.returncode == 0, r.stderr[-4000:]
    return os.path.join(_dir.name, f"launch_k{k}")


def run(k, args, state, outputs, modes=None):
    """Run a command with the placeholders "in" (the state, canonical layout),
    "modes" and "out0", "out1", ... replaced by files; the printed values and the
    output states in canonical layout."""
    exe = driver(k)
    with tempfile.TemporaryDirectory() as d:
        path = {x: os.path.join(d, x) for x in ("in", "modes", *(f"out{j}" for j in range(outputs)))}
        emu._layout(state).tofile(path["in"])
        if modes is not None:
            np.ascontiguousarray(np.concatenate([np.asarray(m, np.float64) for m in modes], axis=1)).tofile(path["modes"])
        info = emu._run(exe, [path.get(a, a) if isinstance(a, str) else a for a in args], d)
        return info, [emu._canonical(np.fromfile(path[f"out{j}"]), state.shape) for j in range(outputs)]
