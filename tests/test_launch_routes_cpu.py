"""Memory safety of the kernels on the routes that the launchers take, under
AddressSanitizer and UndefinedBehaviorSanitizer in the host emulation, where
test_kernels_host_sanitized_cpu.py runs another one: FP64 at degree 1 on the
fixed-point kernels, the fused mixed kernel at degree 1 and with 1 and 2 planes per
segment, the limiter's second pass with its own shared memory, one face direction
per block, the spectrum's own transform. Results against the oracle or numpy, with
that file's bars for the same quantities (transform: 1e-14 of the total power, its
own error being some 1e-16)."""
import os
import tempfile

import numpy as np
import pytest

import launch_emulation as le
import oracle
import synthetic as syn
import test_kernels_host_sanitized_cpu as emu

N_MESH = (5, 3, 7)
G = syn.GAMMA
ROUTES = [(0, 0, 4), (1, 0, 4), (2, 0, 4), (1, 1, 1), (1, 1, 2), (1, 1, 4), (2, 1, 1), (2, 1, 2), (3, 1, 2)]


def driving(seed):
    nv = syn.driving_modes(1.0, 2.0)
    return nv, np.random.default_rng(seed).normal(size=(len(nv), 6)) * 0.5


@pytest.mark.parametrize("k,prec,seg", ROUTES)
def test_rhs(k, prec, seg):
    length = (1.0, 0.7, 1.3)
    w = syn.random_state(N_MESH, oracle.nmodes(k), G, seed=40 + k, high=0.01)
    o = oracle.Oracle(N_MESH, k, G, length)
    modes = driving(k)
    o.set_forcing(*modes)
    args = ["rhs", *N_MESH, prec, repr(G), *map(repr, length), "in", "out0", len(modes[0]), "modes", seg]
    info, (R,) = le.run(k, args, w, 1, modes)
    assert info["err"] == "0"
    assert emu.normwise(R, o.rhs(w)) <= (1e-12 if prec == 0 else 2e-5)


@pytest.mark.parametrize("k,prec,seg", ROUTES)
def test_step_and_reset(k, prec, seg):
    """FP64 with the limiter at work; mixed with smaller high modes, which leave it
    idle (the FP32 increments of a state at the floor are off by more than the bar)."""
    w = syn.random_state(N_MESH, oracle.nmodes(k), G, seed=50 + k, high=0.3 if prec == 0 else 0.03)
    o = oracle.Oracle(N_MESH, k, G)
    modes = driving(60 + k)
    o.set_forcing(*modes)
    st, dt = o.cfl_dt(w, 0.3)
    st, w1 = o.step(w, dt)
    assert st == 0
    st, w2, dref = o.energy_reset(w1, 0.7, 1.0)
    assert st == 0
    args = ["step", *N_MESH, prec, repr(G), 1e-12, 1e-12, 0, "in", "out0", repr(dt), len(modes[0]), "modes", 0.7, 1.0,
            seg]
    info, (y,) = le.run(k, args, w, 1, modes)
    assert info["err"] == "0" and info["n_flag"] == "0"
    bar = 1e-9 if prec == 0 else 1e-5
    assert emu.normwise(y, w2) <= bar
    assert abs(float(info["dissipated"]) - dref) <= bar * abs(dref)


@pytest.mark.parametrize("M", [32, 64])
def test_own_transform(M):
    rng = np.random.default_rng(M)
    v = rng.normal(size=(M, M, M))
    v[M // 2] *= 1e-9  # lines far apart in magnitude, and some that vanish
    v[M // 4, :M // 2] = 0.0
    with tempfile.TemporaryDirectory() as d:
        fin, fout = os.path.join(d, "in"), os.path.join(d, "out")
        v.tofile(fin)
        emu._run(le.driver(1), ["fft", M, fin, fout], d)
        bins = np.fromfile(fout)
    n = np.fft.fftfreq(M, 1.0 / M)
    shell = np.floor(np.sqrt(n[:, None, None] ** 2 + n[None, :, None] ** 2 + n[None, None, :] ** 2) + 0.5).astype(int)
    p = np.abs(np.fft.fftn(v)) ** 2 / float(M) ** 6
    ref = np.bincount(shell.ravel(), weights=p.ravel(), minlength=len(bins))
    assert len(bins) == len(ref)
    assert np.max(np.abs(bins - ref)) <= 1e-14 * ref.sum()
