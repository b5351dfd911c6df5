"""The limiter's FP32 screens in other units: a step and a reset of a state in
other units are the step and the reset in other units, whatever the floors are
set to (dg_set_eps). With powers of two every operation of the FP64 path scales
exactly, so the results agree bit for bit: rho' = a rho, m' = a b m, E' = a b^2 E,
floors a eps_rho and a b^2 eps_p, dt' = dt / b, c_iso' = b c_iso, rho0' = a rho0.
2^-80 is about 1e-24 (a density in g / cm^3), 2^70 about 1e21; 2^-200 lies below
the range of binary32. The states need the limiter, or their mean pressure turns
negative in a stage, which has to be reported."""
import numpy as np
import pytest

import launch_emulation as le
import oracle
import synthetic as syn

N_MESH = (5, 4, 3)
G = syn.GAMMA
EPS = 2.0 ** -40
UNITS = [(2.0 ** -80, 1.0), (2.0 ** -80, 2.0 ** 10), (2.0 ** 70, 1.0), (2.0 ** -200, 2.0 ** -20)]


def scaled(w, a, b):
    return w * np.array([a, a * b, a * b, a * b, a * b * b])[:, None]


def state(k, seed, high=0.3):
    return syn.random_state(N_MESH, oracle.nmodes(k), G, seed=seed, high=high)


@pytest.mark.parametrize("a,b", UNITS)
@pytest.mark.parametrize("k", [1, 3])
@pytest.mark.parametrize("entry", ["queue", "limit"])
def test_limiter_in_other_units(k, a, b, entry):
    w = state(k, 30 + k)
    outs = ["out0", "out1"] if entry == "queue" else ["out0"]

    def run(a, b):
        args = [entry, *N_MESH, repr(G), repr(EPS * a), repr(EPS * a * b * b), 0, "in", *outs]
        return le.run(k, args, scaled(w, a, b), len(outs))

    info, ref = run(1.0, 1.0)
    assert np.any(ref[0] != w)  # cells were limited
    got_info, got = run(a, b)
    assert got_info["err"] == info["err"]
    for x, y in zip(got, ref):
        np.testing.assert_array_equal(x, scaled(y, a, b))


@pytest.mark.parametrize("a,b", [UNITS[0], UNITS[3]])
@pytest.mark.parametrize("k,dt", [(1, 0.01), (2, 0.01), (3, 0.005), (2, 0.4)])
def test_step_in_other_units(k, dt, a, b):
    """dt = 0.4 is some twenty times the CFL time step: mean pressures turn
    negative, which the error word has to say (the state is then void)."""
    w = state(k, 40 + k)

    def run(a, b):
        args = ["step", *N_MESH, 0, repr(G), repr(EPS * a), repr(EPS * a * b * b), 0, "in", "out0", repr(dt / b), 0,
                "none", repr(0.7 * b if dt < 0.1 else 0.0), repr(a), 4]
        return le.run(k, args, scaled(w, a, b), 1)

    info, (ref,) = run(1.0, 1.0)
    got_info, (got,) = run(a, b)
    assert got_info["err"] == info["err"] and got_info["n_flag"] == "0"
    assert (info["err"] == "0") == (dt < 0.1)
    if dt < 0.1:
        assert int(info["queued"]) > 0
        np.testing.assert_array_equal(got, scaled(ref, a, b))
