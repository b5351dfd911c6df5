"""The queued limiter (limit_list_kernel, point values in 64-bit fixed point)
against the FP64 limiter of one cell (limit_cell) on cells with one strong mode
that needs limiting and all others at noise level, as a grid-aligned shock
leaves them: every low limb of the coefficients is then arbitrary, and at the
face points where all basis functions are positive their products add up.

Bound: theta1 = (mean - eps) / (mean - rmin) and tau come from point values
with a few roundings each (2^-53 of the values), divided by differences that
are a tenth of them at least here: 1e-13 of a variable's largest coefficient
covers both sides (a wrapped sum is off by 3.8e-6)."""
import numpy as np
import pytest

import launch_emulation as le
import oracle
import synthetic as syn

N_MESH = (8, 5, 4)


def noisy_state(k, noise, seed, rho_dip):
    """Means near 1 with a strong gradient along a random axis (of the density,
    or of the energy) that needs limiting; the other modes N(0, noise), in one
    quarter of the cells all negative."""
    rng = np.random.default_rng(seed)
    N = oracle.nmodes(k)
    shp = N_MESH[::-1]
    w = rng.normal(size=shp + (5, N)) * noise
    w[:, :, ::4] = -np.abs(w[:, :, ::4])
    rho = rng.uniform(0.8, 1.2, shp)
    v = rng.uniform(-0.3, 0.3, shp + (3,))
    p = rng.uniform(0.5, 1.0, shp)
    w[..., 0, 0] = rho
    w[..., 1:4, 0] = rho[..., None] * v
    w[..., 4, 0] = p / (syn.GAMMA - 1) + 0.5 * rho * np.sum(v * v, axis=-1)
    axis = rng.integers(1, 4, shp)
    sign = rng.choice([-1.0, 1.0], shp)
    var = 0 if rho_dip else 4
    for a in (1, 2, 3):
        m = axis == a
        w[m, var, a] = (sign * w[..., var, 0] * rng.uniform(0.62, 0.9, shp))[m]
    return w


@pytest.mark.parametrize("k,noise,rho_dip,lim_vol", [(1, 1e-13, True, 0), (2, 1e-13, False, 1), (2, 1e-10, True, 0),
                                                     (3, 1e-13, True, 0), (3, 1e-13, False, 1), (3, 1e-12, False, 0),
                                                     (3, 1e-10, True, 1), (3, 1e-3, True, 0)])
def test_queued_limiter_equals_cell_limiter(k, noise, rho_dip, lim_vol):
    w = noisy_state(k, noise, 7 * k + int(-np.log10(noise)), rho_dip)
    info, (got, ref) = le.run(k, ["queue", *N_MESH, repr(syn.GAMMA), 1e-12, 1e-12, lim_vol, "in", "out0", "out1"], w, 2)
    assert info["err"] == info["plain_err"] == "0" and info["n_flag"] == "0"
    assert int(info["deep"]) > 0.9 * w[..., 0, 0].size  # nearly all of them need it
    scale = np.max(np.abs(ref), axis=-1, keepdims=True)
    assert np.max(np.abs(got - ref) / scale) <= 1e-13
