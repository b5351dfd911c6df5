"""Which cells the stage and the reset queue for the limiter (dg_limiter_counts):
those that fail the FP64 bounds of the modal test, not those that only the FP32
screen in front of it cannot clear. Reset states of a uniform density and one
momentum mode m_x = a Pt_1(x) have e = a^2/2 + c2g as energy mean and a^2 as its
excursion bound, so the pressure bound is (gamma - 1) (c2g - 2 a^2): a puts cells on
both sides of it within 3e-5 of the terms, where the FP32 screen clears none
(margin 1e-5 of terms that add up to five times that), and none needs limiting.
The expected counts apply the FP64 test to the state left behind (which no limiter
has changed); a time step of 1e-14 leaves it as it is to 1e-12.

FP64: FP64 sums, borderline cells within 1e-9 excluded from the state. Mixed (reset
only): FP32 sums widened by 1e-5, whose rounding (at most 1e-6) brackets the count."""
import numpy as np
import pytest

import launch_emulation as le
import oracle
import synthetic as syn

N_MESH = (8, 5, 4)
G = syn.GAMMA
EPS = 1e-12


def state(k):
    rng = np.random.default_rng(k)
    shp = N_MESH[::-1]
    w = np.zeros(shp + (5, oracle.nmodes(k)))
    c2g = 0.7 ** 2 / (G - 1)
    d = rng.uniform(1e-9, 3e-5, shp) * rng.choice([-1.0, 1.0], shp)
    a = np.sqrt(0.5 * c2g) * (1 + d)
    w[..., 0, 0] = 1.0
    w[..., 1, 1] = a
    w[..., 4, 0] = 0.5 * a * a + c2g
    w[..., 4, 4] = a * a / np.sqrt(5.0)  # mode (2, 0, 0)
    return w


def failing(w, widen=0.0):
    lmax = np.array([np.sqrt((2 * u + 1) * (2 * v + 1) * (2 * q + 1)) for u, v, q in
                     [(u, v, D - u - v) for D in range(4) for u in range(D, -1, -1) for v in range(D - u, -1, -1)]])
    m = w[..., 0]
    s = (np.abs(w[..., 1:]) * lmax[1:w.shape[-1]]).sum(axis=-1) * (1 + widen)
    rlo = m[..., 0] - s[..., 0]
    kin = 0.5 * np.sum((np.abs(m[..., 1:4]) + s[..., 1:4]) ** 2, axis=-1) / rlo
    p = (G - 1) * (m[..., 4] - s[..., 4] - kin)
    return int(np.sum(~(p >= EPS + 1e-13 * (G - 1) * (np.abs(m[..., 4]) + s[..., 4] + kin))))


@pytest.mark.parametrize("k", [2, 3])
@pytest.mark.parametrize("prec", [0, 1])
def test_counts(k, prec):
    w = state(k)
    args = ["step", *N_MESH, prec, repr(G), EPS, EPS, 0, "in", "out0", 1e-14, 0, "none", 0.7, 1.0, 4]
    info, (got,) = le.run(k, args, w, 1)
    assert info["err"] == "0"
    assert np.max(np.abs(got - w)) <= (1e-11 if prec == 0 else 1e-6)  # nothing was limited
    queued, full = int(info["queued"]), int(info["full"])
    n = w[..., 0, 0].size
    if prec == 0:
        assert 0 < failing(got) < n
        assert queued == 3 * failing(w) and full - queued == failing(got)
    else:
        assert failing(got, 1e-5 - 1e-6) <= full - queued <= failing(got, 1e-5 + 1e-6) < n
