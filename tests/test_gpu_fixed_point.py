"""The FP64 path's fixed-point contractions at the edges of their exponent
handling, through dg_rhs: unequal box lengths (a multiplier per direction),
states whose variables lie many binades from 1 or vanish, driving far weaker
and stronger than the fluxes, non-finite input.

Scaling by powers of two is exact in every operation of the method: with
rho' = a rho, m' = a b m, E' = a b^2 E (a an even power of two, b any) R' is
(a b, a b^2, a b^2, a b^2, a b^3) R bit for bit, whatever exponents the
contractions choose, as long as nothing leaves the exponent range. Against the
oracle: 1e-12 normwise, the FP64 path's bar."""
import numpy as np
import pytest

import oracle
import synthetic as syn

pytestmark = pytest.mark.gpu
G = syn.GAMMA
# standard deviation of the high modes, such that density and pressure stay
# positive at every quadrature point (the flux is undefined elsewhere)
HIGH = {1: 0.03, 2: 0.03, 3: 0.015, 4: 0.007}


@pytest.fixture(scope="module")
def dg():
    import torch
    assert torch.cuda.is_available()
    import paper_1602_09079_gb300 as m
    m.load()
    return m


def solver(dg, n, order, length, w, forcing=None):
    s = dg.Solver(n, order, G, length=length, forcing=forcing is not None)
    if forcing is not None:
        s.set_forcing(*forcing)
    s.set_state(w)
    return s


def normwise(a, b):
    return max(np.max(np.abs(a[..., i, :] - b[..., i, :])) / np.max(np.abs(b[..., i, :])) for i in range(5))


def scaled(w, a, b):
    f = np.array([a, a * b, a * b, a * b, a * b * b])
    return w * f[:, None]


@pytest.mark.parametrize("order", [1, 2, 3, 4])
@pytest.mark.parametrize("n,length", [((5, 4, 3), (1.0, 0.7, 1.3)), ((33, 1, 2), (2.0, 1.0, 3.0)), ((4, 4, 4), (1.0, 1.0, 1.0))])
def test_scaling_is_exact(dg, order, n, length):
    N = oracle.nmodes(order - 1)
    w = syn.random_state(n, N, G, seed=order, high=HIGH[order])
    R = solver(dg, n, order, length, w).rhs()
    assert np.all(np.isfinite(R))
    for a, b in ((2.0 ** -240, 2.0 ** 33), (2.0 ** 120, 2.0 ** -61), (1.0, 2.0 ** -100)):
        got = solver(dg, n, order, length, scaled(w, a, b)).rhs()
        np.testing.assert_array_equal(got, scaled(R, a, b) * b)


@pytest.mark.parametrize("order", [2, 3, 4])
@pytest.mark.parametrize("amp", [0.0, 1e-9, 1e4])
def test_boxes_and_driving_match_oracle(dg, order, amp):
    n, length = (6, 5, 7), (1.0, 0.3, 5.0)
    N = oracle.nmodes(order - 1)
    w = syn.random_state(n, N, G, seed=20 + order, high=HIGH[order])
    w[..., 2, :] = 0.0  # a variable that vanishes everywhere
    w[:3, ..., 3, 1:] *= 1e-14  # and modes far below their means
    nv = syn.driving_modes(1.0, 2.0)
    ah = np.random.default_rng(7).normal(size=(len(nv), 6)) * amp
    o = oracle.Oracle(n, order - 1, G, length)
    forcing = None
    if amp:
        forcing = (nv, ah)
        o.set_forcing(nv, ah)
    assert normwise(solver(dg, n, order, length, w, forcing).rhs(), o.rhs(w)) <= 1e-12


@pytest.mark.parametrize("order", [2, 3, 4])
@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
def test_non_finite_input_shows(dg, order, value):
    n = (6, 5, 4)
    N = oracle.nmodes(order - 1)
    w = syn.random_state(n, N, G, seed=3, high=HIGH[order])
    w[1, 2, 3, 4, N - 1] = value
    R = solver(dg, n, order, (1.0, 1.0, 1.0), w).rhs()
    assert not np.all(np.isfinite(R[1, 2, 3, 4]))  # the cell itself
    assert np.all(np.isfinite(R[3, 4, 0]))  # no neighbour of it
    s = solver(dg, n, order, (1.0, 1.0, 1.0), w)
    s.step(1e-4)
    with pytest.raises(dg.DGError):
        s.check()
