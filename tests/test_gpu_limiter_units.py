"""dg_step and dg_energy_reset of the FP64 path in other units, the floors
(dg_set_eps) with them: powers of two scale every operation exactly, so the
results agree bit for bit with those in units of 1 (rho' = a rho, m' = a b m, E' =
a b^2 E, dt' = dt / b), with the limiter at work; and a mean pressure that turns
negative is reported whatever the units."""
import numpy as np
import pytest

import oracle
import synthetic as syn

pytestmark = pytest.mark.gpu
G = syn.GAMMA
EPS = 2.0 ** -40
N_MESH = (20, 9, 7)


@pytest.fixture(scope="module")
def dg():
    import torch
    assert torch.cuda.is_available()
    import paper_1602_09079_gb300 as m
    m.load()
    return m


def scaled(w, a, b):
    return w * np.array([a, a * b, a * b, a * b, a * b * b])[:, None]


def solver(dg, order, w, a, b):
    s = dg.Solver(N_MESH, order, G)
    dg.dg_set_eps(s.ctx, EPS * a, EPS * a * b * b)
    s.set_state(scaled(w, a, b))
    return s


@pytest.mark.parametrize("a,b", [(2.0 ** -80, 1.0), (2.0 ** 70, 1.0), (2.0 ** -200, 2.0 ** -20)])
@pytest.mark.parametrize("order", [2, 3, 4])
def test_units(dg, order, a, b):
    w = syn.random_state(N_MESH, oracle.nmodes(order - 1), G, seed=50 + order, high=0.3)

    def run(a, b):
        s = solver(dg, order, w, a, b)
        s.step(2e-3 / b)
        s.energy_reset(0.7 * b, a)
        s.check()
        return s.get_state(), dg.dg_limiter_counts(s.ctx)[0]

    ref, queued = run(1.0, 1.0)
    assert queued > 0
    np.testing.assert_array_equal(run(a, b)[0], scaled(ref, a, b))
    s = solver(dg, order, w, a, b)
    s.step(0.4 / b)
    with pytest.raises(dg.DGError):
        s.check()
