"""The fused FP32-mixed stage kernel at the edges of its tiles: meshes of one
cell, one row or one plane, tiles cut at both sides, segments of one and two
planes and a last segment that is shorter; orders 2 to 4, both fluxes, with
and without driving, the limiter at rest. Against the oracle with the FP32-mixed
path's bars: R 2e-5, a step's state 1e-6."""
import numpy as np
import pytest

import oracle
import synthetic as syn

pytestmark = pytest.mark.gpu
G = syn.GAMMA
HIGH = {2: 0.02, 3: 0.012, 4: 0.006}  # density and pressure stay positive at every point


def normwise(a, b):
    return max(np.max(np.abs(a[..., i, :] - b[..., i, :])) / np.max(np.abs(b[..., i, :])) for i in range(5))


@pytest.mark.parametrize("order", [2, 3, 4])
@pytest.mark.parametrize("n", [(1, 1, 1), (17, 1, 2), (1, 9, 3), (8, 8, 1), (9, 7, 5), (24, 17, 37)])
@pytest.mark.parametrize("flux,force", [(0, False), (0, True), (1, True)])
def test_step_and_rhs(order, n, flux, force):
    import torch
    assert torch.cuda.is_available()
    import paper_1602_09079_gb300 as dg
    N = oracle.nmodes(order - 1)
    w = syn.random_state(n, N, G, seed=order, high=HIGH[order])
    s = dg.Solver(n, order, G, forcing=force)
    o = oracle.Oracle(n, order - 1, G, flux=flux)
    s.set_precision(dg.DG_PREC_MIXED)
    s.set_flux(flux)
    if force:
        nv = syn.driving_modes(1.0, 2.0)
        ah = np.random.default_rng(5).normal(size=(len(nv), 6)) * 0.2
        s.set_forcing(nv, ah)
        o.set_forcing(nv, ah)
    s.set_state(w)
    assert normwise(s.rhs(), o.rhs(w)) <= 2e-5
    st, dt = o.cfl_dt(w, 0.3)
    assert st == 0
    st, w1 = o.step(w, dt)
    assert st == 0
    s.step(dt)
    s.check()
    assert normwise(s.get_state(), w1) <= 1e-6
