"""The fused FP32-mixed stage kernel at the edges of its tiles: meshes of one
cell, one row or one plane, tiles cut at both sides, segments of one and two
planes and a last segment that is shorter; orders 2 to 4, both fluxes, with
and without driving, the limiter at rest. Against the oracle with the FP32-mixed
path's bars: R 2e-5, a step's state 1e-6."""
import os
import subprocess
import sys

import numpy as np
import pytest

import oracle
import synthetic as syn

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
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


@pytest.mark.parametrize("order", [2, 3, 4])
def test_step_after_noalloc_call_came_first(order):
    """In a new process the first call of an order is dg_rhs_noalloc, which
    uploads the order's tables; the mixed step that follows finds the fused
    kernels' tables as well. Against the FP64 step, whose own bar is 1e-12."""
    code = f"""
import sys
sys.path[:0] = [{ROOT!r}, {ROOT!r} + "/tests"]
import numpy as np, torch, synthetic as syn, paper_1602_09079_gb300 as dg
n, order = (9, 7, 5), {order}
N = order * (order + 1) * (order + 2) // 6
y = torch.ones(5 * N * 315, dtype=torch.float64, device="cuda")
R = torch.empty_like(y)
dg.dg_rhs_noalloc(n, order, syn.GAMMA, dg.DG_PREC_MIXED, y, R, 0)
torch.cuda.synchronize()
w = syn.random_state(n, N, syn.GAMMA, seed=order, high={HIGH[order]})
out = []
for prec in (dg.DG_PREC_FP64, dg.DG_PREC_MIXED):
    s = dg.Solver(n, order, syn.GAMMA)
    s.set_precision(prec)
    s.set_state(w)
    s.step(1e-3)
    s.check()
    out.append(s.get_state())
for i in range(5):
    a, b = out[1][..., i, :], out[0][..., i, :]
    assert np.max(np.abs(a - b)) <= 1e-6 * np.max(np.abs(b)), i
"""
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
