"""Contexts that use one scratch buffer in turn: the scratch holds no result of an
earlier call that a later one of the other context depends on. dg_cfl_dt of a slow
flow after that of a fast one (and back) gives what each gives on its own scratch,
and the limiter's queue (its count is the control block's fourth word) is empty
between the calls; the unfused stages empty it themselves."""
import numpy as np
import pytest

import oracle
import synthetic as syn

pytestmark = pytest.mark.gpu
N_MESH = (9, 8, 7)


@pytest.fixture(scope="module")
def dg():
    import torch
    assert torch.cuda.is_available()
    import paper_1602_09079_gb300 as m
    m.load()
    return m


def bind(dg, s, scratch):
    dg.dg_bind(s.ctx, s.y, scratch, scratch.numel(), s.stream.cuda_stream)


@pytest.mark.parametrize("order", [1, 3])
def test_cfl_in_turn(dg, order):
    solvers, own = [], []
    for j, v in enumerate((3.0, 0.1)):
        s = dg.Solver(N_MESH, order, syn.GAMMA)
        s.set_state(syn.random_state(N_MESH, oracle.nmodes(order - 1), syn.GAMMA, seed=j, high=0.01,
                                     v_mean=(-v, v)))
        own.append(s.cfl_dt(0.3))
        solvers.append(s)
    assert own[0] < 0.8 * own[1]
    for s in solvers:
        bind(dg, s, solvers[0].scratch)
    for j in (0, 1, 1, 0, 1, 0, 0, 1):
        assert solvers[j].cfl_dt(0.3) == own[j]


@pytest.mark.parametrize("order", [1, 2, 3, 4])
@pytest.mark.parametrize("mixed", [False, True])
def test_queue_between_calls(dg, order, mixed):
    import torch
    w = syn.random_state(N_MESH, oracle.nmodes(order - 1), syn.GAMMA, seed=9, high=0.2)

    def run(left):
        s = dg.Solver(N_MESH, order, syn.GAMMA)
        if mixed:
            s.set_precision(dg.DG_PREC_MIXED)
        s.set_state(w)
        word = s.scratch[:16].view(torch.int32)
        s.step(1e-3)  # the queue's list holds cells from here on
        assert int(word[3]) == 0
        s.energy_reset(0.7, 1.0)
        assert int(word[3]) == 0
        if not mixed:
            word[3] = left
        s.step(1e-3)
        assert int(word[3]) == 0
        s.check()
        return s.get_state(), dg.dg_limiter_counts(s.ctx)

    (a, na), (b, nb) = run(0), run(5)
    np.testing.assert_array_equal(a, b)
    assert na == nb
