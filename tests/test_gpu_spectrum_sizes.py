"""Velocity spectra where the transform's path changes: the smallest and larger
power-of-two grids (own fixed-point transform, odd and even number of radix-4
passes), their neighbours below 32 and between powers of two (cuFFT), against
numpy on the oracle's samples; a flow whose mean and smallest scales lie 10
binades apart keeps every shell."""
import numpy as np
import pytest

import oracle
import synthetic as syn

pytestmark = pytest.mark.gpu
G = syn.GAMMA


@pytest.mark.parametrize("n,sub,order", [(16, 1, 3), (4, 8, 2), (32, 1, 4), (8, 4, 1), (24, 2, 3), (16, 4, 3), (13, 5, 2),
                                         (32, 4, 2)])
@pytest.mark.parametrize("mean", [0.0, 300.0])
def test_shell_sums(n, sub, order, mean):
    import torch
    assert torch.cuda.is_available()
    import paper_1602_09079_gb300 as dg
    N = oracle.nmodes(order - 1)
    w = syn.random_state((n, n, n), N, G, seed=n + order, high=0.01)
    w[..., 1, 0] += mean * w[..., 0, 0]
    s = dg.Solver((n, n, n), order, G)
    s.set_state(w)
    got = s.velocity_spectrum(sub)
    ref = oracle.Oracle((n, n, n), order - 1, G).velocity_spectrum(w, sub)
    # 1e-12 of the total power, as for every size; a shell's own rounding noise
    # is below 1e-13 of the total amplitude
    assert len(got) == len(ref)
    assert np.max(np.abs(got - ref)) <= 1e-12 * np.sum(ref)
    keep = ref > 1e-8 * np.sum(ref)
    assert np.max(np.abs(got[keep] - ref[keep]) / ref[keep]) <= 1e-9
