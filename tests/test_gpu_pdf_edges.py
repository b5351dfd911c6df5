"""Density histogram where its FP32 bin position does not decide: very many and
very narrow bins, samples exactly on bin edges, densities far from 1. Counts
equal the definition's, floor((ln rho - lo) / (hi - lo) n_bins) in FP64, on
uniform cells (one density per cell, so that the reference needs no
quadrature); every sub-division gives sub^3 samples per cell."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order,sub", [(1, 1), (2, 3), (3, 4), (4, 8)])
@pytest.mark.parametrize("lo,hi,nb", [(-0.5, 0.5, 100), (-0.5, 0.5, 4096), (-1e-6, 1e-6, 7), (-30.0, 30.0, 60),
                                      (3.0, 3.5, 1)])
def test_counts_of_uniform_cells(order, sub, lo, hi, nb):
    import torch
    assert torch.cuda.is_available()
    import paper_1602_09079_gb300 as dg
    n = 6
    s = dg.Solver((n, n, n), order, 5.0 / 3.0)
    rng = np.random.default_rng(order)
    rho = np.exp(rng.uniform(lo - 0.2 * (hi - lo), hi + 0.2 * (hi - lo), n ** 3))
    edge = lo + (hi - lo) * np.arange(nb + 1) / nb  # densities at bin edges, 1, and far outside
    rho[:50] = np.exp(rng.choice(edge, 50))
    rho[50:54] = [1.0, 1e-200, 1e200, np.nextafter(np.exp(lo), 2)]
    w = np.zeros(s.state_shape)
    w[..., 0, 0] = rho.reshape(n, n, n)
    w[..., 4, 0] = 1.0
    s.set_state(w)
    t = np.log(rho)
    b = 1 + np.minimum(np.floor((t - lo) / (hi - lo) * nb), nb - 1)
    b = np.where(t < lo, 0, np.where(t >= hi, nb + 1, b)).astype(int)
    np.testing.assert_array_equal(s.density_pdf(sub, lo, hi, nb), np.bincount(b, minlength=nb + 2) * sub ** 3)
