"""R of the FP64 path where one direction's fluxes are far above another's and
cancel: what the weaker direction (or the driving) contributes has to keep its own
precision. The kernels run in the host emulation; degrees 1 to 3.

Each case compares R with itself on scaled input, where the method is exact or
nearly so:
- a flow constant along axis d with a momentum m_d = s f: a passively carried
  quantity, so R_{m_d} / s does not depend on s. Its modes constant along d get
  nothing from the pressure, which sits in the flux along d only and is the same on
  both faces. Between s = 2^-30 and 2^-20 the pressure itself changes by
  m_d^2 / (2 rho) < 2^-42 of E (E is kept), so the bar is 1e-11 of the largest value.
- a one-dimensional flow in a box 2^10 times as long: R falls by 2^10, bit for bit
  in the modes constant across it, whose cross-stream fluxes cancel exactly.
- uniform gas at rest under driving of 2^-40 the strength: the means of R follow
  bit for bit."""
import numpy as np
import pytest

import launch_emulation as le
import oracle
import synthetic as syn

N_MESH = (5, 4, 3)
G = syn.GAMMA
HIGH = {1: 0.03, 2: 0.03, 3: 0.01}
EXPS = [(u, v, D - u - v) for D in range(4) for u in range(D, -1, -1) for v in range(D - u, -1, -1)]


def rhs(k, w, length=(1.0, 1.0, 1.0), modes=None):
    args = ["rhs", *N_MESH, 0, repr(G), *map(repr, length), "in", "out0", 0 if modes is None else len(modes[0]),
            "modes", 4]
    info, (R,) = le.run(k, args, w, 1, modes)
    assert info["err"] == "0"
    return R


def constant_along(w, axes):
    """The state made constant along the axes (0 = x)."""
    w = w.copy()
    for a in axes:
        ax = 2 - a  # arrays are [z][y][x]
        w[:] = np.take(w, [0], axis=ax)
        for l, e in enumerate(EXPS[:w.shape[-1]]):
            if e[a]:
                w[..., l] = 0.0
    return w


def plane_modes(N, axes):
    return [l for l, e in enumerate(EXPS[:N]) if not any(e[a] for a in axes)]


@pytest.mark.parametrize("d", [0, 1, 2])
@pytest.mark.parametrize("k", [1, 2, 3])
def test_weak_momentum(k, d):
    N = oracle.nmodes(k)
    w = constant_along(syn.random_state(N_MESH, N, G, seed=60 + k, high=HIGH[k]), [d])
    R = []
    for s in (2.0 ** -30, 2.0 ** -20):
        ws = w.copy()
        ws[..., 1 + d, :] *= s
        R.append(rhs(k, ws)[..., 1 + d, plane_modes(N, [d])] / s)
    assert np.max(np.abs(R[0] - R[1])) <= 1e-11 * np.max(np.abs(R[1]))


@pytest.mark.parametrize("d", [0, 1, 2])
@pytest.mark.parametrize("k", [1, 2, 3])
def test_long_box(k, d):
    N = oracle.nmodes(k)
    across = [a for a in range(3) if a != d]
    w = constant_along(syn.random_state(N_MESH, N, G, seed=70 + k, high=HIGH[k]), across)
    l0, l1 = [1.0, 0.7, 1.3], [1.0, 0.7, 1.3]
    l1[d] *= 1024.0
    m = plane_modes(N, across)
    np.testing.assert_array_equal(rhs(k, w, l1)[..., m] * 1024.0, rhs(k, w, l0)[..., m])


@pytest.mark.parametrize("k", [1, 2, 3])
def test_weak_driving(k):
    N = oracle.nmodes(k)
    w = np.zeros(N_MESH[::-1] + (5, N))
    w[..., 0, 0], w[..., 4, 0] = 1.0, 3.7
    nv = syn.driving_modes(1.0, 2.0)
    ah = np.random.default_rng(5).normal(size=(len(nv), 6))
    R = [rhs(k, w, modes=(nv, ah * s)) / s for s in (1.0, 2.0 ** -40)]
    assert np.max(np.abs(R[0][..., 1:4, 0])) > 0.1
    np.testing.assert_array_equal(R[1][..., 1:4, 0], R[0][..., 1:4, 0])
