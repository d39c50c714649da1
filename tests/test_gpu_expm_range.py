"""Propagators of a one-body matrix with a large common shift: U = exp(-i dt h)
halves its argument at most 16 times and squares as often, in every form of the
exponential (up to 12 and 32 rows in one CTA or a cluster, larger ones as
products) and in its adjoint (2 N rows).

A shift h + lambda 1 multiplies T by a phase and cancels in I, so that rho and
the gradients do not depend on it.  dt lambda = 7e4 lies between 2^16 and 2^17.
Tolerance: 2^16 squarings' growth of 2^-53 is 7e-12, the rounding of the phase
itself 7e4 2^-53 = 8e-12; a few of each: 1e-9 for T, 1e-6 for gradients (steps
multiply both, and lambda rho is rounded at 2e-10)."""
import numpy as np
import pytest

import gkba_inputs as gi

pytestmark = pytest.mark.gpu
DT, LAM = 0.05, 1.4e6


@pytest.fixture(scope="module")
def P():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1905_01180_gb300 import build as b
    b.build()
    import paper_1905_01180_gb300 as p
    return p


@pytest.mark.parametrize("precision", ["fp64", "tf32"])
@pytest.mark.parametrize("N", [8, 12, 13, 32, 33])
def test_propagator(P, N, precision):
    s = gi.system(N, 8, seed=N)
    h = s["h"] + LAM * np.eye(N)
    with P.Context(h, np.zeros((N,) * 4), s["d"], s["rho0"], DT, max_steps=1, precision=precision) as c:
        c.step(0.0, 0.0)
        T = c.get_history()[2][0]
    e, q = np.linalg.eigh(s["h"])
    U = np.exp(-1j * DT * LAM) * (q * np.exp(-1j * DT * e)) @ q.conj().T
    assert np.abs(T - U).max() < 1e-9


@pytest.mark.parametrize("N", [4, 13, 17])
def test_gradients(P, N):
    s = gi.system(N, 8, seed=N)
    E = [0.1, -0.2, 0.3, 0.1]
    out = []
    for lam in (0.0, LAM):
        with P.Context(s["h"] + lam * np.eye(N), s["v"], s["d"], s["rho0"], DT, max_steps=3) as c:
            for k in range(3):
                rho, _, _ = c.step(E[k], E[k + 1])
            out.append((rho,) + tuple(c.adjoint(s["d"])))
    for a, b in zip(*out):
        assert np.abs(a - b).max() <= 1e-6 * np.abs(a).max()
