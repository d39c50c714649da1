"""A unit's FP64 self-energy depends on the unit alone: bit for bit the same among
other units, in a workspace that holds two units at a time, and with less free
device memory; likewise a collision integral whatever points of weight zero
come with it (the products P_k, the propagation of T)."""
import numpy as np
import pytest

import gkba_inputs as gi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1905_01180_gb300 import build as b
    b.build()
    import paper_1905_01180_gb300 as p
    return p


@pytest.mark.parametrize("N,U", [(4, 300), (10, 200), (13, 40), (24, 60), (33, 12), (48, 4)])
def test_sigma(P, N, U):
    s = gi.system(N, 8, seed=N)
    pairs = [gi.random_pair(N, seed=u) for u in range(3)]
    G = np.stack([pairs[u % 3][0] for u in range(U)])
    Gb = np.stack([pairs[u % 3][1] for u in range(U)])
    args = (s["h"], s["v"], s["d"], s["rho0"], 0.05)
    with P.Context(*args) as c:
        many = c.sigma(G, Gb)
        alone = [c.sigma(*pairs[u]) for u in range(3)]
    with P.Context(*args, workspace_bytes=int(2.5 * 8 * 10 * N ** 4) + 200_000) as c:
        few = c.sigma(G[:6], Gb[:6])
    for u in range(U):
        assert np.array_equal(many[u], alone[u % 3]), u
    assert np.array_equal(few, many[:6])


@pytest.mark.parametrize("precision", ["fp64", "tf32"])
@pytest.mark.parametrize("N", [10, 33])
def test_collision_points(P, N, precision):
    L = 40
    s = gi.system(N, 8, seed=N)
    rho, T = gi.history(N, L, 0.02, seed=5)
    w = np.zeros(L)
    w[L - 2:] = 0.02, 0.01
    with P.Context(s["h"], s["v"], s["d"], s["rho0"], 0.02, precision=precision) as c:
        assert np.array_equal(c.collision(rho, T, w), c.collision(rho[L - 2:], T[L - 2:], w[L - 2:]))
