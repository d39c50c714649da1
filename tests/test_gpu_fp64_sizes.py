"""Sizes and branches of the FP64 path that no other test reaches: up to eleven
column blocks and several K windows in every stage (N > 48, S1 from N = 97 on),
the gradient's three slot derivatives as one batch, one after the other and in a
workspace too small for one batch, and the units-a-block of the density-density
kernel at every N that it serves."""
import numpy as np
import pytest

import gkba_inputs as gi
import oracle as O
from _check import check

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


@pytest.mark.parametrize("N", [65, 97, 128])
def test_large_bases(P, N):
    # against the four contractions in complex FP64; a stage's error is at most 2 N 2^-53 of
    # its largest products on each side: 2 x 4 x 256 x 1.1e-16 = 2.3e-13
    import torch
    g = torch.Generator(device="cuda").manual_seed(N)
    B = torch.randn(4, N, N, generator=g, dtype=torch.float64, device="cuda")
    B = (B + B.transpose(1, 2)).reshape(4, N * N) / N
    v = (B.T @ B).reshape(N, N, N, N).permute(0, 2, 3, 1).contiguous()
    G, Gb = (torch.randn(N, N, generator=g, dtype=torch.complex128, device="cuda") for _ in range(2))
    one = torch.eye(N, dtype=torch.complex128, device="cuda")
    with P.Context(one, v, one, 0.5 * one, 0.05) as c:
        S = c.sigma(G, Gb)
    c16 = torch.complex128
    x = (2.0 * v - v.permute(1, 0, 2, 3)).permute(3, 0, 1, 2).reshape(N ** 3, N).to(c16) @ Gb  # [j m q][r]
    x = G @ x.reshape(N * N, N, N)                                                               # [j m][p][r]
    x = (G @ x.reshape(N, N, N * N)).reshape(N, N ** 3)                                          # [j][n p r]
    vi = v.permute(0, 3, 2, 1).reshape(N, N ** 3)                                                # [i][n p r]
    ref = torch.complex(vi @ x.real.T, vi @ x.imag.T)
    check(S.cpu().numpy(), ref.cpu().numpy(), 2.3e-13, f"N={N}")


def test_gradient_branches(P):
    # a point's part of the gradient does not depend on the points beside it: 14 points of N = 24
    # (above the limit of the one-batch form) against 7 and 7, and 7 in a workspace of 20 units
    N, L = 24, 14
    s = gi.system(N, 8, seed=1)
    rho, T = gi.history(N, L, 0.02, seed=2)
    w = np.linspace(0.01, 0.02, L)
    r = np.random.default_rng(3)
    Ib = r.normal(size=(N, N)) + 1j * r.normal(size=(N, N))
    args = (s["h"], s["v"], s["d"], s["rho0"], 0.02)
    with P.Context(*args) as c:
        whole = c.collision_vjp(rho, T, Ib, w)
        halves = [c.collision_vjp(rho[k:k + 7], T[k:k + 7], Ib, w[k:k + 7]) for k in (0, 7)]
    with P.Context(*args, workspace_bytes=20 * (32 * N ** 4 + 400 * N * N)) as c:
        small = c.collision_vjp(rho[:7], T[:7], Ib, w[:7])
    for i in range(2):
        assert np.array_equal(whole[i], np.concatenate([h[i] for h in halves]))
        assert np.array_equal(small[i], halves[0][i])


@pytest.mark.parametrize("N", range(1, 26))
def test_density_density_units(P, N):
    c = gi.chain(N, "symmetric", U=0.8)
    pairs = [gi.random_pair(N, seed=u) for u in range(17)]
    G, Gb = np.array([p[0] for p in pairs]), np.array([p[1] for p in pairs])
    with P.Context(c["h"], c["v"], c["d"], c["rho0"], 0.05, interaction="symmetric") as ctx:
        S = ctx.sigma(G, Gb)
    for u in range(17):
        check(S[u], O.sigma_symmetric(c["v"], G[u], Gb[u]), 1e-12)
