"""The FP64 contraction on the FP16 tensor cores (csrc/oz_gemm.cu) at the
edges of its tiles: bases around the 16-wide K step, the 32-column block, the
single K window (2 N <= 96) and partial row tiles, against the oracle; exact
scaling by powers of two; non-finite operands.

Tolerance: a stage's error is at most K 2^-53 of its largest products
(tests/oz_digits_check.cpp), four stages with K <= 2 N: 4 x 98 x 1.1e-16 =
4e-14 at N = 49, gated at 1e-13."""
import numpy as np
import pytest

import gkba_inputs as gi
import oracle as O
from _check import check

pytestmark = pytest.mark.gpu

TOL = 1e-13


@pytest.fixture(scope="module")
def P():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1905_01180_gb300 import build as b
    b.build()
    import paper_1905_01180_gb300 as p
    return p


def setup(P, N, U, seed=3):
    s = gi.system(N, 8, seed=seed)
    ctx = P.Context(s["h"], s["v"], s["d"], s["rho0"], 0.05)
    pairs = [gi.random_pair(N, seed=seed + u) for u in range(U)]
    return s, ctx, np.stack([p[0] for p in pairs]), np.stack([p[1] for p in pairs])


@pytest.mark.parametrize("N,U", [(1, 3), (2, 2), (4, 40), (5, 3), (6, 1), (6, 5), (8, 3), (9, 2), (16, 3), (17, 2), (24, 5), (32, 2),
                                 (33, 1), (40, 2), (48, 1), (49, 2), (64, 1)])
def test_sigma_edges(P, N, U):
    s, ctx, G, Gb = setup(P, N, U)
    S = ctx.sigma(G, Gb)
    ref = O.sigma_independent(s["v"], G, Gb)
    for u in range(U):
        e = check(S[u], ref[u], TOL, f"N={N} unit {u}")
    print(f"N={N} rel err {e:.2e}")
    ctx.close()


def test_powers_of_two_scale_exactly(P):
    s, ctx, G, Gb = setup(P, 13, 2)
    S = ctx.sigma(G, Gb)
    assert np.array_equal(ctx.sigma(G * 2.0 ** 120, Gb * 2.0 ** -300), S * 2.0 ** -60)
    ctx.close()


def test_non_finite_operands_reach_their_unit_only(P):
    s, ctx, G, Gb = setup(P, 16, 4)
    S = ctx.sigma(G, Gb)
    for bad in (np.nan, np.inf):
        G2, Gb2 = G.copy(), Gb.copy()
        G2[1, 3, 5] = bad
        Gb2[2, 0, 7] = bad
        S2 = ctx.sigma(G2, Gb2)
        assert not np.isfinite(S2[1]).any() and not np.isfinite(S2[2]).all()
        assert np.array_equal(S2[0], S[0]) and np.array_equal(S2[3], S[3])
    ctx.close()
