"""Split-TF32 stages of small bases (padded N <= 48): two MMA issuers and two
epilogue groups over rings of accumulation windows.  Every window length, with
an even and an odd number of windows per tile, one and several tiles per CTA
pair, and unit changes inside a pair's range; against the FP64 path, repeated
bit for bit; non-finite operands.

Tolerance: that of the split-TF32 self-energy (tests/test_gpu_parity.py), 2e-5;
a window of 16 instead of 8 adds two truncated additions of 2^-24 to a sum."""
import numpy as np
import pytest

import gkba_inputs as gi
from _check import check

pytestmark = pytest.mark.gpu

TOL_TC = 2e-5


@pytest.fixture(scope="module")
def P():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1905_01180_gb300 import build as b
    b.build()
    import paper_1905_01180_gb300 as p
    return p


def inputs(N, U):
    s = gi.system(N, 8, seed=N)
    pairs = [gi.random_pair(N, seed=11 * N + u) for u in range(U)]
    return s, np.stack([p[0] for p in pairs]), np.stack([p[1] for p in pairs])


@pytest.mark.parametrize("window", [8, 16, 32])
@pytest.mark.parametrize("N,U", [(1, 1), (3, 150), (16, 1), (16, 40), (17, 9), (32, 3), (33, 1), (48, 3)])
def test_windows(P, N, U, window):
    s, G, Gb = inputs(N, U)
    ref = P.Context(s["h"], s["v"], s["d"], s["rho0"], 0.05)
    R = ref.sigma(G, Gb)
    ref.close()
    ctx = P.Context(s["h"], s["v"], s["d"], s["rho0"], 0.05, precision="tf32", acc_window=window)
    S = ctx.sigma(G, Gb)
    for u in range(U):
        check(S[u], R[u], TOL_TC, f"N={N} window={window} unit {u}")
    for _ in range(3):
        assert np.array_equal(ctx.sigma(G, Gb), S)
    ctx.close()


@pytest.mark.parametrize("N", [16, 33, 64])
def test_non_finite_operands_reach_their_unit_only(P, N):
    s, G, Gb = inputs(N, 4)
    ctx = P.Context(s["h"], s["v"], s["d"], s["rho0"], 0.05, precision="tf32")
    S = ctx.sigma(G, Gb)
    for bad in (np.nan, np.inf):
        G2, Gb2 = G.copy(), Gb.copy()
        G2[1, 3, 5] = bad
        Gb2[2, 0, 7] = bad
        S2 = ctx.sigma(G2, Gb2)
        assert not np.isfinite(S2[1]).all() and not np.isfinite(S2[2]).all()
        assert np.array_equal(S2[0], S[0]) and np.array_equal(S2[3], S[3])
    ctx.close()
