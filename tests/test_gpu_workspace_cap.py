"""workspace_bytes caps what an FP64 context allocates for its contractions.  Two
units of the largest buffers (X1/X3 and X2, 2 x 16 N^4 bytes a unit), the forms
and the reduction scratch (384 N^2) fit a cap of their size; the digit images
and S4's partial sums share them."""
import math

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


def two_units(N):
    return 2 * (32 * N ** 4 + 368 * N * N + 16 * N * N * math.ceil(N ** 3 / 8192) + 8)


@pytest.mark.parametrize("history", ["sum", "time_linear"])
@pytest.mark.parametrize("N", [1, 2, 3, 4, 5, 13, 24])
def test_two_units_are_enough(P, N, history):
    s = gi.system(N, 8, seed=N)
    pairs = [gi.random_pair(N, seed=u) for u in range(5)]
    G, Gb = np.stack([p[0] for p in pairs]), np.stack([p[1] for p in pairs])
    rho, T = gi.history(N, 6, 0.02, seed=5)
    out = []
    for ws in (0, two_units(N)):
        with P.Context(s["h"], s["v"], s["d"], s["rho0"], 0.02, max_steps=7, workspace_bytes=ws, history=history) as c:
            c.set_history(5, rho, T)
            out.append((c.sigma(G, Gb), c.step(0.1, 0.2)[0]))
    assert np.array_equal(out[0][0], out[1][0])
    assert np.abs(out[0][1] - out[1][1]).max() < 1e-13  # the history is summed in other batches


def test_cap_holds(P):
    # N = 5: 59 kB and at most 4 KiB of alignment a context; device memory comes in 2 MiB steps
    import torch
    N, n = 5, 800
    s = gi.system(N, 8, seed=1)
    G, Gb = gi.random_pair(N, seed=1)
    ctxs = [P.Context(s["h"], s["v"], s["d"], s["rho0"], 0.02, workspace_bytes=two_units(N)) for _ in range(n)]
    for c in ctxs[:1]:
        c.sigma(G, Gb)
    free = torch.cuda.mem_get_info()[0]
    for c in ctxs[1:]:
        c.sigma(G, Gb)
    used = free - torch.cuda.mem_get_info()[0]
    for c in ctxs:
        c.close()
    assert used <= (n - 1) * (two_units(N) + 4096) + (4 << 20), used / (n - 1) / two_units(N)
