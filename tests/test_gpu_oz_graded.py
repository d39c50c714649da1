"""FP64 self-energies of graded operands (csrc/oz_gemm.cu): elements of very
different size in one row, imaginary parts far below the real ones, blocks that
hardly couple, results below the normal range.  The FP64 path is as accurate as
FMA chains there, componentwise.

Tolerance: the four contractions are restated on the real and imaginary planes
with absolute values, which gives sum |terms| of each component of S.  A stage's
error is at most 50 2^-53 of that where the digits are taken (K <= 96), K 2^-53 in
an FMA chain, on either side of the comparison: 2 x 4 x 96 x 1.1e-16 = 8.5e-14,
and N^3 terms in windows of 96 add 2^-53 sqrt(N^3 / 96): gated at 1e-13."""
import numpy as np
import pytest

import gkba_inputs as gi

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


def chain(v, G, Gb, absolute=False):
    """Planes (Re, Im) of S, or of the sum of the absolute values of their terms."""
    w = 2.0 * v - v.transpose(1, 0, 2, 3)  # w_mqsj
    if absolute:
        v, w = np.abs(v), np.abs(v) * 2.0 + np.abs(v).transpose(1, 0, 2, 3)
        G, Gb = (np.abs(G.real), np.abs(G.imag)), (np.abs(Gb.real), np.abs(Gb.imag))
    else:
        G, Gb = (G.real, G.imag), (Gb.real, Gb.imag)
    sg = 1.0 if absolute else -1.0

    def mul(spec, x):
        e = lambda a, b: np.einsum(spec, a, b, optimize=True)
        return e(G[0], x[0]) + sg * e(G[1], x[1]), e(G[0], x[1]) + e(G[1], x[0])

    x = tuple(np.einsum("mqsj,sr->jrmq", w, g, optimize=True) for g in Gb)
    x = mul("pq,jrmq->jrpm", x)
    x = mul("nm,jrpm->jnrp", x)
    return tuple(np.einsum("irpn,jnrp->ij", v, p, optimize=True) for p in x)


def case(kind, N, seed):
    r = np.random.default_rng(seed)
    v = gi.system(N, 8, seed=seed)["v"]
    G, Gb = gi.random_pair(N, seed=seed)
    if kind == "graded":            # G -> D G D, v -> the same in every index
        d = 10.0 ** r.permutation(np.linspace(-6.0, 6.0, N))
        G, Gb = G * np.outer(d, d), Gb * np.outer(d, d)
    elif kind == "graded_v":
        d = 10.0 ** r.permutation(np.linspace(-4.0, 4.0, N))
        v = v * np.einsum("i,j,k,l->ijkl", d, d, d, d)
    elif kind == "nearly_real":
        G, Gb = G.real + 1e-8j * G.imag, Gb.real + 1e-13j * Gb.imag
    elif kind == "blocks":          # two halves that couple by 1e-17
        b = np.arange(N) < N // 2
        m = np.where(np.equal.outer(b, b), 1.0, 1e-17)
        G, Gb = G * m, Gb * m
    elif kind == "real":
        G, Gb = G.real + 0j, Gb.real + 0j
    return v, G, Gb


@pytest.mark.parametrize("kind", ["graded", "graded_v", "nearly_real", "blocks", "real", "plain"])
@pytest.mark.parametrize("N", [3, 4, 10, 13, 24, 33, 50])
def test_components(P, kind, N):
    v, G, Gb = case(kind, N, 11 + N)
    s = gi.system(N, 8, seed=1)
    with P.Context(s["h"], v, s["d"], s["rho0"], 0.05) as ctx:
        S = ctx.sigma(G, Gb)
    ref, mag = chain(v, G, Gb), chain(v, G, Gb, absolute=True)
    for plane, r, m in ((S.real, ref[0], mag[0]), (S.imag, ref[1], mag[1])):
        assert np.all(np.abs(plane - r) <= TOL * m), (np.abs(plane - r) / np.where(m > 0, m, 1.0)).max()


def test_results_below_the_normal_range(P):
    # S of order 2^-1050: kept, in units of 2^-1074 (X3 has them as well: N^3 terms v X3)
    N = 10
    v, G, Gb = case("plain", N, 3)
    s = gi.system(N, 8, seed=1)
    with P.Context(s["h"], v, s["d"], s["rho0"], 0.05) as ctx:
        S = ctx.sigma(G, Gb)
        t = ctx.sigma(G * 2.0 ** -350, Gb * 2.0 ** -350)
    unit = 2.0 ** -1074
    assert np.abs(t.real - S.real * 2.0 ** -1050).max() <= unit * (1 + 0.5 * np.abs(v).sum((1, 2, 3)).max())
    assert np.abs(t.real).max() > 1e3 * unit
