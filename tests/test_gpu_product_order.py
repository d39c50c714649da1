"""Order of the FP64 sums that feed split-TF32 operands.  T(t, t_k), P_k and rho~
of a split-TF32 context are rounded to FP32 for the tensor cores, so their last
FP64 bit counts: an element that crosses an FP32 rounding boundary moves a
collision integral by up to 1e-8.  Every such sum has a fixed order and form,
whatever else the launch computes, which is restated here in exact arithmetic:

  product       acc_x += fma(a_x, b_x, -(a_y b_y)), acc_y += fma(a_y, b_x, a_x b_y), k in order
  exponential   X = -i dt h / 2^s, Y <- X Y / k + I for k = 18 .. 1, s squarings
  Heun stage    k = -i (h rho - rho h) - (I + I^+), y = rho + (a k)
  history sum   ranges of two units in order (257 .. 512 units)

With v = 0 and no field, h_HF = h and I = 0, so that the propagators of a run
follow from h alone.  All comparisons are bit for bit."""
import math
from fractions import Fraction as F

import numpy as np
import pytest

import gkba_inputs as gi

pytestmark = pytest.mark.gpu
DT = 0.02


@pytest.fixture(scope="module")
def P():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1905_01180_gb300 import build as b
    b.build()
    import paper_1905_01180_gb300 as p
    return p


def fma(a, b, c):
    return float(F(a) * F(b) + F(c))


def entry(A, B, i, j):
    x = y = 0.0
    for k in range(A.shape[1]):
        a, b = complex(A[i, k]), complex(B[k, j])
        x += fma(a.real, b.real, -(a.imag * b.imag))
        y += fma(a.imag, b.real, a.real * b.imag)
    return complex(x, y)


def product(A, B):
    n = len(A)
    return np.array([[entry(A, B, i, j) for j in range(n)] for i in range(n)])


def propagator(h):
    n = len(h)
    nrm = 0.0
    for j in range(n):
        s = 0.0
        for i in range(n):
            s += DT * abs(complex(h[i, j]))
        nrm = max(nrm, s)
    s = 0
    while math.ldexp(nrm, -s) > 0.5:
        s += 1
    X = np.array([[complex(DT * z.imag, -DT * z.real) * math.ldexp(1.0, -s) for z in row] for row in h])
    Y = np.eye(n, dtype=complex)
    for k in range(18, 0, -1):
        Z = product(X, Y)
        al = 1.0 / k
        Y = np.array([[complex(al * Z[i, j].real + (i == j), al * Z[i, j].imag) for j in range(n)] for i in range(n)])
    for _ in range(s):
        Y = product(Y, Y)
    return Y


def free_run(P, N, steps):
    """Two Heun steps of a random h with v = 0: h, rho_k and the rows T(t_n, .)."""
    g = np.random.default_rng(N)
    h = g.normal(size=(N, N)) + 1j * g.normal(size=(N, N))
    h = h + h.conj().T
    q = np.linalg.qr(g.normal(size=(N, N)) + 1j * g.normal(size=(N, N)))[0]
    rho = (q * g.random(N)) @ q.conj().T
    rho = 0.5 * (rho + rho.conj().T)
    T = []
    with P.Context(h, np.zeros((N,) * 4), np.zeros((N, N), complex), rho, DT, max_steps=steps, precision="tf32") as c:
        for _ in range(steps):
            c.step(0.0, 0.0)
            _, rhos, t = c.get_history()
            T.append(t)
    return h, rhos, T


@pytest.mark.parametrize("N", [5, 16, 26, 34])
def test_propagator_rows(P, N):
    _, _, T = free_run(P, N, 2)
    U0, U1 = T[0][0], T[1][1]  # T(t_1, t_0) and T(t_2, t_1)
    for i in (0, N // 2, N - 1):
        for j in range(0, N, 3):
            assert T[1][0][i, j] == entry(U1, U0, i, j), (i, j)


@pytest.mark.parametrize("N", [5, 13, 33])
def test_exponential(P, N):
    h, _, T = free_run(P, N, 1)
    assert np.array_equal(T[0][0], propagator(h))


@pytest.mark.parametrize("N", [5, 17])
def test_heun_stages(P, N):
    h, rhos, _ = free_run(P, N, 1)
    rho = rhos[0]

    def slope(r):
        a, b = product(h, r), product(r, h)
        return (a.imag - b.imag) + 1j * -(a.real - b.real)

    def update(k, a):
        return (rho.real + a * k.real) + 1j * (rho.imag + a * k.imag)

    k1 = slope(rho)
    k2 = slope(update(k1, DT))
    assert np.array_equal(rhos[1], update(k1 + k2, 0.5 * DT))


def test_history_sum(P):
    # one weight at a time gives a range's value exactly; L = 150 has ranges of one point
    N, L = 8, 150
    s = gi.system(N, 8, seed=2)
    rho, T = gi.history(N, L, 0.02, seed=5)
    w = np.full(L, 0.02)
    with P.Context(s["h"], s["v"], s["d"], s["rho0"], 0.02, precision="tf32") as c:
        whole = c.collision(rho, T, w)
        acc = np.zeros((N, N), complex)
        for k in range(L):
            acc = acc + c.collision(rho, T, np.where(np.arange(L) == k, w, 0.0))
    assert np.array_equal(whole, acc)
