"""The tables and the epilogue of the tensor-core Brillouin sweep in numpy: real rows of
the stored (re, im) words times signed powers of two, the classes 1 and 3 kept times i, and the
real spin combinations of the epilogue give the defining sum over the 80 directions."""
import itertools

import numpy as np
import pytest

RHO = (0, 64 / 432, 16 / 432, 4 / 432, 1 / 432)
LAM = (0, 8 / 64, 4 / 64, 2 / 64, 1 / 64)
DIRS = [d for d in itertools.product((-1, 0, 1), repeat=4) if any(d)]


def _gammas():
    s = np.array([[[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]]])
    g = np.zeros((4, 4, 4), complex)
    for mu in range(4):
        B = np.eye(2) if mu == 3 else -1j * s[mu]
        g[mu, :2, 2:], g[mu, 2:, :2] = B, B.conj().T
    return g


def _pair(d, j, im):
    """Coefficients of the two words of an A row: class j, its real or imaginary part; whether the
    words (re, im) are swapped first."""
    k = sum(map(abs, d))
    c = 2.0 ** (1 - k) if j == 0 else 4.0 ** (1 - k) * d[j - 1]
    times_i = j in (1, 3)
    first = -c if times_i and not im else c
    second = -c if times_i or not im else c
    return (first, second), bool(im) != times_i


@pytest.mark.parametrize("dagger", [False, True])
def test_sweep_from_its_tables(dagger):
    rng = np.random.default_rng(7)
    W = {d: rng.standard_normal((3, 3)) + 1j * rng.standard_normal((3, 3)) for d in DIRS}
    psi = {d: rng.standard_normal((4, 3)) + 1j * rng.standard_normal((4, 3)) for d in DIRS}
    gam, sg = _gammas(), -1.0 if dagger else 1.0
    want = np.zeros((4, 3), complex)
    for d in DIRS:
        k = sum(map(abs, d))
        M = sg * RHO[k] * sum(d[m] * gam[m] for m in range(4)) - 0.5 * LAM[k] * np.eye(4)
        want += M @ psi[d] @ W[d].T
    X = np.zeros((5, 4, 3), complex)   # T_j, those of j = 1 and 3 times i
    for j, im in itertools.product(range(5), (0, 1)):
        acc = np.zeros((4, 3))
        for d in DIRS:
            co, swap = _pair(d, j, im)
            w = (W[d].imag, W[d].real) if swap else (W[d].real, W[d].imag)
            acc += psi[d].real @ (co[0] * w[0]).T + psi[d].imag @ (co[1] * w[1]).T
        X[j] += acc * (1j if im else 1)
    f = sg * 4 / 27
    s1, s2 = (-1, -1, 1, 1), (-1, 1, 1, -1)
    got = np.array([-X[0, s] / 16 + f * (s1[s] * X[1, 3 - s] + s2[s] * X[2, 3 - s] + s2[s] * X[3, s ^ 2] + X[4, s ^ 2])
                    for s in range(4)])
    np.testing.assert_allclose(got, want, rtol=0, atol=1e-12 * np.abs(want).max())
