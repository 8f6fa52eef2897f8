"""The closed forms behind the point-value kernel's EG2 sums, against
quadrature on the CPU: the moments of the powers of the distance from a grid
line over the half circle beyond it, and of their products over the quarter
beyond both lines."""
import numpy as np
import pytest

_X, _W = np.polynomial.legendre.leggauss(40)


def _int(f, t0, t1):
    t = 0.5 * (t0 + t1) + 0.5 * (t1 - t0) * _X
    return 0.5 * (t1 - t0) * np.sum(_W * f(np.cos(t), np.sin(t)))


@pytest.mark.parametrize("a", [0.0, 0.3, 0.9, 0.9999, 1.0])
def test_half_circle_moments(a):
    al, s = np.arccos(a), np.sqrt(1 - a * a)
    q = s * s
    L = {0: 2 * al, 1: 2 * (s - a * al)}
    L[2] = 0.5 * (q * L[0] - 3 * a * L[1])
    N = {0: L[2] + a * L[1]}
    N[1] = 2 / 3 * s ** 3 - a * N[0]
    for m in (1, 2, 3):
        N[m + 1] = (m * q * N[m - 1] - (2 * m + 3) * a * N[m]) / (m + 3)
    C = {1: N[0], 2: 2 * N[1]}
    CN = {m: N[m + 1] + a * N[m] for m in (1, 2, 3)}
    W = {m: 3 * CN[m + 1] / (m + 1) for m in (1, 2)}
    for m in (1, 2):
        for got, w in ((L[m], lambda c, s: 1.0), (N[m], lambda c, s: s * s), (C[m], lambda c, s: c),
                       (CN[m], lambda c, s: c * s * s), (W[m], lambda c, s: s ** 4),
                       (1.5 * L[m] - 2 * N[m], lambda c, s: 2 * c * c - 0.5),
                       (1.5 * N[m] - 2 * W[m], lambda c, s: (2 * c * c - 0.5) * s * s)):
            assert got == pytest.approx(_int(lambda c, s: w(c, s) * (c - a) ** m, -al, al), abs=1e-13)


@pytest.mark.parametrize("a,b", [(0.0, 0.0), (0.4, 0.3), (0.0, 0.95), (0.7, 0.7), (0.8, 0.6)])
def test_quarter_moments(a, b):
    sa, sb = np.sqrt(1 - a * a), np.sqrt(1 - b * b)
    t0, t1 = np.arcsin(b), np.arccos(a)
    k = 1 - a * a - b * b
    q00, q10 = t1 - t0, sa - b - a * (t1 - t0)
    q01 = sb - a - b * q00
    q11 = 0.5 * k - b * (sa - b) - a * (sb - a) + a * b * q00
    h = 0.5 * (k * q00 - a * q10 - b * q01)
    q20, q02 = h - a * q10, h - b * q01
    q12, q21 = (k * q10 - 4 * b * q11 - a * q20) / 3, (k * q01 - 4 * a * q11 - b * q02) / 3
    t = 0.5 * (k * q11 - a * q21 - b * q12)
    q31, q13 = t - a * q21, t - b * q12
    q30 = 2 * (q12 + b * q11) - a * q20
    q22 = (k * q20 - 5 * b * q21 - a * q30) / 4
    D41, D14 = 0.6 * (k * q21 - a * q31 - b * q22), 0.6 * (k * q12 - b * q13 - a * q22)
    E23, E32 = 2 / 3 * D41, 2 / 3 * D14
    q41, q23, q32 = D41 - a * q31, E23 - b * q22, E32 - a * q22
    F, G = 0.5 * (k * q22 - a * q32 - b * q23), (k * q31 - a * q41 - b * q32) / 3
    c, s = (q21 + a * q11, t, q22 + a * q12, E32), (q12 + b * q11, q22 + b * q21, t, E23)
    cc = (t + a * c[0], D41 + a * t, E32 + a * c[2], F + a * E32)
    sc = (s[1] + a * s[0], q32 + b * q31 + a * s[1], E23 + a * t, G + a * E23)
    powers = ((1, 1), (2, 1), (1, 2), (2, 2))
    for got, w in (((q11, q21, q12, q22), lambda c, s: 1.0), (c, lambda c, s: c), (s, lambda c, s: s),
                   (cc, lambda c, s: c * c), (sc, lambda c, s: s * c)):
        for (m, n), x in zip(powers, got):
            want = _int(lambda c, s: w(c, s) * (c - a) ** m * (s - b) ** n, t0, t1)
            assert x == pytest.approx(want, abs=1e-13)
