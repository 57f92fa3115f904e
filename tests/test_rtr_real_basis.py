"""The cosine / sine basis of the coupling kernel (csrc/rtr_tables.cuh), on the CPU against the oracle's dense blocks.

Per degree l and tau: c_0 = sqrt(2) x_0, c_M = x_M + x_-M, s_M = i (x_M - x_-M), tau = 2 times -i.  The rotation
R^l (Wigner small-d with the sign s_mu s_m) splits into a block C on the c and S on the s; with row mu times (-1)^mu
both are symmetric and orthogonal.  e^{i M phi} is a real rotation of (c_M, s_M), and the axial translation sees
c1 +- s2 and c2 +- s1 with A +- i B.
"""

from math import factorial

import numpy as np
import pytest

from oracle import svwf, translation

K = 2.0 * np.pi / 550.0


def small_d(l, mp, m, beta):
    s = 0.0
    for k in range(0, 2 * l + 1):
        a1, a2, a3 = l + m - k, l - k - mp, k - m + mp
        if min(a1, a2, a3) < 0:
            continue
        num = np.sqrt(factorial(l + mp) * factorial(l - mp) * factorial(l + m) * factorial(l - m))
        s += (-1) ** a3 * num / (factorial(a1) * factorial(k) * factorial(a2) * factorial(a3)) \
            * np.cos(beta / 2) ** (2 * l - 2 * k + m - mp) * np.sin(beta / 2) ** (2 * k - m + mp)
    return s


def rot(l, mu, m, theta):
    def sgn(q):
        return (-1) ** q if q >= 0 else 1
    return sgn(mu) * sgn(m) * small_d(l, m, mu, theta)


def block_c(l, theta):
    out = np.zeros((l + 1, l + 1))
    for mu in range(l + 1):
        for m in range(l + 1):
            r = rot(l, mu, m, theta)
            r = r + rot(l, mu, -m, theta) if mu and m else r * (np.sqrt(2.0) if mu != m else 1.0)
            out[mu, m] = (-1) ** mu * r
    return out


def block_s(l, theta):
    return np.array([[(-1) ** mu * (rot(l, mu, m, theta) - rot(l, mu, -m, theta)) for m in range(1, l + 1)]
                     for mu in range(1, l + 1)])


@pytest.mark.parametrize("l", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("theta", [0.0, 0.4, 1.7, np.pi])
def test_rotation_blocks_are_symmetric_and_their_own_inverses(l, theta):
    for b in (block_c(l, theta), block_s(l, theta)):
        assert np.abs(b - b.T).max() <= 1e-13
        assert np.abs(b @ b - np.eye(len(b))).max() <= 1e-13


def row(l, m):
    return l * (l + 1) - 1 + m


def apply_real_basis(L, d, x):
    nh = L * (L + 2)
    dist = np.linalg.norm(d)
    theta, phi = np.arctan2(np.hypot(d[0], d[1]), d[2]), np.arctan2(d[1], d[0])
    C = {(t, l): np.array([np.sqrt(2.0) * x[(t - 1) * nh + row(l, 0)]]
                          + [x[(t - 1) * nh + row(l, m)] + x[(t - 1) * nh + row(l, -m)] for m in range(1, l + 1)])
         * (1 if t == 1 else -1j) for t in (1, 2) for l in range(1, L + 1)}
    S = {(t, l): np.array([1j * (x[(t - 1) * nh + row(l, m)] - x[(t - 1) * nh + row(l, -m)])
                           for m in range(1, l + 1)]) * (1 if t == 1 else -1j)
         for t in (1, 2) for l in range(1, L + 1)}

    def turn(C, S, sign):
        for key in C:
            m = np.arange(1, key[1] + 1)
            c, s = C[key][1:].copy(), S[key].copy()
            C[key][1:] = np.cos(m * phi) * c + sign * np.sin(m * phi) * s
            S[key] = np.cos(m * phi) * s - sign * np.sin(m * phi) * c

    def rotate(C, S):
        for key in C:
            C[key], S[key] = block_c(key[1], theta) @ C[key], block_s(key[1], theta) @ S[key]

    turn(C, S, 1)
    rotate(C, S)
    W = translation.coupling_blocks(L, K, np.array([[0.0, 0.0, dist]]), np.zeros((1, 3)))[0]
    A, B = W[:nh, :nh], W[:nh, nh:]
    Co, So = {k: np.zeros_like(v) for k, v in C.items()}, {k: np.zeros_like(v) for k, v in S.items()}
    for mu in range(L + 1):
        for lo in range(max(1, mu), L + 1):
            for li in range(max(1, mu), L + 1):
                a, b = A[row(lo, mu), row(li, mu)], B[row(lo, mu), row(li, mu)]
                if mu == 0:
                    Co[1, lo][0] += a * C[1, li][0]
                    Co[2, lo][0] += a * C[2, li][0]
                    continue
                c1, c2, s1, s2 = C[1, li][mu], C[2, li][mu], S[1, li][mu - 1], S[2, li][mu - 1]
                u, p = (a + b) / 2 * (c1 + s2), (a + b) / 2 * (c2 - s1)
                v, q = (a - b) / 2 * (c1 - s2), (a - b) / 2 * (c2 + s1)
                Co[1, lo][mu] += u + v
                So[2, lo][mu - 1] += u - v
                Co[2, lo][mu] += p + q
                So[1, lo][mu - 1] += q - p
    rotate(Co, So)
    turn(Co, So, -1)
    y = np.zeros(2 * nh, dtype=complex)
    for t in (1, 2):
        f = 1 if t == 1 else 1j
        for l in range(1, L + 1):
            y[(t - 1) * nh + row(l, 0)] = f * Co[t, l][0] / np.sqrt(2.0)
            for m in range(1, l + 1):
                c, s = f * Co[t, l][m], -1j * f * So[t, l][m - 1]
                y[(t - 1) * nh + row(l, m)] = (c + s) / 2
                y[(t - 1) * nh + row(l, -m)] = (c - s) / 2
    return y


@pytest.mark.parametrize("L", [1, 3, 5])
@pytest.mark.parametrize("d", [(180.0, -240.0, 330.0), (0.0, 0.0, -400.0), (0.0, 500.0, 0.0)])
def test_real_basis_product_equals_the_dense_block(L, d):
    rng = np.random.default_rng(L)
    x = rng.normal(size=2 * L * (L + 2)) + 1j * rng.normal(size=2 * L * (L + 2))
    want = translation.coupling_blocks(L, K, np.array([d]), np.zeros((1, 3)))[0] @ x
    got = apply_real_basis(L, np.array(d), x)
    # rounding of about 1e3 operations in 64 bits, scaled by the largest block entries
    assert np.abs(got - want).max() <= 1e-12 * np.abs(want).max()
