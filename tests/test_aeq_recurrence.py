"""The coefficients a_{l,m} of f^eq as the stage kernels form them, restated step by
step in numpy in either precision: the downward recurrences over m from a starting
order that follows the flow speed, and the 32-node rule where that order passes
the table's end (rslb_device.cuh: AeqTab, aeq_start, aeq_chains, aeq_cell, aeq_far).
With p3_m = A3 S_m D_m, p4_m = A4 S_m E_m: a_{0,m} = p3_m beta^m / pi and a_{1,m} =
3 (p3_m - p4_m) beta^m / pi."""
import functools
import math

import numpy as np
import pytest
from numpy.polynomial.legendre import leggauss

STEPS, MAXM = 128, 13
N, THETA = 1.3, 0.8


def _mp():
    mpmath = pytest.importorskip("mpmath")
    ctx = mpmath.mp.clone()
    ctx.dps = 40
    return ctx


@functools.lru_cache(None)
def _mp_rule(n=96):
    """Gauss-Legendre nodes and weights to 40 digits (Newton from the FP64 nodes)."""
    mp = _mp()
    out = []
    for x in leggauss(n)[0]:
        x = mp.mpf(float(x))
        for _ in range(4):
            p0, p1 = mp.mpf(1), x
            for m in range(1, n):
                p0, p1 = p1, ((2 * m + 1) * x * p1 - m * p0) / (m + 1)
            d = n * (x * p1 - p0) / (x * x - 1)
            x -= p1 / d
        out.append((x, 2 / ((1 - x * x) * d * d)))
    return mp, out


@functools.lru_cache(None)
def _exact(u):
    """a_{l,m} for m < 13 by the defining integral (Eq. aeq_aux) in s = A t, u0 - u c =
    e^{-s}, to ~30 digits (the oracle's FP64 sums are good to ~1e-14 of a_{l,0} at
    m = 12 only)."""
    mp, rule = _mp_rule()
    u = mp.mpf(u)
    A, u0 = mp.asinh(u), mp.sqrt(1 + u * u)
    J = [[mp.mpf(0)] * MAXM for _ in range(2)]
    for t, w in rule:
        s = A * t
        c = (u0 - mp.exp(-s)) / u
        w3 = w * mp.exp(2 * s)
        w4 = w3 * mp.exp(s)
        p0, p1 = mp.mpf(1), c
        for m in range(MAXM):
            J[0][m] += w3 * p0
            J[1][m] += w4 * p0
            p0, p1 = p1, ((2 * m + 3) * c * p1 - (m + 1) * p0) / (m + 2)
    k = mp.mpf(N) * (A / u) / (4 * mp.pi)
    return np.array([[float(k * x) for x in J[0]],
                     [float(3 * k * (x - mp.mpf(THETA) * y)) for x, y in zip(*J)]])


def _table():
    SD, SE = np.ones(STEPS + 3), np.ones(STEPS + 3)
    for m in range(2, STEPS + 2):
        SD[m + 1] = SD[m - 1] * (m + 2) / (m - 1)
    for m in range(3, STEPS + 2):
        SE[m + 1] = SE[m - 1] * (m + 3) / (m - 2)
    aD, aE = np.zeros(STEPS + 2), np.zeros(STEPS + 2)
    for m in range(2, STEPS + 2):
        aD[m] = (2 * m + 1) / (m + 2) * (SD[m] / SD[m - 1])
    for m in range(3, STEPS + 2):
        aE[m] = (2 * m + 1) / (m + 3) * (SE[m] / SE[m - 1])
    return aD, aE, SD, SE


def _start(u, gamma, nm4, T):
    f = np.float32
    r = f(gamma) / (f(gamma) + f(1))
    l2 = max(-np.log2(max(f(u) / (f(gamma) + f(1)), f(1e-30))), f(1e-6))
    need = f(24.53 if T is np.float64 else 11.55) / l2
    return nm4 + int(min(need, f(4096))), r


def _fma(T, a, b, c):
    # FP32: the product is exact in FP64; FP64: two roundings instead of one
    return T(np.float64(a) * np.float64(b) + np.float64(c))


def coefficients(n, theta, u, nomega, T):
    """(a [2][nomega + 1] in FP64, whether the 32-node rule was taken)."""
    aD, aE, SD, SE = (x.astype(T) for x in _table())
    nm = nomega + 1
    nm4 = max(nm, 4)
    gamma = math.sqrt(1.0 + u * u)
    M, r = _start(u, gamma, nm4, T)
    n, theta, u, gamma = T(n), T(theta), T(u), T(gamma)
    if M > (STEPS if T is np.float64 else 96):
        A, J3, J4 = T(np.arcsinh(u)), np.zeros(nm, T), np.zeros(nm, T)
        sh2 = u * u / (gamma + T(1))
        for t, w in zip(*leggauss(32)):
            s = A * T(t)
            c = (sh2 - np.expm1(-s)) / u
            e1 = np.exp(s)
            w3 = T(w) * (e1 * e1)
            w4 = w3 * e1
            p0, p1 = T(1), c
            J3[0] += w3
            J4[0] += w4
            for m in range(1, nm):
                J3[m] += w3 * p1
                J4[m] += w4 * p1
                p0, p1 = p1, (T(2 * m + 1) * c * p1 - T(m) * p0) * T(1.0 / (m + 1))
        X3, X4 = J3 * (A / u), J4 * (A / u)
        p3 = T(0.25) * n * X3.astype(np.float64)
        p4 = T(0.25) * n * theta * X4.astype(np.float64)
        far = True
    else:
        q = u / gamma
        b2 = q * q
        D, E = np.zeros(MAXM, T), np.zeros(MAXM, T)
        for alpha, out in ((aD, D), (aE, E)):
            d1, d0 = T(r), T(1)
            for m in range(M, 2, -1):
                if m < nm4:
                    out[m] = d0
                d1, d0 = d0, _fma(T, -b2, d1, alpha[m] * d0)
            out[2] = d0
            if alpha is aD:
                out[1] = _fma(T, -b2, d1, alpha[2] * d0)
            assert np.isfinite(out).all()
        rD, rE = T(1) / D[1], T(1) / (_fma(T, T(0.25), b2, T(0.75)) * E[2])
        A3 = T(0.5) * n * gamma
        A4 = A3 * (theta * gamma) * _fma(T, T(1.0 / 3.0), b2, T(1))
        E[1] = E[2] * rE
        D[0] = D[1] = E[0] = T(1)
        D[2:] *= rD
        E[2:] *= rE
        qm = np.cumprod(np.concatenate(([T(1)], np.full(nm - 1, q)))).astype(T)
        p3 = (qm * (A3 * (SD[:nm] * D[:nm]))).astype(np.float64)
        p4 = (qm * (A4 * (SE[:nm] * E[:nm]))).astype(np.float64)
        far = False
    return np.vstack([p3, 3.0 * (p3 - p4)]) / math.pi, far


@pytest.mark.parametrize("T", [np.float32, np.float64])
@pytest.mark.parametrize("nomega", [0, 1, 2, 3, 5, 7, 12])
def test_recurrence_against_the_integrals(T, nomega):
    """Bound: a rounding for each of ~20 operations that a coefficient passes through
    (errors of the chains die out downwards), 64 for the 32-node sums of exponentials,
    relative to the isotropic terms."""
    n, theta = N, THETA
    eps = float(np.finfo(T).eps)
    taken = set()
    for u in np.concatenate([[1e-4, 1e-2, 0.3, 1.0, 2.0, 3.0], np.linspace(4.0, 14.0, 41),
                             [20.0, 50.0]]):
        u = float(T(u))
        got, far = coefficients(n, theta, u, nomega, T)
        taken.add(far)
        ref = _exact(u)[:, :nomega + 1]
        gamma = math.sqrt(1.0 + u * u)
        # n X3_0 / (4 pi), and with theta X4_0 for l = 1
        s0 = n * 2.0 * gamma / (4.0 * math.pi)
        s1 = 3.0 * (s0 + n * theta * (2.0 * gamma ** 2 + 2.0 * u ** 2 / 3.0) / (4.0 * math.pi))
        tol = (64 if far else 20) * eps
        assert np.abs(got[0] - ref[0]).max() <= tol * s0, (u, far)
        assert np.abs(got[1] - ref[1]).max() <= tol * s1, (u, far)
    assert taken == {False, True}


def test_chain_stays_in_range_at_the_table_end():
    """The unscaled chains grow at most by the products of their alphas: from order 96
    within FP32, from order 128 within FP64."""
    aD, aE, _, _ = _table()
    for alpha in (aD[2:], aE[3:]):
        assert np.prod(alpha[:96]) < 1e-3 * np.finfo(np.float32).max
        assert np.prod(alpha) < 1e-3 * np.finfo(np.float64).max
