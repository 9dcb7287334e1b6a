"""The pairs of binary32 numbers behind the certified n = 2 pivots (k_lp_df in
csrc/vrm_lp.cu): the operations restated in numpy binary32 (a fused
multiply-add as an exact binary64 product and sum rounded to binary32), their
errors against exact rational arithmetic within the constants the kernel's
running bounds use, and those bounds along whole pivot sequences of the
nine-row tableau of Sec. 4.1 started from the FP64 Vandermonde matrix.

The tolerances are the kernel's own constants (u = 2^-24): 3 u^2 for an offset
split in two, 12 u^2 and 24 u^2 for its products and cubes, 24 u^2 (|t| + |a p|)
for t - a p, 24 u^2 for a quotient; 1.0001 covers the emulated fma's double
rounding."""
from fractions import Fraction

import numpy as np
import pytest

f32 = np.float32
U2 = Fraction(1, 2 ** 48)
SLACK = Fraction(10001, 10000)
M = 9
B = [0, 0, 2, 0, 2, 0, 0, 0, 0]


def fma(a, b, c):
    return f32(np.float64(a) * np.float64(b) + np.float64(c))


def fast_two_sum(a, b):
    s = f32(a + b)
    return s, f32(b - f32(s - a))


def two_sum(a, b):
    s = f32(a + b)
    bb = f32(s - a)
    return s, f32(f32(a - f32(s - bb)) + f32(b - bb))


def residue(a, b, p):
    e = fma(a[0], b[0], -p)
    e = fma(a[0], b[1], e)
    return fma(a[1], b[0], e)


def mul(a, b):
    p = f32(a[0] * b[0])
    return fast_two_sum(p, residue(a, b, p))


def fnma(a, p, t):
    q = f32(a[0] * p[0])
    e = residue(a, p, q)
    s, r = two_sum(t[0], -q)
    return fast_two_sum(s, f32(r + f32(t[1] - e)))


def add(a, b):
    s, r = two_sum(a[0], b[0])
    return fast_two_sum(s, f32(r + f32(a[1] + b[1])))


def rcp(a, ulps):
    r = f32(1.0) / a[0]
    for _ in range(abs(ulps)):  # the hardware estimate is within one ulp
        r = np.nextafter(r, f32(np.inf) if ulps > 0 else f32(0), dtype=f32)
    e = fma(-a[0], r, f32(1))
    e = fma(-a[1], r, e)
    return fast_two_sum(r, f32(r * fma(e, e, e)))


def split(a):
    b = int(np.float64(a).view(np.uint64))
    if b << 1 & (2 ** 64 - 1) == 0:
        return f32(0), f32(0)
    e = (b >> 52 & 0x7FF) - 1023
    sign = b >> 32 & 0x80000000
    h = np.uint32(sign | (e + 127) << 23 | (b >> 29 & 0x7FFFFF)).view(f32)
    scale = np.uint32(sign | (e - 52 + 127) << 23).view(f32)
    return fast_two_sum(h, f32(f32(b & 0x1FFFFFFF) * scale))


def val(a):
    return Fraction(float(a[0])) + Fraction(float(a[1]))


def test_operations_stay_within_their_constants():
    rng = np.random.default_rng(1)
    for k in range(3000):
        x, y, z = rng.uniform(-2.5, 2.5, 3) * 10.0 ** rng.integers(-6, 4, 3)
        if k % 3 == 0:
            z = x * y * (1 + rng.uniform(-1, 1) * 2.0 ** -rng.integers(0, 50))  # cancelling
        a, b, t = split(x), split(y), split(z)
        X, Y = Fraction(x), Fraction(y)
        assert abs(val(a) - X) <= 3 * U2 * abs(X)
        aa, aab = mul(a, b), mul(mul(a, b), b)
        assert abs(val(aa) - X * Y) <= 12 * U2 * abs(X * Y) * SLACK
        assert abs(val(aab) - X * Y * Y) <= 24 * U2 * abs(X * Y * Y) * SLACK
        A, P, T = val(a), val(b), val(t)
        assert abs(val(fnma(a, b, t)) - (T - A * P)) <= 24 * U2 * (abs(T) + abs(A * P)) * SLACK
        q = mul(t, rcp(a, int(rng.integers(-1, 2))))
        assert abs(val(q) - T / A) <= 24 * U2 * abs(T / A) * SLACK
        assert abs(val(add(a, t)) - (A + T)) <= 3 * U2 * (abs(A) + abs(T)) * SLACK


@pytest.mark.parametrize("seed", range(6))
def test_running_bounds_hold_along_the_pivots(seed):
    rng = np.random.default_rng(100 + seed)
    K = int(rng.integers(10, 15))
    ang, rad = rng.uniform(0, 2 * np.pi, K), rng.uniform(0.5, 2.5, K)
    o = np.argsort(rad)
    xi, eta = rad[o] * np.cos(ang[o]), rad[o] * np.sin(ang[o])
    u2 = f32(2.0 ** -48)
    kop = f32(24) * u2
    T, E = [[None] * K for _ in range(M)], [[None] * K for _ in range(M)]
    V, d, Ed = [], [], []
    for k in range(K):
        x, e = np.float64(xi[k]), np.float64(eta[k])
        v = [x, e, x * x, x * e, e * e]
        V.append([Fraction(t) for t in v + [v[2] * x, v[2] * e, x * v[4], v[4] * e]])
        x, e = split(x), split(e)
        w = [x, e, mul(x, x), mul(x, e), mul(e, e)]
        w += [mul(w[2], x), mul(w[2], e), mul(x, w[4]), mul(w[4], e)]
        s, sa, se = (f32(0), f32(0)), f32(0), f32(0)
        for r in range(M):
            T[r][k] = w[r]
            E[r][k] = f32((3 if r < 2 else 12 if r < 5 else 24)) * u2 * abs(w[r][0])
            s, sa, se = add(s, w[r]), f32(sa + abs(w[r][0])), f32(se + E[r][k])
        d.append((-s[0], -s[1]))
        Ed.append(fma(f32(32) * u2, sa, se))
    Tx = [[V[k][r] for k in range(K)] for r in range(M)]
    dx = [-sum(V[k]) for k in range(K)]
    rhs, Eb, rx = [(f32(b), f32(0)) for b in B], [f32(0)] * M, [Fraction(b) for b in B]
    basis, basic = list(range(M)), set()

    def bound(E_, t, a, ea, p, ep):
        aa, ap = abs(a[0]), abs(p[0])
        return fma(kop, fma(aa, ap, abs(t[0])), fma(f32(aa + ea), ep, fma(ea, ap, E_)))

    def check():
        for k in range(K):
            assert all(abs(val(T[r][k]) - Tx[r][k]) <= Fraction(float(E[r][k])) * SLACK for r in range(M))
            assert k in basic or abs(val(d[k]) - dx[k]) <= Fraction(float(Ed[k])) * SLACK
        assert all(abs(val(rhs[r]) - rx[r]) <= Fraction(float(Eb[r])) * SLACK for r in range(M))

    check()
    pivots = 0
    while pivots < 14 and min(basis) < M:
        q = next((k for k in range(K) if k not in basic and dx[k] < Fraction(-1, 10 ** 9)), None)
        rows = [r for r in range(M) if q is not None and Tx[r][q] > Fraction(1, 10 ** 9)]
        if not rows:
            break
        l = min(rows, key=lambda r: (max(rx[r], 0) / Tx[r][q], basis[r]))
        piv, pe = T[l][q], E[l][q]
        P = rcp(piv, 1)
        rho = f32(pe * P[0])
        if not rho <= f32(0.5):
            break  # the kernel hands such a pivot back
        rr = fma(f32(2) * rho, rho, rho)

        def quotient(t, e_):
            p, eP = mul(t, P), f32(e_ * P[0])
            ap = abs(p[0])
            return p, fma(kop, ap, fma(rr, f32(ap + eP), eP))

        prow = [quotient(T[l][k], E[l][k]) if k != q else ((f32(1), f32(0)), f32(0)) for k in range(K)]
        prhs, ebp = quotient(rhs[l], Eb[l])
        col, ecol = [T[r][q] for r in range(M)], [E[r][q] for r in range(M)]
        px = [Tx[l][k] / Tx[l][q] for k in range(K)]
        bx, cx, dq, edq, dqx = rx[l] / Tx[l][q], [Tx[r][q] for r in range(M)], d[q], Ed[q], dx[q]
        for r in range(M):
            if r == l:
                T[r], E[r], rhs[r], Eb[r], Tx[r], rx[r] = [p for p, _ in prow], [e for _, e in prow], prhs, ebp, px, bx
                continue
            for k in range(K):
                E[r][k] = bound(E[r][k], T[r][k], col[r], ecol[r], *prow[k])
                T[r][k] = fnma(col[r], prow[k][0], T[r][k])
            Eb[r] = bound(Eb[r], rhs[r], col[r], ecol[r], prhs, ebp)
            rhs[r] = fnma(col[r], prhs, rhs[r])
            Tx[r] = [Tx[r][k] - cx[r] * px[k] for k in range(K)]
            rx[r] -= cx[r] * bx
        for k in range(K):
            Ed[k] = bound(Ed[k], d[k], dq, edq, *prow[k])
            d[k] = fnma(dq, prow[k][0], d[k])
        dx = [dx[k] - dqx * px[k] for k in range(K)]
        basic.discard(basis[l] - M)
        basic.add(q)
        basis[l] = M + q
        pivots += 1
        check()
    assert pivots >= 3
