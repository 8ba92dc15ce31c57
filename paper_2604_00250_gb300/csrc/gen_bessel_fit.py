"""Writes bessel_fit.h: float32 approximations of the modified Bessel functions
that the Rician NLL (Eq. 9) and its gradient need,
    Q(z) = 1 - I1(z) / I0(z),   L(z) = log(exp(-z) I0(z)),   z >= 0,
as one polynomial of degree DEG per segment of z, so that lanes of a warp with unlike z take
the same instructions. Segment s < 8 covers [s, s + 1] in w = z - s - 1/2; segment 8 covers
z >= 8 in w = 8 / z. With r = 1 / max(z, 8):
    Q = P(w) r            P fits 8 Q for s < 8, z Q for s = 8
    L = G(w) - log(max(z, 8)) / 2
                          G fits L + log(8) / 2, and log(sqrt(z) exp(-z) I0(z)) for s = 8
Q is obtained directly, never as 1 - I1/I0, so it keeps relative accuracy where I1/I0 -> 1.
The fits are weighted least squares in the Chebyshev basis (weights iterated towards the
minimax fit, Lawson 1961) against scipy.special.i0e / i1e (Cephes, float64). Below z = 8 the coefficients
are rounded to float32 one after the other and the rest fitted again (rounded()), so that the
errors of Q z and L, which an objective adds up over millions of measurements, average to zero over a segment: each
coefficient rounded by itself left an error common to a whole segment (up to 2e-8 in Q z, 3e-8 in L), which
moved dJ/dsigma of noisy volumes, where its terms nearly cancel.

Run: python gen_bessel_fit.py > bessel_fit.h
"""
import math

import numpy as np
import scipy.special as sp

NSEG = 9
ZS = 8.0
DEG = 7


def q_of(z):
    """1 - I1(z) / I0(z); above z = 50 by the asymptotic series of I0 and I1 (A&S 9.7.1)."""
    x = 1 / np.maximum(z, 50.0)
    far = x / 2 + x**2 / 8 + x**3 / 8 + 25 * x**4 / 128 + 13 * x**5 / 32 + 1073 * x**6 / 1024
    near = np.minimum(z, 50.0)
    return np.where(z < 50, 1 - sp.i1e(near) / sp.i0e(near), far)


def fit(f, lo, hi, relative, n=3000, iters=60):
    """Power-basis coefficients of the fit of f over w in [lo, hi]."""
    t = np.cos(np.pi * (np.arange(n) + 0.5) / n)
    y = f((t + 1) / 2 * (hi - lo) + lo)
    w0 = 1 / np.abs(y) if relative else np.ones(n)
    B = np.polynomial.chebyshev.chebvander(t, DEG)
    lw = np.ones(n)
    for _ in range(iters):
        c, *_ = np.linalg.lstsq(B * (w0 * np.sqrt(lw))[:, None], y * w0 * np.sqrt(lw), rcond=None)
        e = np.abs((B @ c - y) * w0)
        lw = lw * (e / e.max() + 1e-6)
        lw /= lw.sum() / n
    P = np.polynomial.Polynomial([0.0])
    arg = np.polynomial.Polynomial([-(hi + lo) / (hi - lo), 2 / (hi - lo)])
    for k in np.polynomial.chebyshev.cheb2poly(c)[::-1]:
        P = P * arg + k
    return P.coef


def rounded(f, c, lo, hi, relative, weight, n=3000):
    """float32 coefficients near the fit c: each in turn rounded and the later ones fitted again by least
    squares, with the mean of weight(w) times the error over [lo, hi] held at zero."""
    w = (np.cos(np.pi * (np.arange(n) + 0.5) / n) + 1) / 2 * (hi - lo) + lo
    u = np.linspace(lo, hi, 4001)
    c, y, yu = c.copy(), f(w), f(u)
    w0 = 1 / np.abs(y) if relative else np.ones(n)
    V, U = (x[:, None] ** np.arange(len(c)) for x in (w, u))
    for k in range(len(c)):
        c[k] = np.float32(c[k])
        if k + 1 < len(c):
            scale = 2.0 ** np.arange(k + 1, len(c))   # columns of like size on [-1/2, 1/2]
            A = np.vstack([V[:, k + 1:] * scale * w0[:, None], 1e6 * np.mean(U[:, k + 1:] * scale * weight(u)[:, None], 0)])
            b = np.append((y - V[:, :k + 1] @ c[:k + 1]) * w0, 1e6 * np.mean((yu - U[:, :k + 1] @ c[:k + 1]) * weight(u)))
            c[k + 1:] = np.linalg.lstsq(A, b, rcond=None)[0] * scale
    return c


def table():
    """[DEG + 1][NSEG][2]: the coefficients of P and G."""
    tab = np.zeros((DEG + 1, NSEG, 2))
    for s in range(NSEG - 1):
        def p(w):
            return 8 * q_of(w + s + 0.5)

        def g(w):
            return np.log(sp.i0e(w + s + 0.5)) + 1.5 * float(np.float32(math.log(2.0)))   # as the kernel subtracts it
        tab[:, s, 0] = rounded(p, fit(p, -0.5, 0.5, True), -0.5, 0.5, True, lambda w: w + s + 0.5)
        tab[:, s, 1] = rounded(g, fit(g, -0.5, 0.5, False), -0.5, 0.5, False, np.ones_like)

    def z_of(x):
        return ZS / np.maximum(x, 1e-7)
    tab[:, NSEG - 1, 0] = fit(lambda x: z_of(x) * q_of(z_of(x)), 0.0, 1.0, True)
    tab[:, NSEG - 1, 1] = fit(lambda x: np.log(sp.i0e(z_of(x)) * np.sqrt(z_of(x))), 0.0, 1.0, False)
    return tab


def main():
    tab = table()
    print("/* Generated by gen_bessel_fit.py -- do not edit. */")
    print("#pragma once")
    print(f"#define PRISM_BESSEL_NSEG {NSEG}")
    print(f"#define PRISM_BESSEL_DEG {DEG}")
    print("/* [j][segment]: {P, G coefficients of w^(2j), P, G coefficients of w^(2j+1)} */")
    print(f"__device__ const float4 k_bessel_tab[{(DEG + 1) // 2 * NSEG}] = {{")
    for j in range((DEG + 1) // 2):
        row = ["{%s}" % ", ".join(f"{float(v):.9e}f" for v in (*tab[2 * j, s], *tab[2 * j + 1, s])) for s in range(NSEG)]
        print("  " + ",\n  ".join(row) + ",")
    print("};")


if __name__ == "__main__":
    main()
