"""The NLL's Bessel tables (bessel_fit.h), evaluated in float32 as the kernels do, against scipy in
float64 over every segment and its edges, and against the error of the two-branch form they replaced."""
import os
import re

import numpy as np
import pytest

sp = pytest.importorskip("scipy.special")
f32 = np.float32
HDR = os.path.join(os.path.dirname(__file__), "..", "paper_2604_00250_gb300", "csrc", "bessel_fit.h")


def _table():
    src = open(HDR).read()
    nseg, deg = (int(re.search(rf"PRISM_BESSEL_{n} (\d+)", src).group(1)) for n in ("NSEG", "DEG"))
    rows = re.findall(r"\{(-?\d[^{}]*)\}", src)
    t = np.array([[float(x.strip(" f")) for x in r.split(",")] for r in rows], f32)
    assert t.shape == ((deg + 1) // 2 * nseg, 4)
    t = t.reshape((deg + 1) // 2, nseg, 2, 2)                      # [j][segment][parity][P or G]
    return t.transpose(0, 2, 1, 3).reshape(deg + 1, nseg, 2)


def _fma(a, b, c):
    return (a.astype(np.float64) * b.astype(np.float64) + c.astype(np.float64)).astype(f32)


def _evaluate(z):
    tab = _table()
    zm = np.maximum(z, f32(8))
    r = (1 / zm.astype(np.float64)).astype(f32)
    zh = np.minimum(z, f32(8)) - f32(0.5)
    seg = (zh + f32(12582912)) - f32(12582912)
    i = seg.astype(int)
    assert i.min() >= 0 and i.max() <= 8
    w = np.where(z < 8, zh - seg, f32(8) * r).astype(f32)
    out = []
    for c in (0, 1):
        p = tab[-1, i, c]
        for k in range(len(tab) - 2, -1, -1):
            p = _fma(p, w, tab[k, i, c])
        out.append(p)
    lg = np.log2(zm.astype(np.float64)).astype(f32)
    return out[0] * r, _fma(np.full_like(z, -0.5 * np.log(2.0)), lg, out[1])


def test_bessel_tables_cover_every_z():
    edges = np.concatenate([[0.0], np.nextafter(f32(np.arange(1, 10)), f32(0)), np.arange(1, 10),
                            np.nextafter(f32(np.arange(1, 10)), f32(99)), [1e-30, 1e-6, 1e6, 1e20]])
    z = np.concatenate([edges, np.linspace(1e-4, 16, 200001),
                        np.exp(np.random.default_rng(0).uniform(np.log(8), np.log(3e4), 50000))]).astype(f32)
    Q, L = _evaluate(z)
    zd = z.astype(np.float64)
    far = zd >= 50
    zf, zn = np.where(far, zd, 50.0), np.where(far, 1.0, zd)
    Qr = np.where(far, 1 / (2 * zf) + 1 / (8 * zf**2) + 1 / (8 * zf**3) + 25 / (128 * zf**4) + 13 / (32 * zf**5),
                  1 - sp.i1e(zn) / sp.i0e(zn))
    Lr = np.log(sp.i0e(zd))
    # fit error (5e-8, 1e-9) and float32 rounding of a degree-7 chain with |coefficients| that sum to
    # at most 2 |P|: 4 roundings of 6e-8; L's logarithm: 6e-8 of its value
    assert np.max(np.abs(Q - Qr) / Qr) <= 3e-7
    assert np.max(np.abs(L - Lr) / np.maximum(1.0, np.abs(Lr))) <= 3e-7


def test_errors_average_out_over_a_segment():
    """An objective adds the terms of millions of measurements, so an error common to a segment of z counts where
    rounding does not: the mean error of z Q and of L over each segment below z = 8. Bound: a coefficient rounded last
    leaves 1e-9 at most, 100,001 roundings of 1e-7 an average of 3e-10."""
    for s in range(8):
        z = np.linspace(s, s + 1, 100003)[1:-1].astype(f32)
        zd = z.astype(np.float64)
        Q, L = _evaluate(z)
        assert abs(np.mean((Q - (1 - sp.i1e(zd) / sp.i0e(zd))) * zd)) <= 1.3e-9, s
        assert abs(np.mean(L - np.log(sp.i0e(zd)))) <= 1.3e-9, s
