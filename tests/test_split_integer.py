"""The split-integer reciprocal of the FP64 sum (fix_term in gpp_terms_fix.cuh), evaluated with
numpy's 32-bit integers and floats over its whole declared range, against the reciprocal in
extended precision: U + gamma within 2^-52 of the largest |1/A| of the pair's range (a few
2^-53, the FP64 form's own error), |U| below 2^31, and the residual inside its 32-bit window.
"""

import numpy as np
import pytest

F = np.float32
KAPPA = 1.0 - 2.0 ** -12


def fma(a, b, c):
    """FP32 fused multiply-add (product exact in FP64; one rounding there, one to FP32)."""
    return (a.astype(np.float64) * b.astype(np.float64) + np.asarray(c, np.float64)).astype(F)


def split(v, h):
    s = np.ldexp(v, h)
    r = np.rint(s)
    lo = np.rint((s - r) * 4294967296.0)
    over = lo >= 2147483648.0
    return (r + over).astype(np.int64), (lo - 4294967296.0 * over).astype(np.int64)


def fsplit(v, ge):
    r = np.rint(np.ldexp(v, -ge)) * 2.0 ** ge
    return r.astype(F), (v - r).astype(F)


def wrap(v):
    return ((v + 2 ** 31) % 2 ** 32) - 2 ** 31


def fix_term(x, wr, wi, E, ks, side_a, rng):
    h = 30 - E
    xh, xl = split(x, h)
    wh, wl = split(wr, h)
    ih, il = split(wi, h)
    xa, xb = fsplit(x, E - 23)
    w1, w2 = fsplit(wr, E - 23)
    i1 = wi.astype(F)
    i2 = (wi - i1).astype(F)
    n1, n2 = fsplit(wi * wi, 2 * E - 21)
    sgn = -1 if side_a else 1
    a64 = (xh * 2 ** 32 + xl) + sgn * (wh * 2 ** 32 + wl)
    Al = wrap(a64 % 2 ** 32)
    Ah = (a64 - Al) >> 32
    A1 = xa + F(sgn) * w1
    A2 = xb + F(sgn) * w2
    N1 = fma(A1, A1, n1)
    Nm = fma(A1, A1, n1 - N1) + n2
    Nm = fma(A1 + A1, A2, Nm)
    rho = F(1) / fma(N1, np.full_like(N1, 1 + 2.0 ** -12), Nm)
    rho = np.nextafter(rho, rho * F(1) + rng.choice([-1, 1], size=rho.shape).astype(F))  # 1 ulp off
    eps = fma(-rho, N1, np.full_like(N1, KAPPA))
    eps = fma(-rho, Nm, eps)
    s = np.ldexp(F(1), ks).astype(F)
    rs = rho * s
    re = rs * eps
    p = A1 * rs
    cr = fma(A2, rs, fma(A1, re, fma(A1, rs, -p)))
    q = i1 * rs
    ci = fma(i2, rs, fma(i1, re, fma(i1, rs, -q)))
    i64 = lambda f: np.rint(f.astype(np.float64)).astype(np.int64)  # noqa: E731
    Ur, Ui = i64(p) + i64(cr), i64(q) + i64(ci)
    ur, ui = p + cr, q + ci
    Er = 1 + ((Al * Ur) >> 32) + ((il * Ui) >> 32) + Ah * Ur + ih * Ui
    Ei = 1 + ((Al * Ui) >> 32) + ((-il * Ur) >> 32) + Ah * Ui - ih * Ur
    full = np.ldexp(KAPPA, ks + h)     # what A U is near: a multiple of 2^32
    room = np.maximum(np.abs(Er.astype(np.longdouble) - full), np.abs(Ei.astype(np.longdouble)))
    Er, Ei = wrap(Er), wrap(Ei)
    c = np.ldexp(F(-1.0 / F(KAPPA)), -(h + ks)).astype(F)
    fr, fi = Er.astype(F) * c, Ei.astype(F) * c
    gr = fma(ur, fr, -ui * fi)
    gi = fma(ur, fi, ui * fr)
    return Ur, Ui, gr, gi, room


@pytest.mark.parametrize("E", [2, 3, 4, 5, 6])
@pytest.mark.parametrize("side_a", [True, False])
def test_reciprocal_over_the_range(E, side_a):
    rng = np.random.Generator(np.random.PCG64(10 * E + side_a))
    n = 60000
    xmax = 0.75 * 2.0 ** E
    x = rng.uniform(0.0, xmax, n)
    lo, hi = 2.0 ** (E - 7), 1.375 * 2.0 ** E - xmax
    mod = np.exp(rng.uniform(np.log(lo), np.log(hi), n))
    mod[:50], mod[50:100] = lo * (1 + 1e-12), hi * (1 - 1e-12)
    ph = np.where(rng.random(n) < 0.5, rng.uniform(-0.1, 0.1, n), rng.uniform(-1.57, 1.57, n))
    wr, wi = mod * np.cos(ph), mod * np.sin(ph)
    near = rng.random(n) < 0.3         # next to |x - w| = 1/2, where |u| is largest
    xn = wr + np.sqrt(np.maximum(0.25 * (1 + np.exp(rng.uniform(-25, -2, n))) - wi * wi, 0))
    x = np.where(near & (xn <= xmax) & (np.abs(wi) < 0.5), xn, x)
    x[100:110] = xmax
    x[110:120] = 0.0
    A = (x - wr if side_a else x + wr).astype(np.longdouble)
    N = A * A + wi.astype(np.longdouble) ** 2
    keep = N > 0.25 if side_a else N > 0
    x, wr, wi, A, N = (v[keep] for v in (x, wr, wi, A, N))
    d = np.full(x.shape, 0.5) if side_a else np.sqrt(wr * wr + wi * wi)
    ks = 31 + np.floor(np.log2(d * (1 + 1e-15))).astype(np.int64)
    Ur, Ui, gr, gi, room = fix_term(x, wr, wi, E, ks, side_a, rng)
    assert np.abs(Ur).max() < 2 ** 31 and np.abs(Ui).max() < 2 ** 31
    assert room.max() < 2 ** 31 - 8, float(room.max())
    s = np.ldexp(np.longdouble(KAPPA), ks)
    err = np.hypot((Ur + gr.astype(np.longdouble)) / s - A / N,
                   (Ui + gi.astype(np.longdouble)) / s - wi / N)
    assert float((err * d).max()) <= 2.0 ** -52
