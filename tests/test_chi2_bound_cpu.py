"""The FP32 bound of the chi-square pair tile against exact rationals.

The tile adds two terms with one reciprocal, fma(fma(t1 t1, u0, (t0 t0) u1), 1 / (u0 u1), acc), with
the denominators u clamped from below at 2^-50. Here each step runs in correctly rounded float32 (an
FMA rounds once: exact rationals, then one rounding) and the reciprocal, which the hardware gives to
2^-23, is pushed to either end of that. |D32 - D| <= (d + 16) 2^-23 D + d 2^-48 has to hold on
histograms, exact zero bins, wide ranges up to 2^40 and values around and below the clamp.
"""

from fractions import Fraction as F

import numpy as np
import pytest

FLOOR = np.float32(2.0 ** -50)


def rn(x):
    """Fraction -> float32, to nearest even, subnormals included."""
    if x == 0:
        return np.float32(0)
    s, x = (-1, -x) if x < 0 else (1, x)
    e = x.numerator.bit_length() - x.denominator.bit_length()
    if F(2) ** e > x:
        e -= 1
    q = F(2) ** max(e - 23, -149)
    n = x / q
    k = n.numerator // n.denominator
    r = n - k
    k += 1 if r > F(1, 2) or (r == F(1, 2) and k & 1) else 0
    return np.float32(s * float(k * q))


def fr(x):
    return F(float(x))


def tile_chi2(a, b, tilt, floor=FLOOR):
    acc = np.float32(0)
    pad = len(a) % 2
    a, b = np.append(a, np.zeros(pad, np.float32)), np.append(b, np.zeros(pad, np.float32))
    for k in range(0, len(a), 2):
        t = [rn(fr(a[k + i]) - fr(b[k + i])) for i in (0, 1)]
        u = [max(rn(fr(a[k + i]) + fr(b[k + i])), floor) for i in (0, 1)]
        m = [rn(fr(x) * fr(x)) for x in t]
        p = rn(fr(u[0]) * fr(u[1]))
        r = rn(1 / fr(p) * (1 + F(tilt) / 2 ** 24))   # with its own rounding: within 2^-23
        n = rn(fr(m[1]) * fr(u[0]) + fr(rn(fr(m[0]) * fr(u[1]))))
        acc = rn(fr(n) * fr(r) + fr(acc))
    return acc


def exact_chi2(a, b):
    return sum((fr(x) - fr(y)) ** 2 / (fr(x) + fr(y)) for x, y in zip(a, b) if fr(x) + fr(y) > 0)


def rows(kind, g, d):
    if kind == "hist":
        x = g.dirichlet(np.full(d, 0.5), 2)
    elif kind == "zeros":
        x = np.clip(g.normal(0.01, 0.02, (2, d)), 0, None)
    elif kind == "wide":
        x = np.exp2(g.uniform(-60, 40, (2, d)))
    elif kind == "near":
        x = g.random((1, d)).repeat(2, 0)
        x[1] *= 1 + 1e-6 * g.random(d)
    else:   # around and below the clamp
        x = np.exp2(g.uniform(-80, -40, (2, d))) * (g.random((2, d)) < 0.8)
    return x.astype(np.float32)


@pytest.mark.parametrize("kind", ["hist", "zeros", "wide", "near", "tiny"])
@pytest.mark.parametrize("d", [1, 2, 31, 128])
def test_bound_holds(kind, d):
    g = np.random.default_rng(77 + d)
    worst = 0.0
    for _ in range(12):
        a, b = rows(kind, g, d)
        want = exact_chi2(a, b)
        lim = (d + 16) * F(1, 2 ** 23) * want + d * F(1, 2 ** 48)
        for tilt in (-1, 0, 1):
            off = abs(fr(tile_chi2(a, b, tilt)) - want)
            assert off <= lim, (kind, d, float(off), float(lim))
            worst = max(worst, float(off / lim) if lim else 0.0)
    assert worst < 1.0
