"""The anchored arithmetic of the mixed-precision traversal (trace_mixed.cu, Sec. 6.2-6.3's per-cell decisions taken in
single precision around an anchor) against exact rationals: the exit-face screen, the double-float exit time, the
position bits of a descent, the opacity polynomial and the quotients of the pixel ray. CPU only; the FP32 and FP64
operations are rebuilt here, no code is shared with the kernels.

Tolerances are the bounds the kernel's comments derive: a screen that decides must be right for the exact values its
words represent; the exit time within 2^-44 |t| + 2^-24 ih; the opacity within 2.5 * 2^-24 relative."""
import math
import random
from fractions import Fraction as Q

import numpy as np
import pytest

from test_screens import add, fma, mul, r32, sub

EPS_F, EPS_X, EPS_U = Q(6, 2 ** 24), Q(12, 2 ** 24), Q(1, 2 ** 20)


def split_inv(d):
    """1 / d (FP64) in units of 2^-31 canvas sides as the leading 24 bits and the rest in binary32."""
    inv = Q(1.0 / d)
    e = math.frexp(float(inv))[1] - 1
    ulp = Q(2) ** (e - 23)
    hi = (inv // ulp) * ulp
    return hi / 2 ** 31, r32(inv - hi) / 2 ** 31


def rest_time(rest, ih, il):
    """The anchor's rest below a unit as a time, from both words of the reciprocal."""
    f = r32(rest)
    return -fma(f, ih, mul(f, il))


def floor_bits(q, e):
    lo, hi = sub(q, e), add(q, e)
    return lo.numerator // lo.denominator, hi.numerator // hi.denominator


def axis(rng, dist_bits):
    """(D, ih, il, rr, exact time of the plane): a plane D units from an anchor with a rest of up to half a unit."""
    d = math.exp(rng.uniform(math.log(1e-3), 0.0))
    ih, il = split_inv(d)
    rest = Q(rng.uniform(-0.5, 0.5))
    D = rng.randrange(1, 2 ** dist_bits)
    return D, ih, il, rest_time(rest, ih, il), (D - rest) * (ih + il)


@pytest.mark.parametrize("dist_bits", [3, 12, 24, 31])
def test_exit_screen_and_time(dist_bits):
    rng = random.Random(dist_bits)
    decided = 0
    for _ in range(3000):
        D, ih, il, rr, t = axis(rng, dist_bits)
        # a second axis whose plane is met within 2^-16 to 2^-26 of the same time
        d2 = math.exp(rng.uniform(math.log(1e-3), 0.0))
        ih2, il2 = split_inv(d2)
        x2 = t / (ih2 + il2) * (1 + Q(rng.choice((-1, 1))) * Q(2) ** -rng.randint(16, 26))
        D2 = int(x2) + rng.randint(0, 1)
        if not 1 <= D2 < 2 ** 31:
            continue
        rest2 = D2 - x2
        rr2 = rest_time(rest2, ih2, il2)
        t2 = (D2 - rest2) * (ih2 + il2)
        F, F2 = fma(r32(Q(D)), ih, rr), fma(r32(Q(D2)), ih2, rr2)
        gscr = Q(1, 2 ** 10) * max(ih, ih2)
        b, s = min(F, F2), max(F, F2)
        if sub(s, b) > fma(EPS_F, add(abs(s), abs(b)), gscr):
            decided += 1
            assert (t < t2) == (F < F2)
        # the double-float time
        dh = r32(Q(D))
        dl = r32(Q(D) - dh)
        p = mul(dh, ih)
        lo = add(fma(dh, il, fma(dl, ih, fma(dh, ih, -p))), rr)
        hi = add(p, lo)
        lo = sub(lo, sub(hi, p))
        assert abs(hi + lo - t) <= Q(1, 2 ** 44) * abs(t) + Q(1, 2 ** 24) * ih
    assert decided > 500 or dist_bits == 3


@pytest.mark.parametrize("way_bits,cell_bits", [(6, 4), (14, 10), (22, 12), (28, 20), (30, 7)])
def test_position_bits(way_bits, cell_bits):
    """Bits that the interval leaves closed are the bits of the exact position's floor."""
    rng = random.Random(way_bits * 100 + cell_bits)
    closed = 0
    for _ in range(4000):
        d = math.exp(rng.uniform(math.log(1e-3), 0.0))
        ih, il = split_inv(d)
        rest = Q(rng.uniform(-0.5, 0.5))
        rr = rest_time(rest, ih, il)
        A = rng.randrange(2 ** 30, 2 ** 30 + 2 ** 20)
        way = Q(rng.uniform(0, 2 ** way_bits))
        if rng.random() < 0.7:   # near a mid-plane of the cell, within the screen's reach
            pos = A + rest + way
            m = Q(2 ** (cell_bits - 1))
            pos = round(pos / m) * m + Q(rng.uniform(-1, 1)) * way * Q(1, 2 ** 21) + Q(rng.uniform(-1, 1)) / 2 ** 20
            way = pos - A - rest
            if way < 0:
                continue
        t = way * (ih + il)
        th = r32(t)
        rcp = (1 / ih) * (1 + Q(rng.uniform(-1, 1)) / 2 ** 23)
        x = mul(sub(th, rr), r32(rcp))
        e = fma(abs(x), EPS_X, EPS_U)
        l, h = floor_bits(x, e)
        exact = A + rest + way
        f = exact.numerator // exact.denominator
        for bit in range(cell_bits):
            if ((A + l) ^ (A + h)) >> bit == 0:
                closed += 1
                assert (A + l) >> bit == f >> bit
    assert closed > 0   # the sampling meets decided bits


def test_opacity_polynomial():
    rng = np.random.default_rng(3)
    x = np.concatenate([rng.random(20000), np.exp(rng.uniform(-30, 0, 20000))]).astype(np.float32)
    c = [np.float32(v) for v in (0.000129130945, -0.00130112655, 0.0082762083, -0.0416474678, 0.166663662, -0.499999851, 1.0)]
    p = np.full_like(x, c[0])
    for v in c[1:]:
        p = (p.astype(np.float64) * x.astype(np.float64) + np.float64(v)).astype(np.float32)
    got, want = (x * p).astype(np.float64), -np.expm1(-x.astype(np.float64))
    assert float(np.max(np.abs(got / want - 1.0))) <= 2.5 * 2.0 ** -24


def rd(x):
    """A Fraction rounded to binary64 (int / int division rounds to nearest)."""
    return Q(x.numerator / x.denominator)


def test_pixel_quotients():
    """(2 i + 1) / W by the rounded reciprocal and one exact-remainder correction is the rounded quotient."""
    rng = random.Random(9)
    for W in [1, 2, 3, 5, 7, 37, 255, 256, 719, 1080, 1512, 2160, 4095, 65537, 2 ** 31 - 1] + [rng.randrange(1, 2 ** 31) for _ in range(60)]:
        r = Q(1.0 / W)
        for i in [0, W - 1, W // 2] + [rng.randrange(W) for _ in range(40)]:
            a = Q(2 * i + 1)
            q = rd(a * r)
            q = rd(rd(a - W * q) * r + q)
            assert q == Q((2 * i + 1) / W)


def fma64(a, b, c):
    return rd(a * b + c)


def test_norm_square_root():
    """sqrt by two coupled Newton steps from an approximation of 20 bits and the exact-remainder correction is the
    rounded square root, and its reciprocal is within two ulps."""
    rng = random.Random(4)
    for k in range(1500):
        x = Q(rng.choice((1.0, 4.0, 2.25, 1.0 + 2.0 ** -52)) if k < 8 else math.exp(rng.uniform(0.0, 12.0)))
        y = Q(float(1.0 / math.sqrt(float(x))) * (1.0 + rng.uniform(-1, 1) * 2.0 ** -20))
        g, h = rd(x * y), rd(y / 2)
        for _ in range(2):
            r = fma64(-g, h, Q(1, 2))
            g, h = fma64(g, r, g), fma64(h, r, h)
        g = fma64(fma64(-g, g, x), h, g)
        assert float(g) == math.sqrt(float(x))
        h = 2 * h
        r = fma64(h, fma64(-g, h, Q(1)), h)
        assert abs(r * g - 1) <= Q(1, 2 ** 51)
