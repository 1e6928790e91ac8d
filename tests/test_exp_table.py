"""The FP64 kernels' e^-u (its table, constants and error), reciprocal and
polynomial tail."""
import os
import re
from fractions import Fraction

import mpmath
import numpy as np

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                   "paper_2102_01734_gb300", "csrc", "fs64_step.cuh")


def _constants():
    src = open(SRC).read()
    body = re.search(r"kPow2\[64\] = \{(.*?)\};", src, re.S).group(1)
    whole, frac = re.search(r"kLn2Int = (0x\w+)ULL;.*?kLn2Frac = (0x\w+)u;", src, re.S).groups()
    return [float(x) for x in body.split(",")], int(whole, 16), int(frac, 16)


def test_table_is_correctly_rounded():
    tab, whole, frac = _constants()
    assert len(tab) == 64
    with mpmath.workdps(50):
        assert tab == [float(mpmath.mpf(2) ** (-mpmath.mpf(j) / 64)) for j in range(64)]
        assert (whole << 32) + frac == int(mpmath.floor(mpmath.log(2) / 64 * mpmath.mpf(2) ** 96))


def test_error_of_one_minus_exp():
    """The fixed-point steps as integers, g exact to 2^-44 of itself: the table's
    rounding (2^-54) and the last one (2^-55 below 1/2) over 1 - e^-u >= 0.393."""
    tab, whole, frac = _constants()
    worst = 0.0
    with mpmath.workdps(40):
        for u in np.concatenate([[0.5, 37.4999], np.random.default_rng(1).uniform(0.5, 37.5, 1500),
                                 (np.arange(48, 200) + 0.5) * np.log(2) / 64]):
            u = float(u)
            n = int(np.rint(np.float32(np.float32(u) * np.float32(92.33248))))
            m, e = np.frexp(u)
            mant = int(m * 2 ** 53)
            r = ((mant << (int(e) + 11)) - n * whole - (n * frac >> 32)) % 2 ** 64
            r -= 2 ** 64 * (r >> 63)
            assert abs(r) <= np.log(2) / 128 * (1 + 2.0 ** -9) * 2 ** 64
            x = mpmath.mpf(r) / 2 ** 64
            rh, rl = r >> 34, (r >> 2) & 0xffffffff
            assert abs(rh) < 2 ** 23 and (rh << 34) + (rl << 2) + (r & 3) == r
            g = x * x * (0.5 + x * (mpmath.mpf(-1) / 6 + x * (mpmath.mpf(1) / 24 - x / 120)))
            g1 = int(mpmath.nint(g * 2 ** 40))
            assert 0 <= g1 <= 2 ** 24
            P = (g1 << 24) + int(mpmath.nint((g * (1 + mpmath.mpf(2) ** -44) - mpmath.mpf(g1) / 2 ** 40) * 2 ** 64)) - r
            T = int(tab[n & 63] * 2 ** 63)
            E = T * (2 ** 63 + (P >> 1)) >> 64
            e0 = 2 ** 62 - (E >> (n >> 6))
            d = (e0 + 256 >> 9) * 2.0 ** -53 if e0 >= 2 ** 61 else (e0 + 128 >> 8) * 2.0 ** -54
            worst = max(worst, float(abs(mpmath.mpf(d) / (1 - mpmath.exp(-mpmath.mpf(u))) - 1)))
    assert worst < (2.0 ** -54 + 2.0 ** -55) / 0.393 * 1.01


def _rd(x):
    """A fraction rounded to FP32."""
    return Fraction(float(np.float32(float(x))))


def test_reciprocal():
    """recip64 step by step, each FP32 operation rounded once, from a seed one
    FP32 unit off either way: at most 0.52 units in the last place."""
    rng = np.random.default_rng(2)
    x = np.concatenate([[1.0, np.nextafter(1.0, 2), np.nextafter(2.0, 1), 1.5, 1 + 2.0 ** -24, 2 - 2.0 ** -24],
                        1 + rng.uniform(0, 1, 2000)])
    worst = 0.0
    for i, v in enumerate(x):
        m = Fraction(float(v))
        k = int(m * 2 ** 52)
        xh, xl, xt = Fraction(k >> 29, 2 ** 23), Fraction(k & 0x1fffffe0, 2 ** 52), Fraction(k & 31, 2 ** 52)
        assert xh + xl + xt == m and _rd(xl) == xl
        r0 = np.float32(float(1 / xh))
        r0 = Fraction(float([r0, np.nextafter(r0, np.float32(0)), min(np.nextafter(r0, np.float32(2)), np.float32(1))][i % 3]))
        ph = _rd(xh * r0)
        pl = _rd(xh * r0 - ph)
        q = _rd(xl * r0)
        ql = _rd(xl * r0 - q)
        a = _rd(1 - ph)
        s1 = _rd(a - q)
        eh = _rd(s1 - pl)
        el = _rd(_rd(_rd((a - q - s1) + (s1 - pl - eh)) - ql) - xt * r0)
        f = _rd(eh * eh + el)
        ch = _rd(r0 * eh)
        cl = _rd(r0 * f + _rd(r0 * eh - ch))
        c1 = round(ch * 2 ** 44)
        c2 = round(_rd(_rd(ch - Fraction(c1, 2 ** 44)) + cl) * 2 ** 60)
        fix = (int(r0 * 2 ** 24) << 36) + (c1 << 16) + c2
        assert abs(c1) < 2 ** 23 and abs(c2) < 2 ** 24
        assert 2 ** 59 <= fix + 64 <= 2 ** 60 + 128
        worst = max(worst, abs(float(Fraction((fix + 64) >> 7, 2 ** 53) * m - 1)) * 2 ** 53 / float(m) * 1.0)
    assert worst < 0.52


def test_tail_weight():
    """What Horner64 evaluates in float-float (2^-45 of itself) is below 2^-9 of p(u) on
    [0, 1/2], and its terms of degree 8 and 9, in FP32, below 2^-29; p's high bit is
    that of 1/4 and the corrections' integers fit."""
    c = {m: 2.0 / float(mpmath.factorial(m + 3)) for m in range(10)}
    p = 1 / 3 - 0.5 / 12
    assert c[3] * 0.5 ** 3 < 2.0 ** -9 * p and c[8] * 0.5 ** 8 < 2.0 ** -29 * p
    assert p > 0.25 and c[3] * 2 ** 30 < 2 ** 22 and 2.0 ** -31 * 2 ** 56 <= 2 ** 25
