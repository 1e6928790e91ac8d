"""The FP64 kernels' e^-u (its table, constants and error), reciprocal and
polynomial tail, on the sources' own constants and functions."""
import os
import re

import mpmath
import numpy as np
import pytest

import kernel_text
from kernel_text import ptr

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                   "paper_2102_01734_gb300", "csrc", "fs64_step.cuh")


@pytest.fixture(scope="module")
def functions(tmp_path_factory):
    """recip, 1 - e^-u, e^-u and the interval functions e0, a, d of an array."""
    lib = kernel_text.build(tmp_path_factory.mktemp("arith"))

    def call(x, ulp=0):
        lib.mode(0, ulp)
        out = [np.empty_like(x) for _ in range(6)]
        lib.fs64(len(x), ptr(x), *[ptr(o) for o in out])
        return out

    return call


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


def test_error_of_one_minus_exp(functions):
    """The fixed-point steps as integers, g exact to 2^-44 of itself, and the function
    itself: the table's rounding (2^-54), the cut of the series (r^6/720 < 3.5e-17,
    times e^-u <= 0.607) and the last rounding (2^-55 below 1/2) over 1 - e^-u >=
    0.393."""
    tab, whole, frac = _constants()
    worst = 0.0
    us = np.concatenate([[0.5, 37.4999], np.random.default_rng(1).uniform(0.5, 37.5, 1500),
                         (np.arange(48, 200) + 0.5) * np.log(2) / 64])
    with mpmath.workdps(40):
        for u, e0_function in zip(us, functions(us)[1]):
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
            exact = 1 - mpmath.exp(-mpmath.mpf(u))
            worst = max(worst, *(float(abs(mpmath.mpf(float(v)) / exact - 1)) for v in (d, e0_function)))
    assert worst < (2.0 ** -54 + 2.0 ** -55 + 0.607 * 3.5e-17) / 0.393


def test_reciprocal(functions):
    """From a seed up to one FP32 unit off either way: at most 0.52 units in the last
    place, for every exponent that takes this way and IEEE division outside."""
    rng = np.random.default_rng(2)
    x = np.concatenate([[1.0, np.nextafter(1.0, 2), np.nextafter(2.0, 1), 1.5, 1 + 2.0 ** -24, 2 - 2.0 ** -24],
                        1 + rng.uniform(0, 1, 2000), 2.0 ** rng.uniform(-1021, 1020, 1000)])
    for ulp in (-1, 0, 1):
        got = functions(x, ulp)[0]
        with mpmath.workdps(40):
            err = [float(abs(mpmath.mpf(float(g)) - 1 / mpmath.mpf(float(v)))) for g, v in zip(got, x)]
        assert np.max(np.array(err) / np.spacing(1.0 / x)) < 0.52
    with np.errstate(all="ignore"):
        edge = np.array([0.0, -0.0, np.inf, np.nan, 5e-324, 1e-310, 2.0 ** 1021, 1.7e308])
        assert np.array_equal(functions(edge)[0], 1.0 / edge, equal_nan=True)


def test_tail_weight():
    """What Horner64 evaluates in float-float (2^-45 of itself) is below 2^-9 of p(u) on
    [0, 1/2], and its terms of degree 8 and 9, in FP32, below 2^-29; p's high bit is
    that of 1/4 and the corrections' integers fit."""
    body = open(SRC).read()
    body = body[body.index("IntervalDE interval64("):]
    c = [abs(float(x)) for x in re.findall(r"fma\(p, u, (-?[\d.e-]+)\)", body)[:10]][::-1]
    p = 1 / 3 - 0.5 / 12  # p(1/2) to 1 %
    assert len(c) == 10 and abs(c[0] - 1 / 3) < 1e-15
    assert c[3] * 0.5 ** 3 < 2.0 ** -9 * p and c[8] * 0.5 ** 8 < 2.0 ** -29 * p
    assert p > 0.25 and c[3] * 2 ** 30 < 2 ** 22 and 2.0 ** -31 * 2 ** 56 <= 2 ** 25
