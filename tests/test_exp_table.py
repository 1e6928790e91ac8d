"""The table and constants of the FP64 kernels' e^-u, and its error."""
import os
import re

import mpmath
import numpy as np

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                   "paper_2102_01734_gb300", "csrc", "fs64_step.cuh")


def _constants():
    src = open(SRC).read()
    body = re.search(r"kPow2\[64\] = \{(.*?)\};", src, re.S).group(1)
    hi, lo = re.search(r"kLn2Hi = (\S+), kLn2Lo = (\S+);", src).groups()
    return [float(x) for x in body.split(",")], float(hi), float(lo)


def test_table_is_correctly_rounded():
    tab, hi, lo = _constants()
    assert len(tab) == 64
    with mpmath.workdps(50):
        assert tab == [float(mpmath.mpf(2) ** (-mpmath.mpf(j) / 64)) for j in range(64)]
        ln2 = mpmath.log(2) / 64
        assert hi == float(ln2) and lo == float(ln2 - mpmath.mpf(hi))


def test_error_of_exp_neg():
    """Every operation in exact arithmetic rounded once (as the fused ones
    are): the table's rounding, e^-r's and the last product's, each 2^-53."""
    tab, hi, lo = _constants()
    m = mpmath.mpf
    rd = lambda x: float(x)
    worst = 0.0
    with mpmath.workdps(40):
        for u in np.concatenate([[0.5, 37.4999], np.random.default_rng(1).uniform(0.5, 37.5, 1500),
                                 (np.arange(48, 200) + 0.5) * np.log(2) / 64]):
            u = float(u)
            n = int(np.rint(np.float32(np.float32(u) * np.float32(92.33248))))
            r = rd(m(u) - n * m(hi))
            r = rd(m(r) - n * m(lo))
            assert abs(r) <= np.log(2) / 128 * (1 + 2.0 ** -9)
            q = rd(m(r) * m(-1.0 / 120) + m(1.0 / 24))
            q = rd(m(r) * m(q) + m(-1.0 / 6))
            q = rd(m(r) * m(q) + m(0.5))
            P = rd(m(rd(m(r) * m(r))) * m(q) - m(r))
            T = tab[n & 63]
            E = rd(m(T) * m(P) + m(T)) * 2.0 ** -(n >> 6)
            worst = max(worst, float(abs(m(E) * mpmath.exp(m(u)) - 1)))
    assert worst < 2.5 * 2.0 ** -53


def test_short_polynomials():
    """What the branches below 2^-6 and 2^-10 leave out of p(u) (leading term
    1/3) stays below a fiftieth of its last bit."""
    c = {m: 2.0 / float(mpmath.factorial(m + 3)) for m in range(5, 10)}
    assert 3 * c[7] * 2.0 ** (-6 * 7) < 2.0 ** -53 / 50
    assert 3 * c[5] * 2.0 ** (-10 * 5) < 2.0 ** -53 / 50
