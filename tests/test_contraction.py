"""The float-float and FP64 arithmetic of the kernels, their own source text run on
the CPU with FP32 operations that are contracted as a compiler may: a product that
is added or subtracted anywhere later is either rounded first or fused into the
sum. The stated error bounds hold whatever is fused, since what must be rounded is
written with __fmul_rn, __fadd_rn and __fsub_rn."""
import mpmath
import numpy as np
import pytest

import kernel_text
from kernel_text import ptr as _ptr


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return kernel_text.build(tmp_path_factory.mktemp("arith"))


FUSE = [0, 1, 2, 3]


@pytest.mark.parametrize("fuse", FUSE)
@pytest.mark.parametrize("ulp", [-1, 0, 1])
def test_fp64(lib, fuse, ulp):
    lib.mode(fuse, ulp)
    rng = np.random.default_rng(3)
    x = np.concatenate([[1.0, np.nextafter(1.0, 2), np.nextafter(2.0, 1), 1.5, 1 + 2.0 ** -24, 0.5, 37.4999],
                        rng.uniform(1, 2, 400), 10.0 ** rng.uniform(-12, 2, 400), rng.uniform(0.4, 38, 400)])
    out = [np.empty_like(x) for _ in range(6)]
    lib.fs64(len(x), _ptr(x), *[_ptr(o) for o in out])
    worst = np.zeros(6)
    with mpmath.workdps(60):
        for i, v in enumerate(x):
            u = mpmath.mpf(float(v))
            e0 = -mpmath.expm1(-u)
            a = 1 - e0 / u
            exact = [1 / u, e0, mpmath.exp(-u), e0, a, (2 * a - e0) / u]
            for k in range(6):
                if k in (1, 2) and not 0.5 <= v < 37.5:
                    continue
                # d is a difference of terms of a's size
                err = abs(out[k][i] - exact[k]) / abs(exact[4 if k == 5 else k])
                worst[k] = max(worst[k], float(err) * 2.0 ** 53)
    # 1/x: 0.52 units in the last place (twice as many 2^-53 of a value just above a
    # power of two). 1 - e^-u: the table's rounding (2^-54), the series' cut (r^6/720 <
    # 0.31 2^-53, times e^-u <= 0.607) and the last rounding (2^-55 below 1/2), over
    # 0.393; e^-u: the table's rounding and the last one, each up to 2^-53, and the
    # cut. At u = 1/2 a = 1 - e0/u = 0.213 is good to 0.94 2 + 0.41 + 0.13 and
    # d = (2a - e0)/u to (2 2.4 + 0.94) 2, in 2^-53
    assert np.all(worst < [1.04, 2.4, 2.4, 2.4, 11.4, 54.0]), worst


@pytest.mark.parametrize("fuse", FUSE)
@pytest.mark.parametrize("ulp", [-1, 0, 1])
def test_float_float(lib, fuse, ulp):
    lib.mode(fuse, ulp)
    rng = np.random.default_rng(4)
    n = 2000
    x, y = (10.0 ** rng.uniform(-4, 4, n) for _ in range(2))
    z = x * y * 10.0 ** rng.uniform(0, 3, n)
    small = x * 10.0 ** rng.uniform(-4, 0, n)
    split = lambda v: v.astype(np.float32).astype(np.longdouble) + (
        v - v.astype(np.float32)).astype(np.float32).astype(np.longdouble)
    X, Y, Z, M = split(x), split(y), split(z), split(small)
    out = np.empty(n)
    for op, b, exact, bound in [(0, y, X + Y, 4), (1, y, X * Y, 4), (2, y, X * Y, 8), (3, y, X * Y + Z, 6),
                                (4, y, X * Y + Z, 8), (5, y, X * Y + Z, 6), (6, y, 1 / X, 8), (7, small, X + M, 4)]:
        lib.fflt(op, n, _ptr(x), _ptr(b), _ptr(z), _ptr(out))
        # units of 2^-48: lo * lo and the roundings of the low part
        err = np.max(np.abs(out - exact) / exact) * 2.0 ** 48
        assert err < bound, (op, err)
