"""The float-float and FP64 arithmetic of the kernels, their own source text run on
the CPU with FP32 operations that are contracted as a compiler may: a product that
is added or subtracted anywhere later is either rounded first or fused into the
sum. The stated error bounds hold whatever is fused, since what must be rounded is
written with __fmul_rn, __fadd_rn and __fsub_rn."""
import ctypes
import os
import re
import subprocess

import mpmath
import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2102_01734_gb300", "csrc")

PRELUDE = r"""
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#define __device__
#define __forceinline__ inline
using std::max;
static int fuse = 0;      // 0 never, 1 always (left operand first), 2 always (right first), 3 at random
static int seed_ulp = 0;  // error of the reciprocal's approximation in units in the last place
static uint64_t rnd = 1;
static bool taken() {
    rnd = rnd * 6364136223846793005ULL + 1442695040888963407ULL;
    return fuse == 1 || fuse == 2 || (fuse == 3 && (rnd >> 40 & 1));
}
struct F {  // an FP32 value, with its factors while it is a product nobody has rounded
    float v, a, b;
    bool prod;
    F() : v(0), a(0), b(0), prod(false) {}
    template <typename T> F(T x) : v((float)x), a(0), b(0), prod(false) {}
    explicit operator double() const { return v; }
    explicit operator int() const { return (int)v; }
    F operator-() const {
        F r = *this;
        r.v = -r.v;
        r.a = -r.a;
        return r;
    }
};
static F mul(F x, F y) {
    F r(x.v * y.v);
    r.a = x.v;
    r.b = y.v;
    r.prod = true;
    return r;
}
static F add(F x, F y) {
    const bool left = fuse != 2;
    for (int i = 0; i < 2; ++i) {
        F &p = (i == 0) == left ? x : y, &q = (i == 0) == left ? y : x;
        if (p.prod && taken()) return F(std::fmaf(p.a, p.b, q.v));
    }
    return F(x.v + y.v);
}
static F operator*(F x, F y) { return mul(x, y); }
static F operator+(F x, F y) { return add(x, y); }
static F operator-(F x, F y) { return add(x, -y); }
static bool operator>(F x, F y) { return x.v > y.v; }
static F fmaf(F x, F y, F z) { return F(std::fmaf(x.v, y.v, z.v)); }
static F __fmul_rn(F x, F y) { return F(x.v * y.v); }
static F __fadd_rn(F x, F y) { return F(x.v + y.v); }
static F __fsub_rn(F x, F y) { return F(x.v - y.v); }
static F rcp_approx(F x) {
    float r = (float)(1.0 / (double)x.v);
    for (int i = 0; i < std::abs(seed_ulp); ++i) r = std::nextafterf(r, seed_ulp < 0 ? 0.0f : 2.0f * r);
    return F(r);
}
template <typename T, typename S> static T bits(S s) {
    T t;
    static_assert(sizeof t == sizeof s, "");
    std::memcpy(&t, &s, sizeof t);
    return t;
}
static int __float2int_rn(F x) { return (int)std::lrintf(x.v); }
static F __double2float_rn(double x) { return F((float)x); }
static F __uint_as_float(unsigned u) { return F(bits<float>(u)); }
static int __float_as_int(F x) { return bits<int>(x.v); }
static int __double2hiint(double x) { return (int)(bits<uint64_t>(x) >> 32); }
static int __double2loint(double x) { return (int)bits<uint64_t>(x); }
static double __hiloint2double(int h, int l) { return bits<double>((uint64_t)(unsigned)h << 32 | (unsigned)l); }
static double __longlong_as_double(long long x) { return bits<double>(x); }
static long long __double_as_longlong(double x) { return bits<long long>(x); }
static unsigned long long __umul64hi(unsigned long long a, unsigned long long b) {
    return (unsigned long long)((unsigned __int128)a * b >> 64);
}
static int __clzll(long long x) { return __builtin_clzll((unsigned long long)x); }
static struct { unsigned x; } threadIdx;
static void __syncthreads() {}
"""

CALLS = r"""
using namespace rt3d;
extern "C" {
void mode(int f, int ulp) { fuse = f; seed_ulp = ulp; rnd = 1; }
void fs64(int n, const double *x, double *recip, double *one_minus, double *exp_neg, double *e0, double *a, double *d) {
    static unsigned long long tab[64];
    for (threadIdx.x = 0; threadIdx.x < 64; ++threadIdx.x) exp_table(tab);
    for (int i = 0; i < n; ++i) {
        recip[i] = recip64(x[i]);
        const bool in = x[i] >= 0.5 && x[i] < 37.5;
        one_minus[i] = in ? one_minus_exp64(x[i], tab) : 0.0;
        exp_neg[i] = in ? exp_neg64(x[i], tab) : 0.0;
        const IntervalDE f = interval64<false>(x[i], 0.0, tab);
        e0[i] = f.e0;
        a[i] = f.a;
        d[i] = f.d;
    }
}
// op: 0 x + y, 1 x y, 2 x y (raw), 3 x y + z with |z| >= |x y|, 4 the same raw, 5 x y + z, 6 1 / x, 7 x + y with
// |x| >= |y|
void fflt(int op, int n, const double *x, const double *y, const double *z, double *out) {
    for (int i = 0; i < n; ++i) {
        const ff X = ff_split(x[i]), Y = ff_split(y[i]), Z = ff_split(z[i]);
        const ff r = op == 0 ? ff_add(X, Y) : op == 1 ? ff_mul(X, Y) : op == 2 ? ff_mul_raw(X, Y)
                   : op == 3 ? ff_fma_big(X, Y, Z) : op == 4 ? ff_fma_big_raw(X, Y, Z) : op == 5 ? ff_fma(X, Y, Z)
                   : op == 6 ? ff_recip(X) : ff_add_big(X, Y);
        out[i] = (double)r.hi.v + (double)r.lo.v;
    }
}
}
"""


def _text(name):
    src = open(os.path.join(CSRC, name)).read()
    src = src[src.index("namespace rt3d {"):]
    src = re.sub(r'asm\("rcp\.approx\.ftz\.f32.*?;\n', "r = rcp_approx(x.hi);\n", src)
    return re.sub(r"\bfloat\b", "F", src)


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("arith")
    cpp, so = str(d / "arith.cpp"), str(d / "arith.so")
    with open(cpp, "w") as f:
        f.write(PRELUDE + _text("ff.cuh") + _text("fs64_step.cuh") + CALLS)
    subprocess.run(["g++", "-O1", "-std=c++17", "-ffp-contract=off", "-fno-fast-math", "-w", "-shared", "-fPIC",
                    cpp, "-o", so, "-lm"], check=True)
    return ctypes.CDLL(so)


def _ptr(a):
    return a.ctypes.data_as(ctypes.POINTER(ctypes.c_double))


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
