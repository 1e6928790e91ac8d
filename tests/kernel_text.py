"""The kernels' FP64 and float-float arithmetic (ff.cuh, fs64_step.cuh), their own
text compiled for the CPU with an FP32 type that fuses products into sums on
demand: build(folder) returns the library, whose calls are

  mode(fuse, ulp)  products entering a sum: 0 rounded first, 1 fused (the left
                   operand's first), 2 fused (the right one's first), 3 at random;
                   ulp: error of the reciprocal's approximation
  fs64, fflt       see CALLS
"""
import ctypes
import os
import re
import subprocess

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


def build(folder):
    cpp, so = os.path.join(str(folder), "arith.cpp"), os.path.join(str(folder), "arith.so")
    with open(cpp, "w") as f:
        f.write(PRELUDE + _text("ff.cuh") + _text("fs64_step.cuh") + CALLS)
    subprocess.run(["g++", "-O1", "-std=c++17", "-ffp-contract=off", "-w", "-shared", "-fPIC", cpp, "-o", so, "-lm"],
                   check=True)
    return ctypes.CDLL(so)


def ptr(a):
    return a.ctypes.data_as(ctypes.POINTER(ctypes.c_double))
