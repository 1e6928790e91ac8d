// FP64 per-point arithmetic of the formal solutions without Lambda*,
// shared by the Cartesian kernel (fs.cu) and the spherical one (sph.cu). The
// FP64 pipe is the bound, so everything that can leave it does (an FP64
// instruction holds its pipe for 64 cycles, in which 64 others issue): branch
// tests on the high word of non-negative doubles (integer compares), reciprocals,
// the polynomial's smaller terms, halving, widening by integer moves. The interval functions follow
// the construction documented at the top of fs.cu (Olson & Kunasz 1987
// weights; the update in difference form).
#pragma once
#include "fs_step.cuh"

namespace rt3d {

// Whether x < b for a double x >= 0 and a bound b > 0 whose low word is
// zero, given the high word of b: an unsigned compare of the high words, so
// a NaN of either sign (0 * Inf where a zero-opacity interval meets a zero
// one) counts as not below.
__device__ __forceinline__ bool hi_below(double x, int b_hi) {
    return (unsigned)__double2hiint(x) < (unsigned)b_hi;
}

// a + b = s + t exactly (Knuth). Here and below, what has to be rounded by itself is
// written with __fmul_rn, __fadd_rn and __fsub_rn: the compiler fuses none of them.
__device__ __forceinline__ float sum_exact(float a, float b, float &t) {
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    t = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return s;
}

// 1/x for x > 0, without the FP64 pipe. With x = 2^k m, 1 <= m < 2, m is split
// by integer moves into its first 24 bits, the next 24 and the last 5 (xh, xl,
// xt); r0 is the FP32 reciprocal of xh. The residual e = 1 - m r0 (|e| < 2^-21) is
// collected as a pair of FP32 values (eh, el) whose error is below 2^-66, the
// correction r0 (e + e^2) likewise (the next term, e^3, is below 2^-63), and the
// sum r0 + correction is formed and rounded in fixed point (units of 2^-60): within
// 0.52 units in the last place of 1/x. For 0, subnormal, infinite and NaN x and x from
// 2^1021 on: IEEE division.
__device__ __forceinline__ double recip64(double x) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const unsigned ex = hi >> 20;
    if (ex - 1u > 2042u) return 1.0 / x;
    const float xh = __uint_as_float(0x3f800000u | ((hi & 0xfffffu) << 3) | (lo >> 29));
    const float xl = (float)(lo & 0x1fffffe0u) * 0x1p-52f, xt = (float)(lo & 31u) * 0x1p-52f;
    const float r0 = rcp_approx(xh);
    const float ph = __fmul_rn(xh, r0), pl = fmaf(xh, r0, -ph);
    const float q = __fmul_rn(xl, r0), ql = fmaf(xl, r0, -q);
    float t1, t2;
    const float s1 = sum_exact(__fsub_rn(1.0f, ph), -q, t1);
    const float eh = sum_exact(s1, -pl, t2);
    const float el = fmaf(-xt, r0, (t1 + t2) - ql);
    const float f = fmaf(eh, eh, el);
    const float ch = __fmul_rn(r0, eh), cl = fmaf(r0, f, fmaf(r0, eh, -ch));
    // r0 2^60, the correction's first 23 bits and the rest
    const int c1 = __float2int_rn(ch * 0x1p44f);
    const int c2 = __float2int_rn((fmaf((float)c1, -0x1p-44f, ch) + cl) * 0x1p60f);
    const long long fix = ((long long)__float2int_rn(r0 * 0x1p24f) << 36) + ((long long)c1 << 16) + c2;
    // 2^59 <= fix <= 2^60: 53 bits, rounded; 1 carries into the exponent
    const long long bits = ((fix + 64) >> 7) + (1021LL << 52) - ((long long)((int)ex - 1023) << 52);
    return __longlong_as_double(bits);
}

// (h, l) = c + u (h, l) in float-float, |c| > |u h|
__device__ __forceinline__ void horner_ff(float &h, float &l, float uh, float ul, double c) {
    const float chi = (float)c, clo = (float)(c - (double)chi);  // folded at compile time
    const float p = __fmul_rn(uh, h);
    const float e = fmaf(uh, l, fmaf(ul, h, fmaf(uh, h, -p)));
    const float s = __fadd_rn(chi, p);
    l = __fadd_rn(__fsub_rn(p, __fsub_rn(s, chi)), __fadd_rn(e, clo));
    h = s;
}
// |x| as a pair of FP32 values, x = +-(h + l) to 2^-48 of it, by integer moves;
// both 0 below 2^-38, for |x| < 2^127.
__device__ __forceinline__ void split_ff(double x, float &h, float &l) {
    const unsigned hi = (unsigned)__double2hiint(x) & 0x7fffffffu, lo = (unsigned)__double2loint(x);
    const unsigned ex = hi >> 20;
    const bool tiny = ex < 985u;
    h = tiny ? 0.0f : __uint_as_float(((hi - 0x38000000u) << 3) | (lo >> 29));
    l = tiny ? 0.0f : (float)(lo & 0x1fffffffu) * __uint_as_float((ex - 948u) << 23);
}

// 2^(-j/64), j = 0 .. 63, correctly rounded.
__device__ const double kPow2[64] = {
    1.0, 0.9892280131939755, 0.9785720620877001, 0.9680308967461472,
    0.9576032806985737, 0.9472879907934828, 0.93708381705515, 0.9269895625416927,
    0.9170040432046712, 0.9071260877501994, 0.8973545375015536, 0.8876882462632606,
    0.8781260801866497, 0.8686669176368531, 0.859309649061239, 0.8500531768592617,
    0.8408964152537145, 0.8318382901633682, 0.8228777390769825, 0.8140137109286739,
    0.8052451659746271, 0.7965710756711335, 0.7879904225539432, 0.7795022001189185,
    0.7711054127039704, 0.7627990753722692, 0.7545822137967114, 0.7464538641456324,
    0.7384130729697497, 0.7304588970903235, 0.7225904034885233, 0.714806669195985,
    0.7071067811865476, 0.6994898362691556, 0.691954940981916, 0.6845012114872953,
    0.6771277734684463, 0.6698337620266515, 0.6626183215798707, 0.6554806057623822,
    0.6484197773255048, 0.6414350080393891, 0.6345254785958666, 0.6276903785123455,
    0.620928906036742, 0.614240268053435, 0.6076236799902345, 0.6010783657263515,
    0.5946035575013605, 0.5881984958251406, 0.5818624293887887, 0.5755946149764913,
    0.5693943173783458, 0.5632608093041209, 0.5571933712979462, 0.5511912916539204,
    0.5452538663326288, 0.5393803988785599, 0.5335702003384118, 0.5278225891802786,
    0.5221368912137069, 0.5165124395106142, 0.5109485743270583, 0.5054446430258502};
// ln2 / 64 in units of 2^-64: the integer part and the next 32 bits
constexpr unsigned long long kLn2Int = 0x2c5c85fdf473de6ULL;
constexpr unsigned kLn2Frac = 0xaf278eceu;

// The table in shared memory, in units of 2^-63 (every thread of the block must
// call it).
__device__ __forceinline__ void exp_table(unsigned long long *tab) {
    if (threadIdx.x < 64) {
        const unsigned long long b = (unsigned long long)__double_as_longlong(kPow2[threadIdx.x]);
        tab[threadIdx.x] = ((b & 0xfffffffffffffULL) | 1ULL << 52) << (threadIdx.x ? 10 : 11);
    }
    __syncthreads();
}

// x >= 0 in units of 2^-64, modulo 2^64, truncated
__device__ __forceinline__ unsigned long long fixed64(double x) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const unsigned long long m = (unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32 | lo;
    const int sh = (int)(hi >> 20) - 1011;
    return sh >= 0 ? m << sh : (sh > -64 ? m >> -sh : 0ULL);
}

// e^-u for 1/2 <= u < 37.5 as E 2^-62 2^-k (Tang's table-driven method in fixed
// point, no FP64 operation): n = nearest integer to 64 u / ln2 (found in FP32; a
// neighbour of it near a tie only widens r's range), r = u - n ln2/64 modulo 1 in
// units of 2^-64 (exact but for the last two), |r| <= ln2/128 (1 + 2^-9), e^-r - 1 =
// -r + g with g from the Taylor polynomial of degree 5 (truncation r^6/720 < 4e-17;
// g, below 2^-15, in float-float), e^-u = 2^-(n div 64) 2^-((n mod 64)/64) e^-r.
__device__ __forceinline__ unsigned long long exp_fixed64(double u, const unsigned long long *tab,
                                                          int &k) {
    const unsigned hi = (unsigned)__double2hiint(u), lo = (unsigned)__double2loint(u);
    const float uf = __uint_as_float(((hi - 0x38000000u) << 3) | (lo >> 29));
    const float t = fmaf(uf, 92.33248f, 12582912.0f);  // 1.5 2^23: n in the low bits
    const int n = __float_as_int(t) - 0x4B400000;
    const unsigned long long m = (unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32 | lo;
    const unsigned long long nl =
        (unsigned long long)n * kLn2Int + ((unsigned long long)n * kLn2Frac >> 32);
    const long long r = (long long)((m << ((int)(hi >> 20) - 1011)) - nl);
    const float rh = (float)(int)(r >> 34) * 0x1p-30f;
    const float rl = (float)(unsigned)(r >> 2) * 0x1p-62f;  // the low 34 bits
    float h = fmaf(rh, (float)(-1.0 / 120.0), (float)(1.0 / 24.0)), l = 0.0f;
    horner_ff(h, l, rh, rl, -1.0 / 6.0);
    horner_ff(h, l, rh, rl, 0.5);
    const float p = __fmul_rn(rh, rh), e = fmaf(rh, 2.0f * rl, fmaf(rh, rh, -p));  // r^2
    const float gh = __fmul_rn(p, h), gl = fmaf(e, h, fmaf(p, l, fmaf(p, h, -gh)));
    const int g1 = __float2int_rn(gh * 0x1p40f);
    const int g2 = __float2int_rn((fmaf((float)g1, -0x1p-40f, gh) + gl) * 0x1p64f);
    const long long P = ((long long)g1 << 24) + g2 - r;  // e^-r - 1
    k = n >> 6;
    return __umul64hi(tab[n & 63], (1ULL << 63) + (unsigned long long)(P >> 1));
}
// 1 - e^-u and e^-u, rounded once: within 2.4 2^-53 of themselves (the table's
// rounding, the cut of the series and the last rounding)
__device__ __forceinline__ double one_minus_exp64(double u, const unsigned long long *tab) {
    int k;
    const unsigned long long E = exp_fixed64(u, tab, k);
    const unsigned long long e0 = (1ULL << 62) - (E >> k);  // units of 2^-62
    const bool half = e0 >= 1ULL << 61;
    return __longlong_as_double((half ? 1021LL << 52 : 1020LL << 52) +
                                (long long)(half ? (e0 + 256) >> 9 : (e0 + 128) >> 8));
}
__device__ __forceinline__ double exp_neg64(double u, const unsigned long long *tab) {
    int k;
    const unsigned long long E = exp_fixed64(u, tab, k);
    const int sh = 11 - __clzll((long long)E);  // 53 bits stay
    return __longlong_as_double(((long long)(1012 + sh - k) << 52) +
                                (long long)((E + (1ULL << (sh - 1))) >> sh));
}

// Horner's rule for p(u) = e2/u^3, 0 <= u < 1/2, degree 9, without an FP64 operation:
// degrees 9 and 8 in FP32, 7 to 3 in float-float (below 2^-9 of p in all), 2 to 0 in
// fixed point (units of 2^-64, alternating signs), rounded once: 1/4 < p < 1/2.
struct Horner64 {
    int next;  // degree of the next coefficient, known at compile time
    float h, l;
    unsigned long long v;

    __device__ __forceinline__ friend Horner64 fma(Horner64 p, double u, double c) {
        float uh, ul;
        split_ff(u, uh, ul);
        const int degree = p.next--;
        if (degree >= 8) {
            p.h = fmaf(uh, p.h, (float)c);
        } else if (degree >= 3) {
            horner_ff(p.h, p.l, uh, ul, c);
        } else {
            if (degree == 2) {  // the sum of the higher terms, negative
                const int t1 = __float2int_rn(p.h * -0x1p30f);
                const int t2 = __float2int_rn((fmaf((float)t1, -0x1p-30f, -p.h) - p.l) * 0x1p56f);
                p.v = (unsigned long long)(((long long)t1 << 34) + ((long long)t2 << 8));
            }
            p.v = (unsigned long long)(fabs(c) * 0x1p64) - __umul64hi(fixed64(u), p.v);
        }
        return p;
    }
    __device__ __forceinline__ double value() const {
        return __longlong_as_double((1020LL << 52) + (long long)((v + 512) >> 10));
    }
};

// u / 2 for finite u >= 0, by integer moves: one less in the exponent, or (below
// 2^-1021, truncated to the smallest subnormal) the whole pattern shifted.
__device__ __forceinline__ double half64(double u) {
    const unsigned hi = (unsigned)__double2hiint(u), lo = (unsigned)__double2loint(u);
    const bool low = hi < 0x00200000u;
    return __hiloint2double((int)(low ? hi >> 1 : hi - 0x00100000u), (int)(low ? lo >> 1 | hi << 31 : lo));
}

// Interval functions in FP64 (as interval(double)); for u < 1/2 p(u) =
// e2/u^3 is a degree-9 polynomial fitted to the exact function (least squares
// in relative error at 300 Chebyshev nodes of [0, 1/2]). It and 1 - e^-u are
// evaluated off the FP64 pipe (Horner64, one_minus_exp64). From 37.5 on e^-u is below
// 2^-54, and e0 = 1 (a NaN u goes there and reaches a through ru). ru = 1/u
// for u >= 1/2 (carried from the previous step, or computed here if CARRY is
// false). Returns e0, a, d for the update in difference form.
struct IntervalDE {
    double e0, a, d;
};
template <bool CARRY>
__device__ __forceinline__ IntervalDE interval64(double u, double ru, const unsigned long long *tab) {
    IntervalDE r;
    if (hi_below(u, 0x3FE00000)) {
        Horner64 p{9, 0.0f, 0.0f, 0ULL};
        p = fma(p, u, -3.4475018036590732e-09);
        p = fma(p, u, 4.9354831016668725e-08);
        p = fma(p, u, -5.507115670485655e-07);
        p = fma(p, u, 5.511310234105578e-06);
        p = fma(p, u, -4.9603140878306714e-05);
        p = fma(p, u, 3.9682539230545495e-04);
        p = fma(p, u, -2.777777777429071e-03);
        p = fma(p, u, 1.6666666666652976e-02);
        p = fma(p, u, -8.333333333333312e-02);
        p = fma(p, u, 3.333333333333333e-01);
        const double b = u * p.value();
        const double hu = half64(u);
        const double a = fma(-hu, b, hu);
        r.e0 = fma(-u, a, u);
        r.a = a;
        r.d = a - b;
    } else {
        if (!CARRY) ru = recip64(u);
        double e0 = 1.0;
        if (hi_below(u, 0x4042C000)) e0 = one_minus_exp64(u, tab);
        const double a = fma(-e0, ru, 1.0);
        r.e0 = e0;
        r.a = a;
        r.d = fma(2.0, a, -e0) * ru;
    }
    return r;
}

// The same with E = e^-u and a0 = e0 - a, for the kernel with Lambda*.
struct IntervalD {
    double E, a0, a, d;
};
__device__ __forceinline__ IntervalD interval64_w(double u, const unsigned long long *tab) {
    IntervalD r;
    if (hi_below(u, 0x3FE00000)) {
        const IntervalDE f = interval64<false>(u, 0.0, tab);
        r.E = 1.0 - f.e0;
        r.a0 = f.e0 - f.a;
        r.a = f.a;
        r.d = f.d;
    } else {
        r.E = hi_below(u, 0x4042C000) ? exp_neg64(u, tab) : exp(-u);
        const double ru = recip64(u), e0 = 1.0 - r.E;
        r.a = fma(-e0, ru, 1.0);
        r.a0 = fma(-(1.0 + u), r.E, 1.0) * ru;
        r.d = fma(2.0, r.a, -e0) * ru;
    }
    return r;
}

}  // namespace rt3d
