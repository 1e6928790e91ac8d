// FP64 per-point arithmetic of the formal solutions without Lambda*,
// shared by the Cartesian kernel (fs.cu) and the spherical one (sph.cu). The
// FP64 pipe is the bound, so everything that can leave it does: branch tests
// on the high word of non-negative doubles (integer compares), reciprocals
// seeded in FP32, widening by integer moves. The interval functions follow
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

// 1/x for x > 0. Seed: x truncated to FP32 by integer moves (for x and 1/x
// inside the FP32 normal range: exponent field 897..1148), its FP32
// reciprocal, widened back; then one third-order Newton-Raphson step
// r = r0 + r0 (e + e^2), e = 1 - x r0, which takes the seed's relative error
// (< 2^-21, the hardware approximation's 2^-23 and the truncation) to below 2^-63, so the result is within an ulp or so of 1/x.
// Outside that range (and for 0, Inf, NaN): IEEE division.
__device__ __forceinline__ double recip64(double x) {
    const unsigned hi = (unsigned)__double2hiint(x);
    if (((hi >> 20) & 0x7ffu) - 897u > 251u || (hi >> 31)) return 1.0 / x;
    const unsigned lo = (unsigned)__double2loint(x);
    const float xf = __uint_as_float(((hi - 0x38000000u) << 3) | (lo >> 29));
    const double r0 = widen_f32(rcp_approx(xf));
    const double e = fma(-x, r0, 1.0);
    return fma(r0, fma(e, e, e), r0);
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
// ln2 / 64 as the sum of two doubles
constexpr double kLn2Hi = 0.010830424696249145, kLn2Lo = 3.623510646634843e-19;

// The table in shared memory (every thread of the block must call it).
__device__ __forceinline__ void exp_table(double *tab) {
    if (threadIdx.x < 64) tab[threadIdx.x] = kPow2[threadIdx.x];
    __syncthreads();
}

// e^-u for 1/2 <= u < 37.5 (Tang's table-driven method): n = nearest integer
// to 64 u / ln2 (found in FP32; a neighbour of it near a tie only widens r's
// range), r = u - n ln2/64, |r| <= ln2/128 (1 + 2^-9), e^-r by its Taylor
// polynomial of degree 5 (truncation r^6/720 < 4e-17), e^-u = 2^-(n div 64)
// 2^-((n mod 64)/64) e^-r. Eight FP64 operations, about half of the library's
// exp, whose accuracy over the whole range e^-u does not need here: the caller
// takes 1 - e^-u.
__device__ __forceinline__ double exp_neg64(double u, const double *tab) {
    const unsigned hi = (unsigned)__double2hiint(u), lo = (unsigned)__double2loint(u);
    const float uf = __uint_as_float(((hi - 0x38000000u) << 3) | (lo >> 29));
    const float t = fmaf(uf, 92.33248f, 12582912.0f);  // 1.5 2^23: n in the low bits
    const int n = __float_as_int(t) - 0x4B400000;
    const double nd = widen_f32(t - 12582912.0f);
    const double r = fma(-nd, kLn2Lo, fma(-nd, kLn2Hi, u));
    double q = fma(r, -1.0 / 120.0, 1.0 / 24.0);
    q = fma(r, q, -1.0 / 6.0);
    q = fma(r, q, 0.5);
    const double P = fma(r * r, q, -r);  // e^-r - 1
    const double T = tab[n & 63];
    const double E = fma(T, P, T);
    return __hiloint2double(__double2hiint(E) - ((n >> 6) << 20), __double2loint(E));
}

// Interval functions in FP64 (as interval(double)); for u < 1/2 p(u) =
// e2/u^3 is a degree-9 polynomial fitted to the exact function (least squares
// in relative error at 300 Chebyshev nodes of [0, 1/2]; FP64 Horner error
// 1.6e-16 relative, the rounding of its leading coefficient 1/3). The terms of
// degree 7 to 9 are left out below 2^-6 and those of degree 5 and 6 below 2^-10,
// where they are under 4e-19 and 2e-18 of the sum. From 37.5 on e^-u is below
// 2^-54, and e0 = 1 (a NaN u goes there and reaches a through ru). ru = 1/u
// for u >= 1/2 (carried from the previous step, or computed here if CARRY is
// false). Returns e0, a, d for the update in difference form.
struct IntervalDE {
    double e0, a, d;
};
template <bool CARRY>
__device__ __forceinline__ IntervalDE interval64(double u, double ru, const double *tab) {
    IntervalDE r;
    if (hi_below(u, 0x3FE00000)) {
        double p = -3.4475018036590732e-09;
        if (hi_below(u, 0x3F900000)) {
            p = 5.511310234105578e-06;
        } else {
            p = fma(p, u, 4.9354831016668725e-08);
            p = fma(p, u, -5.507115670485655e-07);
            p = fma(p, u, 5.511310234105578e-06);
        }
        if (hi_below(u, 0x3F500000)) {
            p = 3.9682539230545495e-04;
        } else {
            p = fma(p, u, -4.9603140878306714e-05);
            p = fma(p, u, 3.9682539230545495e-04);
        }
        p = fma(p, u, -2.777777777429071e-03);
        p = fma(p, u, 1.6666666666652976e-02);
        p = fma(p, u, -8.333333333333312e-02);
        p = fma(p, u, 3.333333333333333e-01);
        const double b = u * p;
        const double hu = 0.5 * u;
        const double a = fma(-hu, b, hu);
        r.e0 = fma(-u, a, u);
        r.a = a;
        r.d = a - b;
    } else {
        if (!CARRY) ru = recip64(u);
        double e0 = 1.0;
        if (hi_below(u, 0x4042C000)) e0 = 1.0 - exp_neg64(u, tab);
        const double a = fma(-e0, ru, 1.0);
        r.e0 = e0;
        r.a = a;
        r.d = fma(2.0, a, -e0) * ru;
    }
    return r;
}

}  // namespace rt3d
