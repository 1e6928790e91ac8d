// Float-float ("double-float") arithmetic on the FP32 pipe: a value is the
// unevaluated sum hi + lo of two FP32 numbers with |lo| <= ulp(hi)/2, about
// 48 significant bits. The error-free transformations are Knuth's two-sum,
// Dekker's fast two-sum (|a| >= |b|) and the FMA-based exact product; the
// compound operations follow the "sloppy" double-double algorithms of Hida,
// Li and Bailey (2001): relative error a few units of 2^-48 except under
// cancellation, where the error stays a few units of 2^-48 of the operands.
// What has to be rounded by itself is written with __fmul_rn, __fadd_rn and
// __fsub_rn, which the compiler does not fuse (a plain product may be fused into
// whatever sum it enters, here or in a caller, and the error terms then count its
// low part twice).
#pragma once

namespace rt3d {

struct ff {
    float hi, lo;
};

__device__ __forceinline__ ff ff_of(float x) { return ff{x, 0.0f}; }

// nearest float-float of a double (the two FP32 conversions run on the FP64
// pipe: for per-voxel or per-step preprocessing, not per-segment work)
__device__ __forceinline__ ff ff_split(double x) {
    const float h = __double2float_rn(x);
    return ff{h, __double2float_rn(x - (double)h)};
}

__device__ __forceinline__ ff two_sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    const float v = __fsub_rn(s, a);
    return ff{s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, v)), __fsub_rn(b, v))};
}

__device__ __forceinline__ ff quick_two_sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    return ff{s, __fsub_rn(b, __fsub_rn(s, a))};
}

__device__ __forceinline__ ff two_prod(float a, float b) {
    const float p = __fmul_rn(a, b);
    return ff{p, fmaf(a, b, -p)};
}

__device__ __forceinline__ ff ff_neg(ff x) { return ff{-x.hi, -x.lo}; }

__device__ __forceinline__ ff ff_add(ff x, ff y) {
    const ff s = two_sum(x.hi, y.hi);
    return quick_two_sum(s.hi, s.lo + (x.lo + y.lo));
}

__device__ __forceinline__ ff ff_sub(ff x, ff y) { return ff_add(x, ff_neg(y)); }

// x + y and x - y for |x| >= |y| (three operations fewer)
__device__ __forceinline__ ff ff_add_big(ff x, ff y) {
    const ff s = quick_two_sum(x.hi, y.hi);
    return quick_two_sum(s.hi, s.lo + (x.lo + y.lo));
}
__device__ __forceinline__ ff ff_sub_big(ff x, ff y) { return ff_add_big(x, ff_neg(y)); }

__device__ __forceinline__ ff ff_add_f(ff x, float y) {
    const ff s = two_sum(x.hi, y);
    return quick_two_sum(s.hi, s.lo + x.lo);
}

__device__ __forceinline__ ff ff_mul(ff x, ff y) {
    const ff p = two_prod(x.hi, y.hi);
    return quick_two_sum(p.hi, fmaf(x.hi, y.lo, fmaf(x.lo, y.hi, p.lo)));
}

__device__ __forceinline__ ff ff_mul_f(ff x, float y) {
    const ff p = two_prod(x.hi, y);
    return quick_two_sum(p.hi, fmaf(x.lo, y, p.lo));
}

// x * y without the last renormalisation: the same sum, its low part up to an
// ulp of the high one. As a factor or an addend of a further operation, which
// drops only lo * lo (2^-46 of the product at most).
__device__ __forceinline__ ff ff_mul_raw(ff x, ff y) {
    const ff p = two_prod(x.hi, y.hi);
    return ff{p.hi, fmaf(x.hi, y.lo, fmaf(x.lo, y.hi, p.lo))};
}

// x * y + z for |z| >= |x y|; the same without the last renormalisation
__device__ __forceinline__ ff ff_fma_big_raw(ff x, ff y, ff z) {
    const ff p = two_prod(x.hi, y.hi);
    const float e = fmaf(x.hi, y.lo, fmaf(x.lo, y.hi, p.lo));
    const ff s = quick_two_sum(z.hi, p.hi);
    return ff{s.hi, s.lo + (e + z.lo)};
}
__device__ __forceinline__ ff ff_fma_big(ff x, ff y, ff z) {
    const ff s = ff_fma_big_raw(x, y, z);
    return quick_two_sum(s.hi, s.lo);
}

// x * y + z
__device__ __forceinline__ ff ff_fma(ff x, ff y, ff z) {
    const ff p = two_prod(x.hi, y.hi);
    const float e = fmaf(x.hi, y.lo, fmaf(x.lo, y.hi, p.lo));
    const ff s = two_sum(p.hi, z.hi);
    return quick_two_sum(s.hi, s.lo + (e + z.lo));
}

// exact scaling by a power of two (no overflow or underflow in range)
__device__ __forceinline__ ff ff_scale(ff x, float p2) { return ff{x.hi * p2, x.lo * p2}; }

// 1/x for x > 0: r the FP32 approximation (relative error e <= 2^-23), then
// r (1 + e + e^2) with e = 1 - x r formed by two fused operations (it is exact
// to 2^-24 of itself, as the product with r is): 2^-47 in all, and nine
// instructions where a float-float residual and a correctly rounded r took
// about 28 for the same accuracy.
__device__ __forceinline__ ff ff_recip(ff x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x.hi));
    const float e = fmaf(-x.lo, r, fmaf(-x.hi, r, 1.0f));
    const float g = fmaf(e, e, e), s = fmaf(r, g, r);
    return ff{s, fmaf(r, g, __fsub_rn(r, s))};
}

// FP64 value of a float-float (the widening of each part is exact; the sum
// rounds once, on the FP64 pipe)
__device__ __forceinline__ double ff_to_double(ff x) { return (double)x.hi + (double)x.lo; }

}  // namespace rt3d
