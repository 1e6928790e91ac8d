// Per-point arithmetic of the FP32 formal solutions: with one, two and four
// characteristics a thread, and with the weights of Lambda* (fs.cu); one
// characteristic a thread also serves the batched wavelengths (batch.cu) and the
// shell (sph.cu). The interval functions and the update follow the construction
// documented at the top of fs.cu (Olson & Kunasz 1987 weights with the
// limited parabola; the update in difference form).
#pragma once
#include "rt3d_internal.cuh"

namespace rt3d {

// FP32 interval functions for the formal solution without Lambda*: e0, a
// and d of the interval of optical depth u (the update in difference form
// needs neither E nor a0). For u < 1, p(u) = e2/u^3 is a degree-5 polynomial
// fitted to the exact function (least squares in relative error at 200
// Chebyshev nodes of [0, 1]; FP32 Horner error 1.2e-7 relative, as for the
// 9-term Taylor series). For u >= 1 the caller passes ru = 1/u.
struct IntervalE {
    float e0, a, d;
};
__device__ __forceinline__ IntervalE interval_fast(float u, float ru) {
    IntervalE r;
    if (u < 1.0f) {
        float p = -3.569704858819023e-05f;
        p = fmaf(p, u, 3.819821577053517e-04f);
        p = fmaf(p, u, -2.770215505734086e-03f);
        p = fmaf(p, u, 1.6664894297719002e-02f);
        p = fmaf(p, u, -8.333317935466766e-02f);
        p = fmaf(p, u, 3.333333432674408e-01f);
        const float b = u * p;
        const float hu = 0.5f * u;
        const float a = fmaf(-hu, b, hu);
        r.e0 = fmaf(-u, a, u);
        r.a = a;
        r.d = a - b;
    } else {
        const float e0 = 1.0f - __expf(-u);
        const float a = fmaf(-e0, ru, 1.0f);
        r.e0 = e0;
        r.a = a;
        r.d = fmaf(2.0f, a, -e0) * ru;
    }
    return r;
}

// x as an FP64 value, by moving the fields of its IEEE binary32 encoding
// into binary64 with the exponent rebiased by 1023 - 127: exact for every
// normal x; a zero or subnormal x becomes +-2^-127 (1 + m 2^-23), below
// 1.2e-38 in magnitude. Infinities and NaNs are not preserved: the kernel
// below checks the intensity at the end of each characteristic instead
// (a non-finite value persists along the recurrence). Integer instructions
// only, where the conversion instruction would load the FP64 pipe.
__device__ __forceinline__ double widen_f32(float x) {
    const unsigned b = __float_as_uint(x);
    const unsigned lo = b << 29;
    // the shift copies the sign into the three bits below it: masked off
    const unsigned hi = ((unsigned)((int)b >> 3) & 0x8fffffffu) + 0x38000000u;
    return __hiloint2double((int)hi, (int)lo);
}

template <bool WIDEN> __device__ __forceinline__ double to_f64(float x) {
    if (WIDEN) return widen_f32(x);
    return (double)x;
}

// ---- Two characteristics per thread in packed FP32x2 arithmetic ----
// The sm_100 family executes add, sub, mul and fma on a pair of FP32 values
// in one instruction (each component rounded as its scalar operation). The
// pair kernel gives a thread the characteristics of face cells (x0, y) and
// (x0, y + 1): component .x and .y of every float2 below.

__device__ __forceinline__ float2 pk(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ float2 pk1(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ unsigned long long f2_bits(float2 a) {
    return ((unsigned long long)__float_as_uint(a.y) << 32) | __float_as_uint(a.x);
}
__device__ __forceinline__ float2 f2_from_bits(unsigned long long r) {
    return make_float2(__uint_as_float((unsigned)r), __uint_as_float((unsigned)(r >> 32)));
}
// a - b per component
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
    unsigned long long r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(f2_bits(a)), "l"(f2_bits(b)));
    return f2_from_bits(r);
}
// MUFU approximations (PTX rcp.approx / ex2.approx, subnormals flushed)
__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float ex2_approx(float x) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

struct IntervalE2 {
    float2 e0, a, d;
};
// interval_fast's polynomial branch (u < 1) on both components
__device__ __forceinline__ IntervalE2 interval_poly2(float2 u) {
    float2 p = fma2(pk1(-3.569704858819023e-05f), u, pk1(3.819821577053517e-04f));
    p = fma2(p, u, pk1(-2.770215505734086e-03f));
    p = fma2(p, u, pk1(1.6664894297719002e-02f));
    p = fma2(p, u, pk1(-8.333317935466766e-02f));
    p = fma2(p, u, pk1(3.333333432674408e-01f));
    const float2 b = mul2(u, p);
    const float2 hu = mul2(u, pk1(0.5f));
    IntervalE2 r;
    r.a = mul2(hu, sub2(pk1(1.0f), b));       // u (1 - b) / 2
    r.e0 = mul2(u, sub2(pk1(1.0f), r.a));     // u (1 - a)
    r.d = sub2(r.a, b);
    return r;
}
// interval_fast's exponential branch (u >= 1) on both components, given
// nru = -1/u
__device__ __forceinline__ IntervalE2 interval_exp2(float2 u, float2 nru) {
    const float2 t = mul2(u, pk1(-1.4426950408889634f));  // -u log2(e)
    IntervalE2 r;
    r.e0 = sub2(pk1(1.0f), pk(ex2_approx(t.x), ex2_approx(t.y)));
    r.a = fma2(r.e0, nru, pk1(1.0f));                    // 1 - e0/u
    r.d = mul2(fma2(r.a, pk1(-2.0f), r.e0), nru);         // (2a - e0)/u
    return r;
}
// Per component the branch of interval_fast; a thread whose two intervals
// fall on different sides of u = 1 evaluates both and selects (a NaN u takes
// the exponential branch, as in the scalar form).
__device__ __forceinline__ IntervalE2 interval2(float2 u, float2 nru) {
    const bool sx = u.x < 1.0f, sy = u.y < 1.0f;
    if (sx && sy) return interval_poly2(u);
    if (!sx && !sy) return interval_exp2(u, nru);
    const IntervalE2 p = interval_poly2(u), e = interval_exp2(u, nru);
    IntervalE2 r;
    r.e0 = pk(sx ? p.e0.x : e.e0.x, sy ? p.e0.y : e.e0.y);
    r.a = pk(sx ? p.a.x : e.a.x, sy ? p.a.y : e.a.y);
    r.d = pk(sx ? p.d.x : e.d.x, sy ? p.d.y : e.d.y);
    return r;
}

// State of a pair of characteristics: intensity, optical depth u of the
// interval ending at the current point and -1/u, half optical depth of the
// current point's chord, S at the previous and current points, their difference
// (-1/u is the form the exponential branch and q use).
struct RayP {
    float2 I, u, nru, hc, Sp, Sc, dS;
};

// One point of a pair of characteristics, given c, the pair-packed (chi, S)
// of the next point, and hl, the pair (l/2, l/2) of its chord: the update in
// difference form on both characteristics (the parabolic correction always
// evaluated, its blend weight 0 where the linear form applies), and the
// advance to the next point. Returns the intensities at the current point.
// The two divisions share one reciprocal: with
// X = wf (u + wf), 1/wf = (u + wf)/X and u/(u + wf) = u wf/X, where wf is
// the next interval floored at 1e-15 (so X >= 1e-30 stays a normal FP32
// number; a zero-opacity interval gets q = 0 or blend weight 0).
template <bool PARAB>
__device__ __forceinline__ float2 pair_advance_c(RayP &s, const float4 &c, float2 hl) {
    const float2 hn = mul2(pk(c.x, c.y), hl);
    const float2 Sn = pk(c.z, c.w);
    const float2 dSn = sub2(Sn, s.Sc);
    const float2 w = add2(s.hc, hn);
    const IntervalE2 f = interval2(s.u, s.nru);
    float2 In = fma2(f.e0, sub2(s.Sp, s.I), s.I);
    In = fma2(f.a, s.dS, In);
    const float2 nwf = pk(fminf(-w.x, -1e-15f), fminf(-w.y, -1e-15f));  // -wf
    float2 nrw;
    if (PARAB) {
        const float2 nuw = sub2(nwf, s.u);                 // -(u + wf)
        const float2 X = mul2(nwf, nuw);                   // wf (u + wf)
        const float2 R = pk(rcp_approx(X.x), rcp_approx(X.y));
        nrw = mul2(nuw, R);                                // -1/wf
        const float2 nq = mul2(s.u, nrw);                  // -q
        const float2 fw = mul2(pk(__saturatef(fmaf(-2.0f, s.u.x, 2.0f)),
                                  __saturatef(fmaf(-2.0f, s.u.y, 2.0f))),
                               pk(__saturatef(fmaf(0.5f, nq.x, 2.0f)),
                                  __saturatef(fmaf(0.5f, nq.y, 2.0f))));
        const float2 ns = mul2(mul2(s.u, nwf), R);         // -u/(u + wf)
        const float2 cd = fma2(nq, dSn, s.dS);             // dS - q dSn
        const float2 g = mul2(mul2(fw, f.d), ns);          // -f s d
        In = sub2(In, mul2(g, cd));
    } else {
        nrw = pk(rcp_approx(nwf.x), rcp_approx(nwf.y));
    }
    s.I = In;
    s.u = w;
    s.nru = nrw;
    s.hc = hn;
    s.Sp = s.Sc;
    s.Sc = Sn;
    s.dS = dSn;
    return In;
}

// The last point of a pair (linear form): its intensities.
__device__ __forceinline__ float2 pair_last(const RayP &s) {
    const IntervalE2 f = interval2(s.u, s.nru);
    return fma2(f.a, s.dS, fma2(f.e0, sub2(s.Sp, s.I), s.I));
}

// A pair at its first point: the entry interval has chi_{-1} l_{-1} = 0 and
// S_{-1} = S_0; c = pair-packed (chi, S) of the first point, hl = l/2 of its
// chord, (Ia, Ib) the boundary intensities.
__device__ __forceinline__ void pair_init(RayP &s, const float4 &c, float2 hl, float Ia, float Ib) {
    s.I = pk(Ia, Ib);
    s.hc = mul2(pk(c.x, c.y), hl);
    s.u = s.hc;
    s.Sc = pk(c.z, c.w);
    s.Sp = s.Sc;
    s.dS = pk1(0.0f);
    s.nru = pk(rcp_approx(fminf(-s.hc.x, -1e-15f)), rcp_approx(fminf(-s.hc.y, -1e-15f)));
}

// ---- The same for the four-characteristic kernel, two pairs at a time ----
// The branches are taken by the warp (votes): all intervals below 1 (the
// polynomials, the parabolic blend), all from 1 on (the exponential; the blend
// is 0 there and left out), or both kinds, where both are evaluated. The signs
// are chosen so that every product is a plain fused multiply-add (a packed
// operand has no free negation): the state keeps nD = Sp - Sc, and the interval
// functions are e0, -a and d.
struct RayN {
    float2 I, u, hc, Sp, Sc, nD;
};
struct IntervalN2 {
    float2 e0, na, d;
};
__device__ __forceinline__ IntervalN2 interval_thin(float2 u) {
    float2 np = fma2(pk1(3.569704858819023e-05f), u, pk1(-3.819821577053517e-04f));  // -p(u)
    np = fma2(np, u, pk1(2.770215505734086e-03f));
    np = fma2(np, u, pk1(-1.6664894297719002e-02f));
    np = fma2(np, u, pk1(8.333317935466766e-02f));
    np = fma2(np, u, pk1(-3.333333432674408e-01f));
    const float2 nb = mul2(u, np);             // -b
    const float2 nhu = mul2(u, pk1(-0.5f));
    IntervalN2 r;
    r.na = fma2(nhu, nb, nhu);                 // -u (1 - b) / 2
    r.e0 = fma2(u, r.na, u);                   // u (1 - a)
    r.d = sub2(nb, r.na);                      // a - b
    return r;
}
__device__ __forceinline__ IntervalN2 interval_thick(float2 u) {
    const float2 t = mul2(u, pk1(-1.4426950408889634f));  // -u log2(e)
    IntervalN2 r;
    r.e0 = sub2(pk1(1.0f), pk(ex2_approx(t.x), ex2_approx(t.y)));
    r.na = fma2(r.e0, pk(rcp_approx(u.x), rcp_approx(u.y)), pk1(-1.0f));  // -(1 - e0/u)
    r.d = pk1(0.0f);  // enters with blend weight 0 only
    return r;
}
__device__ __forceinline__ IntervalN2 interval_both(float2 u) {
    const IntervalN2 p = interval_thin(u), e = interval_thick(u);
    const bool x = u.x < 1.0f, y = u.y < 1.0f;
    IntervalN2 r;
    r.e0 = pk(x ? p.e0.x : e.e0.x, y ? p.e0.y : e.e0.y);
    r.na = pk(x ? p.na.x : e.na.x, y ? p.na.y : e.na.y);
    r.d = pk(x ? p.d.x : 0.0f, y ? p.d.y : 0.0f);
    return r;
}
// I + e0 (Sp - I) + a (Sc - Sp)
__device__ __forceinline__ float2 linear_n(const RayN &s, const IntervalN2 &f) {
    return fma2(f.na, s.nD, fma2(f.e0, sub2(s.Sp, s.I), s.I));
}
// The blend weight f given -q
__device__ __forceinline__ float2 blend_n(float2 u, float2 nq) {
    return mul2(pk(__saturatef(fmaf(-2.0f, u.x, 2.0f)), __saturatef(fmaf(-2.0f, u.y, 2.0f))),
                pk(__saturatef(fmaf(0.5f, nq.x, 2.0f)), __saturatef(fmaf(0.5f, nq.y, 2.0f))));
}
// f s d (dS - q dSn), both factors negated, added to In; w the next interval.
// The two divisions share one reciprocal: with X = wf (u + wf), u/wf = u (u +
// wf)/X and u/(u + wf) = u wf/X, wf = w floored at 1e-15 (X stays a normal FP32
// number; a zero-opacity interval gets q = 0 or blend weight 0).
__device__ __forceinline__ float2 parabola_n(const RayN &s, const IntervalN2 &f, float2 w, float2 nDn,
                                             float2 In) {
    const float2 nwf = pk(fminf(-w.x, -1e-15f), fminf(-w.y, -1e-15f));
    const float2 nuw = sub2(nwf, s.u);  // -(u + wf)
    const float2 X = mul2(nwf, nuw);
    const float2 uR = mul2(s.u, pk(rcp_approx(X.x), rcp_approx(X.y)));
    const float2 nq = mul2(nuw, uR), ns = mul2(nwf, uR);  // -u/wf, -u/(u + wf)
    return fma2(mul2(mul2(blend_n(s.u, nq), f.d), ns), fma2(nq, nDn, s.nD), In);
}
// The same ratios, -u/w and -u/(u + w), over the whole range of optical depths: a
// reciprocal each, w floored near the smallest normal number only. Bounded by 4
// (from there on the blend weight is 0) and 1, they are finite for infinite u and w
// and for w = 0 too, so that a zero blend weight leaves nothing. (From one
// reciprocal of w (u + w), as above, the floor has to be 1e-15, below which the
// parabola of a transparent cell is lost: there up to 0.3 % of its emission.)
__device__ __forceinline__ void ratios_n(float2 u, float2 w, float2 &nq, float2 &ns) {
    const float2 nw = pk(fminf(-w.x, -1e-37f), fminf(-w.y, -1e-37f));
    const float2 nuw = sub2(nw, u);
    const float2 q = mul2(u, pk(rcp_approx(nw.x), rcp_approx(nw.y)));
    const float2 s = mul2(u, pk(rcp_approx(nuw.x), rcp_approx(nuw.y)));
    nq = pk(fmaxf(q.x, -4.0f), fmaxf(q.y, -4.0f));
    ns = pk(fmaxf(s.x, -1.0f), fmaxf(s.y, -1.0f));
}
// One point of two pairs (all lanes of the warp): s[j].I becomes the
// intensities at the current point, the rest moves to the next point (c[j] its
// pair-packed (chi, S), hl its (l/2, l/2)).
template <bool PARAB>
__device__ __forceinline__ void quad_advance(RayN (&s)[2], const float4 (&c)[2], float2 hl) {
    float2 hn[2], Sn[2], nDn[2], w[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        hn[j] = mul2(pk(c[j].x, c[j].y), hl);
        Sn[j] = pk(c[j].z, c[j].w);
        nDn[j] = sub2(s[j].Sc, Sn[j]);
        w[j] = add2(s[j].hc, hn[j]);
    }
    const float hi = fmaxf(fmaxf(s[0].u.x, s[0].u.y), fmaxf(s[1].u.x, s[1].u.y));
    if (__all_sync(0xffffffffu, hi < 1.0f)) {
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const IntervalN2 f = interval_thin(s[j].u);
            const float2 In = linear_n(s[j], f);
            s[j].I = PARAB ? parabola_n(s[j], f, w[j], nDn[j], In) : In;
        }
    } else {
        const float lo = fminf(fminf(s[0].u.x, s[0].u.y), fminf(s[1].u.x, s[1].u.y));
        if (__all_sync(0xffffffffu, lo >= 1.0f)) {
#pragma unroll
            for (int j = 0; j < 2; ++j) s[j].I = linear_n(s[j], interval_thick(s[j].u));
        } else {
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const IntervalN2 f = interval_both(s[j].u);
                const float2 In = linear_n(s[j], f);
                s[j].I = PARAB ? parabola_n(s[j], f, w[j], nDn[j], In) : In;
            }
        }
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        s[j].u = w[j];
        s[j].hc = hn[j];
        s[j].Sp = s[j].Sc;
        s[j].Sc = Sn[j];
        s[j].nD = nDn[j];
    }
}
// A pair at its first point: the entry interval has chi_{-1} l_{-1} = 0 and
// S_{-1} = S_0.
__device__ __forceinline__ void quad_start(RayN &s, const float4 &c, float2 hl, float Ia, float Ib) {
    s.I = pk(Ia, Ib);
    s.hc = mul2(pk(c.x, c.y), hl);
    s.u = s.hc;
    s.Sc = pk(c.z, c.w);
    s.Sp = s.Sc;
    s.nD = pk1(0.0f);
}

// ---- The same with the weights of Lambda*'s window ----
// E = e^-u, al, be and ga: the derivatives of I_k by I_{k-1}, S_{k-1}, S_k and
// S_{k+1} over its own interval.
struct WeightsN {
    float2 E, al, be, ga;
};
// Interval functions with E and al of the linear form: below 1 from the 9-term
// series of p(u), as in the one-characteristic kernel with Lambda*, and e0 - a in
// the form u ((1 + b)/2 - a), which does not cancel.
__device__ __forceinline__ IntervalN2 interval_thin_w(float2 u, WeightsN &w) {
    float2 np = pk1((float)(-2.0 / 39916800.0));  // -p(u), the Taylor polynomial
    np = fma2(np, u, pk1((float)(2.0 / 3628800.0)));
    np = fma2(np, u, pk1((float)(-2.0 / 362880.0)));
    np = fma2(np, u, pk1((float)(2.0 / 40320.0)));
    np = fma2(np, u, pk1((float)(-2.0 / 5040.0)));
    np = fma2(np, u, pk1((float)(2.0 / 720.0)));
    np = fma2(np, u, pk1((float)(-2.0 / 120.0)));
    np = fma2(np, u, pk1((float)(2.0 / 24.0)));
    np = fma2(np, u, pk1((float)(-2.0 / 6.0)));
    const float2 nb = mul2(u, np);
    const float2 nhu = mul2(u, pk1(-0.5f));
    IntervalN2 r;
    r.na = fma2(nhu, nb, nhu);
    r.e0 = fma2(u, r.na, u);
    r.d = sub2(nb, r.na);
    w.E = sub2(pk1(1.0f), r.e0);
    w.al = mul2(u, add2(fma2(nb, pk1(-0.5f), pk1(0.5f)), r.na));
    return r;
}
__device__ __forceinline__ IntervalN2 interval_thick_w(float2 u, WeightsN &w) {
    const float2 t = mul2(u, pk1(-1.4426950408889634f));
    w.E = pk(ex2_approx(t.x), ex2_approx(t.y));
    const float2 ru = pk(rcp_approx(u.x), rcp_approx(u.y));
    IntervalN2 r;
    r.e0 = sub2(pk1(1.0f), w.E);
    r.na = fma2(r.e0, ru, pk1(-1.0f));
    r.d = pk1(0.0f);
    w.al = sub2(mul2(r.e0, ru), w.E);
    return r;
}
// f, w: the thin form's; the thick form's where u >= 1
__device__ __forceinline__ IntervalN2 select_w(float2 u, IntervalN2 f, WeightsN &w) {
    WeightsN h;
    const IntervalN2 e = interval_thick_w(u, h);
    const bool x = u.x < 1.0f, y = u.y < 1.0f;
    IntervalN2 r;
    r.e0 = pk(x ? f.e0.x : e.e0.x, y ? f.e0.y : e.e0.y);
    r.na = pk(x ? f.na.x : e.na.x, y ? f.na.y : e.na.y);
    r.d = pk(x ? f.d.x : 0.0f, y ? f.d.y : 0.0f);
    w.E = pk(x ? w.E.x : h.E.x, y ? w.E.y : h.E.y);
    w.al = pk(x ? w.al.x : h.al.x, y ? w.al.y : h.al.y);
    return r;
}
// quad_advance with the weights; false when all intervals are thick (ga = 0).
template <bool PARAB>
__device__ __forceinline__ bool quad_advance_w(RayN (&s)[2], const float4 (&c)[2], float2 hl,
                                               WeightsN (&wt)[2]) {
    float2 hn[2], Sn[2], nDn[2], w[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        hn[j] = mul2(pk(c[j].x, c[j].y), hl);
        Sn[j] = pk(c[j].z, c[j].w);
        nDn[j] = sub2(s[j].Sc, Sn[j]);
        w[j] = add2(s[j].hc, hn[j]);
    }
    const float lo = fminf(fminf(s[0].u.x, s[0].u.y), fminf(s[1].u.x, s[1].u.y));
    const bool all_thick = __all_sync(0xffffffffu, lo >= 1.0f);
    if (all_thick) {
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const IntervalN2 f = interval_thick_w(s[j].u, wt[j]);
            wt[j].be = sub2(pk1(0.0f), f.na);
            wt[j].ga = pk1(0.0f);
            s[j].I = linear_n(s[j], f);
        }
    } else {
        const float hi = fmaxf(fmaxf(s[0].u.x, s[0].u.y), fmaxf(s[1].u.x, s[1].u.y));
        const bool all_thin = __all_sync(0xffffffffu, hi < 1.0f);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const float2 u = s[j].u;
            IntervalN2 f = interval_thin_w(u, wt[j]);
            if (!all_thin) f = select_w(u, f, wt[j]);
            float2 In = linear_n(s[j], f);
            float2 g = pk1(0.0f), qg = pk1(0.0f);  // -f s d and q f s d
            if (PARAB) {
                float2 nq, ns;
                ratios_n(u, w[j], nq, ns);
                g = mul2(mul2(blend_n(u, nq), f.d), ns);
                qg = mul2(nq, g);
                In = fma2(g, fma2(nq, nDn[j], s[j].nD), In);
            }
            wt[j].al = add2(wt[j].al, g);
            wt[j].be = sub2(qg, add2(f.na, g));
            wt[j].ga = sub2(pk1(0.0f), qg);
            s[j].I = In;
        }
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        s[j].u = w[j];
        s[j].hc = hn[j];
        s[j].Sp = s[j].Sc;
        s[j].Sc = Sn[j];
        s[j].nD = nDn[j];
    }
    return !all_thick;
}
// The last point's (linear form).
__device__ __forceinline__ void quad_last_w(RayN &s, WeightsN &w) {
    const IntervalN2 f = select_w(s.u, interval_thin_w(s.u, w), w);
    w.be = sub2(pk1(0.0f), f.na);
    w.ga = pk1(0.0f);
    s.I = linear_n(s, f);
}

// ---- One characteristic, two successive points at a time ----
// Components .x and .y are points k and k + 1 of the same characteristic: all
// that does not depend on the intensity is evaluated for both in one packed
// instruction stream, and only I + e0 (Sp - I) + B remains in sequence. The
// chain a point waits for is halved, which is what counts where few warps are
// left (small grids, scattered rays). Against the point-by-point form (one
// packed lane unused): box 33^3, 128 angles 107 -> 88 us, shell 65 x 33 x 65,
// 512 angles 2.17 -> 2.07 ms, eight batched wavelengths on 33^3 134 -> 127 ms a
// solve; large boxes gain nothing (97^3 4.74 ms both), but they run four
// characteristics a thread.
struct RayT {
    float I, u, hc, Sp, Sc;
};
__device__ __forceinline__ void twin_start(RayT &s, float2 cs, float hl, float I0) {
    s.I = I0;
    s.hc = cs.x * hl;
    s.u = s.hc;  // the entry interval: chi_{-1} l_{-1} = 0
    s.Sc = cs.y;
    s.Sp = cs.y;  // S_{-1} = S_0
}
// e0 and B = a (Sc - Sp) + f s d (dS - q dSn) of two points with intervals u,
// the next ones w, nD = Sp - Sc and nDn = Sc - Sn.
template <bool PARAB>
__device__ __forceinline__ void twin_coef(float2 u, float2 w, float2 nD, float2 nDn, float2 &e0,
                                          float2 &B) {
    IntervalN2 f;
    const bool tx = !(u.x < 1.0f), ty = !(u.y < 1.0f);
    if (tx && ty) {
        f = interval_thick(u);
        e0 = f.e0;
        B = mul2(f.na, nD);
        return;
    }
    f = tx || ty ? interval_both(u) : interval_thin(u);
    e0 = f.e0;
    B = mul2(f.na, nD);
    if (PARAB) {
        float2 nq, ns;
        ratios_n(u, w, nq, ns);
        B = fma2(mul2(mul2(blend_n(u, nq), f.d), ns), fma2(nq, nDn, nD), B);
    }
}
// Points k and k + 1, given (chi, S) of points k + 1 and k + 2 and their half
// chords; moves on to k + 2 and returns the two intensities.
template <bool PARAB>
__device__ __forceinline__ float2 twin_advance(RayT &s, float2 c1, float2 c2, float l1, float l2) {
    const float2 h = mul2(pk(c1.x, c2.x), pk(l1, l2));
    const float2 w = add2(pk(s.hc, h.x), h);
    const float2 nD = sub2(pk(s.Sp, s.Sc), pk(s.Sc, c1.y));
    const float2 nDn = pk(nD.y, c1.y - c2.y);
    float2 e0, B;
    twin_coef<PARAB>(pk(s.u, w.x), w, nD, nDn, e0, B);
    const float I1 = fmaf(e0.x, s.Sp - s.I, s.I) + B.x;
    const float I2 = fmaf(e0.y, s.Sc - I1, I1) + B.y;
    s.I = I2;
    s.u = w.y;
    s.hc = h.y;
    s.Sp = c1.y;
    s.Sc = c2.y;
    return pk(I1, I2);
}
// Point k alone; then the last point (linear form).
template <bool PARAB>
__device__ __forceinline__ float twin_single(RayT &s, float2 c1, float l1) {
    const float h = c1.x * l1, w = s.hc + h, nD = s.Sp - s.Sc, nDn = s.Sc - c1.y;
    float2 e0, B;
    twin_coef<PARAB>(pk1(s.u), pk1(w), pk1(nD), pk1(nDn), e0, B);
    s.I = fmaf(e0.x, s.Sp - s.I, s.I) + B.x;
    s.u = w;
    s.hc = h;
    s.Sp = s.Sc;
    s.Sc = c1.y;
    return s.I;
}
__device__ __forceinline__ float twin_last(RayT &s) {
    const IntervalE f = interval_fast(s.u, __fdividef(1.0f, s.u));
    s.I = fmaf(f.a, s.Sc - s.Sp, fmaf(f.e0, s.Sp - s.I, s.I));
    return s.I;
}

// A whole characteristic of K points from entry intensity I0: record k gives
// (offset, J weight, l/2), chiS + base the gathers, Jd + base the reductions
// (W0, W1: integer widening of even and odd points' contributions). The next
// two points' records are loaded a trip ahead; loading their gathers ahead as
// well changed nothing on the box (33^3 96 us either way) and cost the shell 1 %.
template <bool PARAB, bool W0, bool W1>
__device__ __forceinline__ void twin_ray(const float4 *__restrict__ rec, int K,
                                         const float2 *__restrict__ chiS, double *__restrict__ Jd,
                                         float I0) {
    RayT s;
    float4 r0 = __ldg(rec);
    int v0 = __float_as_int(r0.x);
    twin_start(s, chiS[v0], r0.z, I0);
    int k = 0;
    float4 r1 = __ldg(rec + min(1, K - 1)), r2 = __ldg(rec + min(2, K - 1));
    for (; k + 2 < K; k += 2) {
        const int v1 = __float_as_int(r1.x), v2 = __float_as_int(r2.x);
        const float2 c1 = chiS[v1], c2 = chiS[v2];
        const float4 q1 = __ldg(rec + min(k + 3, K - 1)), q2 = __ldg(rec + min(k + 4, K - 1));
        const float2 I = twin_advance<PARAB>(s, c1, c2, r1.z, r2.z);
        atomicAdd(Jd + v0, to_f64<W0>(r0.y * I.x));
        atomicAdd(Jd + v1, to_f64<W1>(r1.y * I.y));
        r0 = r2;
        v0 = v2;
        r1 = q1;
        r2 = q2;
    }
    if (k + 1 < K) {
        const int v1 = __float_as_int(r1.x);
        atomicAdd(Jd + v0, to_f64<W0>(r0.y * twin_single<PARAB>(s, chiS[v1], r1.z)));
        r0 = r1;
        v0 = v1;
    }
    atomicAdd(Jd + v0, to_f64<W1>(r0.y * twin_last(s)));
    if (!(fabsf(s.I) <= 3.402823466e38f))  // non-finite: make J NaN
        atomicAdd(Jd + v0, __longlong_as_double(0x7ff8000000000000LL));
}

// FP32 contribution to FP64 for a reduction: CONV 1 integer moves, else the
// conversion instruction.
template <int CONV> __device__ __forceinline__ double pair_widen(float x) {
    return CONV == 1 ? widen_f32(x) : (double)x;
}

}  // namespace rt3d
