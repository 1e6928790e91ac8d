// Formal solution J = Lambda S (Eq. frmsol) by long characteristics on the
// periodic Cartesian box, with the optional non-local Lambda* band (Sec. 4:
// "computing the Lambda* operator (only in the first iteration)"), following
// the per-slot steps of the paper's Listing 1: gather the previous and next S
// and chi, compute dtau, compute alpha/beta/gamma, fix up at the boundary,
// store Lambda* data, compute Delta I and exp(-dtau).
//
// Mapping: one thread integrates one characteristic (all nx*ny
// characteristics of a solid angle are translates of the cached one, so the
// threads of a warp walk neighbouring voxels of the same layer in lock step:
// the (chi, S) gathers of a warp hit one or two 128-byte lines). Blocks are
// (ray bundle, solid angle) with angles ordered longest first. Contributions
// are accumulated in FP64 (red.global.add.f64), also in the FP32 mode.
//
// Interval functions. For the interval of optical depth u between points
// k-1 and k, with e0 = 1 - e^-u, e1 = u - e0, e2 = u^2 - 2 e1 (Olson &
// Kunasz 1987), the kernel works with
//   a = e1/u, b = e2/u^2, a0 = e0 - a, d = a - b,
// which stay O(1) or O(u) at both ends of the range. Small u: e2 = u^3 p(u)
// with p(u) = 2 sum_m (-1)^m u^m / (m+3)!, from the Taylor series of exp,
// then a = u (1 - b)/2, e0 = u (1 - a), E = 1 - e0. Large u: E = exp(-u),
// a = 1 - e0/u, a0 = (1 - (1+u) E)/u, d = (2a - e0)/u.
// Coefficients (s = u/(u+w), q = u/w, w the next interval):
//   linear:    alpha = a0, beta = a, gamma = 0
//   parabolic: beta + gamma = a + f s d, gamma = -f q s d, alpha = a0 - f s d,
// where f = clamp(2 - 2u, 0, 1) clamp(2 - q/2, 0, 1) blends the Olson-Kunasz
// parabola (f = 1: u <= 1/2 and q <= 2) continuously into the linear form
// (f = 0: u >= 1 or q >= 4), which keeps every weight of an optically thick
// interval non-negative (the OS matrix stays diagonally dominant),
// and I_k = E I_{k-1} + alpha S_{k-1} + (beta+gamma) S_k + gamma (S_{k+1} - S_k)
// so that large |gamma| (short next interval) multiplies a difference instead
// of cancelling between two products. The kernels without Lambda* use the
// same update in difference form, I_k = I_{k-1} + e0 (S_{k-1} - I_{k-1}) +
// a (S_k - S_{k-1}) + f s d ((S_k - S_{k-1}) - q (S_{k+1} - S_k)), which
// needs neither E nor a0. The last point of a characteristic is
// linear; the entry point has S_{-1} = S_0 and chi_{-1} l_{-1} = 0.
#include <algorithm>

#include "fs_step.cuh"
#include "fs64_step.cuh"

namespace rt3d {

namespace {

template <typename R> struct V2;
template <> struct V2<float> { using T = float2; };
template <> struct V2<double> { using T = double2; };

// A contribution as the FP64 value its reduction adds: FP32 values widened by
// integer moves (widen_f32), keeping the FP64 pipe free.
__device__ __forceinline__ double red_value(float x) { return widen_f32(x); }
__device__ __forceinline__ double red_value(double x) { return x; }

// Taylor coefficients of p(u) = e2/u^3 = 2 sum_m (-1)^m u^m / (m+3)!.
constexpr double fact(int n) { return n <= 1 ? 1.0 : n * fact(n - 1); }
constexpr double pc(int m) { return (m % 2 ? -2.0 : 2.0) / fact(m + 3); }
template <int M> struct PCf { static constexpr float v = (float)pc(M); };

struct IntervalF {
    float E, a0, a, d;
};

__device__ __forceinline__ IntervalF interval(float u, const unsigned long long *) {
    IntervalF r;
    if (u < 1.0f) {
        // Horner, m = 8 .. 0: truncation < 1.3e-8 relative at u = 1
        float p = PCf<8>::v;
        p = fmaf(p, u, PCf<7>::v);
        p = fmaf(p, u, PCf<6>::v);
        p = fmaf(p, u, PCf<5>::v);
        p = fmaf(p, u, PCf<4>::v);
        p = fmaf(p, u, PCf<3>::v);
        p = fmaf(p, u, PCf<2>::v);
        p = fmaf(p, u, PCf<1>::v);
        p = fmaf(p, u, PCf<0>::v);
        const float b = u * p;
        const float a = 0.5f * u * (1.0f - b);
        const float e0 = u * (1.0f - a);
        r.E = 1.0f - e0;
        r.a = a;
        r.a0 = e0 - a;
        r.d = a - b;
    } else {
        const float E = __expf(-u);
        const float ru = __fdividef(1.0f, u);
        const float e0 = 1.0f - E;
        const float a = fmaf(-e0, ru, 1.0f);
        r.E = E;
        r.a = a;
        r.a0 = fmaf(-(1.0f + u), E, 1.0f) * ru;
        r.d = fmaf(2.0f, a, -e0) * ru;
    }
    return r;
}

__device__ __forceinline__ IntervalD interval(double u, const unsigned long long *tab) {
    return interval64_w(u, tab);
}

template <typename R> __device__ __forceinline__ R div_fast(R x, R y);
template <> __device__ __forceinline__ float div_fast<float>(float x, float y) {
    return __fdividef(x, y);
}
template <> __device__ __forceinline__ double div_fast<double>(double x, double y) {
    return x * recip64(y);
}

template <typename R> __device__ __forceinline__ R clamp01(R x) {
    return x < R(0) ? R(0) : (x > R(1) ? R(1) : x);
}

__device__ __forceinline__ int voxel_of(uint32_t c, int x0, int y0, int nx, int ny) {
    int x = x0 + (int)(c & 0x7ffu);
    int y = y0 + (int)((c >> 11) & 0x7ffu);
    if (x >= nx) x -= nx;
    if (y >= ny) y -= ny;
    return x + nx * (y + ny * (int)(c >> 22));
}

// index of the same point in the 2 x 2-replicated packed (chi, S) array
__device__ __forceinline__ int rep_of(uint32_t c, int x0, int y0, int nx, int ny) {
    return (int)rep_index(x0 + (int)(c & 0x7ffu), y0 + (int)((c >> 11) & 0x7ffu), (int)(c >> 22),
                          nx, ny);
}

// One characteristic a thread, with Lambda* (FP64: the FP64 pipe bounds it; 33^3
// voxels, 128 angles 3.24 ms with the library's exp, divisions and an 18-term
// series, 1.98 ms with interval64_w and recip64; parabolic 4.98 -> 3.23 ms. Error of
// Lambda* against 64 bits 7.8e-16 -> 7.1e-16).
template <typename R, bool PARAB>
__global__ void __launch_bounds__(128) fs_kernel(FsParams p) {
    using R2 = typename V2<R>::T;
    __shared__ unsigned long long tab[64];
    if (sizeof(R) == 8) exp_table(tab);
    const int nray = p.nx * p.ny;
    const int ray = blockIdx.x * blockDim.x + threadIdx.x;
    if (ray >= nray) return;
    const int o = p.order[blockIdx.y];
    const int x0 = ray % p.nx, y0 = ray / p.nx;
    const long long t0 = p.toff[o];
    const int K = p.tlen[o];
    const uint32_t *__restrict__ code = p.code + t0;
    const R *__restrict__ len = static_cast<const R *>(p.len) + t0;
    const R *__restrict__ cw = static_cast<const R *>(p.cw) + t0;
    const R2 *__restrict__ chiS = static_cast<const R2 *>(p.chiS);
    const long long N = (long long)nray * p.nz;

    double I0 = 0.0;
    if (!p.homogeneous)
        I0 = entry_intensity(p.up[o], p.mu, o, ray, p.top_face, p.bot_face, p.bot_grad, p.I_top,
                             p.I_bot);
    R I = (R)I0;

    int v = voxel_of(__ldg(code), x0, y0, p.nx, p.ny);
    R2 cs = chiS[rep_of(__ldg(code), x0, y0, p.nx, p.ny)];
    R chil_c = cs.x * __ldg(len);
    R chil_p = R(0);
    R S_c = cs.y, S_p = cs.y;
    R ring[kWin];
#pragma unroll
    for (int i = 0; i < kWin; ++i) ring[i] = R(0);

    for (int k = 0; k < K; ++k) {
        const R u = R(0.5) * (chil_p + chil_c);
        const auto f = interval(u, tab);
        const bool has_next = (k + 1 < K);
        int vn = v;
        R chil_n = R(0), S_n = S_c;
        if (has_next) {
            const uint32_t cn = __ldg(code + k + 1);
            vn = voxel_of(cn, x0, y0, p.nx, p.ny);
            const R2 c2 = chiS[rep_of(cn, x0, y0, p.nx, p.ny)];
            chil_n = c2.x * __ldg(len + k + 1);
            S_n = c2.y;
        }
        R al = f.a0, bg = f.a, ga = R(0);
        if (PARAB && has_next) {
            const R w = R(0.5) * (chil_c + chil_n);
            if (w > R(0)) {
                const R q = div_fast(u, w);
                const R fw = clamp01(R(2) - R(2) * u) * clamp01(R(2) - R(0.5) * q);
                if (fw > R(0)) {
                    const R sd = fw * div_fast(u, u + w) * f.d;
                    bg = f.a + sd;
                    ga = -q * sd;
                    al = f.a0 - sd;
                }
            }
        }
        I = f.E * I + al * S_p + bg * S_c + ga * (S_n - S_c);
        const R c = __ldg(cw + k);
        atomicAdd(p.J + v, red_value(c * I));
        // ring[i] = dI_k / dS_{k-7+i}
#pragma unroll
        for (int i = 0; i < kWin - 1; ++i) ring[i] = f.E * ring[i + 1];
        const R be = bg - ga;
        if (k == 0) ring[7] += al;  // S_{-1} = S_0 at the entry point
        else ring[6] += al;
        ring[7] += be;
        ring[8] = ga;
        const uint64_t wc = __ldg(reinterpret_cast<const unsigned long long *>(p.win + t0 + k));
#pragma unroll
        for (int i = 0; i < kWin; ++i) {
            const unsigned dc = (unsigned)(wc >> (5 * i)) & 31u;
            if (dc != kWinNone) atomicAdd(p.lstar + (long long)dc * N + v, red_value(c * ring[i]));
        }
        chil_p = chil_c;
        chil_c = chil_n;
        S_p = S_c;
        S_c = S_n;
        v = vn;
    }
    // the widening does not carry a non-finite value: a non-finite intensity
    // (it persists along the recurrence) makes J of the last point NaN
    if (!(fabs((double)I) <= 1.79769313486231570e308))
        atomicAdd(p.J + v, __longlong_as_double(0x7ff8000000000000LL));
}

// FP32 formal solution without Lambda* (every iteration after the first),
// one characteristic per thread, two points at a time (twin_ray; the
// autotuner's pick on small grids). Per point: one 8-byte (chi, S) gather, the
// interval arithmetic, and one FP64 reduction (red.global.add.f64) into the
// replicated J, folded afterwards; the FP32 contribution is widened by integer
// moves, by the conversion instruction (which runs on the FP64 pipe), or
// alternately by both (the autotuner picks). FP64 accumulation keeps the
// operator's error at the level of its FP32 arithmetic (an FP32 reduction
// over ~10^3 contributions per voxel and angle group was measured to cost
// the refinement a fourth FP64 formal solution and 60 more FP32 ones at
// 129^3).
// CONV: how FP32 contributions become FP64 for the reduction: 0 the
// conversion instruction (FP64 pipe), 1 integer moves, 2 alternating between
// the two from point to point (both pipes half loaded).
template <bool PARAB, int CONV>
__global__ void __launch_bounds__(256) fs_fast_kernel(FsParams p) {
    const int nray = p.nx * p.ny;
    const int ray = blockIdx.x * blockDim.x + threadIdx.x;
    if (ray >= nray) return;
    const int o = p.order[blockIdx.y];
    const int K = p.tlen[o];
    const float4 *__restrict__ rec = p.rec32 + p.toff[o];
    const float2 *__restrict__ chiS = static_cast<const float2 *>(p.chiS);
    double *__restrict__ Jd = p.Jrep;
    constexpr bool W0 = CONV == 1, W1 = CONV >= 1;

    const int base = ray % p.nx + 2 * p.nx * (ray / p.nx);
    double I0 = 0.0;
    if (!p.homogeneous)
        I0 = entry_intensity(p.up[o], p.mu, o, ray, p.top_face, p.bot_face, p.bot_grad, p.I_top,
                             p.I_bot);
    twin_ray<PARAB, W0, W1>(rec, K, chiS + base, Jd + base, (float)I0);
}

// FP32 formal solution without Lambda*, two characteristics per thread in
// packed FP32x2 arithmetic (pair_advance_c): face cells (x0, y0) and
// (x0, y0 + 1) with y0 even. Both sit at the same offset of the cached
// characteristic, so one 16-byte load of the pair-packed (chi, S) (p.pairs)
// serves both, and the step record (one 16-byte broadcast load per point) is
// shared. Lanes of a warp take consecutive x0 of one row pair: the gathers of
// a warp cover one contiguous run of 16-byte elements. Per point and
// characteristic one FP64 reduction into the replicated J, as in
// fs_fast_kernel (CONV: 0 both contributions widened by the conversion
// instruction, 1 both by integer moves, 2 the first by conversion and the
// second by integer moves).
// The next point's step record and pair-packed (chi, S) are loaded one point
// ahead, so the gather's L2 latency overlaps the arithmetic of a point.
template <bool PARAB, int CONV>
__global__ void __launch_bounds__(256) fs_pair_kernel(FsParams p) {
    const int nyh = (p.ny + 1) >> 1;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= p.nx * nyh) return;
    const int o = p.order[blockIdx.y];
    const int K = p.tlen[o];
    const float4 *__restrict__ rec = p.rec32 + p.toff[o];
    const int x0 = t % p.nx, y0 = 2 * (t / p.nx);
    const bool lb = y0 + 1 < p.ny;  // row y0 + 1 exists (ny odd: not in the last pair)
    const int base = x0 + 2 * p.nx * y0;
    const float4 *__restrict__ P = p.pairs + base;
    double *__restrict__ Ja = p.Jrep + base;
    double *__restrict__ Jb = Ja + 2 * p.nx;
    constexpr int CA = CONV == 1 ? 1 : 0, CB = CONV >= 1 ? 1 : 0;

    float Ia = 0.0f, Ib = 0.0f;
    if (!p.homogeneous) {
        const bool up = p.up[o];
        const int fa = y0 * p.nx + x0;
        Ia = (float)entry_intensity(up, p.mu, o, fa, p.top_face, p.bot_face, p.bot_grad, p.I_top,
                                    p.I_bot);
        if (lb)
            Ib = (float)entry_intensity(up, p.mu, o, fa + p.nx, p.top_face, p.bot_face, p.bot_grad,
                                        p.I_top, p.I_bot);
    }
    RayP s;
    const float4 r0 = __ldg(rec);
    int vc = __float_as_int(r0.x);
    pair_init(s, __ldg(P + vc), pk(r0.z, r0.w), Ia, Ib);
    float cwc = r0.y;
    float4 rq = __ldg(rec + (K > 1 ? 1 : 0));
    float4 cq = __ldg(P + __float_as_int(rq.x));
#pragma unroll 2
    for (int k = 1; k < K; ++k) {
        const float4 rn = rq, cn = cq;
        rq = __ldg(rec + (k + 1 < K ? k + 1 : k));
        cq = __ldg(P + __float_as_int(rq.x));
        const float2 cI = mul2(pair_advance_c<PARAB>(s, cn, pk(rn.z, rn.w)), pk1(cwc));
        atomicAdd(Ja + vc, pair_widen<CA>(cI.x));
        if (lb) atomicAdd(Jb + vc, pair_widen<CB>(cI.y));
        vc = __float_as_int(rn.x);
        cwc = rn.y;
    }
    // the last point: linear form
    const float2 In = pair_last(s);
    const float2 cI = mul2(In, pk1(cwc));
    const double nan = __longlong_as_double(0x7ff8000000000000LL);
    atomicAdd(Ja + vc, pair_widen<CA>(cI.x));
    if (!(fabsf(In.x) <= 3.402823466e38f)) atomicAdd(Ja + vc, nan);  // non-finite: make J NaN
    if (lb) {
        atomicAdd(Jb + vc, pair_widen<CB>(cI.y));
        if (!(fabsf(In.y) <= 3.402823466e38f)) atomicAdd(Jb + vc, nan);
    }
}

// ---- Four characteristics per thread, the J contributions of successive
// points summed in registers before the FP64 reduction.
//
// One FP64 reduction a segment is what bounds the kernels above: 6.3e11 a
// second at 129^3, and 5.9e11 to 7e11 whatever their width in a loop of
// reductions alone. All characteristics of an angle are translates: when they
// step along an axis, each enters the voxel that its neighbour on that axis
// leaves. So a thread takes four neighbours along the axis the angle steps along
// most (rows; x0 or y0 + 0..3), keeps an FP32 sum for the voxel of each row, and
// on a step along that axis moves the sums one row over and reduces only the
// one whose voxel no row holds any more; any other step reduces all four. On
// average 0.54 reductions a segment are left. The lanes take consecutive cells
// of the other axis, so that loads and reductions stay contiguous: the angles
// that step along x more than along y run on arrays with x and y exchanged
// (pairs_t, Jrep_t, offsets of their records).
// Measured against the pair kernel: 129^3, 2048 angles 45.8 -> 38.1 ms (7.7e11
// segments/s), 97^3, 512 angles 4.23 -> 3.42 ms, 65^3 1.35 -> 1.18 ms; at 33^3,
// 128 angles 0.166 against 0.088 ms (one per thread), where the longest
// characteristic's latency counts. Bound by FP32 issue: 80 warp instructions per
// point of two warps' worth of segments (99 without the votes and the sums), 35
// of them FP32, 66 % of the issue slots at 24 warps a SM (80 registers).
// A sum holds at most the contributions of the rows that pass its voxel at
// successive points. Rows past the face (its last quad) are integrated like the
// others; their sums are never reduced and never move into an existing row.
constexpr int kQuadOffBits = 29;
constexpr unsigned kQuadOffMask = (1u << kQuadOffBits) - 1u;

template <bool PARAB, int CONV>
__global__ void __launch_bounds__(256, 3) fs_quad_kernel(FsParams p) {
    const int o = p.order4[blockIdx.y];
    const bool tr = p.swap[o];
    const int nm = tr ? p.ny : p.nx, nd = tr ? p.nx : p.ny;  // lanes' axis, rows' axis
    const int nlive = nm * ((nd + 3) >> 2);
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t - (threadIdx.x & 31) >= nlive) return;  // the whole warp is past the face
    const int tt = min(t, nlive - 1);
    const int K = p.tlen[o];
    const float4 *__restrict__ rec = p.rec4 + p.toff[o];
    const int m0 = tt % nm, d0 = 4 * (tt / nm);
    const int rowp = 2 * nm;  // one replicated row
    const int base = m0 + rowp * d0;
    // the second pair, or the first one's data again where it is past the face
    const float4 *__restrict__ P0 = (tr ? p.pairs_t : p.pairs) + base;
    const float4 *__restrict__ P1 = d0 + 2 < nd ? P0 + 2 * rowp : P0;
    double *__restrict__ J0 = (tr ? p.Jrep_t : p.Jrep) + base;
    // the quad's last existing row (-1: a lane past the face)
    const int rtop = t < nlive ? min(3, nd - 1 - d0) : -1;

    float Iv[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    if (!p.homogeneous) {
        const bool up = p.up[o];
#pragma unroll
        for (int r = 0; r < 4; ++r)
            if (d0 + r < nd) {
                const int f = tr ? d0 + r + p.nx * m0 : m0 + p.nx * (d0 + r);
                Iv[r] = (float)entry_intensity(up, p.mu, o, f, p.top_face, p.bot_face, p.bot_grad,
                                               p.I_top, p.I_bot);
            }
    }
    RayN s[2];
    const float4 r0 = __ldg(rec);
    int vc = (int)(__float_as_uint(r0.x) & kQuadOffMask);
    quad_start(s[0], __ldg(P0 + vc), pk(r0.z, r0.w), Iv[0], Iv[1]);
    quad_start(s[1], __ldg(P1 + vc), pk(r0.z, r0.w), Iv[2], Iv[3]);
    float2 A01 = pk1(0.0f), A23 = pk1(0.0f);  // sums of the rows' current voxels
    float cwc = r0.y;
    auto reduce_all = [&](double *__restrict__ j) {
        if (rtop >= 0) atomicAdd(j, pair_widen<CONV>(A01.x));
        if (rtop >= 1) atomicAdd(j + rowp, pair_widen<CONV>(A01.y));
        if (rtop >= 2) atomicAdd(j + 2 * rowp, pair_widen<CONV>(A23.x));
        if (rtop >= 3) atomicAdd(j + 3 * rowp, pair_widen<CONV>(A23.y));
    };
    // the next point's record and data are loaded one point ahead
    float4 rn = __ldg(rec + 1);
    float4 c[2] = {__ldg(P0 + (__float_as_uint(rn.x) & kQuadOffMask)),
                   __ldg(P1 + (__float_as_uint(rn.x) & kQuadOffMask))};
// three points per trip: the carried values rotate with that period
#pragma unroll 3
    for (int k = 1; k < K; ++k) {
        const float4 rq = __ldg(rec + k + 1);
        const unsigned oq = __float_as_uint(rq.x) & kQuadOffMask;
        const float4 q[2] = {__ldg(P0 + oq), __ldg(P1 + oq)};
        quad_advance<PARAB>(s, c, pk(rn.z, rn.w));
        A01 = fma2(s[0].I, pk1(cwc), A01);
        A23 = fma2(s[1].I, pk1(cwc), A23);
        // the move from the current points (offset vc) to the next
        const unsigned type = __float_as_uint(rn.x) >> kQuadOffBits;
        double *__restrict__ j = J0 + vc;
        if (type == 0u) {  // one row up: row 0's voxel leaves
            if (rtop >= 0) atomicAdd(j, pair_widen<CONV>(A01.x));
            A01 = pk(A01.y, A23.x);
            A23 = pk(A23.y, 0.0f);
            if (rtop < 3) {  // the last existing row enters a voxel no sum of this lane holds
                if (rtop == 2) A23.x = 0.0f;
                else if (rtop == 1) A01.y = 0.0f;
                else A01.x = 0.0f;
            }
        } else if (type == 1u) {  // one row down: the last existing row's voxel leaves
            const float v = rtop == 3 ? A23.y : (rtop == 2 ? A23.x : (rtop == 1 ? A01.y : A01.x));
            if (rtop >= 0) atomicAdd(j + rtop * rowp, pair_widen<CONV>(v));
            A23 = pk(A01.y, A23.x);
            A01 = pk(0.0f, A01.x);
        } else {  // all four leave
            reduce_all(j);
            A01 = pk1(0.0f);
            A23 = pk1(0.0f);
        }
        vc = (int)(__float_as_uint(rn.x) & kQuadOffMask);
        cwc = rn.y;
        rn = rq;
        c[0] = q[0];
        c[1] = q[1];
    }
    // the last point: linear form
    const float2 I0 = linear_n(s[0], interval_both(s[0].u)), I1 = linear_n(s[1], interval_both(s[1].u));
    A01 = fma2(I0, pk1(cwc), A01);
    A23 = fma2(I1, pk1(cwc), A23);
    double *__restrict__ j = J0 + vc;
    reduce_all(j);
    // a non-finite intensity persists along the recurrence: make J NaN
    const double nan = __longlong_as_double(0x7ff8000000000000LL);
    if (rtop >= 0 && !(fabsf(I0.x) <= 3.402823466e38f)) atomicAdd(j, nan);
    if (rtop >= 1 && !(fabsf(I0.y) <= 3.402823466e38f)) atomicAdd(j + rowp, nan);
    if (rtop >= 2 && !(fabsf(I1.x) <= 3.402823466e38f)) atomicAdd(j + 2 * rowp, nan);
    if (rtop >= 3 && !(fabsf(I1.y) <= 3.402823466e38f)) atomicAdd(j + 3 * rowp, nan);
}

// FP32 formal solution with Lambda*, four characteristics a thread as above.
// With one characteristic a thread (fs_kernel) the L2's reduction rate is the
// bound: J and four to five window entries a segment, 81 % of the rate at 65 x 65
// x 257. Three of the entries follow the axis of the rows: the voxel itself and,
// where the step before or after is along that axis, the neighbour up or down a
// row. Their sums (and J's) ride along in registers, move with the rows and are
// reduced when a voxel is left; the other entries are reduced at once. The
// voxel's own entry, by far the largest, carries what its sum loses by rounding.
// Angles that step along x more run on arrays with x and y exchanged (band_t: the
// 27 planes and J), added to the others afterwards (band_merge_kernel, 0.16 ms at
// 97^3). 154 registers: six blocks of 64 a SM without spills; four blocks of 128
// spill and are no faster. With both kernels and 512 angles: 65 x 65 x 257 27.4 ->
// 22.6 ms, 97^3 21.2 -> 17.2 ms; at 65 x 65 x 257 the L2's atomic input is 72 %
// busy, issue 54 %. Error of Lambda* against 64 bits at 65^3: 6.83e-9 -> 6.80e-9 (interval
// functions from the 9-term series, alpha without cancellation: with the
// polynomials of the kernel above and e0 - a it was 7.6e-9).
template <bool PARAB>
__global__ void __launch_bounds__(64, 6) fs_lstar_quad_kernel(FsParams p) {
    const int o = p.order4[blockIdx.y];
    const bool tr = p.swap[o];
    const int nm = tr ? p.ny : p.nx, nd = tr ? p.nx : p.ny;
    const int nlive = nm * ((nd + 3) >> 2);
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t - (threadIdx.x & 31) >= nlive) return;  // the whole warp is past the face
    const int tt = min(t, nlive - 1);
    const int K = p.tlen[o];
    const float4 *__restrict__ rec = p.rec4 + p.toff[o];
    const uint32_t *__restrict__ code = p.code + p.toff[o];
    const unsigned long long *__restrict__ win =
        reinterpret_cast<const unsigned long long *>(p.win + p.toff[o]);
    const int m0 = tt % nm, d0 = 4 * (tt / nm);
    const int rowp = 2 * nm;
    const float4 *__restrict__ P = (tr ? p.pairs_t : p.pairs) + m0 + rowp * d0;
    const unsigned row2 = d0 + 2 < nd ? 2 * rowp : 0;
    const unsigned N = (unsigned)(p.nx * p.ny * p.nz);  // 27 N < 2^31
    double *__restrict__ band = tr ? p.band_t : p.lstar;
    double *__restrict__ Jd = tr ? p.band_t + 27ull * N : p.J;
    const int rtop = t < nlive ? min(3, nd - 1 - d0) : -1;
    // plane of the neighbour one row up (in the planes' own x, y order)
    const unsigned up_plane = 13u + (tr ? 1u : 3u), down_plane = 26u - up_plane;

    float Iv[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    if (!p.homogeneous) {
        const bool up = p.up[o];
#pragma unroll
        for (int r = 0; r < 4; ++r)
            if (d0 + r < nd) {
                const int f = tr ? d0 + r + p.nx * m0 : m0 + p.nx * (d0 + r);
                Iv[r] = (float)entry_intensity(up, p.mu, o, f, p.top_face, p.bot_face, p.bot_grad,
                                               p.I_top, p.I_bot);
            }
    }
    RayN s[2];
    float2 ring[2][kWin];
#pragma unroll
    for (int i = 0; i < kWin; ++i) ring[0][i] = ring[1][i] = pk1(0.0f);
    const float4 r0 = __ldg(rec);
    {
        const unsigned v = __float_as_uint(r0.x) & kQuadOffMask;
        quad_start(s[0], __ldg(P + v), pk(r0.z, r0.w), Iv[0], Iv[1]);
        quad_start(s[1], __ldg(P + (v + row2)), pk(r0.z, r0.w), Iv[2], Iv[3]);
    }
    // sums of the rows' current voxels: J, the voxel's own plane, the planes up
    // and down; used: which of the last two hold anything since the last flush
    float2 A[4][2];
#pragma unroll
    for (int q = 0; q < 4; ++q) A[q][0] = A[q][1] = pk1(0.0f);
    float2 B[2] = {pk1(0.0f), pk1(0.0f)};  // what A[1] lost by rounding
    bool used_up = false, used_down = false;
    unsigned v[4];  // the rows' current voxels
    auto locate = [&](uint32_t c) {
        const int x = (int)(c & 0x7ffu), y = (int)((c >> 11) & 0x7ffu);
        int m = m0 + (tr ? y : x), d = d0 + (tr ? x : y);
        if (m >= nm) m -= nm;
        if (d >= nd) d -= nd;
        const unsigned z = (unsigned)(nd * (int)(c >> 22));
#pragma unroll
        for (int r = 0; r < 4; ++r) v[r] = m + nm * ((d + r >= nd ? d + r - nd : d + r) + z);
    };
    auto row = [](const float2 (&a)[2], int r) {
        return r == 0 ? a[0].x : (r == 1 ? a[0].y : (r == 2 ? a[1].x : a[1].y));
    };
    auto reduce = [&](double *__restrict__ to, float2 a, float2 b) {  // all rows
        if (rtop >= 0) atomicAdd(to + v[0], widen_f32(a.x));
        if (rtop >= 1) atomicAdd(to + v[1], widen_f32(a.y));
        if (rtop >= 2) atomicAdd(to + v[2], widen_f32(b.x));
        if (rtop >= 3) atomicAdd(to + v[3], widen_f32(b.y));
    };
    auto target = [&](int q) -> double * {
        return q == 0 ? Jd : band + N * (q == 1 ? 13u : (q == 2 ? up_plane : down_plane));
    };
    // the contributions of the current point: weight cw, window wc, types of
    // the moves from the previous point and to the next (2: none along the rows)
    auto contribute = [&](const WeightsN (&wt)[2], float cw, unsigned long long wc, bool first,
                          unsigned prev, unsigned next, bool ahead) {
        const float2 c2 = pk1(cw);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
#pragma unroll
            for (int i = 0; i < kWin - 1; ++i) ring[j][i] = mul2(wt[j].E, ring[j][i + 1]);
            if (first) ring[j][7] = add2(ring[j][7], wt[j].al);  // S_{-1} = S_0
            else ring[j][6] = add2(ring[j][6], wt[j].al);
            ring[j][7] = add2(ring[j][7], wt[j].be);
            ring[j][8] = wt[j].ga;
            A[0][j] = fma2(s[j].I, c2, A[0][j]);
            const float2 sum = fma2(ring[j][7], c2, A[1][j]);
            B[j] = add2(B[j], fma2(ring[j][7], c2, sub2(A[1][j], sum)));
            A[1][j] = sum;
        }
        // the next point's entry (zero where ga is)
        if (ahead) {
            const unsigned dc = (unsigned)(wc >> 40) & 31u;
            if (next < 2u) {
                if (next == 0u) {
                    A[2][0] = fma2(ring[0][8], c2, A[2][0]);
                    A[2][1] = fma2(ring[1][8], c2, A[2][1]);
                    used_up = true;
                } else {
                    A[3][0] = fma2(ring[0][8], c2, A[3][0]);
                    A[3][1] = fma2(ring[1][8], c2, A[3][1]);
                    used_down = true;
                }
            } else if (dc != kWinNone) {
                reduce(band + N * dc, mul2(ring[0][8], c2), mul2(ring[1][8], c2));
            }
        }
        // the previous point's, then the others as long as the run goes on
        const unsigned d6 = (unsigned)(wc >> 30) & 31u;
        if (d6 == kWinNone) return;
        if (prev == 0u) {  // it came one row up: the voxel it left lies down
            A[3][0] = fma2(ring[0][6], c2, A[3][0]);
            A[3][1] = fma2(ring[1][6], c2, A[3][1]);
            used_down = true;
        } else if (prev == 1u) {
            A[2][0] = fma2(ring[0][6], c2, A[2][0]);
            A[2][1] = fma2(ring[1][6], c2, A[2][1]);
            used_up = true;
        } else {
            reduce(band + N * d6, mul2(ring[0][6], c2), mul2(ring[1][6], c2));
        }
#pragma unroll
        for (int i = 5; i >= 0; --i) {
            const unsigned dc = (unsigned)(wc >> (5 * i)) & 31u;
            if (dc == kWinNone) break;
            reduce(band + N * dc, mul2(ring[0][i], c2), mul2(ring[1][i], c2));
        }
    };
    auto flush = [&]() {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (q == 2 && !used_up) continue;
            if (q == 3 && !used_down) continue;
            if (q == 1) {
                double *to = band + N * 13u;
                if (rtop >= 0) atomicAdd(to + v[0], widen_f32(A[1][0].x) + widen_f32(B[0].x));
                if (rtop >= 1) atomicAdd(to + v[1], widen_f32(A[1][0].y) + widen_f32(B[0].y));
                if (rtop >= 2) atomicAdd(to + v[2], widen_f32(A[1][1].x) + widen_f32(B[1].x));
                if (rtop >= 3) atomicAdd(to + v[3], widen_f32(A[1][1].y) + widen_f32(B[1].y));
                B[0] = B[1] = pk1(0.0f);
            } else {
                reduce(target(q), A[q][0], A[q][1]);
            }
            A[q][0] = A[q][1] = pk1(0.0f);
        }
        used_up = used_down = false;
    };

    locate(__ldg(code));
    unsigned prev = 2u;
    float cwc = r0.y;
    float4 rn = __ldg(rec + 1);
    const unsigned on = __float_as_uint(rn.x) & kQuadOffMask;
    float4 c[2] = {__ldg(P + on), __ldg(P + (on + row2))};
    for (int k = 1; k < K; ++k) {
        const float4 rq = __ldg(rec + k + 1);
        const unsigned oq = __float_as_uint(rq.x) & kQuadOffMask;
        const float4 q[2] = {__ldg(P + oq), __ldg(P + (oq + row2))};
        const unsigned long long wc = __ldg(win + k - 1);
        const uint32_t cn = __ldg(code + k);
        WeightsN wt[2];
        const bool ahead = quad_advance_w<PARAB>(s, c, pk(rn.z, rn.w), wt);
        const unsigned next = __float_as_uint(rn.x) >> kQuadOffBits;
        contribute(wt, cwc, wc, k == 1, prev, next, PARAB && ahead);
        if (next == 0u) {  // one row up: row 0's voxel leaves
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (i == 2 && !used_up) continue;
                if (i == 3 && !used_down) continue;
                if (rtop >= 0)
                    atomicAdd(target(i) + v[0], i == 1 ? widen_f32(A[1][0].x) + widen_f32(B[0].x)
                                                       : widen_f32(A[i][0].x));
                A[i][0] = pk(A[i][0].y, A[i][1].x);
                A[i][1] = pk(A[i][1].y, 0.0f);
                if (rtop < 3) {  // the last existing row enters a voxel no sum holds
                    if (rtop == 2) A[i][1].x = 0.0f;
                    else if (rtop == 1) A[i][0].y = 0.0f;
                    else A[i][0].x = 0.0f;
                }
            }
            B[0] = pk(B[0].y, B[1].x);
            B[1] = pk(B[1].y, 0.0f);
            if (rtop == 2) B[1].x = 0.0f;
            else if (rtop == 1) B[0].y = 0.0f;
            else if (rtop == 0) B[0].x = 0.0f;
        } else if (next == 1u) {  // one row down: the last existing row's voxel leaves
            const unsigned vt = rtop == 3 ? v[3] : (rtop == 2 ? v[2] : (rtop == 1 ? v[1] : v[0]));
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (i == 2 && !used_up) continue;
                if (i == 3 && !used_down) continue;
                if (rtop >= 0)
                    atomicAdd(target(i) + vt, i == 1 ? widen_f32(row(A[1], rtop)) + widen_f32(row(B, rtop))
                                                     : widen_f32(row(A[i], rtop)));
                A[i][1] = pk(A[i][0].y, A[i][1].x);
                A[i][0] = pk(0.0f, A[i][0].x);
            }
            B[1] = pk(B[0].y, B[1].x);
            B[0] = pk(0.0f, B[0].x);
        } else {
            flush();
        }
        prev = next;
        locate(cn);
        cwc = rn.y;
        rn = rq;
        c[0] = q[0];
        c[1] = q[1];
    }
    WeightsN wt[2];
    quad_last_w(s[0], wt[0]);
    quad_last_w(s[1], wt[1]);
    contribute(wt, cwc, __ldg(win + K - 1), K == 1, prev, 2u, false);
    flush();
    // a non-finite intensity persists along the recurrence: make J NaN
    const double nan = __longlong_as_double(0x7ff8000000000000LL);
    if (rtop >= 0 && !(fabsf(s[0].I.x) <= 3.402823466e38f)) atomicAdd(Jd + v[0], nan);
    if (rtop >= 1 && !(fabsf(s[0].I.y) <= 3.402823466e38f)) atomicAdd(Jd + v[1], nan);
    if (rtop >= 2 && !(fabsf(s[1].I.x) <= 3.402823466e38f)) atomicAdd(Jd + v[2], nan);
    if (rtop >= 3 && !(fabsf(s[1].I.y) <= 3.402823466e38f)) atomicAdd(Jd + v[3], nan);
}

// The exchanged planes (grid z = 27 nz + z: the plane, J last, and the layer)
// transposed onto the others, 32 x 32 at a time, and zeroed for the next call.
__global__ void __launch_bounds__(256) band_merge_kernel(int nx, int ny, int nz, double *__restrict__ band_t,
                                                         double *__restrict__ lstar,
                                                         double *__restrict__ J) {
    __shared__ double tile[32][33];
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int x0 = blockIdx.x * 32, y0 = blockIdx.y * 32;
    const long long n = (long long)nx * ny;
    for (int l = blockIdx.z; l < 28 * nz; l += gridDim.z) {
        double *__restrict__ from = band_t + n * l + y0 + tx;
        double *__restrict__ to = (l < 27 * nz ? lstar + n * l : J + n * (l - 27 * nz)) + x0 + tx;
        double a[4], b[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {  // all loads first
            const int x = x0 + ty + 8 * i, y = y0 + ty + 8 * i;
            a[i] = x < nx && y0 + tx < ny ? from[(long long)ny * x] : 0.0;
            b[i] = y < ny && x0 + tx < nx ? to[(long long)nx * y] : 0.0;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) tile[ty + 8 * i][tx] = a[i];
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int x = x0 + ty + 8 * i, y = y0 + ty + 8 * i;
            if (x < nx && y0 + tx < ny) from[(long long)ny * x] = 0.0;
            if (y < ny && x0 + tx < nx) to[(long long)nx * y] = b[i] + tile[tx][ty + 8 * i];
        }
        __syncthreads();
    }
}

// Records of the four-characteristic kernel: (offset | step type << 29,
// J weight, l/2, l/2), offsets with x and y exchanged for the angles that swap
// them, the step type of the move from the previous point: 0 one row up, 1 one
// row down, 2 anything else (the first point too).
__global__ void quad_rec_kernel(int nx, int ny, const long long *__restrict__ toff,
                                const int *__restrict__ tlen, const signed char *__restrict__ swap,
                                const uint32_t *__restrict__ code,
                                const float4 *__restrict__ rec32, float4 *__restrict__ rec4) {
    const int o = blockIdx.x;
    const long long t0 = toff[o];
    const int K = tlen[o];
    const bool tr = swap[o];
    const int nm = tr ? ny : nx, nd = tr ? nx : ny;
    for (int i = threadIdx.x; i <= K; i += blockDim.x) {
        const int k = min(i, K - 1);  // one record more: the last point again, to load ahead
        auto split = [&](uint32_t c, int &m, int &d, int &z) {
            const int x = (int)(c & 0x7ffu), y = (int)((c >> 11) & 0x7ffu);
            m = tr ? y : x;
            d = tr ? x : y;
            z = (int)(c >> 22);
        };
        int m1, d1, z1;
        split(code[t0 + k], m1, d1, z1);
        unsigned type = 2u;
        if (k > 0) {
            int m0, d0, z0;
            split(code[t0 + k - 1], m0, d0, z0);
            int dd = d1 - d0;
            if (dd == nd - 1) dd = -1;  // wrapped offsets: a step across the
            if (dd == 1 - nd) dd = 1;   // periodic boundary
            if (m1 == m0 && z1 == z0 && (dd == 1 || dd == -1)) type = dd == 1 ? 0u : 1u;
        }
        const float4 r = rec32[t0 + k];
        const unsigned off = (unsigned)rep_index(m1, d1, z1, nm, nd);
        rec4[t0 + i] = make_float4(__uint_as_float(off | (type << kQuadOffBits)), r.y, r.z, r.w);
    }
}

// p.pairs_t from the replicated FP32 (chi, S): the pair-packed arrays with x
// and y exchanged, element y + 2 ny (x + 2 nx z) the values of columns x and
// x + 1 at y; transposed 32 x 32 at a time through shared memory.
__global__ void __launch_bounds__(256) pair_pack_t_kernel(int nx, int ny, const float2 *__restrict__ chiS,
                                                          float4 *__restrict__ P) {
    __shared__ float2 tile[32][34];
    const int wx = 2 * nx, wy = 2 * ny, tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const long long layer = (long long)wx * wy * blockIdx.z;
    const int x0 = blockIdx.x * 32, y0 = blockIdx.y * 32;
    for (int j = ty; j < 32; j += 8)
        for (int i = tx; i < 33; i += 32)
            if (y0 + j < wy) {
                const int x = x0 + i < wx ? x0 + i : x0 + i - wx;  // the last column pairs with the first
                if (x < wx) tile[j][i] = chiS[layer + x + (long long)wx * (y0 + j)];
            }
    __syncthreads();
    for (int i = ty; i < 32; i += 8)
        if (x0 + i < wx && y0 + tx < wy) {
            const float2 a = tile[tx][i], b = tile[tx][i + 1];
            P[layer + y0 + tx + (long long)wy * (x0 + i)] = make_float4(a.x, b.x, a.y, b.y);
        }
}

// p.pairs from the replicated FP32 (chi, S): at every replicated index the
// values of that row and the next one, (chi(y), chi(y+1), S(y), S(y+1)); the
// last replicated row of a layer pairs with the layer's first (never read by
// an existing characteristic: the pair kernel reads rows <= 2 ny - 2).
__global__ void pair_pack_kernel(int nx, int ny, int nz, const float2 *__restrict__ chiS,
                                 float4 *__restrict__ P) {
    const int rows = 2 * ny * nz, w = 2 * nx;
    for (int row = blockIdx.x; row < rows; row += gridDim.x) {
        const long long i0 = (long long)row * w;
        const long long next = (row % (2 * ny) + 1 < 2 * ny) ? w : w - 2LL * ny * w;
        for (int x = threadIdx.x; x < w; x += blockDim.x) {
            const float2 a = chiS[i0 + x], b = chiS[i0 + next + x];
            P[i0 + x] = make_float4(a.x, b.x, a.y, b.y);
        }
    }
}

// ---- FP64 formal solution without Lambda* (refinement residuals, FP64 mode
// after the first iteration). The FP64 pipe is the bound, so what can leave it
// does: branch tests on the high word of non-negative doubles (integer compares),
// reciprocals, the interval polynomial and 1 - e^-u, widening by integer moves
// (fs64_step.cuh: hi_below, recip64, interval64). 10 FP64 instructions a point
// remain in the linear form below u = 1/2 and 17 in the parabolic one, of 19 and 34.
// 33^3 voxels, 128 angles, linear: 1303 us with three FP64 operations a reciprocal,
// nine for the polynomial and eight for e^-u; 947 us with the smaller terms of both
// in float-float; 618 us with the rest in fixed point.

// One thread per characteristic; per point: the replicated offset (FP32
// record), the FP64 (l/2, J weight) record, the (chi, S) gather, and one
// red.global.add.f64 into the replicated J (folded afterwards). The
// parabolic blend f = clamp(2 - 2u) clamp(2 - q/2) is taken apart on integer
// tests: f > 0 iff u < 1 and q < 4, each factor is 1 below 1/2 (resp. 2) and
// one FMA between.
template <bool PARAB>
__global__ void __launch_bounds__(128) fs64_fast_kernel(FsParams p) {
    __shared__ unsigned long long tab[64];
    exp_table(tab);
    const int nray = p.nx * p.ny;
    const int ray = blockIdx.x * blockDim.x + threadIdx.x;
    if (ray >= nray) return;
    const int o = p.order[blockIdx.y];
    const int K = p.tlen[o];
    const long long t0 = p.toff[o];
    const float4 *__restrict__ rec = p.rec32 + t0;
    const double2 *__restrict__ rd = p.rec64 + t0;
    const double2 *__restrict__ chiS = static_cast<const double2 *>(p.chiS);
    double *__restrict__ J = p.Jrep;
    const int x0 = ray % p.nx, y0 = ray / p.nx;
    const int base = x0 + 2 * p.nx * y0;

    double I = 0.0;
    if (!p.homogeneous)
        I = entry_intensity(p.up[o], p.mu, o, ray, p.top_face, p.bot_face, p.bot_grad, p.I_top,
                            p.I_bot);
    int vc = base + __float_as_int(__ldg(&rec[0].x));
    double2 r = __ldg(rd);
    const double2 cs = chiS[vc];
    double hc = cs.x * r.x;  // half the optical depth of the chord of the point
    double cwc = r.y;
    double u = hc;  // the entry interval: chi_{-1} l_{-1} = 0
    double Sc = cs.y, Sp = cs.y, dS = 0.0;  // S_{-1} = S_0
    double ru = PARAB ? recip64(hc) : 0.0;
    for (int k = 1; k < K; ++k) {
        const int vn = base + __float_as_int(__ldg(&rec[k].x));
        const double2 rn = __ldg(rd + k);
        const double2 cn = chiS[vn];
        const double hn = cn.x * rn.x;
        const double dSn = cn.y - Sc;
        const double w = hc + hn;
        const IntervalDE f = interval64<PARAB>(u, ru, tab);
        // difference form of the update (as in the FP32 kernel)
        double In = fma(f.e0, Sp - I, I);
        In = fma(f.a, dS, In);
        if (PARAB) {
            const double rw = recip64(w);
            const double q = u * rw;
            if (hi_below(u, 0x3FF00000) && hi_below(q, 0x40100000)) {
                double sd = u * recip64(u + w) * f.d;
                if (!hi_below(u, 0x3FE00000)) sd *= fma(-2.0, u, 2.0);
                if (!hi_below(q, 0x40000000)) sd *= fma(-0.5, q, 2.0);
                In = fma(sd, fma(-q, dSn, dS), In);
            }
            ru = rw;
        }
        I = In;
        atomicAdd(J + vc, cwc * I);
        u = w;
        hc = hn;
        Sp = Sc;
        Sc = cn.y;
        dS = dSn;
        vc = vn;
        cwc = rn.y;
    }
    const IntervalDE f = interval64<PARAB>(u, ru, tab);
    I = fma(f.a, dS, fma(f.e0, Sp - I, I));
    atomicAdd(J + vc, cwc * I);
}

// J[v] = sum of the four replicas of v in Jrep (FP64), and of the four in
// Jrep_t (x and y exchanged) where it is given; both zeroed for the next launch.
__global__ void fold_kernel(int nx, int ny, int nz, double *__restrict__ Jrep,
                            double *__restrict__ Jrep_t, double *__restrict__ J) {
    const long long n = (long long)nx * ny * nz;
    const long long dy = 2LL * nx * ny;
    for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < n;
         v += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(v % nx), y = (int)((v / nx) % ny), z = (int)(v / ((long long)nx * ny));
        const long long i0 = rep_index(x, y, z, nx, ny);
        double sum = (Jrep[i0] + Jrep[i0 + nx]) + (Jrep[i0 + dy] + Jrep[i0 + dy + nx]);
        if (Jrep_t) {
            const long long t0 = rep_index(y, x, z, ny, nx);
            sum += (Jrep_t[t0] + Jrep_t[t0 + ny]) + (Jrep_t[t0 + dy] + Jrep_t[t0 + dy + ny]);
            Jrep_t[t0] = 0.0;
            Jrep_t[t0 + ny] = 0.0;
            Jrep_t[t0 + dy] = 0.0;
            Jrep_t[t0 + dy + ny] = 0.0;
        }
        J[v] = sum;
        Jrep[i0] = 0.0;
        Jrep[i0 + nx] = 0.0;
        Jrep[i0 + dy] = 0.0;
        Jrep[i0 + dy + nx] = 0.0;
    }
}

template <typename R, bool PARAB>
cudaError_t launch_t(const FsParams &p, cudaStream_t s) {
    const int threads = 128;
    dim3 grid((p.nx * p.ny + threads - 1) / threads, p.nangles);
    fs_kernel<R, PARAB><<<grid, threads, 0, s>>>(p);
    return cudaGetLastError();
}

}  // namespace

template <bool PARAB>
void launch_fast_w(const FsParams &p, dim3 grid, int block, int widen, cudaStream_t s) {
    if (widen == 0) fs_fast_kernel<PARAB, 0><<<grid, block, 0, s>>>(p);
    else if (widen == 1) fs_fast_kernel<PARAB, 1><<<grid, block, 0, s>>>(p);
    else fs_fast_kernel<PARAB, 2><<<grid, block, 0, s>>>(p);
}

template <bool PARAB>
void launch_quad_w(const FsParams &p, dim3 grid, int block, int widen, cudaStream_t s) {
    if (widen == 1) fs_quad_kernel<PARAB, 1><<<grid, block, 0, s>>>(p);
    else fs_quad_kernel<PARAB, 0><<<grid, block, 0, s>>>(p);
}

template <bool PARAB>
void launch_pair_w(const FsParams &p, dim3 grid, int block, int widen, cudaStream_t s) {
    if (widen == 0) fs_pair_kernel<PARAB, 0><<<grid, block, 0, s>>>(p);
    else if (widen == 1) fs_pair_kernel<PARAB, 1><<<grid, block, 0, s>>>(p);
    else fs_pair_kernel<PARAB, 2><<<grid, block, 0, s>>>(p);
}

// groups of four characteristics of one angle, the larger of the two splits
static int lane_count(const FsParams &p) {
    return std::max(p.nx * ((p.ny + 3) / 4), p.ny * ((p.nx + 3) / 4));
}

cudaError_t launch_fs_lstar_quad(const FsParams &p, bool parabolic, cudaStream_t s) {
    const int rows = 2 * p.ny * p.nz;
    const float2 *chiS = static_cast<const float2 *>(p.chiS);
    pair_pack_kernel<<<rows < 65536 ? rows : 65536, 256, 0, s>>>(p.nx, p.ny, p.nz, chiS, p.pairs);
    pair_pack_t_kernel<<<dim3((2 * p.nx + 31) / 32, (2 * p.ny + 31) / 32, p.nz), 256, 0, s>>>(
        p.nx, p.ny, chiS, p.pairs_t);
    const dim3 grid((lane_count(p) + 63) / 64, p.nangles);
    if (parabolic) fs_lstar_quad_kernel<true><<<grid, 64, 0, s>>>(p);
    else fs_lstar_quad_kernel<false><<<grid, 64, 0, s>>>(p);
    band_merge_kernel<<<dim3((p.nx + 31) / 32, (p.ny + 31) / 32, std::min(28 * p.nz, 65535)), 256, 0, s>>>(
        p.nx, p.ny, p.nz, p.band_t, p.lstar, p.J);
    return cudaGetLastError();
}

// Below about 3.5 waves of groups (384 of them resident per SM) the coarser
// split leaves the last wave too empty: at 65^3 voxels the kernel takes 1.60 ms
// against 1.56 with one characteristic a thread for 141,000 groups (8 x 16
// angles), 3.13 against 3.47 for 318,000 (12 x 24) and 5.4 against 6.3 for 566,000
// (16 x 32); at 33^3 1.26 against 1.27 for 152,000. Sides of one or two
// voxels are left out: there the neighbours up and down a row coincide.
bool lstar_quad_applicable(const FsParams &p) {
    const long long groups = (long long)lane_count(p) * p.nangles;
    return quad_applicable(p) && std::min(p.nx, p.ny) >= 4 && 27LL * p.nx * p.ny * p.nz < (1LL << 31) &&
           2 * groups >= 7LL * 384 * device_sm_count();
}

bool quad_applicable(const FsParams &p) {
    return p.rec4 != nullptr && 4LL * p.nx * p.ny * p.nz <= (long long)kQuadOffMask;
}

cudaError_t launch_quad_rec(const Template &t, int nx, int ny, float4 *rec4, cudaStream_t s) {
    quad_rec_kernel<<<t.nangles, 256, 0, s>>>(nx, ny, t.toff, t.tlen, t.swap, t.code, t.rec32, rec4);
    return cudaGetLastError();
}

bool fs_shape_valid(const FsShape &sh) {
    return (sh.block == 64 || sh.block == 128 || sh.block == 256) &&
           (sh.rays_per_thread == 1 || sh.rays_per_thread == 2 || sh.rays_per_thread == 4) &&
           sh.widen >= 0 && sh.widen <= 2 &&
           (sh.branchless == 0 || sh.branchless == 1);
}

cudaError_t launch_fs_fast(const FsParams &p, bool parabolic, const FsShape &sh, cudaStream_t s) {
    if (!fs_shape_valid(sh)) return cudaErrorInvalidValue;
    if (sh.rays_per_thread >= 2) {
        if (!p.pairs) return cudaErrorInvalidValue;
        if (sh.rays_per_thread == 4 && !quad_applicable(p)) return cudaErrorInvalidValue;
        const int rows = 2 * p.ny * p.nz;
        pair_pack_kernel<<<rows < 65536 ? rows : 65536, 256, 0, s>>>(
            p.nx, p.ny, p.nz, static_cast<const float2 *>(p.chiS), p.pairs);
        if (sh.rays_per_thread == 4) {
            pair_pack_t_kernel<<<dim3((2 * p.nx + 31) / 32, (2 * p.ny + 31) / 32, p.nz), 256, 0, s>>>(
                p.nx, p.ny, static_cast<const float2 *>(p.chiS), p.pairs_t);
            dim3 grid((lane_count(p) + sh.block - 1) / sh.block, p.nangles);
            if (parabolic) launch_quad_w<true>(p, grid, sh.block, sh.widen, s);
            else launch_quad_w<false>(p, grid, sh.block, sh.widen, s);
            return cudaGetLastError();
        }
        const int npair = p.nx * ((p.ny + 1) / 2);
        dim3 grid((npair + sh.block - 1) / sh.block, p.nangles);
        if (parabolic) launch_pair_w<true>(p, grid, sh.block, sh.widen, s);
        else launch_pair_w<false>(p, grid, sh.block, sh.widen, s);
        return cudaGetLastError();
    }
    dim3 grid((p.nx * p.ny + sh.block - 1) / sh.block, p.nangles);
    if (parabolic) launch_fast_w<true>(p, grid, sh.block, sh.widen, s);
    else launch_fast_w<false>(p, grid, sh.block, sh.widen, s);
    return cudaGetLastError();
}

cudaError_t launch_fs64_fast(const FsParams &p, bool parabolic, cudaStream_t s) {
    const int threads = 128;
    dim3 grid((p.nx * p.ny + threads - 1) / threads, p.nangles);
    if (parabolic) fs64_fast_kernel<true><<<grid, threads, 0, s>>>(p);
    else fs64_fast_kernel<false><<<grid, threads, 0, s>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_fold(int nx, int ny, int nz, double *Jrep, double *J, cudaStream_t s,
                        double *Jrep_t) {
    const long long n = (long long)nx * ny * nz;
    long long b = (n + 255) / 256;
    const long long cap = 16LL * device_sm_count();
    if (b > cap) b = cap;
    fold_kernel<<<(int)b, 256, 0, s>>>(nx, ny, nz, Jrep, Jrep_t, J);
    return cudaGetLastError();
}

cudaError_t launch_fs_lstar(const FsParams &p, bool fp64, bool parabolic, cudaStream_t s) {
    if (fp64) return parabolic ? launch_t<double, true>(p, s) : launch_t<double, false>(p, s);
    return parabolic ? launch_t<float, true>(p, s) : launch_t<float, false>(p, s);
}

}  // namespace rt3d
