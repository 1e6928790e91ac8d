// Operator-splitting step (Sec. 2.2, Eq. alo) and its Jacobi solver (Sec. 4,
// "OS iteration"), with the reductions of the convergence test.
//
// The OS system for the correction dJ = J_new - J_old is
//   [1 - Lambda*(1 - eps)] dJ = r,  r = J_FS - J_old,
// a 27-point stencil periodic in x and y. os_prep folds (1 - eps) of the
// neighbour into the 26 off-diagonal coefficients a_d(v) = Lambda*[d][v] (1 -
// eps_{v+d}) (FP64, or FP32 in the mixed mode; blocks of 32 voxels with
// their 26 planes contiguous, os_coef_index) and stores 1/diag in FP64.
// A sweep reads the coefficients once (the HBM stream that bounds it), the
// neighbours of dJ through L1/L2, and writes dJ^{m+1} with the two maxima
// of the stop test. A grid whose coefficients fit in the chip's shared memory is
// solved in one cooperative launch (os_resident_kernel); elsewhere sweeps are
// launched back to back (Gauss-Seidel: two launches a sweep), each reads the
// previous sweep's maxima and returns at once after the stop test is met, so a
// fixed launch sequence serves any sweep count.
#include <cooperative_groups.h>

#include <algorithm>
#include <type_traits>

#include "rt3d_internal.cuh"

namespace rt3d {

namespace {

__device__ __forceinline__ unsigned long long dbits(double x) {
    return (unsigned long long)__double_as_longlong(x);
}
__device__ __forceinline__ double bitsd(unsigned long long x) {
    return __longlong_as_double((long long)x);
}

// block-wide max of a non-negative double (NaN propagates: its bit pattern
// is above +inf), then one atomicMax per block.
__device__ __forceinline__ void block_max_atomic(double x, unsigned long long *dst) {
    __shared__ unsigned long long sm[32];
    unsigned long long b = dbits(fabs(x));
    if (x != x) b = 0x7ff8000000000000ULL;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        unsigned long long o = __shfl_xor_sync(0xffffffffu, b, off);
        b = o > b ? o : b;
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) sm[wid] = b;
    __syncthreads();
    if (wid == 0) {
        const int nw = (blockDim.x + 31) >> 5;
        b = lane < nw ? sm[lane] : 0ULL;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            unsigned long long o = __shfl_xor_sync(0xffffffffu, b, off);
            b = o > b ? o : b;
        }
        if (lane == 0 && b) atomicMax(dst, b);
    }
    __syncthreads();  // sm[] is reused by a following call
}

// Packed (chi, S) written to the four replicas of every voxel.
__global__ void pack_kernel(int nx, int ny, int nz, const double *chi, double scale,
                            const double *S, void *out, bool fp64) {
    const long long n = (long long)nx * ny * nz;
    for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < n;
         v += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(v % nx), y = (int)((v / nx) % ny), z = (int)(v / ((long long)nx * ny));
        const double c = chi[v] * scale, sv = S[v];
        for (int b = 0; b < 2; ++b)
            for (int a = 0; a < 2; ++a) {
                const long long r = rep_index(x + a * nx, y + b * ny, z, nx, ny);
                if (fp64) static_cast<double2 *>(out)[r] = make_double2(c, sv);
                else static_cast<float2 *>(out)[r] = make_float2((float)c, (float)sv);
            }
    }
}

// S = (1 - eps) J + eps B (or (1 - eps) J for the homogeneous problem),
// written into the S half of the four replicas of the packed (chi, S).
__global__ void source_kernel(int nx, int ny, int nz, const double *J, const double *eps,
                              const double *B, void *out, bool fp64, bool homogeneous) {
    const long long n = (long long)nx * ny * nz;
    for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < n;
         v += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(v % nx), y = (int)((v / nx) % ny), z = (int)(v / ((long long)nx * ny));
        const double e = eps[v];
        double sv = (1.0 - e) * J[v];
        if (!homogeneous) sv += e * B[v];
        for (int b = 0; b < 2; ++b)
            for (int a = 0; a < 2; ++a) {
                const long long r = rep_index(x + a * nx, y + b * ny, z, nx, ny);
                if (fp64) static_cast<double2 *>(out)[r].y = sv;
                else static_cast<float2 *>(out)[r].y = (float)sv;
            }
    }
}

// Bottom-face arrays of the LTE diffusion inner boundary (the test cases of
// Sec. 3.1): per column f and wavelength, dB/dtau = (B(z=0) - B(z=1)) /
// (1/2 (chi(z=0) + chi(z=1))), the one-sided difference over the unit centre
// spacing with the trapezoidal optical depth (tau grows inward), and the face
// intensity B(z=0) + 1/2 chi(z=0) dB/dtau, B carried linearly to the face half
// a voxel below the innermost centre; a single layer has gradient 0 and face
// value B(z=0).
__global__ void diffusion_bc_kernel(long long nf, int nz, int nl, const double *chi,
                                    const double *B, double *I_face, double *grad) {
    const long long n = nf * nl, N = nf * nz;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        const long long l = i / nf, f = i - l * nf;
        const double *c = chi + l * N, *b = B + l * N;
        if (nz < 2) {
            grad[i] = 0.0;
            I_face[i] = b[f];
            continue;
        }
        const double dtau = __dmul_rn(0.5, __dadd_rn(c[f], c[nf + f]));
        const double gr = __ddiv_rn(__dsub_rn(b[f], b[nf + f]), dtau);
        grad[i] = gr;
        I_face[i] = __dadd_rn(b[f], __dmul_rn(__dmul_rn(0.5, c[f]), gr));
    }
}

// neighbour index of (x, y, z) + (dx, dy, dz) with the periodic axes wrapped;
// -1 outside a non-periodic axis
__device__ __forceinline__ long long nb_index(int x, int y, int z, int dx, int dy, int dz, int nx,
                                              int ny, int nz, Periodic per) {
    int xx = x + dx, yy = y + dy, zz = z + dz;
    if (xx < 0 || xx >= nx) {
        if (!per.x) return -1;
        xx += xx < 0 ? nx : -nx;
    }
    if (yy < 0 || yy >= ny) {
        if (!per.y) return -1;
        yy += yy < 0 ? ny : -ny;
    }
    if (zz < 0 || zz >= nz) {
        if (!per.z) return -1;
        zz += zz < 0 ? nz : -nz;
    }
    return xx + (long long)nx * (yy + (long long)ny * zz);
}

template <typename A>
__global__ void os_prep_kernel(int nx, int ny, int nz, const double *L, const double *eps, A *a,
                               double *inv_diag, Periodic per, bool colour, ColourGeo cg,
                               double *diag) {
    const long long N = (long long)nx * ny * nz;
    for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < N;
         v += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(v % nx), y = (int)((v / nx) % ny), z = (int)(v / ((long long)nx * ny));
        const double dg = 1.0 - L[13 * N + v] * (1.0 - eps[v]);
        inv_diag[v] = 1.0 / dg;
        if (diag) diag[v] = dg;
        const int c = (x & 1) + 2 * (y & 1) + 4 * (z & 1);
        const long long k = (x >> 1) + (long long)cg.nxc[c] * ((y >> 1) + (long long)cg.nyc[c] * (z >> 1));
        int plane = 0;
        for (int d = 0; d < 27; ++d) {
            if (d == 13) continue;
            const long long u = nb_index(x, y, z, d % 3 - 1, (d / 3) % 3 - 1, d / 9 - 1, nx, ny, nz, per);
            double val = 0.0;
            if (u >= 0) val = L[(long long)d * N + v] * (1.0 - eps[u]);
            a[colour ? os_colour_index(plane, cg.blk[c], k) : os_coef_index(plane, v)] = (A)val;
            ++plane;
        }
    }
}

// Colour c of the eight-colour sweep: every voxel of the colour from its
// neighbours' values of this sweep where their colour comes earlier (in dst,
// already final) and of the last sweep otherwise (in src: later colours, and
// the same colour, which a periodic axis of odd length makes a neighbour
// across the seam); Jacobi inside a colour, as the oracle's sweep defines it.
// In the mixed mode (A = float) the products take the FP32 copies of the
// iterates (src32, dst32; written beside the FP64 values), as the Jacobi
// sweep does, and the stop-test maxima compare FP32 copies.
template <typename A>
__global__ void __launch_bounds__(256) gs_colour_kernel(int nx, int ny, int nz, ColourGeo cg, int c,
                                                        const A *__restrict__ a,
                                                        const double *__restrict__ inv_diag,
                                                        const double *__restrict__ r,
                                                        const double *__restrict__ src,
                                                        double *__restrict__ dst,
                                                        const float *__restrict__ src32,
                                                        float *__restrict__ dst32, int m, double tol,
                                                        OsState *st, Periodic per) {
    constexpr bool f32 = sizeof(A) == 4;
    if (st->done) return;
    if (c == 0 && m >= 2) {
        const double dm = bitsd(st->dmax[m - 1]), jm = bitsd(st->jmax[m - 1]);
        if (dm <= tol * jm) {
            if (blockIdx.x == 0 && threadIdx.x == 0) {
                st->done = 1;
                st->count = m - 1;
            }
            return;
        }
    }
    const int px = c & 1, py = (c >> 1) & 1, pz = c >> 2;
    const int nxc = cg.nxc[c], nyc = cg.nyc[c];
    const long long cnt = cg.cnt[c], blk0 = cg.blk[c];
    const int nxy = nx * ny;
    A dmax = A(0), jmax = A(0);
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < cnt;
         k += (long long)gridDim.x * blockDim.x) {
        const long long kxy = (long long)nxc * nyc;
        const int zi = (int)(k / kxy), rem = (int)(k - zi * kxy), yi = rem / nxc, xi = rem - yi * nxc;
        const int x = 2 * xi + px, y = 2 * yi + py, z = 2 * zi + pz;
        const int v = x + nx * (y + ny * z);
        const int X[3] = {os_nb_lo(x, nx, per.x), x, os_nb_hi(x, nx, per.x)};
        const int Y[3] = {os_nb_lo(y, ny, per.y), y, os_nb_hi(y, ny, per.y)};
        const int Z[3] = {os_nb_lo(z, nz, per.z), z, os_nb_hi(z, nz, per.z)};
        const A *__restrict__ ab = a + os_colour_index(0, blk0, k);
        A acc = A(0);
#pragma unroll
        for (int d = 0, pl = 0; d < 27; ++d) {
            if (d == 13) continue;
            const int xn = X[d % 3], yn = Y[(d / 3) % 3], zn = Z[d / 9];
            const int cn = (xn & 1) + 2 * (yn & 1) + 4 * (zn & 1);
            const int u = xn + nx * yn + nxy * zn;
            A xv;
            if constexpr (f32) xv = cn < c ? dst32[u] : src32[u];
            else xv = cn < c ? dst[u] : src[u];
            acc += ab[pl * 32] * xv;
            ++pl;
        }
        const double nv = (r[v] + (double)acc) * inv_diag[v];
        dst[v] = nv;
        if constexpr (f32) {
            const float nf = (float)nv;
            dst32[v] = nf;
            dmax = fmaxf(dmax, fabsf(nf - src32[v]));
            jmax = fmaxf(jmax, fabsf(nf));
        } else {
            dmax = fmax(dmax, fabs(nv - src[v]));
            jmax = fmax(jmax, fabs(nv));
        }
    }
    block_max_atomic((double)dmax, &st->dmax[m]);
    block_max_atomic((double)jmax, &st->jmax[m]);
}

// Half a sweep of the same iteration in one launch: the four colours of the
// planes with parity pz, one cluster of blocks per plane. Planes of one parity
// are no neighbours (z not periodic, or nz even), so their colours are ordered
// by a barrier of the cluster instead of a launch. Each block owns `band` pairs
// of rows and keeps the iterate of those rows, of the rows beside them and of
// the planes above and below in shared memory, with a column beside either
// edge: all 26 neighbours are read there without index arithmetic. A colour's
// update goes to the copies beside the edges as well (in the neighbouring block
// where the row beside is its own).
// The next voxel's coefficients are loaded while a voxel is computed, across
// the barriers too.
// Sweep at 129^3 149 us with one launch per colour (gs_colour_kernel), 100 us
// here; at 65^3 56 and 35 us. What bounds it is the latency of a voxel's
// instructions at 16 warps per SM: a ring of coefficient blocks in shared memory
// (cp.async) ran at 14 warps and 118 us, two smaller blocks per SM at 110 us,
// prefetches of the next colour's coefficients into the L2 at 117 us.
template <typename A> struct GsShared {
    int pitch, rows;  // row pitch (nx + 2), rows of a plane (2 band + 2)
    __host__ __device__ int plane() const { return rows * pitch; }
    __host__ __device__ size_t bytes() const {
        return (size_t)(3 * plane() + 2 * pitch + 2 * rows) * sizeof(A);
    }
};

template <typename A, bool SEAM>
__global__ void __launch_bounds__(512) gs_plane_kernel(int nx, int ny, int nz, ColourGeo cg, int pz,
                                                       int band, GsShared<A> g, const A *__restrict__ a,
                                                       const double *__restrict__ inv_diag,
                                                       const double *__restrict__ r,
                                                       const double *__restrict__ src,
                                                       double *__restrict__ dst,
                                                       const float *__restrict__ src32,
                                                       float *__restrict__ dst32, int m, double tol,
                                                       OsState *st, Periodic per) {
    namespace coop = cooperative_groups;
    constexpr bool f32 = sizeof(A) == 4;
    if (st->done) return;
    if (pz == 0 && m >= 2) {
        const double dm = bitsd(st->dmax[m - 1]), jm = bitsd(st->jmax[m - 1]);
        if (dm <= tol * jm) {
            if (blockIdx.x == 0 && threadIdx.x == 0) {
                st->done = 1;
                st->count = m - 1;
            }
            return;
        }
    }
    coop::cluster_group cl = coop::this_cluster();
    extern __shared__ __align__(16) unsigned char gs_smem[];
    const int pitch = g.pitch;
    A *const C = reinterpret_cast<A *>(gs_smem);  // this plane: rows y0 - 1 .. y1, columns -1 .. nx
    const int L = g.plane(), H = 2 * L;  // below, above (all as offsets from C)
    const int orow = 3 * L;              // last sweep's rows ny - 1 and 0 (an odd periodic y axis)
    const int ocol = orow + 2 * pitch;   // last sweep's columns nx - 1 and 0 (an odd periodic x axis)
    const int ranks = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    const int zi = blockIdx.x / ranks, z = 2 * zi + pz;
    const int y0 = min(ny, 2 * band * rank), y1 = min(ny, y0 + 2 * band), h = y1 - y0;
    const int nxy = nx * ny, vz = nxy * z;
    const bool seamx = SEAM && per.x && (nx & 1), seamy = SEAM && per.y && (ny & 1);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // 1 / (voxels of a colour's row): the even columns, the odd ones. An index
    // below 2^21 plus a half times it, truncated, is the quotient: the product is
    // within 1.5e-4 of the quotient's value and the half keeps it 1 / (2 1024)
    // away from the next integer.
    const float inv0 = 1.0f / (float)((nx + 1) >> 1), inv1 = 1.0f / (float)max(1, nx >> 1);

    // this block's voxels of colour q: indices [k0, k1) of the colour, its
    // plane's first one at kz
    auto range = [&](int q, int &kz, int &k0, int &k1) {
        const int c = 4 * pz + q, nxc = cg.nxc[c], nyc = cg.nyc[c];
        kz = nxc * nyc * zi;
        k0 = kz + nxc * (y0 >> 1);
        k1 = h > 0 ? kz + nxc * min((y1 - (q >> 1) + 1) >> 1, nyc) : k0;
    };
    // voxel (x, y) of index k
    auto voxel = [&](int q, int k, int kz, int &x, int &y) {
        const int nxc = (nx - (q & 1) + 1) >> 1;
        const int yi = (int)(((float)(k - kz) + 0.5f) * (q & 1 ? inv1 : inv0));
        x = 2 * (k - kz - yi * nxc) + (q & 1);
        y = 2 * yi + (q >> 1);
    };
    struct Item {
        A cf[26];
        double rv, id;
        int x, y;
    };
    auto load = [&](int q, int k, int kz, Item &w) {
        const A *__restrict__ ab = a + os_colour_index(0, cg.blk[4 * pz + q], k);
#pragma unroll
        for (int p = 0; p < 26; ++p) w.cf[p] = ab[p * 32];
        voxel(q, k, kz, w.x, w.y);
        const int gv = w.x + nx * w.y + vz;
        w.rv = r[gv];
        w.id = inv_diag[gv];
    };
    int kz, first, end;
    range(0, kz, first, end);
    int k = first + threadIdx.x;
    bool ok = k < end;
    Item w;
    if (ok) load(0, k, kz, w);

    // the rows: last sweep's values of this plane; of the planes below and
    // above last sweep's for the even planes, this sweep's for the odd ones (a
    // clamped plane, with zero coefficients, is the voxel's own)
    const A *__restrict__ old, *__restrict__ now;
    if constexpr (f32) {
        old = src32;
        now = dst32;
    } else {
        old = src;
        now = dst;
    }
    const A *plane = old + vz;
    const int zl = os_nb_lo(z, nz, per.z), zh = os_nb_hi(z, nz, per.z);
    const A *below = (zl == z || pz == 0 ? old : now) + (long long)nxy * zl;
    const A *above = (zh == z || pz == 0 ? old : now) + (long long)nxy * zh;
    auto edge_x = [&](int xx) {  // the voxel behind column xx of a row
        const int x = xx - 1;
        return x < 0 ? (per.x ? nx - 1 : 0) : (x >= nx ? (per.x ? 0 : nx - 1) : x);
    };
    for (int i = warp; i < (h > 0 ? 3 * (h + 2) : 0); i += (int)(blockDim.x >> 5)) {
        const int p = i / (h + 2), ys = i - p * (h + 2);
        int y = y0 + ys - 1;
        if (y < 0) y = per.y ? ny - 1 : 0;
        if (y >= ny) y = per.y ? 0 : ny - 1;
        const A *from = (p == 0 ? plane : (p == 1 ? below : above)) + y * nx;
        A *to = C + p * g.plane() + ys * pitch;
        for (int xx = lane; xx < pitch; xx += 32) to[xx] = from[edge_x(xx)];
    }
    if (seamy)
        for (int i = threadIdx.x; i < 2 * pitch; i += blockDim.x) {
            const int k = i >= pitch;
            C[orow + i] = plane[edge_x(i - k * pitch) + (k ? 0 : nx * (ny - 1))];
        }
    if (seamx)
        for (int i = threadIdx.x; i < 2 * h; i += blockDim.x) {
            const int k = i >= h, ys = i - k * h;
            C[ocol + k * g.rows + ys + 1] = plane[(k ? 0 : nx - 1) + nx * (y0 + ys)];
        }
    // the copies of this block's first and last row beside other blocks' rows
    // (or its own, where the plane wraps onto the same block)
    const int last = (ny - 1) / (2 * band);  // the rank that owns the last row
    A *lo = nullptr, *hi = nullptr;
    if (h > 0) {
        if (y0 > 0) lo = cl.map_shared_rank(C, rank - 1) + (2 * band + 1) * pitch;
        else if (per.y) lo = cl.map_shared_rank(C, last) + (ny - 2 * band * last + 1) * pitch;
        if (y1 < ny) hi = cl.map_shared_rank(C, rank + 1);
        else if (per.y) hi = cl.map_shared_rank(C, 0);
    }
    cl.sync();
    A dmax = A(0), jmax = A(0);
    // results are stored one voxel later: a barrier waits for the block's
    // stores, and those of its last voxels would be on their way still
    double pv = 0.0;
    int pg = -1;
    auto store = [&]() {
        if (pg < 0) return;
        dst[pg] = pv;
        if constexpr (f32) dst32[pg] = (float)pv;
        pg = -1;
    };
    for (int q = 0, left = -1;;) {
        if (left < 0) left = max(1, (end - first + (int)blockDim.x - 1) / (int)blockDim.x);
        k += blockDim.x;
        int nq = q;
        if (left == 1 && q < 3) {
            range(++nq, kz, first, end);
            k = first + (int)threadIdx.x;
        }
        const bool nok = k < end;
        Item nw;
        if (nok) load(nq, k, kz, nw);
        store();
        if (ok) {
            const int x = w.x, y = w.y;
            const int ys = y - y0 + 1, at = ys * pitch + x;
            const bool ex[3] = {seamx && x == 0, true, seamx && x == nx - 1};
            const bool ey[3] = {seamy && y == 0, true, seamy && y == ny - 1};
            A acc = A(0);
#pragma unroll
            for (int d = 0, p = 0; d < 27; ++d) {
                if (d == 13) continue;
                const int i = d % 3, j = (d / 3) % 3, o = at + (j - 1) * pitch + i;
                A xv;
                if (d < 9) xv = C[L + o];
                else if (d >= 18) xv = C[H + o];
                else if (!SEAM) xv = C[o];
                else {
                    // a neighbour of the same colour (across the seam of an
                    // odd periodic axis): its value of the last sweep
                    const int u = j == 1 ? ocol + (i == 2 ? g.rows : 0) + ys
                                         : orow + (j == 2 ? pitch : 0) + x + i;
                    xv = C[ex[i] && ey[j] ? u : o];
                }
                acc += w.cf[p] * xv;
                ++p;
            }
            const double nv = (w.rv + (double)acc) * w.id;
            pv = nv;
            pg = x + nx * y + vz;
            A val;
            const A was = C[at + 1];
            if constexpr (f32) {
                val = (float)nv;
                dmax = fmaxf(dmax, fabsf(val - was));
                jmax = fmaxf(jmax, fabsf(val));
            } else {
                val = nv;
                dmax = fmax(dmax, fabs(val - was));
                jmax = fmax(jmax, fabs(val));
            }
            if (q < 3) {
                C[at + 1] = val;
                const bool row = y == y0 || y == y1 - 1, col = per.x && (x == 0 || x == nx - 1);
                if (row || col) {
                    const int e = x == 0 ? nx + 1 : 0;
                    if (col) C[ys * pitch + e] = val;
                    if (lo && y == y0) {
                        lo[x + 1] = val;
                        if (col) lo[e] = val;
                    }
                    if (hi && y == y1 - 1) {
                        hi[x + 1] = val;
                        if (col) hi[e] = val;
                    }
                }
            }
        }
        ok = nok;
        w = nw;
        if (--left > 0) continue;
        if (q++ == 3) break;
        cl.sync();
        left = -1;
    }
    store();
    block_max_atomic((double)dmax, &st->dmax[m]);
    block_max_atomic((double)jmax, &st->jmax[m]);
}

// ---- The whole OS solve in one cooperative launch, the coefficients of a
// block kept in its shared memory over all sweeps (grids of up to 64 blocks of
// 32 voxels per SM in FP32, 32 in FP64: 304,000 and 152,000 voxels). A sweep then
// reads the neighbours' values only (from the L2: other blocks wrote them), and
// what remains is the grid barrier, one per Jacobi sweep and one per colour.
// Same arithmetic and stop test as the sweeps launched one by one. A
// Gauss-Seidel sweep at 65^3 takes 24 us (35 us with gs_plane_kernel), eight
// barriers and eight times the latency of 26 loads and their products; whole
// solves with it, the rest unchanged: 65^3 float-float with Gauss-Seidel 269 ->
// 238 ms, 33^3 FP64 with Jacobi 44.7 -> 37.3 ms.
// Block of 32 voxels i warps + w of a thread block is slot i of warp w. Jacobi
// spreads them over 16 warps; Gauss-Seidel has a warp for every block of a
// colour, so that slot i holds colour i, and more registers a thread.
template <typename A, bool GS> struct Resident {
    static constexpr int kBlocks = sizeof(A) == 4 ? 64 : 32;  // per thread block
    static constexpr int kWarps = GS ? kBlocks / 8 : 16;
    static constexpr int kSlots = kBlocks / kWarps;  // per warp
    static constexpr size_t kBytes = (size_t)kBlocks * 26 * 32 * sizeof(A);
};

template <typename A, bool GS>
__global__ void __launch_bounds__(32 * Resident<A, GS>::kWarps, 1)
    os_resident_kernel(int nx, int ny, int nz, ColourGeo cg, const A *__restrict__ a,
                       const double *__restrict__ inv_diag, const double *__restrict__ r, double *buf0,
                       double *buf1, A *val0, A *val1, int max_sweeps, double tol, OsState *st,
                       Periodic per) {
    namespace coop = cooperative_groups;
    using R = Resident<A, GS>;
    coop::grid_group grid = coop::this_grid();
    extern __shared__ __align__(16) unsigned char res_smem[];
    A *const coef = reinterpret_cast<A *>(res_smem);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long N = (long long)nx * ny * nz;
    const int nxy = nx * ny;
    // this thread's voxel of every slot (-1: none), packed as x | y << 11 | z << 22
    int at[R::kSlots];
    double rv[R::kSlots], id[R::kSlots];
#pragma unroll
    for (int i = 0; i < R::kSlots; ++i) {
        const int b = i * R::kWarps + warp;  // block of this thread block
        const int c = GS ? i : 0, j = GS ? warp : b;
        const long long blk = blockIdx.x + (long long)gridDim.x * j;
        const long long k = 32 * blk + lane, cnt = GS ? cg.cnt[c] : N;
        at[i] = -1;
        rv[i] = id[i] = 0.0;
        if (32 * blk < cnt) {
            const A *from = a + (GS ? os_colour_index(0, cg.blk[c] + blk, 0) : os_coef_index(0, 32 * blk));
            const unsigned to = (unsigned)__cvta_generic_to_shared(coef + b * 26 * 32);
            for (int q = 16 * lane; q < 26 * 32 * (int)sizeof(A); q += 512)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(to + q),
                             "l"(reinterpret_cast<const unsigned char *>(from) + q)
                             : "memory");
        }
        if (k < cnt) {
            int x, y, z;
            if (GS) {
                const int nxc = cg.nxc[c], kxy = nxc * cg.nyc[c];
                const int zi = (int)(k / kxy), rem = (int)(k - (long long)zi * kxy), yi = rem / nxc;
                x = 2 * (rem - yi * nxc) + (c & 1);
                y = 2 * yi + ((c >> 1) & 1);
                z = 2 * zi + (c >> 2);
            } else {
                z = (int)(k / nxy);
                const int rem = (int)(k - (long long)z * nxy);
                y = rem / nx;
                x = rem - y * nx;
            }
            at[i] = x | (y << 11) | (z << 22);
            const int v = x + nx * y + nxy * z;
            rv[i] = r[v];
            id[i] = inv_diag[v];
        }
    }
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
    __syncwarp();

    for (int m = 1; m <= max_sweeps; ++m) {
        double *const dst = m & 1 ? buf1 : buf0;
        const A *const src = m & 1 ? val0 : val1;
        A *const now = m & 1 ? val1 : val0;
        A dmax = A(0), jmax = A(0);
#pragma unroll
        for (int i = 0; i < R::kSlots; ++i) {
            const int c = i;  // Gauss-Seidel's colour
            if (at[i] >= 0) {
                // opaque: 26 addresses a slot kept over the sweeps would spill
                int packed = at[i];
                asm volatile("" : "+r"(packed));
                const int x = packed & 0x7ff, y = (packed >> 11) & 0x7ff, z = packed >> 22;
                const int v = x + nx * y + nxy * z;
                const int X[3] = {os_nb_lo(x, nx, per.x), x, os_nb_hi(x, nx, per.x)};
                const int Y[3] = {os_nb_lo(y, ny, per.y), y, os_nb_hi(y, ny, per.y)};
                const int Z[3] = {os_nb_lo(z, nz, per.z), z, os_nb_hi(z, nz, per.z)};
                A xv[26];
#pragma unroll
                for (int d = 0, p = 0; d < 27; ++d) {
                    if (d == 13) continue;
                    const int xn = X[d % 3], yn = Y[(d / 3) % 3], zn = Z[d / 9];
                    const A *from = src;
                    // this sweep's value where the neighbour's colour came earlier
                    if (GS && (xn & 1) + 2 * (yn & 1) + 4 * (zn & 1) < c) from = now;
                    xv[p] = __ldcg(from + (xn + nx * yn + nxy * zn));
                    ++p;
                }
                const A was = __ldcg(src + v);
                const A *cf = coef + (i * R::kWarps + warp) * 26 * 32 + lane;
                A acc = A(0);
#pragma unroll
                for (int p = 0; p < 26; ++p) acc += cf[32 * p] * xv[p];
                const double nv = (rv[i] + (double)acc) * id[i];
                dst[v] = nv;
                const A val = (A)nv;
                if constexpr (sizeof(A) == 4) {
                    now[v] = val;
                    dmax = fmaxf(dmax, fabsf(val - was));
                    jmax = fmaxf(jmax, fabsf(val));
                } else {
                    dmax = fmax(dmax, fabs(val - was));
                    jmax = fmax(jmax, fabs(val));
                }
            }
            if (GS && c < 7) grid.sync();
        }
        block_max_atomic((double)dmax, &st->dmax[m]);
        block_max_atomic((double)jmax, &st->jmax[m]);
        grid.sync();
        const double dm = bitsd(__ldcg(&st->dmax[m])), jm = bitsd(__ldcg(&st->jmax[m]));
        if (dm <= tol * jm) {
            // the stop test of the sweeps launched one by one: met after the
            // last sweep it is not looked at
            if (m < max_sweeps && blockIdx.x == 0 && threadIdx.x == 0) {
                st->done = 1;
                st->count = m;
            }
            return;
        }
    }
}

// ---- BiCGStab (van der Vorst 1992) on A x = r, A = [1 - Lambda*(1 - eps)],
// from x = 0, as the oracle's orc_os_bicgstab: scalars on the device, dot
// products accumulated by the kernels that produce their operands.

// block sum of v (all threads), added to *out by thread 0 of each block
__device__ __forceinline__ void block_sum_atomic(double v, double *out) {
    __shared__ double part[32];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) part[w] = v;
    __syncthreads();
    if (w == 0) {
        v = lane < (int)(blockDim.x >> 5) ? part[lane] : 0.0;
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (lane == 0) atomicAdd(out, v);
    }
}

// (A x)_v = diag_v x_v - sum_d a_d(v) x_{v+d}
template <typename A>
__device__ __forceinline__ double os_apply(const A *a, const double *diag, const double *x, int v,
                                           int nx, int ny, int nz, Periodic per) {
    return diag[v] * x[v] - (double)os_stencil(a, x, v, nx, ny, nz, per);
}

__global__ void bicg_init_kernel(int n, const double *r, BicgVecs vv, BicgState *bs) {
    const int tid = blockIdx.x * blockDim.x + threadIdx.x;
    if (tid == 0) {
        bs->rho = bs->alpha = bs->omega = 1.0;
        bs->rhv = bs->tt = bs->ts = bs->rr = 0.0;
    }
    double acc = 0.0;
    for (int i = tid; i < n; i += gridDim.x * blockDim.x) {
        const double ri = r[i];
        vv.x[i] = 0.0;
        vv.res[i] = ri;
        vv.rh[i] = ri;
        vv.p[i] = 0.0;
        vv.vv[i] = 0.0;
        acc += ri * ri;
    }
    block_sum_atomic(acc, &bs->rr0);
}

// rho1 = rh . res
__global__ void bicg_rho_kernel(int n, BicgVecs v, BicgState *bs) {
    double acc = 0.0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        acc += v.rh[i] * v.res[i];
    block_sum_atomic(acc, &bs->rho1);
}

// p = res + beta (p - omega vv), beta = (rho1/rho)(alpha/omega)
__global__ void bicg_p_kernel(int n, BicgVecs v, BicgState *bs) {
    const double beta = (bs->rho1 / bs->rho) * (bs->alpha / bs->omega), om = bs->omega;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        v.p[i] = v.res[i] + beta * (v.p[i] - om * v.vv[i]);
}

// vv = A p; rhv = rh . vv
template <typename A>
__global__ void __launch_bounds__(256) bicg_vv_kernel(int nx, int ny, int nz, const A *__restrict__ a,
                                                      const double *__restrict__ diag, BicgVecs v,
                                                      BicgState *bs, Periodic per) {
    const int n = nx * ny * nz;
    double acc = 0.0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const double y = os_apply(a, diag, v.p, i, nx, ny, nz, per);
        v.vv[i] = y;
        acc += v.rh[i] * y;
    }
    block_sum_atomic(acc, &bs->rhv);
}

// alpha = rho1 / rhv; sv = res - alpha vv
__global__ void bicg_s_kernel(int n, BicgVecs v, BicgState *bs) {
    const double alpha = bs->rho1 / bs->rhv;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        v.sv[i] = v.res[i] - alpha * v.vv[i];
}

// t = A sv; tt = t . t; ts = t . sv
template <typename A>
__global__ void __launch_bounds__(256) bicg_t_kernel(int nx, int ny, int nz, const A *__restrict__ a,
                                                     const double *__restrict__ diag, BicgVecs v,
                                                     BicgState *bs, Periodic per) {
    const int n = nx * ny * nz;
    double att = 0.0, ats = 0.0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const double y = os_apply(a, diag, v.sv, i, nx, ny, nz, per);
        v.t[i] = y;
        att += y * y;
        ats += y * v.sv[i];
    }
    block_sum_atomic(att, &bs->tt);
    block_sum_atomic(ats, &bs->ts);
}

// omega = ts / tt (0 if tt = 0); x += alpha p + omega sv; res = sv - omega t;
// rr = res . res
__global__ void bicg_x_kernel(int n, BicgVecs v, BicgState *bs) {
    const double alpha = bs->rho1 / bs->rhv;
    const double om = bs->tt > 0.0 ? bs->ts / bs->tt : 0.0;
    double acc = 0.0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        v.x[i] += alpha * v.p[i] + om * v.sv[i];
        const double ri = v.sv[i] - om * v.t[i];
        v.res[i] = ri;
        acc += ri * ri;
    }
    block_sum_atomic(acc, &bs->rr);
}

// end of an iteration: rho = rho1, alpha and omega kept; accumulators of the
// next iteration zeroed (rr stays for the host's stop test)
__global__ void bicg_next_kernel(BicgState *bs) {
    bs->alpha = bs->rho1 / bs->rhv;
    bs->omega = bs->tt > 0.0 ? bs->ts / bs->tt : 0.0;
    bs->rho = bs->rho1;
    bs->rho1 = 0.0;
    bs->rhv = 0.0;
    bs->tt = 0.0;
    bs->ts = 0.0;
}

__global__ void bicg_zero_rr_kernel(BicgState *bs) { bs->rr = 0.0; }

__global__ void os_set_result_kernel(int n, const double *src, double *dst, int k, OsState *st) {
    const int tid = blockIdx.x * blockDim.x + threadIdx.x;
    if (tid == 0) {
        st->done = 1;
        st->count = k;
        st->sweeps_total += (unsigned long long)k;
    }
    if (dst != src)
        for (int i = tid; i < n; i += gridDim.x * blockDim.x) dst[i] = src[i];
}

// r = Jfs - J (+ extra); dJ0 = r / diag; resets the sweep state.
__global__ void os_init_kernel(int n, const double *Jfs, const double *J, const double *extra,
                               const double *inv_diag, double *r, double *dJ0, float *dJ0_32,
                               OsState *st) {
    const int tid = blockIdx.x * blockDim.x + threadIdx.x;
    if (tid == 0) {
        st->done = 0;
        st->count = 0;
    }
    if (tid < 260) {
        st->dmax[tid] = 0ULL;
        st->jmax[tid] = 0ULL;
    }
    for (int v = tid; v < n; v += gridDim.x * blockDim.x) {
        double rv = Jfs ? Jfs[v] : 0.0;
        if (J) rv -= J[v];
        if (extra) rv += extra[v];
        r[v] = rv;
        const double d0 = rv * inv_diag[v];
        dJ0[v] = d0;
        if (dJ0_32) dJ0_32[v] = (float)d0;
    }
}

// One Jacobi sweep dst = (r + sum_d a_d src_{v+d}) / diag over all voxels
// (os_stencil's order), with the stop test of the previous sweep first. The mixed
// mode (A = float) multiplies by the FP32 copy of the previous sweep and
// keeps the iterate, r and 1/diag in FP64; its stop test compares against
// that copy.
// Bound by reading the coefficients (104 bytes a voxel in FP32). With 26 loads a
// thread into registers too few bytes were in flight, and with 2432 thread blocks
// the last wave was half empty; here a warp copies the next blocks of 32 voxels
// (contiguous, 3.3 kB) into a ring in shared memory while it works on one, and
// three thread blocks (two in FP64) stay on an SM, each with a contiguous run of
// voxels (the neighbours' rows are found in its L1). Solves of 50 sweeps, before
// and after: 97^3 2.06 -> 1.56 ms, 129^3 4.23 -> 3.25 ms, 161^3 7.6 -> 5.8 ms; FP64
// 97^3 3.51 -> 3.44 ms, 161^3 13.7 -> 12.7 ms. Rings of three or four stages at two
// blocks, four blocks at 64 registers and blocks of 6 or 16 warps were no faster.
template <typename A> struct SweepRing {
    static constexpr int kWarps = 8, kStages = 2;
    static constexpr int kCtas = sizeof(A) == 4 ? 3 : 2;  // per SM
    static constexpr int kBlock = 26 * 32 * (int)sizeof(A);  // bytes
    static constexpr size_t kBytes = (size_t)kWarps * kStages * kBlock;
};

template <typename A>
__global__ void __launch_bounds__(32 * SweepRing<A>::kWarps, SweepRing<A>::kCtas)
    os_sweep_kernel(int nx, int ny, int nz, const A *__restrict__ a, const double *__restrict__ inv_diag,
                    const double *__restrict__ r, const double *__restrict__ src,
                    double *__restrict__ dst, const float *__restrict__ src32, float *__restrict__ dst32,
                    int m, double tol, OsState *st, Periodic per) {
    using R = SweepRing<A>;
    constexpr bool f32 = sizeof(A) == 4;
    extern __shared__ __align__(16) unsigned char sweep_smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nxy = nx * ny, N = nxy * nz;
    const int nb = (N + 31) >> 5;  // blocks of 32 voxels; a contiguous run of them per thread block
    const int begin = (int)((long long)nb * blockIdx.x / gridDim.x);
    const int end = (int)((long long)nb * (blockIdx.x + 1) / gridDim.x);
    A *const ring = reinterpret_cast<A *>(sweep_smem) + warp * R::kStages * 26 * 32;
    const unsigned to = (unsigned)__cvta_generic_to_shared(ring);
    auto fetch = [&](int b, int stage) {
        if (b < end) {
            const unsigned char *from = reinterpret_cast<const unsigned char *>(a + os_coef_index(0, 32LL * b));
#pragma unroll
            for (int q = 0; q < R::kBlock; q += 512)
                if (q + 512 <= R::kBlock || q + 16 * lane < R::kBlock)
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(to + stage * R::kBlock + q + 16 * lane),
                                 "l"(from + q + 16 * lane)
                                 : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
#pragma unroll
    for (int i = 0; i < R::kStages; ++i) fetch(begin + warp + i * R::kWarps, i);
    bool stop = st->done;
    if (!stop && m >= 2) {
        const double dm = bitsd(st->dmax[m - 1]), jm = bitsd(st->jmax[m - 1]);
        stop = dm <= tol * jm;
        if (stop && blockIdx.x == 0 && threadIdx.x == 0) {
            st->done = 1;
            st->count = m - 1;
        }
    }
    if (stop) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        return;
    }
    // stop-test maxima in A (FP32 in the mixed mode: a 1e-3 relative test)
    A dmax = A(0), jmax = A(0);
    int stage = 0;
    for (int b = begin + warp; b < end; b += R::kWarps) {
        const int v = min(32 * b + lane, N - 1);
        const int z = v / nxy, rem = v - z * nxy, y = rem / nx, x = rem - y * nx;
        const int X[3] = {os_nb_lo(x, nx, per.x), x, os_nb_hi(x, nx, per.x)};
        const int Y[3] = {os_nb_lo(y, ny, per.y) * nx, y * nx, os_nb_hi(y, ny, per.y) * nx};
        const int Z[3] = {os_nb_lo(z, nz, per.z) * nxy, z * nxy, os_nb_hi(z, nz, per.z) * nxy};
        A xv[26];
#pragma unroll
        for (int d = 0, p = 0; d < 27; ++d) {
            if (d == 13) continue;
            const int u = X[d % 3] + Y[(d / 3) % 3] + Z[d / 9];
            if constexpr (f32) xv[p] = src32[u];
            else xv[p] = src[u];
            ++p;
        }
        A was;
        if constexpr (f32) was = src32[v];
        else was = src[v];
        const double rv = r[v], id = inv_diag[v];
        asm volatile("cp.async.wait_group %0;" ::"n"(R::kStages - 1) : "memory");
        __syncwarp();
        const A *c = ring + stage * 26 * 32 + lane;
        A acc = A(0);
#pragma unroll
        for (int p = 0; p < 26; ++p) acc += c[32 * p] * xv[p];
        __syncwarp();  // all lanes have read the stage
        fetch(b + R::kStages * R::kWarps, stage);
        stage = stage + 1 == R::kStages ? 0 : stage + 1;
        const double nv = (rv + (double)acc) * id;
        if (32 * b + lane < N) {
            dst[v] = nv;
            const A val = (A)nv;
            if constexpr (f32) {
                dst32[v] = val;
                dmax = fmaxf(dmax, fabsf(val - was));
                jmax = fmaxf(jmax, fabsf(val));
            } else {
                dmax = fmax(dmax, fabs(val - was));
                jmax = fmax(jmax, fabs(val));
            }
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    block_max_atomic((double)dmax, &st->dmax[m]);
    block_max_atomic((double)jmax, &st->jmax[m]);
}

__global__ void os_finish_kernel(int max_sweeps, double tol, OsState *st) {
    if (!st->done) {
        st->done = 1;
        st->count = max_sweeps;
    }
    st->sweeps_total += (unsigned long long)st->count;
}

// J += dJ (dJ = the final sweep buffer); rel = max |dJ| / |J_new|.
__global__ void ali_update_kernel(int n, double *J, double *const *buf, OsState *st,
                                  double *dJ_out) {
    const double *dJ = buf[st->count & 1];
    double rel = 0.0;
    bool bad = false;
    for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
        const double d = dJ[v];
        const double jn = J[v] + d;
        J[v] = jn;
        if (dJ_out) dJ_out[v] = d;
        if (d != 0.0) rel = fmax(rel, fabs(d) / fabs(jn));
        bad |= !(fabs(jn) <= 1.79e308);
    }
    block_max_atomic(bad ? __longlong_as_double(0x7ff8000000000000LL) : rel, &st->rel);
}

__global__ void copy_buf_kernel(int n, double *const *buf, const OsState *st, double *dst) {
    const double *src = buf[st->count & 1];
    for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x)
        dst[v] = src[v];
}

// J += d; rel = max |d| / |J_new|; amax = max |d|.
__global__ void axpy_rel_kernel(int n, double *J, const double *d, OsState *st) {
    double rel = 0.0;
    bool bad = false;
    for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
        const double jn = J[v] + d[v];
        J[v] = jn;
        if (d[v] != 0.0) rel = fmax(rel, fabs(d[v]) / fabs(jn));
        bad |= !(fabs(jn) <= 1.79e308);
    }
    block_max_atomic(bad ? __longlong_as_double(0x7ff8000000000000LL) : rel, &st->rel);
}

// r = Jfs - J; res = max |r| / |J|.
__global__ void residual_kernel(int n, const double *Jfs, const double *J, double *r,
                                OsState *st) {
    double res = 0.0;
    bool bad = false;
    for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
        const double rv = Jfs[v] - J[v];
        if (r) r[v] = rv;
        if (rv != 0.0) res = fmax(res, fabs(rv) / fabs(J[v]));
        bad |= !(fabs(rv) <= 1.79e308);
    }
    block_max_atomic(bad ? __longlong_as_double(0x7ff8000000000000LL) : res, &st->res);
}

__global__ void compare_kernel(long long n, const double *a, const double *b, OsState *st) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x) {
        if (__double_as_longlong(a[i]) != __double_as_longlong(b[i])) {
            st->changed = 1;
            return;
        }
    }
}

int grid_for(long long n, int threads) {
    long long b = (n + threads - 1) / threads;
    const long long cap = 16LL * device_sm_count();
    if (b > cap) b = cap;
    if (b < 1) b = 1;
    return (int)b;
}

}  // namespace

cudaError_t launch_pack(int nx, int ny, int nz, const double *chi, double scale, const double *S,
                        void *chiS, bool fp64, cudaStream_t s) {
    const long long n = (long long)nx * ny * nz;
    pack_kernel<<<grid_for(n, 256), 256, 0, s>>>(nx, ny, nz, chi, scale, S, chiS, fp64);
    return cudaGetLastError();
}

cudaError_t launch_source(int nx, int ny, int nz, const double *J, const double *eps,
                          const double *B, void *chiS, bool fp64, bool homogeneous,
                          cudaStream_t s) {
    const long long n = (long long)nx * ny * nz;
    source_kernel<<<grid_for(n, 256), 256, 0, s>>>(nx, ny, nz, J, eps, B, chiS, fp64, homogeneous);
    return cudaGetLastError();
}

cudaError_t launch_diffusion_bc(int nx, int ny, int nz, int nl, const double *chi,
                                const double *B, double *I_face, double *grad, cudaStream_t s) {
    const long long nf = (long long)nx * ny;
    diffusion_bc_kernel<<<grid_for(nf * nl, 256), 256, 0, s>>>(nf, nz, nl, chi, B, I_face, grad);
    return cudaGetLastError();
}

ColourGeo colour_geo(int nx, int ny, int nz) {
    ColourGeo cg{};
    long long blk = 0;
    for (int c = 0; c < 8; ++c) {
        const int px = c & 1, py = (c >> 1) & 1, pz = c >> 2;
        cg.nxc[c] = (nx - px + 1) / 2;
        cg.nyc[c] = (ny - py + 1) / 2;
        const long long nzc = (nz - pz + 1) / 2;
        cg.cnt[c] = (long long)cg.nxc[c] * cg.nyc[c] * nzc;
        cg.blk[c] = blk;
        blk += (cg.cnt[c] + 31) >> 5;
    }
    return cg;
}

// Blocks per plane and pairs of rows per block of the plane kernel: the
// smallest cluster that fits its rows into shared memory and gives the GPU a
// block per SM from the planes of one parity, at most 8. False where the
// kernel does not apply: the planes of one parity meet across a periodic z
// axis of odd length, or a plane's rows do not fit.
template <typename A>
static bool gs_plane_shape(int nx, int ny, int nz, Periodic per, int *ranks, int *band,
                           GsShared<A> *g) {
    if (per.z && (nz & 1)) return false;
    const int pairs = (ny + 1) / 2, planes = (nz + 1) / 2;
    for (*ranks = 1; *ranks <= 8; *ranks *= 2) {
        *band = (pairs + *ranks - 1) / *ranks;
        *g = GsShared<A>{nx + 2, 2 * *band + 2};
        const bool full = (long long)planes * *ranks * 4 >= 3LL * device_sm_count();
        if (g->bytes() <= 220 * 1024 && (full || *ranks == 8 || *band == 1)) return true;
    }
    return false;
}

// The planes of both parities in turn; returns how many colours have been launched:
// all eight, or fewer (0, 4) where a launch is refused.
template <typename A, bool SEAM>
static int gs_planes(int nx, int ny, int nz, const ColourGeo &cg, int ranks, int band,
                     const GsShared<A> &g, const A *a, const double *inv_diag, const double *r,
                     const double *src, double *dst, const float *src32, float *dst32, int m, double tol,
                     OsState *st, cudaStream_t s, Periodic per) {
    const size_t shm = g.bytes();
    if (shm > 48 * 1024 &&
        cudaFuncSetAttribute(gs_plane_kernel<A, SEAM>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)shm) != cudaSuccess)
        return 0;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = ranks;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cudaLaunchConfig_t lc{};
    lc.blockDim = dim3(std::min(512, (band * ((nx + 1) / 2) + 31) / 32 * 32));
    lc.dynamicSmemBytes = shm;
    lc.stream = s;
    lc.attrs = &at;
    lc.numAttrs = 1;
    for (int pz = 0; pz < 2 && pz < nz; ++pz) {
        lc.gridDim = dim3((nz - pz + 1) / 2 * ranks);
        if (cudaLaunchKernelEx(&lc, gs_plane_kernel<A, SEAM>, nx, ny, nz, cg, pz, band, g, a, inv_diag, r,
                               src, dst, src32, dst32, m, tol, st, per) != cudaSuccess)
            return 4 * pz;
    }
    return 8;
}

cudaError_t launch_gs_sweep(int nx, int ny, int nz, const ColourGeo &cg, const void *a, bool a64,
                            const double *inv_diag, const double *r, const double *src,
                            double *dst, const float *src32, float *dst32, int m, double tol,
                            OsState *st, cudaStream_t s, Periodic per, int *launches) {
    auto planes = [&](const auto *x) -> int {
        using A = std::remove_const_t<std::remove_pointer_t<decltype(x)>>;
        int ranks = 0, band = 0;
        GsShared<A> g{};
        if (!gs_plane_shape<A>(nx, ny, nz, per, &ranks, &band, &g)) return 0;
        const bool seam = (per.x && (nx & 1)) || (per.y && (ny & 1));
        return seam ? gs_planes<A, true>(nx, ny, nz, cg, ranks, band, g, x, inv_diag, r, src, dst, src32,
                                         dst32, m, tol, st, s, per)
                    : gs_planes<A, false>(nx, ny, nz, cg, ranks, band, g, x, inv_diag, r, src, dst, src32,
                                          dst32, m, tol, st, s, per);
    };
    const int first = a64 ? planes(static_cast<const double *>(a)) : planes(static_cast<const float *>(a));
    *launches = first == 8 && nz == 1 ? 1 : first / 4 + (8 - first);
    if (first == 8) return cudaSuccess;
    // colour by colour, also where a cluster is refused (part of the SMs is not
    // ours); what ails more than the cluster shows in these launches too
    cudaGetLastError();
    for (int c = first; c < 8; ++c) {
        const int blocks = grid_for(cg.cnt[c] > 0 ? cg.cnt[c] : 1, 256);
        if (a64)
            gs_colour_kernel<double><<<blocks, 256, 0, s>>>(nx, ny, nz, cg, c,
                                                            static_cast<const double *>(a), inv_diag,
                                                            r, src, dst, nullptr, nullptr, m, tol,
                                                            st, per);
        else
            gs_colour_kernel<float><<<blocks, 256, 0, s>>>(nx, ny, nz, cg, c,
                                                           static_cast<const float *>(a), inv_diag, r,
                                                           src, dst, src32, dst32, m, tol, st, per);
    }
    return cudaGetLastError();
}

// Whether the resident solve fits, and its number of thread blocks.
template <typename A>
static bool os_resident_shape(long long N, bool gs, const ColourGeo &cg, int *grid) {
    using R = Resident<A, true>;
    long long most = (N + 31) / 32;
    if (gs)
        for (int c = most = 0; c < 8; ++c) most = std::max(most, (cg.cnt[c] + 31) / 32);
    const int per = gs ? R::kWarps : R::kBlocks;
    *grid = (int)std::min<long long>(most, device_sm_count());
    return *grid >= 1 && most <= (long long)per * *grid;
}

template <typename A, bool GS>
static cudaError_t os_resident(int nx, int ny, int nz, ColourGeo cg, int grid, const A *a,
                               const double *inv_diag, const double *r, double *const *buf, A *val0,
                               A *val1, int max_sweeps, double tol, OsState *st, cudaStream_t s,
                               Periodic per) {
    auto *k = os_resident_kernel<A, GS>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)Resident<A, GS>::kBytes);
    if (e != cudaSuccess) return e;
    double *b0 = buf[0], *b1 = buf[1];
    void *args[] = {&nx, &ny, &nz, &cg, &a, &inv_diag, &r, &b0, &b1, &val0, &val1,
                    &max_sweeps, &tol, &st, &per};
    return cudaLaunchCooperativeKernel(reinterpret_cast<void *>(k), dim3(grid),
                                       dim3(32 * Resident<A, GS>::kWarps), args,
                                       Resident<A, GS>::kBytes, s);
}

cudaError_t launch_os_resident(int nx, int ny, int nz, bool gs, const void *a, bool a64,
                               const double *inv_diag, const double *r, double *const *buf,
                               float *const *buf32, int max_sweeps, double tol, OsState *st,
                               cudaStream_t s, Periodic per, bool *ran) {
    const long long N = (long long)nx * ny * nz;
    const ColourGeo cg = colour_geo(nx, ny, nz);
    int grid = 0;
    *ran = nx < 2048 && ny < 2048 && nz < 512 &&
           (a64 ? os_resident_shape<double>(N, gs, cg, &grid) : os_resident_shape<float>(N, gs, cg, &grid));
    if (!*ran) return cudaSuccess;
    cudaError_t e;
    if (a64) {
        const double *x = static_cast<const double *>(a);
        e = gs ? os_resident<double, true>(nx, ny, nz, cg, grid, x, inv_diag, r, buf, buf[0], buf[1],
                                           max_sweeps, tol, st, s, per)
               : os_resident<double, false>(nx, ny, nz, cg, grid, x, inv_diag, r, buf, buf[0], buf[1],
                                            max_sweeps, tol, st, s, per);
    } else {
        const float *x = static_cast<const float *>(a);
        e = gs ? os_resident<float, true>(nx, ny, nz, cg, grid, x, inv_diag, r, buf, buf32[0], buf32[1],
                                          max_sweeps, tol, st, s, per)
               : os_resident<float, false>(nx, ny, nz, cg, grid, x, inv_diag, r, buf, buf32[0], buf32[1],
                                           max_sweeps, tol, st, s, per);
    }
    if (e == cudaErrorCooperativeLaunchTooLarge) {  // part of the SMs is not ours: sweep by sweep
        cudaGetLastError();
        *ran = false;
        return cudaSuccess;
    }
    return e;
}

cudaError_t launch_bicg_init(int n, const double *r, const BicgVecs &v, BicgState *bs,
                             cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(&bs->rr0, 0, sizeof(double), s);
    if (e != cudaSuccess) return e;
    e = cudaMemsetAsync(&bs->rho1, 0, sizeof(double), s);
    if (e != cudaSuccess) return e;
    bicg_init_kernel<<<grid_for(n, 256), 256, 0, s>>>(n, r, v, bs);
    return cudaGetLastError();
}

cudaError_t launch_bicg_iteration(int nx, int ny, int nz, const void *a, bool a64,
                                  const double *diag, const BicgVecs &v, BicgState *bs,
                                  cudaStream_t s, Periodic per) {
    const int n = nx * ny * nz;
    const int b = grid_for(n, 256);
    bicg_rho_kernel<<<b, 256, 0, s>>>(n, v, bs);
    bicg_p_kernel<<<b, 256, 0, s>>>(n, v, bs);
    if (a64) bicg_vv_kernel<double><<<b, 256, 0, s>>>(nx, ny, nz, static_cast<const double *>(a), diag, v, bs, per);
    else bicg_vv_kernel<float><<<b, 256, 0, s>>>(nx, ny, nz, static_cast<const float *>(a), diag, v, bs, per);
    bicg_s_kernel<<<b, 256, 0, s>>>(n, v, bs);
    if (a64) bicg_t_kernel<double><<<b, 256, 0, s>>>(nx, ny, nz, static_cast<const double *>(a), diag, v, bs, per);
    else bicg_t_kernel<float><<<b, 256, 0, s>>>(nx, ny, nz, static_cast<const float *>(a), diag, v, bs, per);
    bicg_zero_rr_kernel<<<1, 1, 0, s>>>(bs);
    bicg_x_kernel<<<b, 256, 0, s>>>(n, v, bs);
    bicg_next_kernel<<<1, 1, 0, s>>>(bs);
    return cudaGetLastError();
}

cudaError_t launch_os_set_result(int n, const double *src, double *dst, int k, OsState *st,
                                 cudaStream_t s) {
    os_set_result_kernel<<<grid_for(n, 256), 256, 0, s>>>(n, src, dst, k, st);
    return cudaGetLastError();
}

cudaError_t launch_os_prep(int nx, int ny, int nz, const double *lstar, const double *eps,
                           void *a, bool a64, double *inv_diag, cudaStream_t s, Periodic per,
                           bool colour, double *diag) {
    const long long N = (long long)nx * ny * nz;
    const ColourGeo cg = colour_geo(nx, ny, nz);
    if (a64)
        os_prep_kernel<double><<<grid_for(N, 256), 256, 0, s>>>(
            nx, ny, nz, lstar, eps, static_cast<double *>(a), inv_diag, per, colour, cg, diag);
    else
        os_prep_kernel<float><<<grid_for(N, 256), 256, 0, s>>>(
            nx, ny, nz, lstar, eps, static_cast<float *>(a), inv_diag, per, colour, cg, diag);
    return cudaGetLastError();
}

cudaError_t launch_os_init(int n, const double *Jfs, const double *J, const double *extra,
                           const double *inv_diag, double *r, double *dJ0, float *dJ0_32,
                           OsState *st, cudaStream_t s) {
    int g = grid_for(n, 256);
    if (g < 2) g = 2;  // >= 260 threads to reset the sweep maxima
    os_init_kernel<<<g, 256, 0, s>>>(n, Jfs, J, extra, inv_diag, r, dJ0, dJ0_32, st);
    return cudaGetLastError();
}

template <typename A>
static cudaError_t os_sweep(int nx, int ny, int nz, const A *a, const double *inv_diag, const double *r,
                            const double *src, double *dst, const float *src32, float *dst32, int m,
                            double tol, OsState *st, cudaStream_t s, Periodic per) {
    using R = SweepRing<A>;
    cudaError_t e = cudaFuncSetAttribute(os_sweep_kernel<A>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)R::kBytes);
    if (e != cudaSuccess) return e;
    const long long nb = ((long long)nx * ny * nz + 31) / 32;
    const int grid = (int)std::min<long long>((nb + R::kWarps - 1) / R::kWarps, R::kCtas * device_sm_count());
    os_sweep_kernel<A><<<grid, 32 * R::kWarps, R::kBytes, s>>>(nx, ny, nz, a, inv_diag, r, src, dst, src32,
                                                               dst32, m, tol, st, per);
    return cudaGetLastError();
}

cudaError_t launch_os_sweep(int nx, int ny, int nz, const void *a, bool a64,
                            const double *inv_diag, const double *r, double *const *buf,
                            float *const *buf32, int m, double tol, OsState *st, cudaStream_t s,
                            Periodic per) {
    // buf, buf32: host arrays of the two device ping-pong buffers (FP64, FP32 copy)
    const double *src = buf[(m - 1) & 1];
    double *dst = buf[m & 1];
    const float *src32 = buf32 ? buf32[(m - 1) & 1] : nullptr;
    float *dst32 = buf32 ? buf32[m & 1] : nullptr;
    return a64 ? os_sweep(nx, ny, nz, static_cast<const double *>(a), inv_diag, r, src, dst, src32, dst32,
                          m, tol, st, s, per)
               : os_sweep(nx, ny, nz, static_cast<const float *>(a), inv_diag, r, src, dst, src32, dst32,
                          m, tol, st, s, per);
}

cudaError_t launch_os_finish(int max_sweeps, double tol, OsState *st, cudaStream_t s) {
    os_finish_kernel<<<1, 1, 0, s>>>(max_sweeps, tol, st);
    return cudaGetLastError();
}

cudaError_t launch_ali_update(int n, double *J, double *const *buf, OsState *st, double *dJ_out,
                              cudaStream_t s) {
    ali_update_kernel<<<grid_for(n, 256), 256, 0, s>>>(n, J, buf, st, dJ_out);
    return cudaGetLastError();
}

cudaError_t launch_copy_buf(int n, double *const *buf, const OsState *st, double *dst,
                            cudaStream_t s) {
    copy_buf_kernel<<<grid_for(n, 256), 256, 0, s>>>(n, buf, st, dst);
    return cudaGetLastError();
}

cudaError_t launch_axpy_rel(int n, double *J, const double *d, OsState *st, cudaStream_t s) {
    axpy_rel_kernel<<<grid_for(n, 256), 256, 0, s>>>(n, J, d, st);
    return cudaGetLastError();
}

cudaError_t launch_residual(int n, const double *Jfs, const double *J, double *r, OsState *st,
                            cudaStream_t s) {
    residual_kernel<<<grid_for(n, 256), 256, 0, s>>>(n, Jfs, J, r, st);
    return cudaGetLastError();
}

cudaError_t launch_compare(long long n, const double *a, const double *b, OsState *st,
                           cudaStream_t s) {
    compare_kernel<<<grid_for(n, 256), 256, 0, s>>>(n, a, b, st);
    return cudaGetLastError();
}

}  // namespace rt3d
