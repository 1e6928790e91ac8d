// Learned warm start: the layers of a small 3D U-Net that predicts log J of
// the converged solution from (log chi, log eps, B, log J_start). Not in the
// paper; the ALI/Krylov solve started from its prediction is certified by the
// same FP64 residual as any other start.
//
// Activations are BF16, channel-last [S][V][C] (S samples, V = nx*ny*nz
// voxels, x fastest, C a multiple of 16). Convolutions are 3x3x3, periodic in
// x and y, zero-padded in z (the geometry of the radiative-transfer box),
// computed as implicit GEMMs on the tensor cores (nn_conv.cu): BF16 operands,
// FP32 accumulation, mma.sync m16n8k16. Weights are stored per
// offset d = (dz+1)*9 + (dy+1)*3 + (dx+1) as Wt[d][Ci][Co] (BF16), with an
// FP32 master copy for the optimiser.
#include <cuda_bf16.h>

#include <type_traits>

#include "nn_conv.cuh"
#include "rt3d_internal.cuh"
#include "../../include/rt3d_nn.h"

namespace rt3d {

namespace {

using bf16 = __nv_bfloat16;

struct Geo {
    int nx, ny, nz;
};

// The elementwise kernels move W channels of a voxel per thread (W = 8: one
// 16-byte access, W = 1 where a pointer or a channel offset is not aligned to
// it; per_thread) and index with I, 32 bits while the element count fits.
// They are bound by their launch and by memory: with one channel a thread and
// 64-bit indices the upsampling of the training box took 43 us, its gradient
// 15 us and the ReLU gradient 14 us.
template <typename T, int W> struct __align__(sizeof(T) * W < 16 ? sizeof(T) * W : 16) Vec {
    T v[W];
};
template <int W, typename T> __device__ __forceinline__ Vec<T, W> vload(const T *p) {
    return *reinterpret_cast<const Vec<T, W> *>(p);
}
template <int W, typename T> __device__ __forceinline__ void vstore(T *p, const Vec<T, W> &v) {
    *reinterpret_cast<Vec<T, W> *>(p) = v;
}

// *p += v, each value atomically: several streams may accumulate into one buffer
template <int W> __device__ __forceinline__ void vadd(float *p, const Vec<float, W> &v) {
    if constexpr (W == 8) {
        atomicAdd(reinterpret_cast<float4 *>(p), make_float4(v.v[0], v.v[1], v.v[2], v.v[3]));
        atomicAdd(reinterpret_cast<float4 *>(p) + 1, make_float4(v.v[4], v.v[5], v.v[6], v.v[7]));
    } else {
        static_assert(W == 1, "one value or eight");
        atomicAdd(p, v.v[0]);
    }
}

// dYpre = dY * (Y > 0)
template <int W, typename I>
__global__ void relu_bwd_kernel(const bf16 *dY, const bf16 *Y, bf16 *out, I n) {
    for (I i = blockIdx.x * (I)blockDim.x + threadIdx.x; i < n; i += (I)gridDim.x * blockDim.x) {
        Vec<bf16, W> g = vload<W>(dY + W * i);
        const Vec<bf16, W> y = vload<W>(Y + W * i);
#pragma unroll
        for (int c = 0; c < W; ++c)
            if (!(__bfloat162float(y.v[c]) > 0.0f)) g.v[c] = __float2bfloat16(0.0f);
        vstore<W>(out + W * i, g);
    }
}

// Coordinates of voxel v of a grid
template <typename I> __device__ __forceinline__ int3 coords(I v, Geo g) {
    const I q = v / (I)g.nx, z = q / (I)g.ny;
    return make_int3((int)(v - q * (I)g.nx), (int)(q - z * (I)g.ny), (int)z);
}
// element i = W channels: channel, sample and voxel of a [S][V][C] tensor
template <int W, typename I>
__device__ __forceinline__ void split(I i, int C, I V, int &c, I &s, I &v) {
    const I cv = (I)(C / W), r = i / cv;
    c = (int)(i - r * cv) * W;
    s = r / V;
    v = r - s * V;
}

// 2x2x2 average (periodic in x, y; a child beyond the top layer counts as 0)
template <int W, typename I>
__global__ void pool_kernel(const bf16 *X, bf16 *P, Geo g, Geo p, int C, int S) {
    const I Vp = (I)p.nx * p.ny * p.nz, n = Vp * (C / W) * S;
    const long long V = (long long)g.nx * g.ny * g.nz;
    for (I i = blockIdx.x * (I)blockDim.x + threadIdx.x; i < n; i += (I)gridDim.x * blockDim.x) {
        int c;
        I s, vp;
        split<W>(i, C, Vp, c, s, vp);
        const int3 q = coords(vp, p);
        float acc[W] = {};
        for (int a = 0; a < 2; ++a) {
            const int zz = 2 * q.z + a;
            if (zz >= g.nz) continue;
            for (int b = 0; b < 2; ++b)
                for (int e = 0; e < 2; ++e) {
                    const int xx = (2 * q.x + e) % g.nx, yy = (2 * q.y + b) % g.ny;
                    const Vec<bf16, W> x = vload<W>(
                        X + (s * V + xx + (long long)g.nx * (yy + (long long)g.ny * zz)) * C + c);
#pragma unroll
                    for (int k = 0; k < W; ++k) acc[k] += __bfloat162float(x.v[k]);
                }
        }
        Vec<bf16, W> o;
#pragma unroll
        for (int k = 0; k < W; ++k) o.v[k] = __float2bfloat16(acc[k] * 0.125f);
        vstore<W>(P + (s * (long long)Vp + vp) * C + c, o);
    }
}

// dX[v] += dP[parent] / 8 over the parents of v: (x/2, y/2, z/2), and on an
// odd axis the last parent, whose second child wraps onto coordinate 0
template <int W, typename I>
__global__ void pool_bwd_kernel(const bf16 *dP, float *dX32, Geo g, Geo p, int C, int S) {
    const I V = (I)g.nx * g.ny * g.nz, n = V * (C / W) * S;
    const long long Vp = (long long)p.nx * p.ny * p.nz;
    for (I i = blockIdx.x * (I)blockDim.x + threadIdx.x; i < n; i += (I)gridDim.x * blockDim.x) {
        int c;
        I s, v;
        split<W>(i, C, V, c, s, v);
        const int3 q = coords(v, g);
        const int px[2] = {q.x / 2, p.nx - 1}, py[2] = {q.y / 2, p.ny - 1};
        const int ex = (g.nx & 1) && q.x == 0 ? 2 : 1, ey = (g.ny & 1) && q.y == 0 ? 2 : 1;
        float *o = dX32 + (s * (long long)V + v) * C + c;
        Vec<float, W> acc{};
        for (int b = 0; b < ey; ++b)
            for (int a = 0; a < ex; ++a) {
                const Vec<bf16, W> d = vload<W>(
                    dP + (s * Vp + px[a] + (long long)p.nx * (py[b] + (long long)p.ny * (q.z / 2))) * C + c);
#pragma unroll
                for (int k = 0; k < W; ++k) acc.v[k] += __bfloat162float(d.v[k]) * 0.125f;
            }
        vadd<W>(o, acc);
    }
}

// U[v][c] = X[parent(v)][c] written into channels [coff, coff + C) of a
// Ctot-channel buffer; the backward pass sums the children of every parent.
template <int W, typename I>
__global__ void up_kernel(const bf16 *X, bf16 *U, Geo g, Geo p, int C, int Ctot, int coff, int S) {
    const I V = (I)g.nx * g.ny * g.nz, n = V * (C / W) * S;
    const long long Vp = (long long)p.nx * p.ny * p.nz;
    for (I i = blockIdx.x * (I)blockDim.x + threadIdx.x; i < n; i += (I)gridDim.x * blockDim.x) {
        int c;
        I s, v;
        split<W>(i, C, V, c, s, v);
        const int3 q = coords(v, g);
        const long long par = q.x / 2 + (long long)p.nx * (q.y / 2 + (long long)p.ny * (q.z / 2));
        vstore<W>(U + (s * (long long)V + v) * Ctot + coff + c, vload<W>(X + (s * Vp + par) * C + c));
    }
}

template <int W, typename I>
__global__ void up_bwd_kernel(const bf16 *dU, float *dX32, Geo g, Geo p, int C, int Ctot, int coff,
                              int S) {
    const I Vp = (I)p.nx * p.ny * p.nz, n = Vp * (C / W) * S;
    const long long V = (long long)g.nx * g.ny * g.nz;
    for (I i = blockIdx.x * (I)blockDim.x + threadIdx.x; i < n; i += (I)gridDim.x * blockDim.x) {
        int c;
        I s, vp;
        split<W>(i, C, Vp, c, s, vp);
        const int3 q = coords(vp, p);
        float *o = dX32 + (s * (long long)Vp + vp) * C + c;
        Vec<float, W> acc{};
        for (int z = 2 * q.z; z < min(2 * q.z + 2, g.nz); ++z)
            for (int y = 2 * q.y; y < min(2 * q.y + 2, g.ny); ++y)
                for (int x = 2 * q.x; x < min(2 * q.x + 2, g.nx); ++x) {
                    const Vec<bf16, W> d = vload<W>(
                        dU + (s * V + x + (long long)g.nx * (y + (long long)g.ny * z)) * Ctot + coff + c);
#pragma unroll
                    for (int k = 0; k < W; ++k) acc.v[k] += __bfloat162float(d.v[k]);
                }
        vadd<W>(o, acc);
    }
}

// copy channels [coff, coff+C) of a Ctot-channel buffer to/from a C-channel one
template <int W, typename I>
__global__ void channel_copy_kernel(const bf16 *src, int Cs, int soff, bf16 *dst, int Cd, int doff,
                                    int C, I n) {
    for (I i = blockIdx.x * (I)blockDim.x + threadIdx.x; i < n; i += (I)gridDim.x * blockDim.x) {
        const I r = i / (I)(C / W);
        const int c = (int)(i - r * (I)(C / W)) * W;
        vstore<W>(dst + (long long)r * Cd + doff + c, vload<W>(src + (long long)r * Cs + soff + c));
    }
}

template <int W, typename I> __global__ void f32_to_bf16_kernel(const float *a, bf16 *b, I n) {
    for (I i = blockIdx.x * (I)blockDim.x + threadIdx.x; i < n; i += (I)gridDim.x * blockDim.x) {
        const Vec<float, W> x = vload<W>(a + W * i);
        Vec<bf16, W> o;
#pragma unroll
        for (int k = 0; k < W; ++k) o.v[k] = __float2bfloat16(x.v[k]);
        vstore<W>(b + W * i, o);
    }
}

template <int W, typename I>
__global__ void add_bf16_f32_kernel(const bf16 *a, const float *b, bf16 *out, I n) {
    for (I i = blockIdx.x * (I)blockDim.x + threadIdx.x; i < n; i += (I)gridDim.x * blockDim.x) {
        const Vec<bf16, W> x = vload<W>(a + W * i);
        const Vec<float, W> y = vload<W>(b + W * i);
        Vec<bf16, W> o;
#pragma unroll
        for (int k = 0; k < W; ++k) o.v[k] = __float2bfloat16(__bfloat162float(x.v[k]) + y.v[k]);
        vstore<W>(out + W * i, o);
    }
}

// Features from the radiative-transfer arrays (FP64 [S][V]) into a 16-channel
// BF16 tensor: log10(chi)/3, log10(eps)/4, B - 1, ln(J0), 12 zero channels.
__global__ void features_kernel(const double *chi, const double *eps, const double *B,
                                const double *J0, bf16 *X, long long rows) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < rows;
         i += (long long)gridDim.x * blockDim.x) {
        float f[16] = {0};
        f[0] = (float)(log10(chi[i]) / 3.0);
        f[1] = (float)(log10(eps[i]) / 4.0);
        f[2] = (float)(B[i] - 1.0);
        f[3] = (float)log(fmax(J0[i], 1e-300));
        for (int c = 0; c < 16; ++c) X[i * 16 + c] = __float2bfloat16(f[c]);
    }
}

// Loss on channel 0 of the FP32 network output y, read as the correction
// ln J - ln J0: L = mean (y - ln(target/J0))^2; the gradient dY (BF16, 16
// channels, zeros beyond channel 0) and the summed squared error are written.
__global__ void mse_kernel(const float *Yf, const double *target, const double *J0, bf16 *dY,
                           float *sse, long long rows, float scale) {
    float acc = 0.0f;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < rows;
         i += (long long)gridDim.x * blockDim.x) {
        const float e = Yf[i * 16] - (float)log(target[i] / J0[i]);
        acc += e * e;
        dY[i * 16] = __float2bfloat16(2.0f * e * scale);
        for (int c = 1; c < 16; ++c) dY[i * 16 + c] = __float2bfloat16(0.0f);
    }
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
    if ((threadIdx.x & 31) == 0) atomicAdd(sse, acc);
}

// J = J0 exp(y) (FP64 out)
__global__ void apply_kernel(const float *Yf, const double *J0, double *J, long long rows) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < rows;
         i += (long long)gridDim.x * blockDim.x)
        J[i] = J0[i] * exp((double)Yf[i * 16]);
}

// Adam on an FP32 master copy, then the BF16 working copy Wt[d][ci][co] and
// its transpose WT[d][co][ci] (for the data gradient).
__global__ void adam_kernel(float *w, const float *gw, float *m, float *v, int n, float lr,
                            float b1, float b2, float eps, float c1, float c2, bf16 *Wt, bf16 *WT,
                            int Ci, int Co) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const float gi = gw[i];
        const float mi = b1 * m[i] + (1.0f - b1) * gi;
        const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        const float wi = w[i] - lr * (mi * c1) / (sqrtf(vi * c2) + eps);
        w[i] = wi;
        if (Wt) {
            Wt[i] = __float2bfloat16(wi);
            const int d = i / (Ci * Co), rem = i % (Ci * Co), ci = rem / Co, co = rem % Co;
            WT[((long long)d * Co + co) * Ci + ci] = __float2bfloat16(wi);
        }
    }
}

// Whether eight channels a thread fit: element counts or channel offsets
// (or-ed into `count`) are multiples of 8 and every pointer is 16-byte aligned.
bool eight(long long count, const void *a, const void *b, const void *c = nullptr) {
    const uintptr_t p = reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b) |
                        reinterpret_cast<uintptr_t>(c);
    return ((count & 7) | (long long)(p & 15)) == 0;
}
// Calls f(W, index type's zero) for n scalars in all.
template <typename F> void per_thread(bool vec, long long n, F f) {
    using W8 = std::integral_constant<int, 8>;
    using W1 = std::integral_constant<int, 1>;
    // the grid-stride index of the last round stays below 2^32 too
    if (n < (1LL << 31)) {
        if (vec) f(W8{}, 0u);
        else f(W1{}, 0u);
    } else {
        if (vec) f(W8{}, 0ull);
        else f(W1{}, 0ull);
    }
}

int gsz(long long n) {
    long long b = (n + 255) / 256;
    const long long cap = 16LL * device_sm_count();
    return (int)(b < 1 ? 1 : (b > cap ? cap : b));
}

}  // namespace

}  // namespace rt3d

using namespace rt3d;

extern "C" {

static rt3d_status nn_err(cudaError_t e) {
    if (e == cudaSuccess) return RT3D_OK;
    set_last_error(cudaGetErrorString(e));
    return RT3D_ECUDA;
}

rt3d_status rt3d_nn_conv3d(const void *X, const void *Wt, const float *bias, void *Y, float *Yf,
                           int S, int nx, int ny, int nz, int Ci, int Co, int relu, int transpose,
                           void *stream) {
    if (Ci <= 0 || Ci % 16 || Ci > 96 || (Co != 16 && Co != 32 && Co != 48 && Co != 64 && Co != 96) ||
        S < 1) {
        set_last_error("conv3d: Ci must be a multiple of 16 up to 96 and Co one of 16/32/48/64/96");
        return RT3D_EINVAL;
    }
    const long long V = (long long)nx * ny * nz;
    if (V <= 0 || V * 64 >= (1LL << 31)) {
        set_last_error("conv3d: bad volume");
        return RT3D_EINVAL;
    }
    return nn_err(launch_conv3d(static_cast<const bf16 *>(X), static_cast<const bf16 *>(Wt), bias,
                                static_cast<bf16 *>(Y), Yf, S, nx, ny, nz, Ci, Co, relu != 0,
                                transpose ? -1 : 1, static_cast<cudaStream_t>(stream)));
}

rt3d_status rt3d_nn_conv3d_wgrad(const void *X, const void *dY, float *dW, float *db, int S, int nx,
                                 int ny, int nz, int Ci, int Co, void *stream) {
    if (Ci <= 0 || Ci % 16 || Ci > 96 || Co <= 0 || Co % 16 || (Ci / 16) * (Co / 16) > 16) {
        set_last_error("conv3d_wgrad: Ci <= 96 and (Ci/16)(Co/16) <= 16");
        return RT3D_EINVAL;
    }
    return nn_err(launch_conv3d_wgrad(static_cast<const bf16 *>(X), static_cast<const bf16 *>(dY), dW,
                                      db, S, nx, ny, nz, Ci, Co, static_cast<cudaStream_t>(stream)));
}

rt3d_status rt3d_nn_relu_bwd(const void *dY, const void *Y, void *out, long long n, void *stream) {
    per_thread(eight(n, dY, Y, out), n, [&](auto w, auto zero) {
        constexpr int W = decltype(w)::value;
        using I = decltype(zero);
        relu_bwd_kernel<W, I><<<gsz(n / W), 256, 0, static_cast<cudaStream_t>(stream)>>>(
            static_cast<const bf16 *>(dY), static_cast<const bf16 *>(Y), static_cast<bf16 *>(out),
            (I)(n / W));
    });
    return nn_err(cudaGetLastError());
}

rt3d_status rt3d_nn_pool(const void *X, void *P, int S, int nx, int ny, int nz, int C, void *stream) {
    Geo g{nx, ny, nz}, p{(nx + 1) / 2, (ny + 1) / 2, (nz + 1) / 2};
    const long long n = (long long)p.nx * p.ny * p.nz * C * S;
    per_thread(eight(C, X, P), n, [&](auto w, auto zero) {
        constexpr int W = decltype(w)::value;
        pool_kernel<W, decltype(zero)><<<gsz(n / W), 256, 0, static_cast<cudaStream_t>(stream)>>>(
            static_cast<const bf16 *>(X), static_cast<bf16 *>(P), g, p, C, S);
    });
    return nn_err(cudaGetLastError());
}

rt3d_status rt3d_nn_pool_bwd(const void *dP, float *dX32, int S, int nx, int ny, int nz, int C,
                             void *stream) {
    Geo g{nx, ny, nz}, p{(nx + 1) / 2, (ny + 1) / 2, (nz + 1) / 2};
    const long long n = (long long)nx * ny * nz * C * S;
    per_thread(eight(C, dP, dX32), n, [&](auto w, auto zero) {
        constexpr int W = decltype(w)::value;
        pool_bwd_kernel<W, decltype(zero)><<<gsz(n / W), 256, 0, static_cast<cudaStream_t>(stream)>>>(
            static_cast<const bf16 *>(dP), dX32, g, p, C, S);
    });
    return nn_err(cudaGetLastError());
}

rt3d_status rt3d_nn_upsample(const void *X, void *U, int S, int nx, int ny, int nz, int C, int Ctot,
                             int coff, void *stream) {
    Geo g{nx, ny, nz}, p{(nx + 1) / 2, (ny + 1) / 2, (nz + 1) / 2};
    const long long n = (long long)nx * ny * nz * C * S;
    per_thread(eight(C | Ctot | coff, X, U), n, [&](auto w, auto zero) {
        constexpr int W = decltype(w)::value;
        up_kernel<W, decltype(zero)><<<gsz(n / W), 256, 0, static_cast<cudaStream_t>(stream)>>>(
            static_cast<const bf16 *>(X), static_cast<bf16 *>(U), g, p, C, Ctot, coff, S);
    });
    return nn_err(cudaGetLastError());
}

rt3d_status rt3d_nn_upsample_bwd(const void *dU, float *dX32, int S, int nx, int ny, int nz, int C,
                                 int Ctot, int coff, void *stream) {
    Geo g{nx, ny, nz}, p{(nx + 1) / 2, (ny + 1) / 2, (nz + 1) / 2};
    const long long n = (long long)p.nx * p.ny * p.nz * C * S;
    per_thread(eight(C | Ctot | coff, dU, dX32), n, [&](auto w, auto zero) {
        constexpr int W = decltype(w)::value;
        up_bwd_kernel<W, decltype(zero)><<<gsz(n / W), 256, 0, static_cast<cudaStream_t>(stream)>>>(
            static_cast<const bf16 *>(dU), dX32, g, p, C, Ctot, coff, S);
    });
    return nn_err(cudaGetLastError());
}

rt3d_status rt3d_nn_channel_copy(const void *src, int Cs, int soff, void *dst, int Cd, int doff, int C,
                                 long long rows, void *stream) {
    per_thread(eight(C | Cs | soff | Cd | doff, src, dst), rows * C, [&](auto w, auto zero) {
        constexpr int W = decltype(w)::value;
        using I = decltype(zero);
        channel_copy_kernel<W, I><<<gsz(rows * (C / W)), 256, 0, static_cast<cudaStream_t>(stream)>>>(
            static_cast<const bf16 *>(src), Cs, soff, static_cast<bf16 *>(dst), Cd, doff, C,
            (I)(rows * (C / W)));
    });
    return nn_err(cudaGetLastError());
}

rt3d_status rt3d_nn_f32_to_bf16(const float *a, void *b, long long n, void *stream) {
    per_thread(eight(n, a, b), n, [&](auto w, auto zero) {
        constexpr int W = decltype(w)::value;
        using I = decltype(zero);
        f32_to_bf16_kernel<W, I><<<gsz(n / W), 256, 0, static_cast<cudaStream_t>(stream)>>>(
            a, static_cast<bf16 *>(b), (I)(n / W));
    });
    return nn_err(cudaGetLastError());
}

rt3d_status rt3d_nn_add_bf16_f32(const void *a, const float *b, void *out, long long n, void *stream) {
    per_thread(eight(n, a, b, out), n, [&](auto w, auto zero) {
        constexpr int W = decltype(w)::value;
        using I = decltype(zero);
        add_bf16_f32_kernel<W, I><<<gsz(n / W), 256, 0, static_cast<cudaStream_t>(stream)>>>(
            static_cast<const bf16 *>(a), b, static_cast<bf16 *>(out), (I)(n / W));
    });
    return nn_err(cudaGetLastError());
}

rt3d_status rt3d_nn_features(const double *chi, const double *eps, const double *B, const double *J0,
                             void *X, long long rows, void *stream) {
    features_kernel<<<gsz(rows), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        chi, eps, B, J0, static_cast<bf16 *>(X), rows);
    return nn_err(cudaGetLastError());
}

rt3d_status rt3d_nn_mse(const float *Yf, const double *target, const double *J0, void *dY, float *sse,
                        long long rows, float grad_scale, void *stream) {
    mse_kernel<<<gsz(rows), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        Yf, target, J0, static_cast<bf16 *>(dY), sse, rows, grad_scale);
    return nn_err(cudaGetLastError());
}

rt3d_status rt3d_nn_apply(const float *Yf, const double *J0, double *J, long long rows, void *stream) {
    apply_kernel<<<gsz(rows), 256, 0, static_cast<cudaStream_t>(stream)>>>(Yf, J0, J, rows);
    return nn_err(cudaGetLastError());
}

rt3d_status rt3d_nn_adam(float *w, const float *g, float *m, float *v, int n, float lr, float b1,
                         float b2, float eps, int step, void *Wt, void *WT, int Ci, int Co,
                         void *stream) {
    const float c1 = 1.0f / (1.0f - powf(b1, (float)step));
    const float c2 = 1.0f / (1.0f - powf(b2, (float)step));
    adam_kernel<<<gsz(n), 256, 0, static_cast<cudaStream_t>(stream)>>>(
        w, g, m, v, n, lr, b1, b2, eps, c1, c2, static_cast<bf16 *>(Wt), static_cast<bf16 *>(WT), Ci, Co);
    return nn_err(cudaGetLastError());
}

}  // extern "C"
