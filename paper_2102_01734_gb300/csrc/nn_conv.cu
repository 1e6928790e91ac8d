// Convolutions of the learned warm start as implicit GEMMs on the tensor
// cores (BF16 operands, FP32 accumulation, mma.sync m16n8k16 fed by ldmatrix
// from shared memory).
//
// A block takes a box of voxels (a tile) and holds in shared memory, for 16
// input channels at a time, the tile with its halo of one voxel (gathered once:
// 2.3 to 2.5 reads of an input value instead of 27) and the 27 taps' weights
// of those channels; a tap is then a shift of the addresses that ldmatrix
// takes, and nothing is staged per tap. The layers are small (16 to 96
// channels), so shared memory bandwidth bounds the inner loop (a 16 x 16
// operand tile feeds two to twelve products) and the tensor cores stay under a
// third busy; at the training box's coarse levels there are fewer tiles than
// SMs and the latency of one tile is what remains, so small volumes get
// smaller tiles (conv_tile). tcgen05 tiles of 128 rows would leave fewer
// tiles still.
//
// Training box 32 x 32 x 193 (device time of a step's launches, before: one
// 16 x 16 operand tile gathered per tap and warp): the 21 forward and data
// gradient convolutions 1460 -> 385 us (16 to 16 channels 62 -> 17 us, 48 to 16
// 113 -> 42 us), the 11 weight gradients 1820 -> 277 us and the bias gradients,
// 168 us in launches of their own, inside them. A whole training step 3.76 ->
// 0.92 ms.
//
// The sums run over blocks of 16 channels, the 27 taps inside. Against gradients
// in 64 bits, over 25 training steps on boxes of different sizes and 22 tensors
// each, the mean error is that of the taps-first order (ratio 0.999, per-tensor
// medians 0.97 to 1.02); a tensor of one step scatters either way, up to a factor of
// a few where its error is small, because BF16 roundings of the activations flip.
#include "nn_conv.cuh"

#include <algorithm>
#include <cstdint>

#include "rt3d_internal.cuh"

namespace rt3d {

namespace {

using bf16 = __nv_bfloat16;

// Tile of 2^lx x 2^ly x 2^lz voxels, its halo box hx x hy x hz, the tiles of
// a sample on each axis.
struct ConvTile {
    int lx, ly, lz, hx, hy, hz, tx, ty, tz;
    __host__ __device__ int halo() const { return hx * hy * hz; }
    __host__ __device__ int tiles() const { return tx * ty * tz; }
};
constexpr int kMaxHalo = 720;

__device__ __forceinline__ unsigned smem_addr(const void *p) {
    return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void cp_async16(unsigned dst, const bf16 *src, bool valid) {
    const int n = valid ? 16 : 0;  // 0: the 16 bytes are zero-filled, src is not read
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n)
                 : "memory");
}
// The same value by value, for arrays whose address is no multiple of 16.
__device__ __forceinline__ void copy16(unsigned dst, const bf16 *src, bool valid) {
    unsigned v[4] = {0u, 0u, 0u, 0u};
    if (valid) {
        const unsigned short *p = reinterpret_cast<const unsigned short *>(src);
#pragma unroll
        for (int i = 0; i < 4; ++i) v[i] = p[2 * i] | (unsigned)p[2 * i + 1] << 16;
    }
    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "r"(v[0]), "r"(v[1]), "r"(v[2]),
                 "r"(v[3])
                 : "memory");
}
// Bits of the kernels' `wide` argument: X, the other operand (weights or dY), and
// the outputs in pairs.
constexpr int kWideX = 1, kWideB = 2, kWideOut = 4;
int wide_operands(const bf16 *X, const bf16 *b) {
    return ((reinterpret_cast<uintptr_t>(X) & 15) == 0 ? kWideX : 0) |
           ((reinterpret_cast<uintptr_t>(b) & 15) == 0 ? kWideB : 0);
}
// at(i, copy) for the pieces i < n of an array, copy as its address allows. (One
// branch for the array: in the loop it cost a training step 3 %.)
template <int THREADS, typename F> __device__ __forceinline__ void stage(int n, bool wide, F at) {
    if (wide)
        for (int i = threadIdx.x; i < n; i += THREADS) at(i, cp_async16);
    else
        for (int i = threadIdx.x; i < n; i += THREADS) at(i, copy16);
}
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
}
__device__ __forceinline__ void ldsm(unsigned (&r)[4], unsigned a) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(a)
                 : "memory");
}
__device__ __forceinline__ void ldsm_t(unsigned (&r)[4], unsigned a) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(a)
                 : "memory");
}
__device__ __forceinline__ void mma(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
        "{%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Byte address of 16-byte half `half` of halo voxel h (32 bytes a voxel; the
// halves of every second group of four voxels are exchanged, so that eight
// consecutive voxels fall on all banks once).
__device__ __forceinline__ unsigned halo_at(int h, int half) {
    return (unsigned)(h * 32 + ((half ^ ((h >> 2) & 1)) << 4));
}
// The same for row k of a [rows][C] operand: 16-byte chunk c of C / 8.
template <int C> __device__ __forceinline__ unsigned row_at(int k, int c) {
    constexpr int shift = C % 64 == 0 ? 0 : (C % 32 == 0 ? 1 : 2);
    constexpr int mask = C % 64 == 0 ? 7 : (C % 32 == 0 ? 3 : 1);
    return (unsigned)(k * (2 * C) + ((c ^ ((k >> shift) & mask)) << 4));
}

// Voxel index of every halo voxel of tile (bx, by, bz), -1 where the padded
// volume is zero (periodic in x and y).
__device__ __forceinline__ void halo_table(int *tab, const ConvTile &t, int bx, int by, int bz,
                                           int nx, int ny, int nz) {
    const int n = t.halo();
    for (int h = threadIdx.x; h < n; h += blockDim.x) {
        const int q = h / t.hx, hx = h - q * t.hx, hz = q / t.hy, hy = q - hz * t.hy;
        int x = (bx << t.lx) + hx - 1, y = (by << t.ly) + hy - 1;
        const int z = (bz << t.lz) + hz - 1;
        const bool in = x <= nx && y <= ny && z >= 0 && z < nz;
        x = x < 0 ? x + nx : (x == nx ? 0 : x);
        y = y < 0 ? y + ny : (y == ny ? 0 : y);
        tab[h] = in ? x + nx * (y + ny * z) : -1;
    }
}

template <int THREADS>
__device__ __forceinline__ void load_halo(unsigned dst, const int *tab, int n, const bf16 *Xs, int Ci,
                                          int c0, bool wide) {
    auto at = [&](int i, auto copy) {
        const int h = i >> 1, half = i & 1, u = tab[h];
        copy(dst + halo_at(h, half), Xs + (long long)(u < 0 ? 0 : u) * Ci + c0 + 8 * half, u >= 0);
    };
    stage<THREADS>(2 * n, wide, at);
}

// Halo index of tile voxel m (the halo voxel of its own position)
__device__ __forceinline__ int halo_of(const ConvTile &t, int m) {
    const int x = m & ((1 << t.lx) - 1), y = (m >> t.lx) & ((1 << t.ly) - 1), z = m >> (t.lx + t.ly);
    return ((z + 1) * t.hy + y + 1) * t.hx + x + 1;
}

// Y[s][v][co] = act(b[co] + sum_{d, ci} Wt[d][ci][co] X[s][v + sign d][ci]):
// four warps, each 16 MT voxels of the tile and all CO channels.
template <int CO, int MT>
__global__ void __launch_bounds__(128) conv_tile_kernel(const bf16 *__restrict__ X,
                                                        const bf16 *__restrict__ Wt,
                                                        const float *__restrict__ bias,
                                                        bf16 *__restrict__ Y, float *__restrict__ Yf,
                                                        ConvTile t, int nx, int ny, int nz, int Ci,
                                                        int relu, int sign, int wide) {
    extern __shared__ __align__(128) unsigned char sm[];
    int *tab = reinterpret_cast<int *>(sm);
    const unsigned sX = smem_addr(sm) + 4 * kMaxHalo, sW = sX + 32 * kMaxHalo;
    const int bx = blockIdx.x % t.tx, by = (blockIdx.x / t.tx) % t.ty, bz = blockIdx.x / (t.tx * t.ty);
    const long long V = (long long)nx * ny * nz;
    const bf16 *Xs = X + blockIdx.y * V * Ci;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n = t.halo();
    halo_table(tab, t, bx, by, bz, nx, ny, nz);

    float acc[MT][CO / 8][4];
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int j = 0; j < CO / 8; ++j)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[i][j][q] = 0.0f;
    // ldmatrix row of this lane: voxel lane & 15 of a 16-voxel block, half lane >> 4
    int hb[MT];
#pragma unroll
    for (int i = 0; i < MT; ++i) hb[i] = halo_of(t, (warp * MT + i) * 16 + (lane & 15));
    const int half = lane >> 4;
    for (int c0 = 0; c0 < Ci; c0 += 16) {
        __syncthreads();
        load_halo<128>(sX, tab, n, Xs, Ci, c0, wide & kWideX);
        stage<128>(27 * 16 * (CO / 8), wide & kWideB, [&](int i, auto copy) {
            const int k = i / (CO / 8), c = i % (CO / 8);  // k = 16 tap + channel
            copy(sW + row_at<CO>(k, c), Wt + ((long long)(k >> 4) * Ci + c0 + (k & 15)) * CO + 8 * c, true);
        });
        cp_async_wait();
        __syncthreads();
        int d = 0;
        for (int dz = -1; dz <= 1; ++dz)
            for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
                for (int dx = -1; dx <= 1; ++dx, ++d) {
                    const int off = sign * ((dz * t.hy + dy) * t.hx + dx);
                    unsigned a[MT][4];
#pragma unroll
                    for (int i = 0; i < MT; ++i) ldsm(a[i], sX + halo_at(hb[i] + off, half));
#pragma unroll
                    for (int j = 0; j < CO / 16; ++j) {
                        unsigned b[4];
                        ldsm_t(b, sW + row_at<CO>(16 * d + (lane & 15), 2 * j + half));
#pragma unroll
                        for (int i = 0; i < MT; ++i) {
                            mma(acc[i][2 * j], a[i], b[0], b[1]);
                            mma(acc[i][2 * j + 1], a[i], b[2], b[3]);
                        }
                    }
                }
    }
    const int g = lane >> 2, c = 2 * (lane & 3);
#pragma unroll
    for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int m = (warp * MT + i) * 16 + g + 8 * r;
            const int x = (bx << t.lx) + (m & ((1 << t.lx) - 1));
            const int y = (by << t.ly) + ((m >> t.lx) & ((1 << t.ly) - 1));
            const int z = (bz << t.lz) + (m >> (t.lx + t.ly));
            if (x >= nx || y >= ny || z >= nz) continue;
            const long long o = (blockIdx.y * V + x + (long long)nx * (y + (long long)ny * z)) * CO + c;
#pragma unroll
            for (int j = 0; j < CO / 8; ++j) {
                float v0 = acc[i][j][2 * r], v1 = acc[i][j][2 * r + 1];
                if (bias) {
                    v0 += __ldg(bias + 8 * j + c);
                    v1 += __ldg(bias + 8 * j + c + 1);
                }
                if (relu) {
                    v0 = fmaxf(v0, 0.0f);
                    v1 = fmaxf(v1, 0.0f);
                }
                if (wide & kWideOut) {
                    if (Y) *reinterpret_cast<__nv_bfloat162 *>(Y + o + 8 * j) = __floats2bfloat162_rn(v0, v1);
                    if (Yf) *reinterpret_cast<float2 *>(Yf + o + 8 * j) = make_float2(v0, v1);
                } else {
                    if (Y) {
                        Y[o + 8 * j] = __float2bfloat16(v0);
                        Y[o + 8 * j + 1] = __float2bfloat16(v1);
                    }
                    if (Yf) {
                        Yf[o + 8 * j] = v0;
                        Yf[o + 8 * j + 1] = v1;
                    }
                }
            }
        }
}

// dW[d][ci][co] += sum_v X[v + d][ci] dY[v][co] for 16 input channels (grid
// y) and NC output channels (grid z); db[co] += sum_v dY[v][co]. Nine warps,
// each the three x-taps of one (dz, dy): its sums stay in registers over all
// tiles of the block and are added to dW once. Tiles of all samples in one
// list, strided over grid x.
template <int NC>
__global__ void __launch_bounds__(288) conv_wgrad_tile_kernel(const bf16 *__restrict__ X,
                                                              const bf16 *__restrict__ dY,
                                                              float *__restrict__ dW,
                                                              float *__restrict__ db, ConvTile t, int S,
                                                              int nx, int ny, int nz, int Ci, int Co,
                                                              int wide) {
    extern __shared__ __align__(128) unsigned char sm[];
    int *tab = reinterpret_cast<int *>(sm);
    const unsigned sX = smem_addr(sm) + 4 * kMaxHalo, sY = sX + 32 * kMaxHalo;
    const unsigned char *gY = sm + 36 * kMaxHalo;
    const long long V = (long long)nx * ny * nz;
    const int c0 = blockIdx.y * 16, n0 = blockIdx.z * NC;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n = t.halo(), P = 1 << (t.lx + t.ly + t.lz);
    const int dz = warp / 3 - 1, dy = warp % 3 - 1;
    const int shift = (dz * t.hy + dy) * t.hx;
    float acc[3][NC / 8][4];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < NC / 8; ++j)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[i][j][q] = 0.0f;
    const bool bias = db && blockIdx.y == 0;
    const int bc = threadIdx.x % NC, bg = threadIdx.x / NC;  // bias sums: channel, group of rows
    float bsum = 0.0f;
    // A = X^T (16 channels x 16 voxels) by transposing loads: this lane's row
    // is voxel ka of a 16-voxel block, channel half ha
    const int ka = (lane & 7) + ((lane >> 4) & 1) * 8, ha = (lane >> 3) & 1;
    for (int it = blockIdx.x; it < t.tiles() * S; it += gridDim.x) {
        const int s = it / t.tiles(), b = it - s * t.tiles();
        const int bx = b % t.tx, by = (b / t.tx) % t.ty, bz = b / (t.tx * t.ty);
        __syncthreads();
        halo_table(tab, t, bx, by, bz, nx, ny, nz);
        __syncthreads();
        load_halo<288>(sX, tab, n, X + s * V * Ci, Ci, c0, wide & kWideX);
        stage<288>(P * (NC / 8), wide & kWideB, [&](int i, auto copy) {
            const int m = i / (NC / 8), c = i % (NC / 8);
            const int x = (bx << t.lx) + (m & ((1 << t.lx) - 1));
            const int y = (by << t.ly) + ((m >> t.lx) & ((1 << t.ly) - 1));
            const int z = (bz << t.lz) + (m >> (t.lx + t.ly));
            const bool in = x < nx && y < ny && z < nz;
            const long long v = in ? x + (long long)nx * (y + (long long)ny * z) : 0;
            copy(sY + row_at<NC>(m, c), dY + (s * V + v) * Co + n0 + 8 * c, in);
        });
        cp_async_wait();
        __syncthreads();
        for (int k0 = 0; k0 < P; k0 += 16) {
            unsigned bf[NC / 16][4];
#pragma unroll
            for (int j = 0; j < NC / 16; ++j)
                ldsm_t(bf[j], sY + row_at<NC>(k0 + (lane & 15), 2 * j + (lane >> 4)));
            const int h = halo_of(t, k0 + ka) + shift;
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                unsigned a[4];
                ldsm_t(a, sX + halo_at(h + i - 1, ha));
#pragma unroll
                for (int j = 0; j < NC / 16; ++j) {
                    mma(acc[i][2 * j], a, bf[j][0], bf[j][1]);
                    mma(acc[i][2 * j + 1], a, bf[j][2], bf[j][3]);
                }
            }
        }
        if (bias && bg < 288 / NC)
            for (int m = bg; m < P; m += 288 / NC)
                bsum += __bfloat162float(*reinterpret_cast<const bf16 *>(
                    gY + row_at<NC>(m, bc >> 3) + 2 * (bc & 7)));
    }
    const int g = lane >> 2, q = 2 * (lane & 3);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        float *w = dW + ((long long)(3 * warp + i) * Ci + c0 + g) * Co + n0 + q;
#pragma unroll
        for (int j = 0; j < NC / 8; ++j) {
            atomicAdd(w + 8 * j, acc[i][j][0]);
            atomicAdd(w + 8 * j + 1, acc[i][j][1]);
            atomicAdd(w + 8 * Co + 8 * j, acc[i][j][2]);
            atomicAdd(w + 8 * Co + 8 * j + 1, acc[i][j][3]);
        }
    }
    if (bias && bg < 288 / NC) atomicAdd(db + n0 + bc, bsum);
}

// The box of 2^p voxels that covers the volume with the least work: products
// of the padded voxels plus the halo's loads.
ConvTile conv_tile(int nx, int ny, int nz, int p) {
    ConvTile best{};
    double cost = 0.0;
    for (int lx = 2; lx <= p; ++lx)
        for (int ly = 0; lx + ly <= p; ++ly) {
            ConvTile t{};
            t.lx = lx;
            t.ly = ly;
            t.lz = p - lx - ly;
            t.hx = (1 << lx) + 2;
            t.hy = (1 << ly) + 2;
            t.hz = (1 << t.lz) + 2;
            if (t.halo() > kMaxHalo) continue;
            t.tx = (nx + (1 << lx) - 1) >> lx;
            t.ty = (ny + (1 << ly) - 1) >> ly;
            t.tz = (nz + (1 << t.lz) - 1) >> t.lz;
            const double c = (double)t.tiles() * ((1 << p) + 0.5 * t.halo());
            if (best.tx && c >= cost) continue;
            cost = c;
            best = t;
        }
    return best;
}

template <int CO, int MT>
cudaError_t conv_go(const bf16 *X, const bf16 *Wt, const float *bias, bf16 *Y, float *Yf, int S, int nx,
                    int ny, int nz, int Ci, bool relu, int sign, cudaStream_t s) {
    const ConvTile t = conv_tile(nx, ny, nz, MT == 4 ? 8 : (MT == 2 ? 7 : 6));
    const size_t shm = 36 * kMaxHalo + 27 * 16 * CO * 2;
    const cudaError_t e = cudaFuncSetAttribute(conv_tile_kernel<CO, MT>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm);
    if (e != cudaSuccess) return e;
    const bool pairs = (reinterpret_cast<uintptr_t>(Y) & 3) == 0 && (reinterpret_cast<uintptr_t>(Yf) & 7) == 0;
    conv_tile_kernel<CO, MT><<<dim3(t.tiles(), S), 128, shm, s>>>(X, Wt, bias, Y, Yf, t, nx, ny, nz, Ci,
                                                                  relu ? 1 : 0, sign,
                                                                  wide_operands(X, Wt) | (pairs ? kWideOut : 0));
    return cudaGetLastError();
}

// Large tiles (256 voxels, 128 from 48 channels on: the accumulators) while
// they give every SM two blocks, else 64 voxels.
template <int CO>
cudaError_t conv_pick(const bf16 *X, const bf16 *Wt, const float *bias, bf16 *Y, float *Yf, int S,
                      int nx, int ny, int nz, int Ci, bool relu, int sign, cudaStream_t s) {
    constexpr int MT = CO <= 32 ? 4 : 2;
    const long long V = (long long)nx * ny * nz * S;
    if (V >= (long long)64 * MT * 2 * device_sm_count())
        return conv_go<CO, MT>(X, Wt, bias, Y, Yf, S, nx, ny, nz, Ci, relu, sign, s);
    return conv_go<CO, 1>(X, Wt, bias, Y, Yf, S, nx, ny, nz, Ci, relu, sign, s);
}

template <int NC>
cudaError_t wgrad_go(const bf16 *X, const bf16 *dY, float *dW, float *db, int S, int nx, int ny, int nz,
                     int Ci, int Co, cudaStream_t s) {
    const int sms = device_sm_count(), parts = (Ci / 16) * (Co / NC);
    const long long V = (long long)nx * ny * nz * S;
    const ConvTile t = conv_tile(nx, ny, nz, V * parts >= 256LL * sms ? 8 : 6);
    const size_t shm = 36 * kMaxHalo + (size_t)(1 << (t.lx + t.ly + t.lz)) * NC * 2;
    const cudaError_t e = cudaFuncSetAttribute(conv_wgrad_tile_kernel<NC>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm);
    if (e != cudaSuccess) return e;
    const long long all = (long long)t.tiles() * S;
    const int gx = (int)std::max(1LL, std::min(all, (long long)(2 * sms + parts - 1) / parts));
    conv_wgrad_tile_kernel<NC><<<dim3(gx, Ci / 16, Co / NC), 288, shm, s>>>(
        X, dY, dW, db, t, S, nx, ny, nz, Ci, Co, wide_operands(X, dY));
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_conv3d(const bf16 *X, const bf16 *Wt, const float *bias, bf16 *Y, float *Yf, int S,
                          int nx, int ny, int nz, int Ci, int Co, bool relu, int sign, cudaStream_t s) {
    switch (Co) {
        case 16: return conv_pick<16>(X, Wt, bias, Y, Yf, S, nx, ny, nz, Ci, relu, sign, s);
        case 32: return conv_pick<32>(X, Wt, bias, Y, Yf, S, nx, ny, nz, Ci, relu, sign, s);
        case 48: return conv_pick<48>(X, Wt, bias, Y, Yf, S, nx, ny, nz, Ci, relu, sign, s);
        case 64: return conv_pick<64>(X, Wt, bias, Y, Yf, S, nx, ny, nz, Ci, relu, sign, s);
        default: return conv_pick<96>(X, Wt, bias, Y, Yf, S, nx, ny, nz, Ci, relu, sign, s);
    }
}

cudaError_t launch_conv3d_wgrad(const bf16 *X, const bf16 *dY, float *dW, float *db, int S, int nx,
                                int ny, int nz, int Ci, int Co, cudaStream_t s) {
    if (Co % 64 == 0) return wgrad_go<64>(X, dY, dW, db, S, nx, ny, nz, Ci, Co, s);
    if (Co % 48 == 0) return wgrad_go<48>(X, dY, dW, db, S, nx, ny, nz, Ci, Co, s);
    if (Co % 32 == 0) return wgrad_go<32>(X, dY, dW, db, S, nx, ny, nz, Ci, Co, s);
    return wgrad_go<16>(X, dY, dW, db, S, nx, ny, nz, Ci, Co, s);
}

}  // namespace rt3d
