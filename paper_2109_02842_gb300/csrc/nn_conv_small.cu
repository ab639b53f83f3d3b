// The learned path's 3 x 3 x 3 convolution for one to four input channels (the
// network's three-channel input layer, the input gradient of its two-channel
// head), walking columns of the volume with mma.sync.
//
// K = 27 Cin is a few steps of 16, so the weights of all steps stay in
// registers, and the floor is the output. A block owns a tile of TX x TY voxels
// of every z slice of a segment and keeps four slices of it (with a one-voxel
// halo, channels interleaved as in memory, rows padded to P = TX + 2 voxels) in
// shared memory. The voxel operand of a product is gathered from there element
// by element: element k of a row is at a fixed offset from the row's voxel, the
// offsets of a lane's elements coming from a table of the four positions the
// slices can have in the ring. (Eight 2-byte shared loads a step and lane take
// less time than the 27-fold copies and index divisions from global memory
// that this kernel replaces.) The sums run in the order of the other kernels.
//
// 96 x 128 x 128 voxels, 3 -> 16 channels: 0.764 -> 0.059 ms, 2 -> 16: 0.516 ->
// 0.043 ms (the output alone: 0.008 ms).
#include <cuda_bf16.h>

#include "common.cuh"
#include "kernels.h"

namespace {

constexpr int kWarps = 8, kThreads = 32 * kWarps;

struct SmallShape {
    int D, H, W, Cout, Kp;
    int TX, TY, nx, ny;           // tile and tiles
    int zlen, nz;                 // slices of a segment, segments
    int srow;                     // elements of a slice buffer
    int relu;
    unsigned inv_p, inv_pc;       // ceil(2^20 / P), ceil(2^20 / (P Cin)): see div20
};

// v / d with inv = ceil(2^20 / d), for v d < 2^20
__device__ __forceinline__ int div20(int v, unsigned inv) { return (int)((unsigned)v * inv >> 20); }

__device__ __forceinline__ void mma16816(float (&d)[4], const unsigned (&a)[4], unsigned b0,
                                         unsigned b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
        "{%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// grid: (columns x segments, blocks of 8 NT output channels)
template <int CIN, int NT, bool OUT_BF16>
__global__ void __launch_bounds__(kThreads, 2)
k_conv3d_small(const __nv_bfloat16 *__restrict__ x, const __nv_bfloat16 *__restrict__ w,
               const float *__restrict__ bias, void *__restrict__ out, const SmallShape s) {
    constexpr int K = 27 * CIN, KS = (K + 15) / 16, CO = 8 * NT;
    extern __shared__ unsigned short sl[];                 // [4][srow]
    __shared__ int tab[4][16 * KS];                        // element offsets for z & 3
    const int P = s.TX + 2;
    const int bx = blockIdx.x % s.nx, by = (blockIdx.x / s.nx) % s.ny, bz = blockIdx.x / (s.nx * s.ny);
    const int x0 = bx * s.TX, y0 = by * s.TY;
    const int z0 = bz * s.zlen, z1 = min(s.D, z0 + s.zlen);
    const int co0 = blockIdx.y * CO;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 2, t = lane & 3;

    for (int i = threadIdx.x; i < 4 * 16 * KS; i += kThreads) {
        const int q = i / (16 * KS), k = i - q * (16 * KS);
        const int tap = min(k, K - 1) / CIN, ci = min(k, K - 1) - tap * CIN;
        const int dz = tap / 9, dy = tap / 3 % 3, dx = tap % 3;
        tab[q][k] = ((q + dz + 3) & 3) * s.srow + (dy * P + dx) * CIN + ci;
    }
    // elements past the slices stay zero
    const int n_el = (s.TY + 2) * P * CIN, slack = s.srow - n_el;
    for (int i = threadIdx.x; i < 4 * slack; i += kThreads)
        sl[(i / slack) * s.srow + n_el + i % slack] = 0;
    // the weights of row n of product j: the output channel whose sum lane
    // t = n / 2 holds, chosen so that a lane's channels are consecutive
    unsigned b[KS][NT][2];
#pragma unroll
    for (int j = 0; j < NT; ++j) {
        const int co = co0 + 2 * NT * (g >> 1) + 2 * j + (g & 1);
#pragma unroll
        for (int st = 0; st < KS; ++st)
#pragma unroll
            for (int h = 0; h < 2; ++h)
                b[st][j][h] = co < s.Cout ? *reinterpret_cast<const unsigned *>(
                                                w + (size_t)co * s.Kp + 16 * st + 8 * h + 2 * t)
                                          : 0u;
    }
    float bs[2 * NT];
#pragma unroll
    for (int k = 0; k < 2 * NT; ++k) {
        const int co = co0 + 2 * NT * t + k;
        bs[k] = (bias && co < s.Cout) ? bias[co] : 0.f;
    }
    const unsigned short *xs = reinterpret_cast<const unsigned short *>(x);
    auto load_slice = [&](int z) {
        const bool zin = z >= 0 && z < s.D;
        unsigned short *dst = sl + (z & 3) * s.srow;
        const unsigned short *src = xs + (zin ? (size_t)z * s.H * s.W * CIN : 0);
#pragma unroll 4
        for (int i = threadIdx.x; i < n_el; i += kThreads) {
            const int r = div20(i, s.inv_pc), e = i - r * (P * CIN);
            const int yy = y0 - 1 + r, xe = (x0 - 1) * CIN + e;      // element of the row
            const bool ok = zin && (unsigned)yy < (unsigned)s.H && (unsigned)xe < (unsigned)(s.W * CIN);
            dst[i] = ok ? src[(size_t)(yy * s.W) * CIN + xe] : (unsigned short)0;
        }
    };
    load_slice(z0 - 1);
    load_slice(z0);
    const int tiles = (s.TY * P + 15) / 16;
    for (int z = z0; z < z1; ++z) {
        load_slice(z + 1);         // over slice z - 3, read two barriers ago
        __syncthreads();
        int off[KS][4];
#pragma unroll
        for (int st = 0; st < KS; ++st)
#pragma unroll
            for (int e = 0; e < 4; ++e)
                off[st][e] = tab[z & 3][16 * st + 2 * t + (e & 1) + 8 * (e >> 1)] + g * CIN;
        for (int tl = warp; tl < tiles; tl += kWarps) {
            const unsigned short *base = sl + tl * 16 * CIN;
            float acc[NT][4] = {};
#pragma unroll
            for (int st = 0; st < KS; ++st) {
                unsigned a[4];
#pragma unroll
                for (int e = 0; e < 2; ++e)          // k halves
#pragma unroll
                    for (int r = 0; r < 2; ++r) {    // rows g, g + 8
                        unsigned lo = base[off[st][2 * e] + 8 * r * CIN];
                        unsigned hi = base[off[st][2 * e + 1] + 8 * r * CIN];
                        const int k = 16 * st + 8 * e + 2 * t;
                        if (16 * st + 16 > K) {      // (the last step's elements past K)
                            if (k >= K) lo = 0;
                            if (k + 1 >= K) hi = 0;
                        }
                        a[2 * e + r] = lo | (hi << 16);
                    }
#pragma unroll
                for (int j = 0; j < NT; ++j) mma16816(acc[j], a, b[st][j][0], b[st][j][1]);
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int p = tl * 16 + g + 8 * h;
                const int row = div20(p, s.inv_p), col = p - row * P;
                const int yy = y0 + row, xx = x0 + col, co = co0 + 2 * NT * t;
                if (row >= s.TY || col >= s.TX || yy >= s.H || xx >= s.W || co >= s.Cout) continue;
                float f[2 * NT];
#pragma unroll
                for (int k = 0; k < 2 * NT; ++k) {
                    f[k] = acc[k >> 1][2 * h + (k & 1)] + bs[k];
                    if (s.relu) f[k] = fmaxf(f[k], 0.f);
                }
                const size_t o = (((size_t)z * s.H + yy) * s.W + xx) * s.Cout + co;
                const bool whole = (s.Cout & (2 * NT - 1)) == 0;   // aligned, all in range
                if (OUT_BF16) {
                    __nv_bfloat16 *po = reinterpret_cast<__nv_bfloat16 *>(out) + o;
                    unsigned u[NT];
#pragma unroll
                    for (int k = 0; k < NT; ++k) {
                        __nv_bfloat162 b2 = __floats2bfloat162_rn(f[2 * k], f[2 * k + 1]);
                        u[k] = *reinterpret_cast<unsigned *>(&b2);
                    }
                    if (whole && NT == 2) *reinterpret_cast<uint2 *>(po) = make_uint2(u[0], u[NT - 1]);
                    else if (whole) *reinterpret_cast<unsigned *>(po) = u[0];
                    else
#pragma unroll
                        for (int k = 0; k < 2 * NT; ++k)
                            if (co + k < s.Cout) po[k] = __float2bfloat16(f[k]);
                } else {
                    float *po = reinterpret_cast<float *>(out) + o;
                    if (whole && NT == 2)
                        *reinterpret_cast<float4 *>(po) = make_float4(f[0], f[1], f[2 * NT - 2], f[2 * NT - 1]);
                    else if (whole) *reinterpret_cast<float2 *>(po) = make_float2(f[0], f[1]);
                    else
#pragma unroll
                        for (int k = 0; k < 2 * NT; ++k)
                            if (co + k < s.Cout) po[k] = f[k];
                }
            }
        }
    }
}

template <int CIN>
cudaError_t launch_cin(const SmallShape &s, const __nv_bfloat16 *x, const __nv_bfloat16 *w,
                       const float *bias, void *out, int out_bf16, cudaStream_t st) {
    const size_t smem = 4 * (size_t)s.srow * 2;
    const dim3 grid(s.nx * s.ny * s.nz, s.Cout <= 8 ? 1 : (s.Cout + 15) / 16);
    if (s.Cout <= 8) {
        if (out_bf16) k_conv3d_small<CIN, 1, true><<<grid, kThreads, smem, st>>>(x, w, bias, out, s);
        else k_conv3d_small<CIN, 1, false><<<grid, kThreads, smem, st>>>(x, w, bias, out, s);
    } else {
        if (out_bf16) k_conv3d_small<CIN, 2, true><<<grid, kThreads, smem, st>>>(x, w, bias, out, s);
        else k_conv3d_small<CIN, 2, false><<<grid, kThreads, smem, st>>>(x, w, bias, out, s);
    }
    return cudaGetLastError();
}

}  // namespace

cudaError_t nn_conv3d_small(const void *x, const void *w, const float *bias, void *out, int D, int H,
                            int W, int Cin, int Cout, int Kp, int relu, int out_bf16, cudaStream_t st) {
    if (Cin < 1 || Cin > 4 || ((uintptr_t)w % 4) || ((uintptr_t)out % 16)) return cudaErrorNotSupported;
    // tiles of about 540 positions (four rounds of the warps, 16 KB of slices
    // with three channels), segments that fill the device twice over
    SmallShape s{};
    s.D = D;
    s.H = H;
    s.W = W;
    s.Cout = Cout;
    s.Kp = Kp;
    s.relu = relu;
    s.nx = (W + 79) / 80;
    s.TX = (W + s.nx - 1) / s.nx;
    const int P = s.TX + 2;
    int ty = 512 / P < 1 ? 1 : 512 / P;
    if (ty > H) ty = H;
    s.ny = (H + ty - 1) / ty;
    s.TY = (H + s.ny - 1) / s.ny;
    const int tiles = (s.TY * P + 15) / 16;
    s.srow = (tiles * 16 + 2 * P + 2) * Cin;
    s.inv_p = ((1u << 20) + P - 1) / P;
    s.inv_pc = ((1u << 20) + P * Cin - 1) / (P * Cin);
    const long long per = (long long)s.nx * s.ny * ((Cout + 15) / 16);
    long long nz = 152ll * 4 / per;
    if (nz > D / 4) nz = D / 4;
    if (nz < 1) nz = 1;
    s.zlen = (int)((D + nz - 1) / nz);
    s.nz = (D + s.zlen - 1) / s.zlen;
    const auto *xb = (const __nv_bfloat16 *)x;
    const auto *wb = (const __nv_bfloat16 *)w;
    switch (Cin) {
        case 1: return launch_cin<1>(s, xb, wb, bias, out, out_bf16, st);
        case 2: return launch_cin<2>(s, xb, wb, bias, out, out_bf16, st);
        case 3: return launch_cin<3>(s, xb, wb, bias, out, out_bf16, st);
        default: return launch_cin<4>(s, xb, wb, bias, out, out_bf16, st);
    }
}
