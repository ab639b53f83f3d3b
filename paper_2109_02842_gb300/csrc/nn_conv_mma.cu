// The learned path's 3 x 3 x 3 convolution for narrow outputs, walking columns
// of the volume with mma.sync (Cin a multiple of 16, any D, H, W and Cout as
// far as weights and slices fit in shared memory; see conv_mma_plan).
//
// A block owns a tile of TX x TY voxels of every z slice of a segment and
// walks the segment: each slice of the tile (with a one-voxel halo) is copied
// once by cp.async into a ring of four, three in use, and serves all 27 taps.
// A slice is a flat list of padded rows, P = TX + 2 voxels each, so a tap is an
// offset dy P + dx into it and the outputs are tiles of 16 flat positions
// without remainders per row (the two padding positions of a row are computed
// and not stored). Voxels lie 32 bytes apart (16 channels), their halves
// swapped in every other group of four, which makes ldmatrix free of bank
// conflicts from any starting voxel. A warp takes groups of MT tiles and all CO
// output channels: per tap and 16 input channels MT + NT / 2 ldmatrix feed MT
// NT products (m16n8k16).
//
// Why not tcgen05: an M = 128, K = 16 product from shared memory takes 69
// cycles whatever N up to 64 (measured; its A rows come at 64 bytes a cycle),
// so with N = 16 it does 475 multiply-adds a cycle where mma.sync does 1024 and
// is bound by ldmatrix at 820: 16 -> 16 channels on 96 x 128 x 128 voxels took
// 0.123 ms that way.
//
// The products of an output are those of the other kernels in the same order
// (tap by tap, 16 channels at a time, FP32 accumulation), so the results are
// theirs bit for bit.
//
// 96 x 128 x 128 voxels, before (nn_tc.cu, which copies each row once per tap)
// and now: 16 -> 16 channels 0.278 and 0.090 ms, 32 -> 16 0.425 and 0.162, 16 ->
// 2 0.320 and 0.070; 48 x 64 x 64, 32 -> 32 0.072 and 0.047; 44 x 72 x 72, 32 ->
// 32 (rows nn_tc.cu does not take) 0.187 and 0.047. Shared memory is 64 % and
// the tensor pipe 50 % busy (16 -> 16), integer work 38 %: the latter halved
// when the sixteen-voxel steps became immediates and divisions reciprocals
// (0.107 -> 0.090).
#include <cuda_bf16.h>

#include "common.cuh"
#include "kernels.h"

namespace {

constexpr int kWarps = 8, kThreads = 32 * kWarps;
constexpr int kMaxSmem = 224 * 1024;

struct MmaShape {
    int D, H, W, Cin, Cout, Kp;
    int TX, TY, nx, ny;           // tile and tiles
    int zlen, nz;                 // slices of a segment, segments
    int n_co;                     // blocks of CO output channels
    int CO, MT;                   // output channels of a block, tiles of 16 a warp takes at once
    int xrows;                    // voxels of a slice buffer (one chunk of 16 channels)
    int chunks;                   // Cin / 16
    int relu;
    unsigned inv_p, inv_c;        // ceil(2^20 / P), ceil(2^20 / (2 chunks)): see div20
};

size_t mma_smem(const MmaShape &s) {
    return 32 * ((size_t)27 * s.chunks * s.CO + 4 * (size_t)s.chunks * s.xrows);
}

// Tile, split and segments of a shape; false where nothing fits. CO: the
// smallest of 8, 16 and 32 that holds Cout, else 32; 16 where 32 leaves no
// room. The tile's rows: as many of the warps' positions used as possible,
// little halo, two blocks an SM where that is possible.
bool conv_mma_plan(int D, int H, int W, int Cin, int Cout, int Kp, MmaShape &best) {
    if (Cin % 16 || Cin < 16) return false;
    MmaShape s{};
    s.D = D;
    s.H = H;
    s.W = W;
    s.Cin = Cin;
    s.Cout = Cout;
    s.Kp = Kp;
    s.chunks = Cin / 16;
    s.nx = (W + 79) / 80;
    s.TX = (W + s.nx - 1) / s.nx;
    const int P = s.TX + 2;
    double best_score = 0;
    int best_occ = 1;
    for (int CO = Cout <= 8 ? 8 : Cout <= 16 ? 16 : 32; CO >= 8; CO /= 2) {
        if (CO < 16 && Cout > 8) break;
        s.CO = CO;
        for (int MT = 4; MT >= 2; MT /= 2) {
            s.MT = MT;
            for (int ty = 1; ty <= H && ty * P <= 1024; ++ty) {      // (div20: at most 1120 positions)
                s.TY = ty;
                s.ny = (H + ty - 1) / ty;
                // (the last group of tiles reads past the tile's own slice)
                const int groups = (ty * P + 16 * MT - 1) / (16 * MT);
                s.xrows = groups * 16 * MT + 2 * P + 2;
                const size_t smem = mma_smem(s);
                if (smem > (size_t)kMaxSmem) break;
                const int occ = smem <= 112 * 1024 ? 2 : 1;
                const int rounds = (groups + kWarps - 1) / kWarps;
                // share of the warps' positions that are outputs, times the
                // loads' and the ldmatrix's efficiency, less one block an SM
                const double use = (double)H * s.TX / ((double)s.ny * rounds * kWarps * 16 * MT);
                const double mem = MT * CO / 8.0 / (MT * CO / 8.0 + 0.25 * (4 * MT + 2 * CO / 8.0));
                const double score = use * mem * ty / (ty + 0.4) * (occ == 2 ? 1.0 : 0.8) *
                                     (CO == 32 || Cout <= CO ? 1.0 : 0.8);
                if (score > best_score) {
                    best_score = score;
                    best = s;
                    best_occ = occ;
                }
            }
        }
    }
    if (best_score == 0) return false;
    best.n_co = (Cout + best.CO - 1) / best.CO;
    const long long per = (long long)best.nx * best.ny * best.n_co;
    long long nz = 152ll * best_occ / per;
    if (nz > D) nz = D;
    if (nz < 1) nz = 1;
    best.zlen = (int)((D + nz - 1) / nz);
    best.nz = (D + best.zlen - 1) / best.zlen;
    best.inv_p = ((1u << 20) + P - 1) / P;
    best.inv_c = ((1u << 20) + 2 * best.chunks - 1) / (2 * best.chunks);
    return true;
}

__device__ __forceinline__ unsigned smem_u32(const void *p) {
    return (unsigned)__cvta_generic_to_shared(p);
}
// 16 bytes to shared memory, zeros where !ok (the source is not read then)
__device__ __forceinline__ void cp16z(unsigned dst, const void *src, bool ok) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src),
                 "r"(ok ? 16 : 0)
                 : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }
__device__ __forceinline__ void ldm_x4(unsigned (&r)[4], unsigned addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}
__device__ __forceinline__ void ldm_x2(unsigned &r0, unsigned &r1, unsigned addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];\n"
                 : "=r"(r0), "=r"(r1)
                 : "r"(addr)
                 : "memory");
}
__device__ __forceinline__ void mma16816(float (&d)[4], const unsigned (&a)[4], unsigned b0,
                                         unsigned b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
        "{%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// v / d with inv = ceil(2^20 / d), for v d < 2^20 (both below 2^14, 2^6 here)
__device__ __forceinline__ int div20(int v, unsigned inv) { return (int)((unsigned)v * inv >> 20); }
// byte offset of half h (8 of 16 channels) of voxel or row v
__device__ __forceinline__ unsigned half_at(int v, int h) {
    return (unsigned)v * 32u + (unsigned)((h ^ (v >> 2)) & 1) * 16u;
}

// grid: (columns x segments, blocks of output channels)
template <int NT, int MT, bool OUT_BF16>
__global__ void __launch_bounds__(kThreads, 2)
k_conv3d_mma(const __nv_bfloat16 *__restrict__ x, const __nv_bfloat16 *__restrict__ w,
             const float *__restrict__ bias, void *__restrict__ out, const MmaShape s) {
    constexpr int CO = 8 * NT;
    extern __shared__ __align__(128) unsigned char sm[];
    const unsigned wbase = smem_u32(sm);                       // [tap][chunk][CO rows] x 32 B
    const unsigned xbase = wbase + 27u * s.chunks * CO * 32u;  // [slice & 3][chunk][xrows] x 32 B
    const unsigned chunk_b = (unsigned)s.xrows * 32u, slice_b = chunk_b * s.chunks;
    const int P = s.TX + 2;
    const int bx = blockIdx.x % s.nx, by = (blockIdx.x / s.nx) % s.ny, bz = blockIdx.x / (s.nx * s.ny);
    const int x0 = bx * s.TX, y0 = by * s.TY;
    const int z0 = bz * s.zlen, z1 = min(s.D, z0 + s.zlen);
    const int co0 = blockIdx.y * CO;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 2, t = lane & 3;

    // weights: row n of a block is the output channel whose sum lane t = n / 2
    // of product n / 8 holds, chosen so that a lane's channels are consecutive
    for (int i = threadIdx.x; i < 27 * s.chunks * CO * 2; i += kThreads) {
        const int h = i & 1, n = (i >> 1) % CO, r = (i >> 1) / CO;
        const int j = n / 8, q = n % 8, co = co0 + 2 * NT * (q >> 1) + 2 * j + (q & 1);
        const bool ok = co < s.Cout;
        cp16z(wbase + (unsigned)r * CO * 32u + half_at(n, h),
              w + (ok ? (size_t)co * s.Kp + 16 * r + 8 * h : 0), ok);
    }
    // the voxels past the slices stay zero
    const int slack = 2 * (s.xrows - (s.TY + 2) * P);
    for (int i = threadIdx.x; i < 4 * s.chunks * slack; i += kThreads) {
        const int b = i / slack, k = i - b * slack;
        *reinterpret_cast<uint4 *>(sm + (xbase - wbase) + (size_t)(b + 1) * chunk_b - 16 * (k + 1)) =
            make_uint4(0u, 0u, 0u, 0u);
    }
    const int per = 2 * s.chunks, n_cp = (s.TY + 2) * P * per;
    auto load_slice = [&](int z) {
        const bool zin = z >= 0 && z < s.D;
        const unsigned dst = xbase + (unsigned)(z & 3) * slice_b;
        const __nv_bfloat16 *src = x + (zin ? (size_t)z * s.H * s.W * s.Cin : 0);
        for (int i = threadIdx.x; i < n_cp; i += kThreads) {
            const int v = div20(i, s.inv_c), c = i - v * per, r = div20(v, s.inv_p);
            const int yy = y0 - 1 + r, xx = x0 - 1 + v - r * P;
            const bool ok = zin && (unsigned)yy < (unsigned)s.H && (unsigned)xx < (unsigned)s.W;
            const size_t at = ok ? (size_t)(yy * s.W + xx) * s.Cin + 8 * c : 0;
            cp16z(dst + (unsigned)(c >> 1) * chunk_b + half_at(v, c & 1), src + at, ok);
        }
    };
    float bs[2 * NT];
#pragma unroll
    for (int k = 0; k < 2 * NT; ++k) {
        const int co = co0 + 2 * NT * t + k;
        bs[k] = (bias && co < s.Cout) ? bias[co] : 0.f;
    }

    load_slice(z0 - 1);
    load_slice(z0);
    load_slice(z0 + 1);
    cp_commit();
    // this lane's row and half of an operand's 16 x 16 block: A rows are
    // voxels (rows 0-7 and 8-15, halves), B rows are output channels
    const int arow = (lane & 7) + ((lane >> 3) & 1) * 8, ahalf = lane >> 4;
    const int brow = (lane & 7) + (lane >> 4) * 8, bhalf = (lane >> 3) & 1;
    const unsigned boff = half_at(brow, bhalf);
    const int groups = (s.TY * P + 16 * MT - 1) / (16 * MT);
    for (int z = z0; z < z1; ++z) {
        cp_wait<0>();
        __syncthreads();       // slices z - 1 .. z + 1 have landed; z - 2 is read
        if (z + 1 < z1) {
            load_slice(z + 2);
            cp_commit();
        }
        for (int gr = warp; gr < groups; gr += kWarps) {
            float acc[MT][NT][4] = {};
            const int v = gr * MT * 16 + arow;
            // operands of two steps: one step's products run while the next
            // step's ldmatrix are in flight
            unsigned fa[2][MT][4], fb[2][2 * NT];
            unsigned wa = wbase + boff;
            int dz = 0, dy = 0, dx = 0, j = 0;             // the step to load
            unsigned sl = xbase + (unsigned)((z - 1) & 3) * slice_b;
            int off = 0;
            auto load = [&](int b) {
                if (NT == 1) {
                    ldm_x2(fb[b][0], fb[b][1], wa);
                } else {
#pragma unroll
                    for (int k = 0; k < NT / 2; ++k) {
                        unsigned q[4];
                        ldm_x4(q, wa + (unsigned)k * 512u);
#pragma unroll
                        for (int e = 0; e < 4; ++e) fb[b][4 * k + e] = q[e];
                    }
                }
                wa += CO * 32;
#pragma unroll
                for (int i = 0; i < MT; ++i)      // (16 voxels on, the halves lie the same)
                    ldm_x4(fa[b][i], sl + half_at(v + off, ahalf) + 512u * i);
                // on to the next 16 channels, or the next tap
                sl += chunk_b;
                if (++j == s.chunks) {
                    j = 0;
                    ++off;
                    sl -= slice_b;
                    if (++dx == 3) {
                        dx = 0;
                        off += P - 3;
                        if (++dy == 3) {
                            dy = 0;
                            off = 0;
                            ++dz;
                            sl = xbase + (unsigned)((z + dz - 1) & 3) * slice_b;
                        }
                    }
                }
            };
            auto products = [&](int b) {
#pragma unroll
                for (int i = 0; i < MT; ++i)
#pragma unroll
                    for (int k = 0; k < NT; ++k)
                        mma16816(acc[i][k], fa[b][i], fb[b][2 * k], fb[b][2 * k + 1]);
            };
            const int steps = 27 * s.chunks;
            load(0);
            int st = 0;
            for (; st + 2 < steps; st += 2) {
                load(1);
                products(0);
                load(0);
                products(1);
            }
            if (st + 1 < steps) {
                load(1);
                products(0);
                products(1);
            } else {
                products(0);
            }
#pragma unroll
            for (int i = 0; i < MT; ++i)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int p = (gr * MT + i) * 16 + g + 8 * h;
                    const int row = div20(p, s.inv_p), col = p - row * P;
                    const int yy = y0 + row, xx = x0 + col, co = co0 + 2 * NT * t;
                    if (row >= s.TY || col >= s.TX || yy >= s.H || xx >= s.W || co >= s.Cout) continue;
                    float f[2 * NT];
#pragma unroll
                    for (int k = 0; k < 2 * NT; ++k) {
                        f[k] = acc[i][k >> 1][2 * h + (k & 1)] + bs[k];
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
                        if (whole && NT == 4) *reinterpret_cast<uint4 *>(po) = make_uint4(u[0], u[1], u[NT > 2 ? 2 : 0], u[NT > 2 ? 3 : 0]);
                        else if (whole && NT == 2) *reinterpret_cast<uint2 *>(po) = make_uint2(u[0], u[NT > 1 ? 1 : 0]);
                        else if (whole) *reinterpret_cast<unsigned *>(po) = u[0];
                        else
#pragma unroll
                            for (int k = 0; k < 2 * NT; ++k)
                                if (co + k < s.Cout) po[k] = __float2bfloat16(f[k]);
                    } else {
                        float *po = reinterpret_cast<float *>(out) + o;
                        if (whole && NT >= 2)
#pragma unroll
                            for (int k = 0; k < NT / 2; ++k)
                                reinterpret_cast<float4 *>(po)[k] =
                                    make_float4(f[4 * k], f[4 * k + 1], f[4 * k + 2], f[4 * k + 3]);
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

template <int NT, int MT>
cudaError_t launch_nt(const MmaShape &s, const __nv_bfloat16 *x, const __nv_bfloat16 *w,
                      const float *bias, void *out, int out_bf16, cudaStream_t st) {
    auto kern = out_bf16 ? k_conv3d_mma<NT, MT, true> : k_conv3d_mma<NT, MT, false>;
    const size_t smem = mma_smem(s);
    cudaError_t e = allow_dynamic_smem(kern, smem);
    if (e != cudaSuccess) return e;
    kern<<<dim3(s.nx * s.ny * s.nz, s.n_co), kThreads, smem, st>>>(x, w, bias, out, s);
    return cudaGetLastError();
}

}  // namespace

cudaError_t nn_conv3d_mma(const void *x, const void *w, const float *bias, void *out, int D, int H,
                          int W, int Cin, int Cout, int Kp, int relu, int out_bf16, cudaStream_t st) {
    MmaShape s;
    if (((uintptr_t)x | (uintptr_t)w | (uintptr_t)out) % 16 ||
        !conv_mma_plan(D, H, W, Cin, Cout, Kp, s))
        return cudaErrorNotSupported;
    s.relu = relu;
    const auto *xb = (const __nv_bfloat16 *)x;
    const auto *wb = (const __nv_bfloat16 *)w;
    if (s.MT == 4) {
        switch (s.CO) {
            case 8: return launch_nt<1, 4>(s, xb, wb, bias, out, out_bf16, st);
            case 16: return launch_nt<2, 4>(s, xb, wb, bias, out, out_bf16, st);
            default: return launch_nt<4, 4>(s, xb, wb, bias, out, out_bf16, st);
        }
    }
    switch (s.CO) {
        case 8: return launch_nt<1, 2>(s, xb, wb, bias, out, out_bf16, st);
        case 16: return launch_nt<2, 2>(s, xb, wb, bias, out, out_bf16, st);
        default: return launch_nt<4, 2>(s, xb, wb, bias, out, out_bf16, st);
    }
}
