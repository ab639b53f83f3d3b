// The learned path's weight and bias gradients: gw[co][tap Cin + ci] += sum_v
// gy[v][co] x[v + off(tap)][ci] and gb[co] += sum_v gy[v][co] of the 3 x 3 x 3
// convolution of nn.cu, channels-last volumes, zero padding.
//
// A contraction over the voxels of two channels-last operands, for 27 shifts
// of one of them: the floor is one read of x and gy. A block owns a tile of
// TX x TY voxels of every z slice of a segment, 16 input channels and up to 64
// output channels, and walks the segment slice by slice. Slices of x (with a
// one-voxel halo) stand in a ring of four shared-memory buffers, three in use
// and one being filled by cp.async; gy in two. A slice is a flat list of
// padded rows, P = TX + 2 voxels each, so that a tap is an offset dy P + dx
// into it and the contraction runs over the flat list in steps of 16 voxels
// without remainders per row (gy is zero in the two padding columns). Warp
// (dz, dy) of nine holds the three taps of its row; both operands reach the
// tensor cores (m16n8k16) through transposing ldmatrix loads, from rows padded
// to 48 (80, 144) bytes, which are free of bank conflicts. Each block writes
// a partial sum every 2048 voxels or so, and a second kernel adds them in a
// fixed order: gradients are bitwise reproducible. (With one partial sum per
// block, chains of 400 steps, gw was off by 2.6e-6 instead of 0.9e-6.) Where gy
// has a zero of its own that is no voxel (padding columns, rows past the tile or
// the volume) x is masked to zero too: a tap's list passes real voxels there that
// are none of its own, and a non-finite one would reach the tap's sum.
//
// 96 x 128 x 128 voxels, 16 -> 16 channels: 0.120 ms with the sums (before, with
// one 16-voxel step of both operands gathered element by element at a time and a
// serial bias sum: 3.70, 0.17 and 0.10 ms). What is left is shared-memory loads:
// three operand blocks of x and one of gy for six products a warp. Of the steps
// (a quarter there) that hold a padding position only those mask x; masking every
// step took 0.130 ms, none 0.110.
#include <cuda_bf16.h>

#include <type_traits>

#include "common.cuh"
#include "kernels.h"

namespace {

constexpr int kWarps = 9, kThreads = 32 * kWarps;
constexpr int kSlack = 24;        // voxels past a slice that the last step may touch (at most 17)
constexpr int kChain = 128;       // steps of 16 voxels of one partial sum
constexpr int kMaxSteps = 48;     // of a slice: 256 rows of three positions

struct WgShape {
    int D, H, W, Cin, Cout, Kp;
    int TX, TY, nx, ny;           // tile and tiles
    int zlen, nz;                 // slices of a segment, segments
    int zsum, nsum;               // slices of a partial sum, partial sums of a segment
    int n_ci, n_co;               // channel blocks of 16 (8) and 16 MT
    int xrows, grows;             // voxel rows of a slice buffer of x and gy
    unsigned inv_p;               // ceil(2^20 / P)
    int parts() const { return nx * ny * nz * nsum; }
};

__host__ __device__ constexpr int x_pitch(int NT) { return NT == 1 ? 8 : 24; }        // BF16 per voxel
__host__ __device__ constexpr int g_pitch(int MT) { return 16 * MT + 8; }

int mt_of(int Cout) { return Cout <= 16 ? 1 : Cout <= 32 ? 2 : 4; }
int nt_of(int Cin) { return Cin <= 8 ? 1 : 2; }
// shared memory a block may take: two blocks an SM up to 32 output channels
// (beside the static sb and live and the 1 KB the system reserves for each)
__host__ __device__ constexpr int max_smem(int MT) { return (MT <= 2 ? 110 : 200) * 1024; }

size_t smem_bytes(const WgShape &s) {
    return 2 * (4 * (size_t)s.xrows * x_pitch(nt_of(s.Cin)) +
                2 * (size_t)s.grows * g_pitch(mt_of(s.Cout)));
}

// Tiles of about 256 voxels, rows of at most 64, fewer rows where two blocks
// would not share an SM's memory (up to 32 output channels) or one would not
// fit; segments of at least four slices (two more are loaded for each), as
// many as fill the device.
WgShape wg_shape(int D, int H, int W, int Cin, int Cout, int Kp) {
    WgShape s{};
    s.D = D;
    s.H = H;
    s.W = W;
    s.Cin = Cin;
    s.Cout = Cout;
    s.Kp = Kp;
    const int MT = mt_of(Cout), NT = nt_of(Cin);
    s.nx = (W + 63) / 64;
    s.TX = (W + s.nx - 1) / s.nx;
    const int P = s.TX + 2;
    int ty = 256 / s.TX < H ? 256 / s.TX : H;
    for (;; --ty) {
        s.ny = (H + ty - 1) / ty;
        s.TY = (H + s.ny - 1) / s.ny;
        s.xrows = (s.TY + 2) * P + kSlack;
        s.grows = (s.TY * P + 15) / 16 * 16;
        if (smem_bytes(s) <= (size_t)max_smem(MT) || ty == 1) break;   // (one row: 64 KB at most)
    }
    s.inv_p = ((1u << 20) + P - 1) / P;
    s.n_ci = (Cin + 8 * NT - 1) / (8 * NT);
    s.n_co = (Cout + 16 * MT - 1) / (16 * MT);
    const int slots = 152 * (MT <= 2 ? 2 : 1);
    const long long per = (long long)s.nx * s.ny * s.n_ci * s.n_co;
    long long nz = slots / per;
    if (nz > D / 4) nz = D / 4;
    if (nz < 1) nz = 1;
    s.zlen = (int)((D + nz - 1) / nz);
    s.nz = (D + s.zlen - 1) / s.zlen;
    // the tensor cores truncate their running sum, so a chain of products is
    // at most kChain steps long
    s.zsum = kChain / (s.grows / 16) < 1 ? 1 : kChain / (s.grows / 16);
    s.nsum = (s.zlen + s.zsum - 1) / s.zsum;
    s.zsum = (s.zlen + s.nsum - 1) / s.nsum;
    return s;
}

__device__ __forceinline__ unsigned smem_u32(const void *p) {
    return (unsigned)__cvta_generic_to_shared(p);
}
// 16 bytes to shared memory, zeros where !ok (the source is not read then)
__device__ __forceinline__ void cp16z(void *dst, const void *src, bool ok) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(smem_u32(dst)), "l"(src),
                 "r"(ok ? 16 : 0)
                 : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

__device__ __forceinline__ void ldm_x4_t(unsigned (&r)[4], unsigned addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}
__device__ __forceinline__ void ldm_x2_t(unsigned &r0, unsigned &r1, unsigned addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];\n"
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

// Running sums: FP32, and a float pair (Knuth's two-sum), rounded once at the end
struct Plain {
    float s = 0.f;
    __device__ __forceinline__ void operator+=(float x) { s += x; }
    __device__ __forceinline__ float value() const { return s; }
};
struct Pair {
    float hi = 0.f, lo = 0.f;
    __device__ __forceinline__ void operator+=(float x) {
        const float s = hi + x, b = s - hi;
        lo += (hi - (s - b)) + (x - b);
        hi = s;
    }
    // (an infinite sum has no low part: it would be NaN)
    __device__ __forceinline__ float value() const { return isinf(hi) ? hi : hi + lo; }
};

// Copies a slice's voxel rows [rows x P] of `C` channels, channels c0 .. c0 +
// CW, into `dst` (pitch elements per voxel): voxel (y0 + r, x0 + c) of slice z,
// zeros outside the volume, past column `cols`, and past channel C. VEC: 16
// bytes at a time by cp.async (C a multiple of 8, 16-byte aligned base).
template <int CW, bool VEC>
__device__ __forceinline__ void load_slice(__nv_bfloat16 *dst, int pitch, const __nv_bfloat16 *src,
                                           const WgShape &s, int C, int c0, int z, int y0, int x0,
                                           int rows, int P, int cols) {
    const bool zin = z >= 0 && z < s.D;
    const __nv_bfloat16 *plane = src + (zin ? (size_t)z * s.H * s.W * C : 0);
    constexpr int CH = VEC ? CW / 8 : CW;
    for (int i = threadIdx.x; i < rows * P * CH; i += kThreads) {
        // (v P < 2^20: v / P by the rounded-up reciprocal is exact)
        const int h = i % CH, v = i / CH, r = (int)((unsigned)v * s.inv_p >> 20), c = v - r * P;
        const int y = y0 + r, x = x0 + c, k = c0 + (VEC ? 8 * h : h);
        const bool ok = zin && (unsigned)y < (unsigned)s.H && (unsigned)x < (unsigned)s.W && c < cols &&
                        k < C;
        const size_t at = ok ? (size_t)(y * s.W + x) * C + k : 0;
        if (VEC) cp16z(dst + (size_t)v * pitch + 8 * h, plane + at, ok);
        else dst[(size_t)v * pitch + h] = ok ? plane[at] : __float2bfloat16(0.f);
    }
}

// grid: (spatial parts, input-channel blocks, output-channel blocks)
template <int NT, int MT, bool XVEC, bool GVEC>
__global__ void __launch_bounds__(kThreads, MT <= 2 ? 2 : 1)
k_wgrad(const __nv_bfloat16 *__restrict__ x, const __nv_bfloat16 *__restrict__ gy,
        float *__restrict__ part, float *__restrict__ bpart, WgShape s) {
    constexpr int XP = x_pitch(NT), GP = g_pitch(MT);
    extern __shared__ __align__(16) __nv_bfloat16 sm[];
    __shared__ float sb[kWarps][16 * MT];                  // the warps' bias sums
    __shared__ uint2 live[kMaxSteps][4];                   // [step][lane & 3]: x's mask
    __shared__ unsigned pads[2];                           // the steps with a zero in it
    __nv_bfloat16 *xs = sm;                                // [4][xrows][XP]
    __nv_bfloat16 *gs = sm + 4 * (size_t)s.xrows * XP;     // [2][grows][GP]
    const int P = s.TX + 2;
    const int bx = blockIdx.x % s.nx, by = (blockIdx.x / s.nx) % s.ny, bz = blockIdx.x / (s.nx * s.ny);
    const int x0 = bx * s.TX, y0 = by * s.TY;
    const int z0 = bz * s.zlen, z1 = min(s.D, z0 + s.zlen);
    const int ci0 = blockIdx.y * 8 * NT, co0 = blockIdx.z * 16 * MT;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 2, t = lane & 3;
    const int dz = warp / 3, dy = warp % 3;
    const bool with_bias = bpart != nullptr && blockIdx.y == 0;

    // the voxels past the slices, and gy's past its rows, stay zero
    for (int i = threadIdx.x; i < 4 * kSlack * XP; i += kThreads) {
        const int b = i / (kSlack * XP), k = i - b * kSlack * XP;
        xs[((size_t)b * s.xrows + s.xrows - kSlack) * XP + k] = __float2bfloat16(0.f);
    }
    const int gtail = s.grows - s.TY * P;
    for (int i = threadIdx.x; i < 2 * gtail * GP; i += kThreads) {
        const int b = i / (gtail * GP), k = i - b * gtail * GP;
        gs[((size_t)b * s.grows + s.TY * P) * GP + k] = __float2bfloat16(0.f);
    }

    // all ones where positions 16 st + 2 t, + 1 (and + 8, + 9) are voxels of the tile
    const int cols = min(s.TX, s.W - x0), rows = min(s.TY, s.H - y0);
    if (threadIdx.x < 2) pads[threadIdx.x] = 0u;
    __syncthreads();
    for (int i = threadIdx.x; i < s.grows / 4; i += kThreads) {
        auto word = [&](int p) {
            unsigned m = 0;
            for (int e = 0; e < 2; ++e) {
                const int r = (p + e) / P, c = p + e - r * P;
                if (r < rows && c < cols) m |= 0xffffu << (16 * e);
            }
            return m;
        };
        const int p = i / 4 * 16 + (i & 3) * 2;
        const uint2 m = make_uint2(word(p), word(p + 8));
        live[i / 4][i & 3] = m;
        if ((m.x & m.y) != ~0u) atomicOr(&pads[i / 128], 1u << (i / 4 % 32));
    }

    auto load_x = [&](int z) {
        load_slice<8 * NT, XVEC>(xs + (size_t)(z & 3) * s.xrows * XP, XP, x, s, s.Cin, ci0, z,
                                 y0 - 1, x0 - 1, s.TY + 2, P, P);
    };
    // rows of the next tile are that tile's: y past this one's rows is past
    // the loop, columns past TX are zero
    auto load_g = [&](int z) {
        load_slice<16 * MT, GVEC>(gs + (size_t)(z & 1) * s.grows * GP, GP, gy, s, s.Cout, co0, z,
                                  y0, x0, s.TY, P, s.TX);
    };

    float acc[3][MT][NT][4] = {};
    // bias sums of output channels g and g + 8, over this lane's voxels of this
    // warp's steps: FP32 additions (products with ones on the tensor cores, which
    // truncate, were twice as far off for a gradient of one sign)
    float bacc[MT][2] = {};

    // writes partial sum f of the segment and clears the accumulators
    auto store_part = [&](int f) {
        const size_t pi = (size_t)blockIdx.x * s.nsum + f;
#pragma unroll
        for (int i = 0; i < MT; ++i) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int co = co0 + i * 16 + g + 8 * h;
                float *row = part + (pi * s.Cout + co) * s.Kp + (9 * dz + 3 * dy) * s.Cin;
#pragma unroll
                for (int k = 0; k < 3; ++k)
#pragma unroll
                    for (int j = 0; j < NT; ++j)
#pragma unroll
                        for (int q = 0; q < 2; ++q) {
                            const int ci = ci0 + 8 * j + 2 * t + q;
                            if (co < s.Cout && ci < s.Cin) row[k * s.Cin + ci] = acc[k][i][j][2 * h + q];
                            acc[k][i][j][2 * h + q] = 0.f;
                        }
                if (with_bias) {
                    float b = bacc[i][h];
                    b += __shfl_xor_sync(0xffffffffu, b, 1);
                    b += __shfl_xor_sync(0xffffffffu, b, 2);
                    if (t == 0) sb[warp][i * 16 + g + 8 * h] = b;
                    bacc[i][h] = 0.f;
                }
            }
        }
        if (!with_bias) return;        // (one answer for the whole block)
        __syncthreads();
        const int c = (int)threadIdx.x, co = co0 + c;
        if (c < 16 * MT && co < s.Cout) {
            Pair b;
            for (int k = 0; k < kWarps; ++k) b += sb[k][c];
            bpart[pi * s.Cout + co] = b.value();
        }
        __syncthreads();
    };

    load_x(z0 - 1);
    load_x(z0);
    load_x(z0 + 1);
    load_g(z0);
    cp_commit();
    // this lane's row and column within an operand's 16 x 16 block
    const int arow = (lane & 7) + ((lane >> 4) & 1) * 8, acol = ((lane >> 3) & 1) * 8;
    const int brow = (lane & 7) + ((lane >> 3) & 1) * 8, bcol = NT == 2 ? (lane >> 4) * 8 : 0;
    for (int z = z0; z < z1; ++z) {
        cp_wait<0>();
        __syncthreads();       // slices z - 1 .. z + 1 have landed; the last ones are read
        if (z + 1 < z1) {
            load_x(z + 2);
            load_g(z + 1);
            cp_commit();
        }
        const unsigned xa = smem_u32(xs + ((size_t)((z + dz - 1) & 3) * s.xrows + dy * P + brow) * XP +
                                     bcol);
        const unsigned ga = smem_u32(gs + ((size_t)(z & 1) * s.grows + arow) * GP + acol);
        const int steps = s.grows / 16;
        int bst = with_bias ? warp : steps;       // this warp's next step of the bias sum
        const unsigned long long padded = pads[0] | (unsigned long long)pads[1] << 32;
        auto step = [&](int st, auto masked) {
            unsigned a[MT][4];
#pragma unroll
            for (int i = 0; i < MT; ++i) ldm_x4_t(a[i], ga + (unsigned)(st * 16 * GP + 16 * i) * 2);
            uint2 lv;
            if constexpr (decltype(masked)::value) lv = live[st][t];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                unsigned b[4];
                const unsigned addr = xa + (unsigned)((st * 16 + k) * XP) * 2;
                if (NT == 2) ldm_x4_t(b, addr);
                else ldm_x2_t(b[0], b[1], addr);
#pragma unroll
                for (int j = 0; j < NT; ++j) {
                    if constexpr (decltype(masked)::value) {
                        b[2 * j] &= lv.x;
                        b[2 * j + 1] &= lv.y;
                    }
#pragma unroll
                    for (int i = 0; i < MT; ++i) mma16816(acc[k][i][j], a[i], b[2 * j], b[2 * j + 1]);
                }
            }
            if (st == bst) {
                bst += kWarps;
                auto lo = [](unsigned v) { return __uint_as_float(v << 16); };
                auto hi = [](unsigned v) { return __uint_as_float(v & 0xffff0000u); };
#pragma unroll
                for (int i = 0; i < MT; ++i)
#pragma unroll
                    for (int h = 0; h < 2; ++h)
                        bacc[i][h] += (lo(a[i][h]) + hi(a[i][h])) + (lo(a[i][h + 2]) + hi(a[i][h + 2]));
            }
        };
        for (int st = 0; st < steps; ++st) {
            if (padded >> st & 1) step(st, std::true_type());
            else step(st, std::false_type());
        }
        if ((z + 1 - z0) % s.zsum == 0 || z + 1 == z1) store_part((z - z0) / s.zsum);
    }
    // a short last segment: its remaining partial sums are zero
    for (int f = (z1 - z0 + s.zsum - 1) / s.zsum; f < s.nsum; ++f) store_part(f);
}

// gw[co][k] += sum over the parts (k < K), gb[co] += sum over the bias parts:
// 32 sums a block, kSumWays threads each (every kSumWays-th part, then in order;
// eight threads with four loads in flight took 0.023 ms for 768 parts).
constexpr int kSumWays = 16;
template <class T>
__device__ __forceinline__ void sum_parts(const float *__restrict__ p, float *__restrict__ o,
                                          float (&s)[kSumWays][32], int nparts, size_t stride,
                                          bool live) {
    const int e = threadIdx.x & 31, q = threadIdx.x >> 5;
    T v;
    if (live) {
#pragma unroll 16
        for (int c = q; c < nparts; c += kSumWays) v += p[(size_t)c * stride];
    }
    s[q][e] = v.value();
    __syncthreads();
    if (q == 0 && live) {
        T r;
        for (int k = 0; k < kSumWays; ++k) r += s[k][e];
        r += *o;
        *o = r.value();
    }
}
__global__ void __launch_bounds__(32 * kSumWays)
k_wgrad_sum(const float *__restrict__ part, const float *__restrict__ bpart, float *__restrict__ gw,
            float *__restrict__ gb, int nparts, int Cout, int K, int Kp, int wblocks) {
    __shared__ float s[kSumWays][32];
    const int e = threadIdx.x & 31;
    if ((int)blockIdx.x < wblocks) {
        const int i = (int)blockIdx.x * 32 + e;
        const size_t at = (size_t)(i / K) * Kp + i % K;
        sum_parts<Plain>(part + at, gw + at, s, nparts, (size_t)Cout * Kp, i < Cout * K);
    } else {
        const int i = ((int)blockIdx.x - wblocks) * 32 + e;
        sum_parts<Pair>(bpart + i, gb + i, s, nparts, (size_t)Cout, i < Cout);
    }
}

template <int NT, int MT, bool XVEC, bool GVEC>
cudaError_t launch_one(const WgShape &s, const __nv_bfloat16 *x, const __nv_bfloat16 *gy, float *part,
                       float *bpart, cudaStream_t st) {
    auto kern = k_wgrad<NT, MT, XVEC, GVEC>;
    const size_t smem = smem_bytes(s);
    // (the same limit whatever the shape: with this call's size, a thread with a
    // smaller shape could lower it between another thread's call and launch)
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem(MT));
    if (e != cudaSuccess) return e;
    kern<<<dim3(s.nx * s.ny * s.nz, s.n_ci, s.n_co), kThreads, smem, st>>>(x, gy, part, bpart, s);
    return cudaGetLastError();
}

template <int NT, int MT>
cudaError_t launch_vec(const WgShape &s, const __nv_bfloat16 *x, const __nv_bfloat16 *gy, float *part,
                       float *bpart, cudaStream_t st) {
    const bool xv = s.Cin % 8 == 0 && (uintptr_t)x % 16 == 0;
    const bool gv = s.Cout % 8 == 0 && (uintptr_t)gy % 16 == 0;
    if (xv) return gv ? launch_one<NT, MT, true, true>(s, x, gy, part, bpart, st)
                      : launch_one<NT, MT, true, false>(s, x, gy, part, bpart, st);
    return gv ? launch_one<NT, MT, false, true>(s, x, gy, part, bpart, st)
              : launch_one<NT, MT, false, false>(s, x, gy, part, bpart, st);
}

}  // namespace

size_t nn_wgrad_work_floats(int D, int H, int W, int Cin, int Cout, int Kp) {
    const WgShape s = wg_shape(D, H, W, Cin, Cout, Kp);
    return (size_t)s.parts() * Cout * (Kp + 1);
}

cudaError_t nn_conv3d_wgrad(const void *x, const void *gy, float *gw, float *gb, float *work,
                            int D, int H, int W, int Cin, int Cout, int Kp, cudaStream_t st) {
    const WgShape s = wg_shape(D, H, W, Cin, Cout, Kp);
    const auto *xb = (const __nv_bfloat16 *)x;
    const auto *gyb = (const __nv_bfloat16 *)gy;
    float *bpart = gb ? work + (size_t)s.parts() * Cout * Kp : nullptr;
    cudaError_t e;
    if (nt_of(Cin) == 1) {
        switch (mt_of(Cout)) {
            case 1: e = launch_vec<1, 1>(s, xb, gyb, work, bpart, st); break;
            case 2: e = launch_vec<1, 2>(s, xb, gyb, work, bpart, st); break;
            default: e = launch_vec<1, 4>(s, xb, gyb, work, bpart, st); break;
        }
    } else {
        switch (mt_of(Cout)) {
            case 1: e = launch_vec<2, 1>(s, xb, gyb, work, bpart, st); break;
            case 2: e = launch_vec<2, 2>(s, xb, gyb, work, bpart, st); break;
            default: e = launch_vec<2, 4>(s, xb, gyb, work, bpart, st); break;
        }
    }
    if (e != cudaSuccess) return e;
    const int K = 27 * Cin;
    const int wblocks = (Cout * K + 31) / 32, bblocks = gb ? (Cout + 31) / 32 : 0;
    k_wgrad_sum<<<wblocks + bblocks, 32 * kSumWays, 0, st>>>(work, bpart, gw, gb, s.parts(), Cout, K, Kp,
                                                   wblocks);
    return cudaGetLastError();
}
