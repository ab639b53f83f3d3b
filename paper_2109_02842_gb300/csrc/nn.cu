// Learned fast path: kernels of a 3-D convolutional encoder-decoder that maps
// features of a cheap reconstruction to the full one (the network is
// described in paper_2109_02842_gb300/learned.py; the paper has no learned
// component).
//
// Volumes are channels-last: x[v][c] with v = (z H + y) W + x. Convolutions
// are 3 x 3 x 3, stride 1, 'same' zero padding; weights w[co][k] with
// k = tap Cin + ci, tap = (dz 3 + dy) 3 + dx reading x[z+dz-1][y+dy-1][x+dx-1],
// rows padded with zeros to a multiple of 16.
//
// The convolution is an implicit GEMM on the tensor cores: out[v][co] =
// sum_k A[v][k] B[k][co] with A the (never materialised) im2col matrix and B
// the weights. Cin of one to four takes nn_conv_small.cu, Cin a multiple of 16
// nn_conv_mma.cu or, wide and in shapes that suit it, the tcgen05 kernel of
// nn_tc.cu; what those refuse (other Cin, unaligned operands) the kernel
// below, BF16 mma.sync m16n8k16 with FP32 accumulation. All sum in the same
// order, K in steps of 16, with equal results bit for bit. A block of 4
// warps owns 64 voxels x (8 NT) output channels; per 16-wide K chunk it
// stages the A tile (one 32-byte row per voxel when Cin is a multiple of 16 and x
// 16-byte aligned, an element gather otherwise) and the B tile in shared memory.
// The backward pass reuses the forward kernel for the input gradient (the
// transposed convolution is a convolution with flipped taps and swapped
// channel roles); the weight gradient is in nn_wgrad.cu.
#include <cuda_bf16.h>

#include "common.cuh"
#include "kernels.h"

namespace {

constexpr int kRowPad = 24;   // bf16 per staged row: 16 + 8 (conflict-free fragment loads)

__device__ __forceinline__ void mma_bf16_16816(float (&d)[4], const unsigned (&a)[4],
                                               const unsigned (&b)[2]) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
        "{%8,%9}, {%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

__device__ __forceinline__ unsigned ld_pair(const __nv_bfloat16 *p) {
    return *reinterpret_cast<const unsigned *>(p);
}

struct Vol {
    int D, H, W;
    __device__ __forceinline__ bool neighbour(int v, int tap, int &nv) const {
        const int x = v % W;
        const int y = (v / W) % H;
        const int z = v / (W * H);
        const int dz = tap / 9 - 1, dy = (tap / 3) % 3 - 1, dx = tap % 3 - 1;
        const int zz = z + dz, yy = y + dy, xx = x + dx;
        if (zz < 0 || zz >= D || yy < 0 || yy >= H || xx < 0 || xx >= W) return false;
        nv = (zz * H + yy) * W + xx;
        return true;
    }
};

// out[v][co] = act(bias[co] + sum_k x~[v][k] w[co][k])
template <int NT, bool OUT_BF16>
__global__ void __launch_bounds__(128)
k_conv3d(const __nv_bfloat16 *__restrict__ x, const __nv_bfloat16 *__restrict__ w,
         const float *__restrict__ bias, void *__restrict__ out, Vol vol, int Cin, int Cout,
         int Kp, int relu, bool xvec, bool wvec) {
    constexpr int NTILE = 8 * NT;
    __shared__ __align__(16) __nv_bfloat16 As[64][kRowPad];
    __shared__ __align__(16) __nv_bfloat16 Bs[NTILE][kRowPad];
    const int V = vol.D * vol.H * vol.W;
    const int v0 = blockIdx.x * 64;
    const int n0 = blockIdx.y * NTILE;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 2, t = lane & 3;
    const int K = 27 * Cin;
    float acc[NT][4];
#pragma unroll
    for (int j = 0; j < NT; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;

    for (int k0 = 0; k0 < Kp; k0 += 16) {
        // A tile: 64 voxels x 16 k
        if (xvec) {
            const int row = threadIdx.x >> 1, half = threadIdx.x & 1;
            const int tap = k0 / Cin, ci0 = k0 - tap * Cin;
            uint4 val = make_uint4(0u, 0u, 0u, 0u);
            int nv;
            if (v0 + row < V && k0 < K && vol.neighbour(v0 + row, tap, nv))
                val = *reinterpret_cast<const uint4 *>(x + (size_t)nv * Cin + ci0 + 8 * half);
            *reinterpret_cast<uint4 *>(&As[row][8 * half]) = val;
        } else {
            for (int e = threadIdx.x; e < 64 * 16; e += 128) {
                const int row = e >> 4, kk = e & 15;
                const int k = k0 + kk;
                __nv_bfloat16 val = __float2bfloat16(0.f);
                int nv;
                if (v0 + row < V && k < K) {
                    const int tap = k / Cin, ci = k - tap * Cin;
                    if (vol.neighbour(v0 + row, tap, nv)) val = x[(size_t)nv * Cin + ci];
                }
                As[row][kk] = val;
            }
        }
        // B tile: NTILE output channels x 16 k (k contiguous per channel)
        if (wvec) {
            for (int e = threadIdx.x; e < NTILE * 2; e += 128) {
                const int n = e >> 1, half = e & 1;
                uint4 val = make_uint4(0u, 0u, 0u, 0u);
                if (n0 + n < Cout)
                    val = *reinterpret_cast<const uint4 *>(w + (size_t)(n0 + n) * Kp + k0 + 8 * half);
                *reinterpret_cast<uint4 *>(&Bs[n][8 * half]) = val;
            }
        } else {
            for (int e = threadIdx.x; e < NTILE * 16; e += 128) {
                const int n = e >> 4, k = e & 15;
                Bs[n][k] = n0 + n < Cout ? w[(size_t)(n0 + n) * Kp + k0 + k] : __float2bfloat16(0.f);
            }
        }
        __syncthreads();
        unsigned a[4];
        const int r0 = warp * 16;
        a[0] = ld_pair(&As[r0 + g][2 * t]);
        a[1] = ld_pair(&As[r0 + g + 8][2 * t]);
        a[2] = ld_pair(&As[r0 + g][2 * t + 8]);
        a[3] = ld_pair(&As[r0 + g + 8][2 * t + 8]);
#pragma unroll
        for (int j = 0; j < NT; ++j) {
            unsigned b[2];
            b[0] = ld_pair(&Bs[j * 8 + g][2 * t]);
            b[1] = ld_pair(&Bs[j * 8 + g][2 * t + 8]);
            mma_bf16_16816(acc[j], a, b);
        }
        __syncthreads();
    }
    // epilogue: rows g, g+8 of this warp's 16 voxels; columns 2t, 2t+1 of each n-tile
#pragma unroll
    for (int j = 0; j < NT; ++j) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int v = v0 + warp * 16 + g + 8 * h;
            if (v >= V) continue;
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int co = n0 + j * 8 + 2 * t + q;
                if (co >= Cout) continue;
                float r = acc[j][2 * h + q] + (bias ? bias[co] : 0.f);
                if (relu) r = fmaxf(r, 0.f);
                if (OUT_BF16)
                    reinterpret_cast<__nv_bfloat16 *>(out)[(size_t)v * Cout + co] = __float2bfloat16(r);
                else
                    reinterpret_cast<float *>(out)[(size_t)v * Cout + co] = r;
            }
        }
    }
}

// wt[ci][tap' Cout + co] = w[co][tap Cin + ci], tap' = 26 - tap
__global__ void k_weight_flip(const __nv_bfloat16 *__restrict__ w, __nv_bfloat16 *__restrict__ wt,
                              int Cin, int Cout, int Kp, int Kpt) {
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= Cin * Kpt) return;
    const int ci = idx / Kpt, k = idx - ci * Kpt;
    __nv_bfloat16 v = __float2bfloat16(0.f);
    if (k < 27 * Cout) {
        const int tp = k / Cout, co = k - tp * Cout;
        v = w[(size_t)co * Kp + (26 - tp) * Cin + ci];
    }
    wt[idx] = v;
}

// The element-wise passes are bound by memory. Eight elements (16 bytes of
// BF16) a thread where every operand is 16-byte aligned, the rest one by one:
// 25 M elements, ReLU backward 0.099 -> 0.027 ms, sum 0.064 -> 0.021 ms (200
// and 150 MB; one element a thread kept too few bytes in flight).
struct bf8 {
    uint4 q;
    __device__ __forceinline__ float get(int i) const {
        const unsigned w = i < 2 ? q.x : i < 4 ? q.y : i < 6 ? q.z : q.w;
        return __uint_as_float((i & 1) ? (w & 0xffff0000u) : (w << 16));
    }
    __device__ static __forceinline__ bf8 of(const float (&f)[8]) {
        unsigned w[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            __nv_bfloat162 h = __floats2bfloat162_rn(f[2 * k], f[2 * k + 1]);
            w[k] = *reinterpret_cast<unsigned *>(&h);
        }
        return {make_uint4(w[0], w[1], w[2], w[3])};
    }
};
__device__ __forceinline__ void load8(const float *p, float (&f)[8]) {
    const float4 a = reinterpret_cast<const float4 *>(p)[0], b = reinterpret_cast<const float4 *>(p)[1];
    f[0] = a.x; f[1] = a.y; f[2] = a.z; f[3] = a.w;
    f[4] = b.x; f[5] = b.y; f[6] = b.z; f[7] = b.w;
}
__device__ __forceinline__ bf8 load8(const __nv_bfloat16 *p) {
    return {*reinterpret_cast<const uint4 *>(p)};
}

// OP 0: out (bf16) = g (f32) where y > 0, else 0; 1: out (bf16) = g; 2: out
// (bf16) = a + b (bf16). n8 groups of eight elements, then up to n.
template <int OP>
__global__ void __launch_bounds__(256)
k_to_bf16(const void *__restrict__ a, const __nv_bfloat16 *__restrict__ b,
          __nv_bfloat16 *__restrict__ out, size_t n8, size_t n) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const float *af = (const float *)a;
    const __nv_bfloat16 *ab = (const __nv_bfloat16 *)a;
    if (i < n8) {
        float f[8];
        if (OP == 2) {
            const bf8 p = load8(ab + 8 * i), q = load8(b + 8 * i);
#pragma unroll
            for (int k = 0; k < 8; ++k) f[k] = p.get(k) + q.get(k);
        } else {
            load8(af + 8 * i, f);
            if (OP == 0) {
                const bf8 y = load8(b + 8 * i);
#pragma unroll
                for (int k = 0; k < 8; ++k) f[k] = y.get(k) > 0.f ? f[k] : 0.f;
            }
        }
        *reinterpret_cast<uint4 *>(out + 8 * i) = bf8::of(f).q;
        return;
    }
    const size_t e = 8 * n8 + (i - n8);
    if (e >= n) return;
    float f;
    if (OP == 0) f = __bfloat162float(b[e]) > 0.f ? af[e] : 0.f;
    else if (OP == 1) f = af[e];
    else f = __bfloat162float(ab[e]) + __bfloat162float(b[e]);
    out[e] = __float2bfloat16(f);
}

__global__ void k_accum_f32(const float *__restrict__ a, float *__restrict__ acc, size_t n) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) acc[i] += a[i];
}

// y[Z][Y][X][c] = mean of the 2x2x2 block of x (D, H, W even)
__global__ void k_avgpool2(const __nv_bfloat16 *__restrict__ x, __nv_bfloat16 *__restrict__ y,
                           int D, int H, int W, int C) {
    const size_t n = (size_t)(D / 2) * (H / 2) * (W / 2) * C;
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int c = (int)(i % C);
    const size_t o = i / C;
    const int X = (int)(o % (W / 2)), Y = (int)((o / (W / 2)) % (H / 2)), Z = (int)(o / ((W / 2) * (H / 2)));
    float s = 0.f;
    for (int d = 0; d < 8; ++d) {
        const int z = 2 * Z + (d >> 2), yy = 2 * Y + ((d >> 1) & 1), xx = 2 * X + (d & 1);
        s += __bfloat162float(x[(((size_t)z * H + yy) * W + xx) * C + c]);
    }
    y[i] = __float2bfloat16(0.125f * s);
}

// the same with 8 channels (16 bytes) per thread, for C a multiple of 8
__global__ void k_avgpool2_v8(const __nv_bfloat16 *__restrict__ x, __nv_bfloat16 *__restrict__ y,
                              int D, int H, int W, int C8) {
    const size_t n = (size_t)(D / 2) * (H / 2) * (W / 2) * C8;
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int c = (int)(i % C8);
    const size_t o = i / C8;
    const int X = (int)(o % (W / 2)), Y = (int)((o / (W / 2)) % (H / 2)), Z = (int)(o / ((W / 2) * (H / 2)));
    float s[8] = {};
#pragma unroll
    for (int d = 0; d < 8; ++d) {
        const int z = 2 * Z + (d >> 2), yy = 2 * Y + ((d >> 1) & 1), xx = 2 * X + (d & 1);
        const bf8 v = load8(x + ((((size_t)z * H + yy) * W + xx) * C8 + c) * 8);
#pragma unroll
        for (int k = 0; k < 8; ++k) s[k] += v.get(k);
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) s[k] *= 0.125f;
    *reinterpret_cast<uint4 *>(y + 8 * i) = bf8::of(s).q;
}

// gx[v] += gy[parent(v)] / 8
__global__ void k_avgpool2_bwd(const float *__restrict__ gy, float *__restrict__ gx, int D, int H,
                               int W, int C) {
    const size_t n = (size_t)D * H * W * C;
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int c = (int)(i % C);
    const size_t v = i / C;
    const int x = (int)(v % W), y = (int)((v / W) % H), z = (int)(v / ((size_t)W * H));
    gx[i] += 0.125f * gy[(((size_t)(z / 2) * (H / 2) + y / 2) * (W / 2) + x / 2) * C + c];
}

// y (2D x 2H x 2W) = nearest x
__global__ void k_upsample2(const __nv_bfloat16 *__restrict__ x, __nv_bfloat16 *__restrict__ y,
                            int D, int H, int W, int C) {
    const size_t n = (size_t)8 * D * H * W * C;
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int c = (int)(i % C);
    const size_t v = i / C;
    const int W2 = 2 * W, H2 = 2 * H;
    const int xx = (int)(v % W2), yy = (int)((v / W2) % H2), zz = (int)(v / ((size_t)W2 * H2));
    y[i] = x[(((size_t)(zz / 2) * H + yy / 2) * W + xx / 2) * C + c];
}

// the same with 8 channels (16 bytes) per thread, for C a multiple of 8
__global__ void k_upsample2_v8(const uint4 *__restrict__ x, uint4 *__restrict__ y, int D, int H,
                               int W, int C8) {
    const size_t n = (size_t)8 * D * H * W * C8;
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int c = (int)(i % C8);
    const size_t v = i / C8;
    const int W2 = 2 * W, H2 = 2 * H;
    const int xx = (int)(v % W2), yy = (int)((v / W2) % H2), zz = (int)(v / ((size_t)W2 * H2));
    y[i] = x[(((size_t)(zz / 2) * H + yy / 2) * W + xx / 2) * C8 + c];
}

// gx[Z][Y][X] = sum of gy over the 8 children (gx has the small size D x H x W)
__global__ void k_upsample2_bwd(const float *__restrict__ gy, float *__restrict__ gx, int D, int H,
                                int W, int C) {
    const size_t n = (size_t)D * H * W * C;
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int c = (int)(i % C);
    const size_t o = i / C;
    const int X = (int)(o % W), Y = (int)((o / W) % H), Z = (int)(o / ((size_t)W * H));
    float s = 0.f;
    for (int d = 0; d < 8; ++d) {
        const int z = 2 * Z + (d >> 2), y = 2 * Y + ((d >> 1) & 1), x = 2 * X + (d & 1);
        s += gy[(((size_t)z * 2 * H + y) * 2 * W + x) * C + c];
    }
    gx[i] = s;
}

// *mx = max |img| (non-negative floats compare as integers)
__global__ void k_absmax(const float2 *__restrict__ img, size_t n, float *mx) {
    float m = 0.f;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (size_t)gridDim.x * blockDim.x)
        m = fmaxf(m, hypotf(img[i].x, img[i].y));
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(reinterpret_cast<int *>(mx), __float_as_int(m));
}

// feat[v] = (Re g / s, Im g / s, |g| / s) as bf16 [v][3]
__global__ void k_features(const float2 *__restrict__ img, const float *__restrict__ scale,
                           __nv_bfloat16 *__restrict__ feat, size_t n) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float2 z = img[i];
    const float a = hypotf(z.x, z.y);
    const float s = *scale > 0.f ? *scale : 1.f;
    feat[3 * i + 0] = __float2bfloat16(z.x / s);
    feat[3 * i + 1] = __float2bfloat16(z.y / s);
    feat[3 * i + 2] = __float2bfloat16(a / s);
}

// sums[0] = sum |target/s|^2, sums[1] = sum |pred - target/s|^2; one block of
// 1024 threads with a fixed-order tree, so the result is reproducible
__global__ void __launch_bounds__(1024)
k_loss_sums(const float *__restrict__ pred, const float2 *__restrict__ tgt,
            const float *__restrict__ scale, size_t n, float *sums) {
    __shared__ float st_s[1024], sd_s[1024];
    const float inv = 1.0f / (*scale > 0.f ? *scale : 1.f);
    float st = 0.f, sd = 0.f;
    for (size_t i = threadIdx.x; i < n; i += blockDim.x) {
        const float tx = tgt[i].x * inv, ty = tgt[i].y * inv;
        const float dx = pred[2 * i] - tx, dy = pred[2 * i + 1] - ty;
        st += tx * tx + ty * ty;
        sd += dx * dx + dy * dy;
    }
    st_s[threadIdx.x] = st;
    sd_s[threadIdx.x] = sd;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) {
            st_s[threadIdx.x] += st_s[threadIdx.x + o];
            sd_s[threadIdx.x] += sd_s[threadIdx.x + o];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        sums[0] = st_s[0];
        sums[1] = sd_s[0];
    }
}

// Acceptance check of a learned correction: out[0] = number of non-finite
// entries of corr ([n][2]), out[1] = sum of corr^2 over the finite ones,
// out[2] = sum |gain img / s|^2 (the scaled cheap image the correction is
// added to). Two passes with fixed orders (reproducible sums): 256 blocks of
// 256 threads write partial sums (block b takes the entries b, b + 256, ...
// in tree order), one block adds the partials in block order.
constexpr int kCheckBlocks = 256;
// the partial sums: a file-scope device array (the check allocates nothing;
// two checks running at the same time on different streams would race on it)
__device__ float g_check_part[3 * kCheckBlocks];
__global__ void __launch_bounds__(256)
k_check_part(const float *__restrict__ corr, const float2 *__restrict__ img,
             const float *__restrict__ scale, float gain, size_t n, float *part) {
    __shared__ float s_bad[256], s_c[256], s_i[256];
    const float k = gain / (*scale > 0.f ? *scale : 1.f);
    float bad = 0.f, sc = 0.f, si = 0.f;
    for (size_t i = (size_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (size_t)kCheckBlocks * 256) {
        const float a = corr[2 * i], b = corr[2 * i + 1];
        if (isfinite(a)) sc += a * a; else bad += 1.f;
        if (isfinite(b)) sc += b * b; else bad += 1.f;
        const float x = k * img[i].x, y = k * img[i].y;
        si += x * x + y * y;
    }
    s_bad[threadIdx.x] = bad;
    s_c[threadIdx.x] = sc;
    s_i[threadIdx.x] = si;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o) {
            s_bad[threadIdx.x] += s_bad[threadIdx.x + o];
            s_c[threadIdx.x] += s_c[threadIdx.x + o];
            s_i[threadIdx.x] += s_i[threadIdx.x + o];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        part[3 * blockIdx.x + 0] = s_bad[0];
        part[3 * blockIdx.x + 1] = s_c[0];
        part[3 * blockIdx.x + 2] = s_i[0];
    }
}

__global__ void __launch_bounds__(256) k_check_sum(const float *__restrict__ part, float *out) {
    __shared__ float s[3][kCheckBlocks];
    for (int q = 0; q < 3; ++q) s[q][threadIdx.x] = part[3 * threadIdx.x + q];
    __syncthreads();
    for (int o = kCheckBlocks / 2; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o)
            for (int q = 0; q < 3; ++q) s[q][threadIdx.x] += s[q][threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x < 3) out[threadIdx.x] = s[threadIdx.x][0];
}

// grad = 2 (pred - target/s) / sum|target/s|^2
__global__ void k_loss_grad(const float *__restrict__ pred, const float2 *__restrict__ tgt,
                            const float *__restrict__ scale, const float *__restrict__ sums,
                            float *__restrict__ grad, size_t n) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float inv = 1.0f / (*scale > 0.f ? *scale : 1.f);
    const float k = 2.0f / fmaxf(sums[0], 1e-30f);
    grad[2 * i] = k * (pred[2 * i] - tgt[i].x * inv);
    grad[2 * i + 1] = k * (pred[2 * i + 1] - tgt[i].y * inv);
}

// pred[v] += gain (Re, Im) of img[v] / s
__global__ void k_residual(float *__restrict__ pred, const float2 *__restrict__ img,
                           const float *__restrict__ scale, float gain, size_t n) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float k = gain / (*scale > 0.f ? *scale : 1.f);
    pred[2 * i] += k * img[i].x;
    pred[2 * i + 1] += k * img[i].y;
}

// img = s (pred.x + j pred.y)
__global__ void k_to_complex(const float *__restrict__ pred, const float *__restrict__ scale,
                             float2 *__restrict__ img, size_t n) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float s = *scale > 0.f ? *scale : 1.f;
    img[i] = make_float2(s * pred[2 * i], s * pred[2 * i + 1]);
}

// Adam (Kingma & Ba 2015), bias-corrected; refreshes the BF16 copy.
__global__ void k_adam(float *__restrict__ p, const float *__restrict__ g, float *__restrict__ m,
                       float *__restrict__ v, __nv_bfloat16 *__restrict__ pb, size_t n, float lr,
                       float b1, float b2, float eps, float c1, float c2) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float pi = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    p[i] = pi;
    if (pb) pb[i] = __float2bfloat16(pi);
}

inline unsigned nblk(size_t n, int t = 256) { return (unsigned)((n + t - 1) / t); }

}  // namespace

// ---------------------------------------------------------------------------
// launch wrappers (declared in kernels.h)
// ---------------------------------------------------------------------------
cudaError_t nn_conv3d(const void *x, const void *w, const float *bias, void *out, int D, int H,
                      int W, int Cin, int Cout, int Kp, int relu, int out_bf16, cudaStream_t st) {
    // one to four channels: the gathering column kernel
    cudaError_t e = nn_conv3d_small(x, w, bias, out, D, H, W, Cin, Cout, Kp, relu, out_bf16, st);
    if (e != cudaErrorNotSupported) return e;
    // wide layers of many tiles of 128 voxels: the tcgen05 kernel. Measured
    // both ways (us, tcgen05 / mma.sync columns): 64 -> 32 on 1536 tiles 133 /
    // 171, 64 -> 128 on 192 tiles 42 / 64; but 64 -> 64 on 192 tiles 39 / 35,
    // 64 -> 128 on 24 tiles 39 / 18, and 32 -> 64 on 1536 tiles 82 / 78. With
    // 128 input channels the columns leave little room in shared memory: 128
    // -> 64 on 192 tiles 71 / (not taken), 128 -> 128 on 24 tiles 70 / 43.
    const bool wide = Cin >= 64 && (long long)D * H * W / 128 * Cout >= 16384;
    const bool tc = nn_conv3d_tc_supported(D, H, W, Cin, Cout, x, w, out);
    if (!(wide && tc)) {
        e = nn_conv3d_mma(x, w, bias, out, D, H, W, Cin, Cout, Kp, relu, out_bf16, st);
        if (e != cudaErrorNotSupported) return e;
    }
    if (tc) return nn_conv3d_tc(x, w, bias, out, D, H, W, Cin, Cout, Kp, relu, out_bf16, st);
    const int V = D * H * W;
    Vol vol{D, H, W};
    const auto *xb = (const __nv_bfloat16 *)x;
    const auto *wb = (const __nv_bfloat16 *)w;
    // 16-byte loads where they are aligned, else single elements
    const bool xv = Cin % 16 == 0 && (uintptr_t)x % 16 == 0, wv = (uintptr_t)w % 16 == 0;
    if (Cout <= 8) {
        dim3 grid((V + 63) / 64, (Cout + 7) / 8);
        if (out_bf16) k_conv3d<1, true><<<grid, 128, 0, st>>>(xb, wb, bias, out, vol, Cin, Cout, Kp, relu, xv, wv);
        else k_conv3d<1, false><<<grid, 128, 0, st>>>(xb, wb, bias, out, vol, Cin, Cout, Kp, relu, xv, wv);
    } else if (Cout <= 16) {
        dim3 grid((V + 63) / 64, (Cout + 15) / 16);
        if (out_bf16) k_conv3d<2, true><<<grid, 128, 0, st>>>(xb, wb, bias, out, vol, Cin, Cout, Kp, relu, xv, wv);
        else k_conv3d<2, false><<<grid, 128, 0, st>>>(xb, wb, bias, out, vol, Cin, Cout, Kp, relu, xv, wv);
    } else {
        dim3 grid((V + 63) / 64, (Cout + 31) / 32);
        if (out_bf16) k_conv3d<4, true><<<grid, 128, 0, st>>>(xb, wb, bias, out, vol, Cin, Cout, Kp, relu, xv, wv);
        else k_conv3d<4, false><<<grid, 128, 0, st>>>(xb, wb, bias, out, vol, Cin, Cout, Kp, relu, xv, wv);
    }
    return cudaGetLastError();
}

cudaError_t nn_weight_flip(const void *w, void *wt, int Cin, int Cout, int Kp, int Kpt,
                           cudaStream_t st) {
    k_weight_flip<<<nblk((size_t)Cin * Kpt), 256, 0, st>>>((const __nv_bfloat16 *)w,
                                                           (__nv_bfloat16 *)wt, Cin, Cout, Kp, Kpt);
    return cudaGetLastError();
}

cudaError_t nn_elementwise(int op, const void *a, const void *b, void *out, size_t n,
                           cudaStream_t st) {
    const bool vec = ((uintptr_t)a | (uintptr_t)(op == 1 || op == 3 ? nullptr : b) | (uintptr_t)out) % 16 == 0;
    const size_t n8 = vec ? n / 8 : 0;
    const unsigned blocks = nblk(n8 + (n - 8 * n8));
    const auto *bb = (const __nv_bfloat16 *)b;
    auto *ob = (__nv_bfloat16 *)out;
    switch (op) {
        case 0: k_to_bf16<0><<<blocks, 256, 0, st>>>(a, bb, ob, n8, n); break;
        case 1: k_to_bf16<1><<<blocks, 256, 0, st>>>(a, bb, ob, n8, n); break;
        case 2: k_to_bf16<2><<<blocks, 256, 0, st>>>(a, bb, ob, n8, n); break;
        case 3: k_accum_f32<<<nblk(n), 256, 0, st>>>((const float *)a, (float *)out, n); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t nn_resample(int op, const void *x, void *y, int D, int H, int W, int C, cudaStream_t st) {
    // D, H, W: the fine (large) size for pooling ops, the coarse size for upsampling ops
    switch (op) {
        case 0:
            if (C % 8 == 0 && (uintptr_t)x % 16 == 0 && (uintptr_t)y % 16 == 0)
                k_avgpool2_v8<<<nblk((size_t)D * H * W * C / 64), 256, 0, st>>>(
                    (const __nv_bfloat16 *)x, (__nv_bfloat16 *)y, D, H, W, C / 8);
            else
                k_avgpool2<<<nblk((size_t)D * H * W * C / 8), 256, 0, st>>>(
                    (const __nv_bfloat16 *)x, (__nv_bfloat16 *)y, D, H, W, C);
            break;
        case 1: k_avgpool2_bwd<<<nblk((size_t)D * H * W * C), 256, 0, st>>>(
                    (const float *)x, (float *)y, D, H, W, C); break;
        case 2:
            if (C % 8 == 0 && (uintptr_t)x % 16 == 0 && (uintptr_t)y % 16 == 0)
                k_upsample2_v8<<<nblk((size_t)D * H * W * C), 256, 0, st>>>(
                    (const uint4 *)x, (uint4 *)y, D, H, W, C / 8);
            else
                k_upsample2<<<nblk((size_t)8 * D * H * W * C), 256, 0, st>>>(
                    (const __nv_bfloat16 *)x, (__nv_bfloat16 *)y, D, H, W, C);
            break;
        case 3: k_upsample2_bwd<<<nblk((size_t)D * H * W * C), 256, 0, st>>>(
                    (const float *)x, (float *)y, D, H, W, C); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t nn_features(const void *img, void *feat, float *scale, size_t n, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(scale, 0, sizeof(float), st);
    if (e != cudaSuccess) return e;
    k_absmax<<<1024, 256, 0, st>>>((const float2 *)img, n, scale);
    k_features<<<nblk(n), 256, 0, st>>>((const float2 *)img, scale, (__nv_bfloat16 *)feat, n);
    return cudaGetLastError();
}

cudaError_t nn_loss(const float *pred, const void *target, const float *scale, float *sums,
                    float *grad, size_t n, cudaStream_t st) {
    k_loss_sums<<<1, 1024, 0, st>>>(pred, (const float2 *)target, scale, n, sums);
    if (grad) k_loss_grad<<<nblk(n), 256, 0, st>>>(pred, (const float2 *)target, scale, sums, grad, n);
    return cudaGetLastError();
}

cudaError_t nn_check(const float *corr, const void *img, const float *scale, float gain, size_t n,
                     float *out, cudaStream_t st) {
    float *part = nullptr;
    cudaError_t e = cudaGetSymbolAddress((void **)&part, g_check_part);
    if (e != cudaSuccess) return e;
    k_check_part<<<kCheckBlocks, 256, 0, st>>>(corr, (const float2 *)img, scale, gain, n, part);
    k_check_sum<<<1, kCheckBlocks, 0, st>>>(part, out);
    return cudaGetLastError();
}

cudaError_t nn_residual(float *pred, const void *img, const float *scale, float gain, size_t n,
                        cudaStream_t st) {
    k_residual<<<nblk(n), 256, 0, st>>>(pred, (const float2 *)img, scale, gain, n);
    return cudaGetLastError();
}

cudaError_t nn_to_complex(const float *pred, const float *scale, void *img, size_t n,
                          cudaStream_t st) {
    k_to_complex<<<nblk(n), 256, 0, st>>>(pred, scale, (float2 *)img, n);
    return cudaGetLastError();
}

cudaError_t nn_adam(float *p, const float *g, float *m, float *v, void *pb, size_t n, float lr,
                    float b1, float b2, float eps, int step, cudaStream_t st) {
    const float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
    k_adam<<<nblk(n), 256, 0, st>>>(p, g, m, v, (__nv_bfloat16 *)pb, n, lr, b1, b2, eps, c1, c2);
    return cudaGetLastError();
}
