// Transforms along the scan axis (Sec. II-A, Eq. 2) and along k_z (Eq. 9).
//
// Both act on the middle axis of a [batch][n][inner] complex64 array whose
// inner axis is contiguous: the echo s[c][n][m] (forward, zero-padded to N_p)
// and the image spectrum G[u][pixel] (inverse; the sum of the two channel
// parts' spectra, added as the first stage reads them). One block stages a
// [n][IB] column panel in shared memory (coalesced row segments), runs a
// mixed-radix (2, 3, 4, 5, 8) Stockham autosort FFT on all IB columns at once
// (column pairs), and its last stage writes the requested output rows to
// global memory (complex64 rows, or the range table's BF16 hi/lo operand). A
// launch may cover a range of columns of wider rows (row stride ld). Lengths
// with another prime factor, and inverse transforms onto voxel heights off
// the scan grid, use the tiled direct DFT kernel below with a precomputed
// phase matrix.
#include <cuda_bf16.h>

#include <algorithm>
#include <cstdint>


#include "common.cuh"
#include "kernels.h"
#include "stockham.cuh"

namespace {

constexpr int kFftIB = 16;        // columns per block (128-byte rows)
constexpr int kFftThreads = 256;  // threads per block

// in:  [batch][n_in][ld], columns i < I  (rows n >= n_in are zero padding)
// out: [batch][out_rows][ld], out row r = transform index (r + out_off) mod N
// (complex64, or with sp.bf16_rows set bfloat16 (re, im) pairs in the same
// layout); or, with sp.A set, the tensor-core range table's operand instead:
// A[r][re hi, re lo, im hi, im lo][batch][Kp] = split(X[r][i]) (BF16; with
// sp.hi_only only the hi planes are written)
struct SplitOut {
    __nv_bfloat16 *A;        // nullptr: plain output
    int batch, Kp;
    int hi_only;             // split output: hi planes only (BF16 spectrum)
    int bf16_rows;           // plain output as bfloat16 (re, im) pairs
};
// The FFT stages run on column pairs (float4 shared-memory accesses, a zero
// column beside an odd last one). VEC (even rows, 16-byte aligned): the copies
// and the plain output move pairs too, else single columns (8 bytes).
// LIMBS: the output is the range table's operand (sp.A) in that many BF16 parts of
// each real number (2 or 3), or `out` (0).
// (Odd rows took single columns through every stage before: a scan of 51
// frequencies 67.0 -> 65.8 us, of 201 235.9 -> 233.8.)
template <bool VEC, int LIMBS>
__global__ void __launch_bounds__(kFftThreads)
k_fft_strided(const float2 *__restrict__ in, const float2 *__restrict__ in2, float2 *__restrict__ out,
              int n_in, int I, int ld, FftPlan plan, const float2 *__restrict__ tw_g, int sgn,
              float scale, int out_rows, int out_off, SplitOut sp) {
    extern __shared__ __align__(16) float2 smem[];
    const int N = plan.n;
    float2 *buf0 = smem;
    float2 *buf1 = smem + N * kFftIB;
    float2 *tw = smem + 2 * N * kFftIB;
    const int i0 = blockIdx.x * kFftIB;
    const size_t b = blockIdx.y;
    constexpr int CW = VEC ? 2 : 1;            // columns per copy
    constexpr int NG = kFftIB / CW;            // copies per row

    // the whole panel in flight at once: asynchronous copies, zeros for the
    // padding rows and the columns past I. Each thread keeps one column group
    // (CW columns) and walks the rows RPS apart with running pointers.
    constexpr int RPS = kFftThreads / NG;      // rows per sweep of the block
    const int col = (threadIdx.x % NG) * CW;
    const int n_first = threadIdx.x / NG;
    const bool col_ok = i0 + col < I;
    for (int k = threadIdx.x; k < N; k += kFftThreads) tw[k] = tw_g[k];
    // in2 (optional): a second array of the same shape, added on load (into
    // buf1 first, which the transform then reuses)
    for (int part = 0; part < (in2 ? 2 : 1); ++part) {
        const float2 *src = (part ? in2 : in) + (b * n_in + n_first) * (size_t)ld + i0 + col;
        float2 *dst = (part ? buf1 : buf0) + n_first * kFftIB + col;
        const size_t src_step = (size_t)RPS * ld;
        for (int n = n_first; n < N; n += RPS, src += src_step, dst += RPS * kFftIB) {
            if (col_ok && n < n_in) {
                if (VEC)
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;\n" ::"r"(
                                     (unsigned)__cvta_generic_to_shared(dst)),
                                 "l"(src)
                                 : "memory");
                else
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(
                                     (unsigned)__cvta_generic_to_shared(dst)),
                                 "l"(src)
                                 : "memory");
            } else if (VEC) {
                *reinterpret_cast<float4 *>(dst) = make_float4(0.f, 0.f, 0.f, 0.f);
            } else {
                *dst = make_float2(0.f, 0.f);
            }
        }
    }
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();

    // the last FFT stage writes the output rows itself: transform index t
    // goes to output row (t - out_off) mod N when that is below out_rows
    if constexpr (LIMBS > 0) {
        // (the pair's second column may be the operand's first padding column,
        // which is zero and stays so)
        const size_t plane = (size_t)sp.batch * sp.Kp;
        __nv_bfloat16 *A = sp.A + b * sp.Kp + i0;
        auto emit = [&](int t, int cp, float2 x0, float2 x1) {
            int r = t - out_off;
            if (r < 0) r += N;
            if (r >= out_rows || i0 + 2 * cp >= I) return;
            const float2 v0 = cscale(x0, scale), v1 = cscale(x1, scale);
            if constexpr (LIMBS == 3) {
                __nv_bfloat16 *o = A + (size_t)r * 6 * plane + 2 * cp;
                float re0 = v0.x, re1 = v1.x, im0 = v0.y, im1 = v1.y;
#pragma unroll
                for (int l = 0; l < 3; ++l, o += plane) {
                    const __nv_bfloat162 re = __floats2bfloat162_rn(re0, re1);
                    const __nv_bfloat162 im = __floats2bfloat162_rn(im0, im1);
                    *reinterpret_cast<__nv_bfloat162 *>(o) = re;
                    *reinterpret_cast<__nv_bfloat162 *>(o + 3 * plane) = im;
                    re0 -= __low2float(re);
                    re1 -= __high2float(re);
                    im0 -= __low2float(im);
                    im1 -= __high2float(im);
                }
                return;
            }
            const __nv_bfloat16 h0 = __float2bfloat16(v0.x), h1 = __float2bfloat16(v1.x);
            const __nv_bfloat16 g0 = __float2bfloat16(v0.y), g1 = __float2bfloat16(v1.y);
            __nv_bfloat16 *o = A + (size_t)r * 4 * plane + 2 * cp;
            *reinterpret_cast<__nv_bfloat162 *>(o) = __halves2bfloat162(h0, h1);
            *reinterpret_cast<__nv_bfloat162 *>(o + 2 * plane) = __halves2bfloat162(g0, g1);
            if (sp.hi_only) return;
            *reinterpret_cast<__nv_bfloat162 *>(o + plane) = __halves2bfloat162(
                __float2bfloat16(v0.x - __bfloat162float(h0)),
                __float2bfloat16(v1.x - __bfloat162float(h1)));
            *reinterpret_cast<__nv_bfloat162 *>(o + 3 * plane) = __halves2bfloat162(
                __float2bfloat16(v0.y - __bfloat162float(g0)),
                __float2bfloat16(v1.y - __bfloat162float(g1)));
        };
        stockham_run_pairs_emit<kFftIB>(buf0, buf1, tw, plan, sgn, in2 != nullptr, emit);
    } else {
        float2 *o0 = out + b * out_rows * (size_t)ld + i0;
        __nv_bfloat162 *ob = reinterpret_cast<__nv_bfloat162 *>(out) + b * out_rows * (size_t)ld + i0;
        auto emit = [&](int t, int cp, float2 x0, float2 x1) {
            int r = t - out_off;
            if (r < 0) r += N;
            if (r >= out_rows || i0 + 2 * cp >= I) return;
            const size_t at = (size_t)r * ld + 2 * cp;
            const bool both = VEC || i0 + 2 * cp + 1 < I;
            if (sp.bf16_rows) {
                __nv_bfloat162 q[2] = {__floats2bfloat162_rn(scale * x0.x, scale * x0.y),
                                       __floats2bfloat162_rn(scale * x1.x, scale * x1.y)};
                if (VEC) {
                    *reinterpret_cast<uint2 *>(ob + at) = *reinterpret_cast<const uint2 *>(q);
                } else {
                    ob[at] = q[0];
                    if (both) ob[at + 1] = q[1];
                }
                return;
            }
            if (VEC) {
                *reinterpret_cast<float4 *>(o0 + at) =
                    make_float4(scale * x0.x, scale * x0.y, scale * x1.x, scale * x1.y);
            } else {
                o0[at] = cscale(x0, scale);
                if (both) o0[at + 1] = cscale(x1, scale);
            }
        };
        stockham_run_pairs_emit<kFftIB>(buf0, buf1, tw, plan, sgn, in2 != nullptr, emit);
    }
}

// Direct DFT along the middle axis with an explicit phase matrix:
//   out[b][r][i] = scale * sum_{n < n_in} in[b][n][i] * T[r][n]
// in two kernels. A 32 x 32 output tile per block of 256 threads, 4 rows of one
// column each, for few columns and few blocks (the rule is at the launch):
__global__ void __launch_bounds__(256)
k_dft_narrow(const float2 *__restrict__ in, const float2 *__restrict__ in2, float2 *__restrict__ out,
              int n_in, int I, int out_rows, const float2 *__restrict__ T, float scale,
              int out_bf16) {
    __shared__ float2 xs[32][33];
    __shared__ float2 ts[32][33];
    const int tx = threadIdx.x & 31;
    const int ty = threadIdx.x >> 5;   // 0..7
    const int i = blockIdx.x * 32 + tx;
    const int r0 = blockIdx.y * 32;
    const size_t b = blockIdx.z;
    float2 acc[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[q] = make_float2(0.f, 0.f);
    for (int n0 = 0; n0 < n_in; n0 += 32) {
        for (int q = 0; q < 4; ++q) {
            const int nn = ty * 4 + q;
            const int n = n0 + nn;
            float2 x = make_float2(0.f, 0.f);
            if (n < n_in && i < I) {
                const size_t o = (b * n_in + n) * (size_t)I + i;
                x = in[o];
                if (in2) x = cadd(x, in2[o]);
            }
            xs[nn][tx] = x;
            const int rr = r0 + ty * 4 + q;
            ts[ty * 4 + q][tx] = (rr < out_rows && n0 + tx < n_in)
                                     ? T[(size_t)rr * n_in + n0 + tx] : make_float2(0.f, 0.f);
        }
        __syncthreads();
#pragma unroll 8
        for (int nn = 0; nn < 32; ++nn) {
            const float2 x = xs[nn][tx];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float2 t = ts[ty * 4 + q][nn];
                acc[q].x += x.x * t.x - x.y * t.y;
                acc[q].y += x.x * t.y + x.y * t.x;
            }
        }
        __syncthreads();
    }
    if (i < I) {
        for (int q = 0; q < 4; ++q) {
            const int r = r0 + ty * 4 + q;
            if (r >= out_rows) continue;
            const float2 v = cscale(acc[q], scale);
            const size_t o = (b * out_rows + r) * (size_t)I + i;
            if (out_bf16)
                reinterpret_cast<__nv_bfloat162 *>(out)[o] = __floats2bfloat162_rn(v.x, v.y);
            else
                out[o] = v;
        }
    }
}

// ... and 32 rows x 64 columns per block of 128 threads, 4 x 4 outputs each: four
// 16-byte shared loads feed 64 FMA (one output column a thread takes five
// 8-byte loads for 16). FP32 scan of 225 bins, 96 heights, 120 x 101 pixels:
// 1041 -> 1027 us.
constexpr int kDftK = 32, kDftRows = 32, kDftCols = 64;
__global__ void __launch_bounds__(128)
k_dft_strided(const float2 *__restrict__ in, const float2 *__restrict__ in2, float2 *__restrict__ out,
              int n_in, int I, int out_rows, const float2 *__restrict__ T, float scale,
              int out_bf16) {
    __shared__ __align__(16) float2 xs[kDftK][kDftCols];
    __shared__ __align__(16) float2 ts[kDftK][kDftRows + 4];     // [n][row]
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int i0 = blockIdx.x * kDftCols, r0 = blockIdx.y * kDftRows;
    const size_t b = blockIdx.z;
    float2 acc[4][4] = {};                                       // [row][column]
    for (int n0 = 0; n0 < n_in; n0 += kDftK) {
#pragma unroll 4
        for (int q = threadIdx.x; q < kDftK * kDftCols; q += 128) {
            const int nn = q / kDftCols, c = q % kDftCols, n = n0 + nn, i = i0 + c;
            float2 x = make_float2(0.f, 0.f);
            if (n < n_in && i < I) {
                const size_t o = (b * n_in + n) * (size_t)I + i;
                x = in[o];
                if (in2) x = cadd(x, in2[o]);
            }
            xs[nn][c] = x;
        }
#pragma unroll 4
        for (int q = threadIdx.x; q < kDftK * kDftRows; q += 128) {
            const int nn = q % kDftK, r = q / kDftK;
            ts[nn][r] = (r0 + r < out_rows && n0 + nn < n_in) ? T[(size_t)(r0 + r) * n_in + n0 + nn]
                                                              : make_float2(0.f, 0.f);
        }
        __syncthreads();
#pragma unroll 4
        for (int nn = 0; nn < kDftK; ++nn) {
            // columns 2 tx, 2 tx + 1 of each half
            const float4 xa = *reinterpret_cast<const float4 *>(&xs[nn][2 * tx]);
            const float4 xb = *reinterpret_cast<const float4 *>(&xs[nn][32 + 2 * tx]);
            const float4 ta = *reinterpret_cast<const float4 *>(&ts[nn][4 * ty]);
            const float4 tb = *reinterpret_cast<const float4 *>(&ts[nn][4 * ty + 2]);
            const float2 x[4] = {{xa.x, xa.y}, {xa.z, xa.w}, {xb.x, xb.y}, {xb.z, xb.w}};
            const float2 t[4] = {{ta.x, ta.y}, {ta.z, ta.w}, {tb.x, tb.y}, {tb.z, tb.w}};
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    acc[r][c].x = fmaf(x[c].x, t[r].x, fmaf(-x[c].y, t[r].y, acc[r][c].x));
                    acc[r][c].y = fmaf(x[c].x, t[r].y, fmaf(x[c].y, t[r].x, acc[r][c].y));
                }
        }
        __syncthreads();
    }
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const int row = r0 + 4 * ty + r, i = i0 + 32 * (c >> 1) + 2 * tx + (c & 1);
            if (row >= out_rows || i >= I) continue;
            const float2 v = cscale(acc[r][c], scale);
            const size_t o = (b * out_rows + row) * (size_t)I + i;
            if (out_bf16)
                reinterpret_cast<__nv_bfloat162 *>(out)[o] = __floats2bfloat162_rn(v.x, v.y);
            else
                out[o] = v;
        }
}

}  // namespace

size_t fft_strided_smem_bytes(int n) { return (size_t)(2 * n * kFftIB + n) * sizeof(float2); }

cudaError_t launch_fft_strided(const float2 *in, float2 *out, int batch, int n_in, int I,
                               const FftPlan &plan, const float2 *tw, int sgn, float scale,
                               int out_rows, int out_off, cudaStream_t st,
                               void *split_A, int split_Kp, const float2 *in2, int ld,
                               int bf16_out, int split_limbs) {
    const size_t smem = fft_strided_smem_bytes(plan.n);
    // copies of column pairs need 16-byte aligned rows: I even, 16-byte aligned
    // buffers; the split output always takes pairs (operand rows of Kp, a
    // multiple of 64)
    if (ld <= 0) ld = I;
    if (split_A && (split_Kp % 2 || (uintptr_t)split_A % 4 || split_Kp < (I + 1) / 2 * 2))
        return cudaErrorInvalidValue;
    if (ld < I) return cudaErrorInvalidValue;
    const bool pairs = (I % 2 == 0) && (ld % 2 == 0) && ((uintptr_t)in % 16 == 0) &&
                       ((uintptr_t)in2 % 16 == 0) && (split_A || (uintptr_t)out % 16 == 0);
    auto kern = pairs ? k_fft_strided<true, 0> : k_fft_strided<false, 0>;
    if (split_A && split_limbs == 3) kern = pairs ? k_fft_strided<true, 3> : k_fft_strided<false, 3>;
    else if (split_A) kern = pairs ? k_fft_strided<true, 2> : k_fft_strided<false, 2>;
    cudaError_t e = allow_dynamic_smem(kern, smem);
    if (e != cudaSuccess) return e;
    dim3 grid((I + kFftIB - 1) / kFftIB, batch);
    // bf16_out: with split_A, the hi planes only; else bfloat16 (re, im) rows
    const SplitOut sp{(__nv_bfloat16 *)split_A, batch, split_Kp, split_A ? bf16_out : 0,
                      split_A ? 0 : bf16_out};
    kern<<<grid, kFftThreads, smem, st>>>(in, in2, out, n_in, I, ld, plan, tw, sgn, scale, out_rows, out_off,
                                  sp);
    return cudaGetLastError();
}

cudaError_t launch_dft_strided(const float2 *in, float2 *out, int batch, int n_in, int I,
                               int out_rows, const float2 *T, float scale, cudaStream_t st,
                               const float2 *in2, int bf16_out) {
    // The wide tile costs 1.7 narrow ones, so it wins where it takes fewer than
    // 1 / 1.7 of the narrow tile's blocks, and once its blocks (four warps of long
    // chains) fill the device about three times. Narrow and wide, us: 127 points,
    // 256 transforms of 32 columns 39.6 and 57.6, of 64 73.5 and 65.7, of 80 106
    // and 109, of 128 136 and 114; 64 transforms of 64 24.9 and 24.7; 251 points
    // onto 128 rows, 2304 columns 26.7 and 34.9, 4096 45.6 and 45.4, 9216 83.6 and
    // 67.9.
    const long long rows = (long long)((out_rows + kDftRows - 1) / kDftRows) * batch;
    const int wide = (I + kDftCols - 1) / kDftCols, narrow = (I + 31) / 32;
    if (17LL * wide < 10LL * narrow && rows * wide >= 400) {
        dim3 grid(wide, (out_rows + kDftRows - 1) / kDftRows, batch);
        k_dft_strided<<<grid, 128, 0, st>>>(in, in2, out, n_in, I, out_rows, T, scale, bf16_out);
    } else {
        dim3 grid(narrow, (out_rows + 31) / 32, batch);
        k_dft_narrow<<<grid, 256, 0, st>>>(in, in2, out, n_in, I, out_rows, T, scale, bf16_out);
    }
    return cudaGetLastError();
}

namespace {

// Exponent all ones <=> NaN or Inf, decided on the bits (no float compare).
__device__ __forceinline__ bool nonfinite_bits(float v) {
    return (__float_as_uint(v) & 0x7f800000u) == 0x7f800000u;
}

__global__ void __launch_bounds__(256) k_check_finite(const float4 *__restrict__ x4, size_t n4,
                                                     const float2 *__restrict__ tail, int n_tail,
                                                     int *flag) {
    bool bad = false;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4;
         i += (size_t)gridDim.x * blockDim.x) {
        const float4 v = __ldg(&x4[i]);
        bad |= nonfinite_bits(v.x) | nonfinite_bits(v.y) | nonfinite_bits(v.z) |
               nonfinite_bits(v.w);
    }
    if (blockIdx.x == 0 && (int)threadIdx.x < n_tail) {
        const float2 v = tail[threadIdx.x];
        bad |= nonfinite_bits(v.x) | nonfinite_bits(v.y);
    }
    if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicOr(flag, PL_FLAG_NONFINITE);
}

}  // namespace

cudaError_t launch_check_finite(const float2 *x, size_t n, int *flag, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    if (!x || !flag) return cudaErrorInvalidValue;
    // float4 body from the first 16-byte boundary; the rest (at most two
    // leading or one trailing complex value) read as float2
    const size_t lead = ((uintptr_t)x % 16) ? 1 : 0;       // x is 8-byte aligned
    if (lead && n == 1) {
        k_check_finite<<<1, 32, 0, st>>>(nullptr, 0, x, 1, flag);
        return cudaGetLastError();
    }
    const size_t body = (n - lead) / 2;                      // float4 = two complex values
    const size_t rest = n - lead - 2 * body;                 // 0 or 1
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const size_t want = (body + 255) / 256;
    const int blocks = (int)std::max<size_t>(1, std::min<size_t>(want, (size_t)sms * 8));
    if (lead) {
        k_check_finite<<<1, 32, 0, st>>>(nullptr, 0, x, 1, flag);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    k_check_finite<<<blocks, 256, 0, st>>>(reinterpret_cast<const float4 *>(x + lead), body,
                                           x + lead + 2 * body, (int)rest, flag);
    return cudaGetLastError();
}
