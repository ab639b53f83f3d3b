// The two comparison algorithms of Sec. III (Table II), on the GPU:
//
//  * exact-sum hybrid ("omega-K-BP", the method without the NUFFT): after the
//    z-FFT, per k_z bin u and pixel
//      G_u(x,y) = sum_c sum_m S[c][u][m] k_m e^{+j kappa_um a_c(x,y)}
//    (Eq. 7 mono, Eq. 19 multistatic, evanescent terms dropped), then the
//    inverse transform over k_z (Eq. 9);
//  * direct back-projection (BP), the time-domain matched filter of the echo
//    model (Eq. 1 / 10) with the k weight:
//      g(x,y,z) = sum_c sum_n sum_m s[c][n][m] k_m e^{+j k_m (R_T + R_R)}.
//
// Both in FP32 with float-float ranges and phases (kappa a and k R reach
// ~2e3 rad; a float-float product reduced modulo 2 pi leaves ~1e-7 rad).
#include "bp_body.cuh"
#include "common.cuh"
#include "kernels.h"

namespace {

struct ff {
    float hi, lo;
};
__device__ __forceinline__ ff ff_of(double v) {
    const float h = (float)v;
    return {h, (float)(v - (double)h)};
}
__device__ __forceinline__ ff quick_two_sum(float a, float b) {
    const float s = a + b;
    return {s, b - (s - a)};
}
__device__ __forceinline__ ff two_sum(float a, float b) {
    const float s = a + b;
    const float bb = s - a;
    return {s, (a - (s - bb)) + (b - bb)};
}
__device__ __forceinline__ ff ff_add(ff x, ff y) {
    ff s = two_sum(x.hi, y.hi);
    return quick_two_sum(s.hi, s.lo + x.lo + y.lo);
}
__device__ __forceinline__ ff ff_neg(ff x) { return {-x.hi, -x.lo}; }
__device__ __forceinline__ ff ff_sqr(ff x) {
    const float p = x.hi * x.hi;
    const float e = fmaf(x.hi, x.hi, -p) + 2.0f * x.hi * x.lo;
    return quick_two_sum(p, e);
}
// sqrt of a positive float pair: one correction step of the float root
__device__ __forceinline__ ff ff_sqrt(ff x) {
    if (!(x.hi > 0.f)) return {0.f, 0.f};
    const float r = sqrtf(x.hi);
    const float p = r * r;
    const float e = fmaf(r, r, -p);
    const float d = ((x.hi - p) - e + x.lo) / (2.0f * r);
    return quick_two_sum(r, d);
}
// |(x, y) - (px, py)| as a float pair
__device__ __forceinline__ ff ff_dist2d(ff x, ff y, ff px, ff py) {
    const ff dx = ff_add(x, ff_neg(px)), dy = ff_add(y, ff_neg(py));
    return ff_sqrt(ff_add(ff_sqr(dx), ff_sqr(dy)));
}

// G[u][pixel] of the exact sum: UT bins x a tile of 16 x 8 pixels per block,
// one pixel per thread.
//
// Bound by the two MUFU operations of a term (16 lanes per cycle and SM). The
// phase kappa a is split at the tile's reference pixel, a = a_ref + delta:
// e^{j kappa a_ref} is common to the block and goes into the term's
// coefficient (k_m S e^{j kappa a_ref}, formed once per block and staged in
// shared memory, the phase as a float pair), so a (pixel, term) costs one
// product kappa delta, a sine and a cosine and four FMA in place of a
// float-float product with its reduction. The launcher keeps kappa delta
// below kMaxSplitPhase, where a rounded FP32 phase is off by at most 1e-5 rad
// and by 1e-6 rad on usual grids, independently from term to term.
// 120 channels, 51 frequencies, 128 bins, 64 x 64 pixels: 4.85 -> 1.65 ms
// (MUFU floor 1.4 ms). Two bins a block: 1.72 ms with four (512 blocks on 152
// SMs leave a part-filled last wave), 2.00 ms with eight.
constexpr int kExTX = 16, kExTY = 8, kExThreads = kExTX * kExTY;
constexpr int kExChunk = 256;                 // frequencies staged at a time
constexpr float kMaxSplitPhase = 128.f;

template <int UT, int MODE>
__global__ void __launch_bounds__(kExThreads)
k_exact_sum(ExactDesc e, const float2 *__restrict__ S, const float2 *__restrict__ kap,
            const float *__restrict__ wum, const float4 *__restrict__ chff, float2 *__restrict__ G) {
    // two buffers: one barrier between the staging and the reading of a chunk
    extern __shared__ float4 sm_terms[];
    __shared__ float2 s_ref[2];
    const int tiles_x = (e.nx + kExTX - 1) / kExTX;
    const int ix = (blockIdx.x % tiles_x) * kExTX + (int)threadIdx.x % kExTX;
    const int iy = (blockIdx.x / tiles_x) * kExTY + (int)threadIdx.x / kExTX;
    const bool live = ix < e.nx && iy < e.ny;
    const int u0 = blockIdx.y * UT;
    // pixels past the edge repeat the last one
    const ff px = ff_of(e.x0 + min(ix, e.nx - 1) * e.dx), py = ff_of(e.y0 + min(iy, e.ny - 1) * e.dy);
    const int ref = kExThreads / 2 + kExTX / 2;
    const int mc_full = min(e.n_f, kExChunk);
    float2 acc[UT];
#pragma unroll
    for (int j = 0; j < UT; ++j) acc[j] = make_float2(0.f, 0.f);
    int buf = 0;
    for (int c = 0; c < e.n_chan; ++c) {
        const float4 t = chff[2 * c], r = chff[2 * c + 1];
        // a = rho (mono: kappa = sqrt(4k^2 - k_z^2) carries the factor 2) or
        // rho_T + rho_R (multi: kappa = sqrt(k^2 - k_z^2 / 4))
        ff a = ff_dist2d(px, py, {t.x, t.y}, {t.z, t.w});
        if (MODE == 1) a = ff_add(a, ff_dist2d(px, py, {r.x, r.y}, {r.z, r.w}));
        // (two slots: the slot of channel c is read before channel c + 1's
        // first barrier, and written again after it)
        if (threadIdx.x == ref) s_ref[c & 1] = make_float2(a.hi, a.lo);
        __syncthreads();
        const float2 ar = s_ref[c & 1];
        const float delta = (a.hi - ar.x) + (a.lo - ar.y);
        for (int m0 = 0; m0 < e.n_f; m0 += kExChunk) {
            const int mc = min(kExChunk, e.n_f - m0);
            float4 *terms = sm_terms + (size_t)buf * UT * mc_full;
            for (int i = threadIdx.x; i < UT * mc; i += kExThreads) {
                const int j = i / mc, m = m0 + i - j * mc, u = u0 + j;
                float4 v = make_float4(0.f, 0.f, 0.f, 0.f);     // evanescent, or past the bins
                if (u < e.n_pad) {
                    const float w = wum[(size_t)u * e.n_f + m];
                    if (w != 0.f) {
                        const float2 k = kap[(size_t)u * e.n_f + m];
                        const float2 s = S[((size_t)c * e.n_pad + u) * e.n_f + m];
                        float sn, cs;
                        sincosf(bp::phase_ff(k.x, k.y, ar.x, ar.y), &sn, &cs);
                        const float sr = s.x * w, si = s.y * w;
                        v = make_float4(fmaf(sr, cs, -si * sn), fmaf(sr, sn, si * cs), k.x, 0.f);
                    }
                }
                terms[i] = v;
            }
            __syncthreads();
#pragma unroll
            for (int j = 0; j < UT; ++j) {
                const float4 *tj = terms + j * mc;
                float2 s = acc[j];
#pragma unroll 4
                for (int m = 0; m < mc; ++m) {
                    const float4 v = tj[m];
                    float sn, cs;
                    __sincosf(v.z * delta, &sn, &cs);
                    s.x = fmaf(v.x, cs, fmaf(-v.y, sn, s.x));
                    s.y = fmaf(v.x, sn, fmaf(v.y, cs, s.y));
                }
                acc[j] = s;
            }
            buf ^= 1;
        }
    }
    if (live) {
        const size_t np = (size_t)e.nx * e.ny, p = (size_t)iy * e.nx + ix;
#pragma unroll
        for (int j = 0; j < UT; ++j)
            if (u0 + j < e.n_pad) G[(size_t)(u0 + j) * np + p] = acc[j];
    }
}

// The same with the whole phase as a float pair in every term, for pixels so
// far apart that kappa delta would pass kMaxSplitPhase.
template <int UT>
__global__ void __launch_bounds__(128)
k_exact_sum_coarse(ExactDesc e, const float2 *__restrict__ S, const float2 *__restrict__ kap,
                   const float *__restrict__ wum, const float4 *__restrict__ chff,
                   float2 *__restrict__ G) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    const int u0 = blockIdx.y * UT;
    const int np = e.nx * e.ny;
    const bool live = p < np;
    const int ix = live ? p % e.nx : 0, iy = live ? p / e.nx : 0;
    const ff px = ff_of(e.x0 + ix * e.dx), py = ff_of(e.y0 + iy * e.dy);
    float2 acc[UT];
#pragma unroll
    for (int j = 0; j < UT; ++j) acc[j] = make_float2(0.f, 0.f);
    for (int c = 0; c < e.n_chan; ++c) {
        const float4 t = chff[2 * c], r = chff[2 * c + 1];
        ff a = ff_dist2d(px, py, {t.x, t.y}, {t.z, t.w});
        if (e.mode == 1) a = ff_add(a, ff_dist2d(px, py, {r.x, r.y}, {r.z, r.w}));
#pragma unroll
        for (int j = 0; j < UT; ++j) {
            const int u = u0 + j;
            if (u >= e.n_pad) break;
            const float2 *Su = S + ((size_t)c * e.n_pad + u) * e.n_f;
            const float2 *ku = kap + (size_t)u * e.n_f;
            const float *wu = wum + (size_t)u * e.n_f;
            for (int m = 0; m < e.n_f; ++m) {
                const float w = wu[m];
                if (w == 0.f) continue;              // evanescent (uniform across the block)
                const float2 k = ku[m];
                const float2 s = Su[m];
                float sn, cs;
                __sincosf(bp::phase_ff(k.x, k.y, a.hi, a.lo), &sn, &cs);
                const float sr = s.x * w, si = s.y * w;
                acc[j].x = fmaf(sr, cs, fmaf(-si, sn, acc[j].x));
                acc[j].y = fmaf(sr, sn, fmaf(si, cs, acc[j].y));
            }
        }
    }
    if (live) {
#pragma unroll
        for (int j = 0; j < UT; ++j)
            if (u0 + j < e.n_pad) G[(size_t)(u0 + j) * np + p] = acc[j];
    }
}

// Direct back-projection of an evenly spaced band: with z = e^{j dk a} the sum
// over the frequencies is e^{j k_0 a} times a polynomial in z, evaluated by
// Horner's rule (four FMA a term, the count of the complex sum itself; forming
// e^{j k_m a} by rotation and weighting every term by k_m took ten).
//
// Bound by the FP32 pipe. A warp owns 128 pixels of one z plane, four a lane,
// worked on in packed pairs (fma.rn.f32x2), so that one shared-memory load of
// a coefficient (k_m s, both halves of a pair filled) serves eight packed FMA.
// The eight warps of a block own the same pixels and every eighth channel, so
// small images also fill the device; their sums are added in warp order at the
// end. Each warp stages its own coefficients (no block barrier): kDirTerms
// terms, several scan positions at a time when the band is short. A band of
// more than kDirPoly frequencies is a sum of polynomials of that many terms,
// each from its own k: the error of z, which the m-th power multiplies by m,
// grows no further. 120 channels, 48 positions, 51 frequencies, 64^3 voxels:
// 43.6 -> 14.3 ms (7.9 ms at the FP32 peak; the rest is the two phases of each
// (voxel, channel, position), 16.2 ms with unpacked FMA).
constexpr int kDirWarps = 8, kDirPx = 128, kDirTerms = 256, kDirPoly = 128;

using bp::f2;

// sqrt(x + y) of float pairs from the reciprocal root: r = s rsqrt(s) is
// within a few ulp, the correction leaves the pair's own rounding. (The sum
// and the root stay unnormalised pairs, |lo| a few ulp of hi, which the phase
// products take as they are.)
__device__ __forceinline__ ff ff_sqrt_sum(ff x, ff y) {
    const ff s = two_sum(x.hi, y.hi);
    const float lo = s.lo + (x.lo + y.lo);
    const float q = rsqrtf(fmaxf(s.hi, 1e-30f));
    const float r = s.hi * q;
    return {r, (fmaf(-r, r, s.hi) + lo) * (0.5f * q)};
}

template <int MODE>
__global__ void __launch_bounds__(32 * kDirWarps, 3)
k_bp_direct_uniform(DirectDesc e, const float2 *__restrict__ s, const float4 *__restrict__ chff,
                    const float2 *__restrict__ zs, const float2 *__restrict__ kff,
                    float2 *__restrict__ img) {
    __shared__ float4 sm_coef[kDirWarps * kDirTerms];   // [warp][term] {re, re, im, im}
    __shared__ float2 sm_dz2[kDirWarps][32];            // (z - z'_n)^2 of the staged positions
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float4 *coef = sm_coef + warp * kDirTerms;
    const int np = e.nx * e.ny, px_blocks = (np + kDirPx - 1) / kDirPx;
    const int iz = (int)(blockIdx.x / px_blocks);
    const int pb = (int)(blockIdx.x - (unsigned)iz * px_blocks) * kDirPx;
    const ff pz = ff_of(e.z0 + iz * e.dz);
    const int p0 = pb + lane;
    const int rows = e.n_f > kDirPoly ? 1 : min(32, kDirTerms / e.n_f);  // positions staged at a time
    // frequency of staged term `lane`, and its step over 32 terms (modulo n_f)
    const int lane_m = lane % e.n_f, step_m = 32 % e.n_f;
    float2 sum[2][2] = {{{0.f, 0.f}, {0.f, 0.f}}, {{0.f, 0.f}, {0.f, 0.f}}};   // [pair][re, im]
    for (int c = warp; c < e.n_chan; c += kDirWarps) {
        const float4 t = chff[2 * c], r = chff[2 * c + 1];
        ff rho_t[4], rho_r[MODE == 1 ? 4 : 1];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int p = min(p0 + 32 * k, np - 1);          // past the image: the last pixel
            const ff px = ff_of(e.x0 + (p % e.nx) * e.dx), py = ff_of(e.y0 + (p / e.nx) * e.dy);
            const ff dxt = ff_add(px, ff_neg({t.x, t.y})), dyt = ff_add(py, ff_neg({t.z, t.w}));
            rho_t[k] = ff_add(ff_sqr(dxt), ff_sqr(dyt));
            if (MODE == 1) {
                const ff dxr = ff_add(px, ff_neg({r.x, r.y})), dyr = ff_add(py, ff_neg({r.z, r.w}));
                rho_r[MODE == 1 ? k : 0] = ff_add(ff_sqr(dxr), ff_sqr(dyr));
            }
        }
        const float2 *sc = s + (size_t)c * e.n_scan * e.n_f;
        for (int n0 = 0; n0 < e.n_scan; n0 += rows) {
            const int nr = min(rows, e.n_scan - n0);
            for (int m0 = 0; m0 < e.n_f; m0 += kDirPoly) {
                const int mc = min(kDirPoly, e.n_f - m0);
                const float2 k0 = kff[m0];
                __syncwarp();                                // the last terms are read
                // (the staged positions' terms are contiguous in the echo)
                const float2 *src = sc + (size_t)n0 * e.n_f + m0;
                for (int i = lane, m = lane_m; i < nr * mc; i += 32) {
                    const float2 x = src[i];
                    const float k = kff[m0 + m].x;
                    coef[i] = make_float4(x.x * k, x.x * k, x.y * k, x.y * k);
                    m += step_m;
                    if (m >= e.n_f) m -= e.n_f;
                }
                if (lane < nr) {
                    const float2 zn = zs[n0 + lane];
                    const ff d = ff_sqr(ff_add(pz, ff_neg({zn.x, zn.y})));
                    sm_dz2[warp][lane] = make_float2(d.hi, d.lo);
                }
                __syncwarp();
                for (int n = 0; n < nr; ++n) {
                    const ff dz2 = {sm_dz2[warp][n].x, sm_dz2[warp][n].y};
                    float cs[4], sn[4], c0[4], s0[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        ff a = ff_sqrt_sum(rho_t[k], dz2);
                        a = MODE == 0 ? ff{a.hi + a.hi, a.lo + a.lo}
                                      : ff_add(a, ff_sqrt_sum(rho_r[MODE == 1 ? k : 0], dz2));
                        __sincosf(bp::phase_ff(e.dk_hi, e.dk_lo, a.hi, a.lo), &sn[k], &cs[k]);
                        __sincosf(bp::phase_ff(k0.x, k0.y, a.hi, a.lo), &s0[k], &c0[k]);
                    }
                    float2 ar[2] = {{0.f, 0.f}, {0.f, 0.f}}, ai[2] = {{0.f, 0.f}, {0.f, 0.f}};
                    const float4 *cn = coef + n * mc;
#pragma unroll 8
                    for (int m = mc - 1; m >= 0; --m) {
                        const float4 v = cn[m];
                        const float2 vr = f2(v.x, v.y), vi = f2(v.z, v.w);
#pragma unroll
                        for (int q = 0; q < 2; ++q) {
                            const float2 zr = f2(cs[2 * q], cs[2 * q + 1]);
                            const float2 zi = f2(sn[2 * q], sn[2 * q + 1]), nzi = f2(-zi.x, -zi.y);
                            const float2 re = __ffma2_rn(ar[q], zr, __ffma2_rn(ai[q], nzi, vr));
                            ai[q] = __ffma2_rn(ar[q], zi, __ffma2_rn(ai[q], zr, vi));
                            ar[q] = re;
                        }
                    }
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        const float2 er = f2(c0[2 * q], c0[2 * q + 1]);
                        const float2 ei = f2(s0[2 * q], s0[2 * q + 1]), ne = f2(-ei.x, -ei.y);
                        sum[q][0] = __ffma2_rn(ar[q], er, __ffma2_rn(ai[q], ne, sum[q][0]));
                        sum[q][1] = __ffma2_rn(ar[q], ei, __ffma2_rn(ai[q], er, sum[q][1]));
                    }
                }
            }
        }
    }
    // the warps' sums, in warp order (the coefficients' storage is free)
    __syncthreads();
    float2 *part = reinterpret_cast<float2 *>(sm_coef);      // [warp][128]
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        part[warp * kDirPx + 64 * q + lane] = f2(sum[q][0].x, sum[q][1].x);
        part[warp * kDirPx + 64 * q + 32 + lane] = f2(sum[q][0].y, sum[q][1].y);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kDirPx; i += 32 * kDirWarps) {
        const int p = pb + i;
        if (p >= np) break;
        float2 g = part[i];
        for (int w = 1; w < kDirWarps; ++w) {
            g.x += part[w * kDirPx + i].x;
            g.y += part[w * kDirPx + i].y;
        }
        img[(size_t)iz * np + p] = g;
    }
}

// Direct back-projection of an uneven band onto the voxel grid: one voxel per
// thread, a phase per term.
__global__ void __launch_bounds__(128)
k_bp_direct(DirectDesc e, const float2 *__restrict__ s, const float4 *__restrict__ chff,
            const float2 *__restrict__ zs, const float2 *__restrict__ kff, float2 *__restrict__ img) {
    const long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long nv = (long long)e.nx * e.ny * e.nz;
    const bool live = v < nv;
    const int ix = live ? (int)(v % e.nx) : 0;
    const int iy = live ? (int)((v / e.nx) % e.ny) : 0;
    const int iz = live ? (int)(v / ((long long)e.nx * e.ny)) : 0;
    const ff px = ff_of(e.x0 + ix * e.dx), py = ff_of(e.y0 + iy * e.dy);
    const ff pz = ff_of(e.z0 + iz * e.dz);
    float2 acc = make_float2(0.f, 0.f);
    for (int c = 0; c < e.n_chan; ++c) {
        const float4 t = chff[2 * c], r = chff[2 * c + 1];
        const ff dxt = ff_add(px, ff_neg({t.x, t.y})), dyt = ff_add(py, ff_neg({t.z, t.w}));
        const ff rho_t = ff_add(ff_sqr(dxt), ff_sqr(dyt));
        ff rho_r = rho_t;
        if (e.mode == 1) {
            const ff dxr = ff_add(px, ff_neg({r.x, r.y})), dyr = ff_add(py, ff_neg({r.z, r.w}));
            rho_r = ff_add(ff_sqr(dxr), ff_sqr(dyr));
        }
        const float2 *sc = s + (size_t)c * e.n_scan * e.n_f;
        for (int n = 0; n < e.n_scan; ++n) {
            const float2 zn = zs[n];
            const ff dz2 = ff_sqr(ff_add(pz, ff_neg({zn.x, zn.y})));
            ff a = ff_sqrt(ff_add(rho_t, dz2));
            a = e.mode == 0 ? ff_add(a, a) : ff_add(a, ff_sqrt(ff_add(rho_r, dz2)));
            const float2 *sn_ = sc + (size_t)n * e.n_f;
            for (int m = 0; m < e.n_f; ++m) {
                const float2 x = sn_[m];
                const float2 k = kff[m];
                float sv, cv;
                __sincosf(bp::phase_ff(k.x, k.y, a.hi, a.lo), &sv, &cv);
                const float sr = x.x * k.x, si = x.y * k.x;
                acc.x = fmaf(sr, cv, fmaf(-si, sv, acc.x));
                acc.y = fmaf(sr, sv, fmaf(si, cv, acc.y));
            }
        }
    }
    if (live) img[v] = acc;
}

template <int UT>
cudaError_t launch_exact_split(const ExactDesc &e, const float2 *S, const float2 *kap,
                               const float *wum, const float4 *chff, float2 *G, cudaStream_t st) {
    const size_t smem = 2 * (size_t)UT * (e.n_f < kExChunk ? e.n_f : kExChunk) * sizeof(float4);
    const int tiles = ((e.nx + kExTX - 1) / kExTX) * ((e.ny + kExTY - 1) / kExTY);
    dim3 grid(tiles, (e.n_pad + UT - 1) / UT);
    if (e.mode == 1) k_exact_sum<UT, 1><<<grid, kExThreads, smem, st>>>(e, S, kap, wum, chff, G);
    else k_exact_sum<UT, 0><<<grid, kExThreads, smem, st>>>(e, S, kap, wum, chff, G);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_exact_sum(const ExactDesc &e, const float2 *S, const float2 *kap,
                             const float *wum, const float4 *chff, float2 *G, cudaStream_t st) {
    // |delta| is at most the distance to the tile's reference pixel (8 and 4
    // steps away), once per range; kappa <= 2 k (mono) or k per range (multi)
    const double far = (e.mode == 1 ? 2.0 : 1.0) * hypot(kExTX / 2 * e.dx, kExTY / 2 * e.dy);
    if (far * e.kappa_max > kMaxSplitPhase) {
        constexpr int UT = 8;
        dim3 grid((e.nx * e.ny + 127) / 128, (e.n_pad + UT - 1) / UT);
        k_exact_sum_coarse<UT><<<grid, 128, 0, st>>>(e, S, kap, wum, chff, G);
        return cudaGetLastError();
    }
    return launch_exact_split<2>(e, S, kap, wum, chff, G, st);
}

cudaError_t launch_bp_direct(const DirectDesc &e, const float2 *s, const float4 *chff,
                             const float2 *zs, const float2 *kff, float2 *img, cudaStream_t st) {
    if (e.uniform) {
        auto kern = e.mode == 1 ? k_bp_direct_uniform<1> : k_bp_direct_uniform<0>;
        const unsigned blocks = (unsigned)((e.nx * e.ny + kDirPx - 1) / kDirPx) * (unsigned)e.nz;
        kern<<<blocks, 32 * kDirWarps, 0, st>>>(e, s, chff, zs, kff, img);
        return cudaGetLastError();
    }
    const long long nv = (long long)e.nx * e.ny * e.nz;
    const unsigned blocks = (unsigned)((nv + 127) / 128);
    k_bp_direct<<<blocks, 128, 0, st>>>(e, s, chff, zs, kff, img);
    return cudaGetLastError();
}
