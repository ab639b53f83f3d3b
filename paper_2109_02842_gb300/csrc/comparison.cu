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

// G[u][pixel] of the exact sum: two bins x 128 consecutive pixels per block, one
// pixel per thread.
//
// Bound by instruction issue (65 % of the slots; FP32 pipe 47 %, MUFU 37 %). The
// terms' coefficients k_m S and wavenumbers are staged in shared memory once per
// block and read by every lane at once. The phase kappa a of each (pixel, term)
// is a float-pair product reduced modulo 2 pi, so that the fast sine and cosine
// see [-pi, pi], where their error is bounded; the two bins' phases are formed
// in packed pairs. 120 channels, 51 frequencies, 128 bins, 64 x 64 pixels: 4.85
// (eight bins a block, terms loaded one by one) -> 1.87 ms, 2.29 with unpacked
// phases (0.67 at the MUFU pipe's rate); 1024 x 1 pixels 4.38 -> 0.62 ms. (Splitting the
// phase at a reference pixel, one FP32 product of up to 128 rad a term, took
// 1.65 ms but raised the image's error from 4.7e-6 to 6.4e-6.)
constexpr int kExThreads = 128;
constexpr int kExChunk = 256;                 // frequencies staged at a time

// bp::phase_ff of two terms at once in packed pairs (same operations, same
// rounding), the nearest integer by adding and taking off 1.5 2^23
__device__ __forceinline__ float2 phase_ff2(float2 kh, float2 kl, float ah, float al) {
    const float2 h = bp::f2(ah, ah), nh = bp::f2(-ah, -ah);
    const float2 np = __fmul2_rn(kh, nh);                      // -p
    float2 e = __ffma2_rn(kh, h, np);
    e = __ffma2_rn(kh, bp::f2(al, al), e);
    e = __ffma2_rn(kl, h, e);
    constexpr float kMagic = 12582912.f;
    const float2 t = __ffma2_rn(np, bp::f2(-bp::kInvTwoPi, -bp::kInvTwoPi), bp::f2(kMagic, kMagic));
    const float2 n = __fadd2_rn(t, bp::f2(-kMagic, -kMagic));
    float2 r = __ffma2_rn(n, bp::f2(bp::kTwoPiHi, bp::kTwoPiHi), np);
    r = __ffma2_rn(n, bp::f2(bp::kTwoPiLo, bp::kTwoPiLo), r);
    return __ffma2_rn(r, bp::f2(-1.f, -1.f), e);
}

template <int MODE>
__global__ void __launch_bounds__(kExThreads)
k_exact_sum(ExactDesc e, const float2 *__restrict__ S, const float2 *__restrict__ kap,
            const float *__restrict__ wum, const float4 *__restrict__ chff, float2 *__restrict__ G) {
    // two buffers: one barrier between the staging and the reading of a chunk
    extern __shared__ float4 sm_terms[];
    const int np = e.nx * e.ny, tiles = (np + kExThreads - 1) / kExThreads;
    const int p = (int)(blockIdx.x % tiles) * kExThreads + (int)threadIdx.x;
    const int u0 = (int)(blockIdx.x / tiles) * 2;
    const bool live = p < np;
    const int ix = live ? p % e.nx : 0, iy = live ? p / e.nx : 0;
    const ff px = ff_of(e.x0 + ix * e.dx), py = ff_of(e.y0 + iy * e.dy);
    const int mc_full = min(e.n_f, kExChunk);
    float2 acc0 = make_float2(0.f, 0.f), acc1 = acc0;
    int buf = 0;
    for (int c = 0; c < e.n_chan; ++c) {
        const float4 t = chff[2 * c], r = chff[2 * c + 1];
        // a = rho (mono: kappa = sqrt(4k^2 - k_z^2) carries the factor 2) or
        // rho_T + rho_R (multi: kappa = sqrt(k^2 - k_z^2 / 4))
        ff a = ff_dist2d(px, py, {t.x, t.y}, {t.z, t.w});
        if (MODE == 1) a = ff_add(a, ff_dist2d(px, py, {r.x, r.y}, {r.z, r.w}));
        for (int m0 = 0; m0 < e.n_f; m0 += kExChunk) {
            const int mc = min(kExChunk, e.n_f - m0);
            // [term][coefficients of both bins (re, re, im, im), wavenumbers
            // (high, high, low, low)]
            float *terms = reinterpret_cast<float *>(sm_terms + (size_t)buf * 2 * mc_full);
            for (int i = threadIdx.x; i < 2 * mc; i += kExThreads) {
                const int j = i >= mc ? 1 : 0, ml = i - j * mc, m = m0 + ml, u = u0 + j;
                float2 s = make_float2(0.f, 0.f), k = s;        // evanescent, or past the bins
                if (u < e.n_pad) {
                    const float w = wum[(size_t)u * e.n_f + m];
                    if (w != 0.f) {
                        k = kap[(size_t)u * e.n_f + m];
                        s = S[((size_t)c * e.n_pad + u) * e.n_f + m];
                        s = make_float2(s.x * w, s.y * w);
                    }
                }
                float *o = terms + 8 * ml + j;
                o[0] = s.x;
                o[2] = s.y;
                o[4] = k.x;
                o[6] = k.y;
            }
            __syncthreads();
            const float4 *tm = reinterpret_cast<const float4 *>(terms);
#pragma unroll 4
            for (int m = 0; m < mc; ++m) {
                const float4 s = tm[2 * m], k = tm[2 * m + 1];
                float sn0, cs0, sn1, cs1;
                const float2 ph = phase_ff2(bp::f2(k.x, k.y), bp::f2(k.z, k.w), a.hi, a.lo);
                __sincosf(ph.x, &sn0, &cs0);
                __sincosf(ph.y, &sn1, &cs1);
                acc0.x = fmaf(s.x, cs0, fmaf(-s.z, sn0, acc0.x));
                acc0.y = fmaf(s.x, sn0, fmaf(s.z, cs0, acc0.y));
                acc1.x = fmaf(s.y, cs1, fmaf(-s.w, sn1, acc1.x));
                acc1.y = fmaf(s.y, sn1, fmaf(s.w, cs1, acc1.y));
            }
            buf ^= 1;
        }
    }
    if (live) {
        G[(size_t)u0 * np + p] = acc0;
        if (u0 + 1 < e.n_pad) G[(size_t)(u0 + 1) * np + p] = acc1;
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
//
// LINES: the 128 voxels of a warp are consecutive over the whole volume, each
// with its own height, for planes of so few pixels that most lanes of a plane's
// block would repeat the last one (the rule is at the launch).
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

template <int MODE, bool LINES>
__global__ void __launch_bounds__(32 * kDirWarps, 3)
k_bp_direct_uniform(DirectDesc e, const float2 *__restrict__ s, const float4 *__restrict__ chff,
                    const float2 *__restrict__ zs, const float2 *__restrict__ kff,
                    float2 *__restrict__ img) {
    __shared__ float4 sm_coef[kDirWarps * kDirTerms];   // [warp][term] {re, re, im, im}
    // (z - z'_n)^2 of the staged positions; LINES: z'_n
    __shared__ float2 sm_dz2[kDirWarps][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float4 *coef = sm_coef + warp * kDirTerms;
    const int np = e.nx * e.ny, px_blocks = LINES ? 1 : (np + kDirPx - 1) / kDirPx;
    const int iz = LINES ? 0 : (int)(blockIdx.x / px_blocks);
    // this block's first pixel of plane iz (LINES: 0, of the voxels from v0 on)
    // and where they end
    const long long v0 = LINES ? (long long)blockIdx.x * kDirPx : (long long)iz * np;
    const int pb = LINES ? 0 : (int)(blockIdx.x - (unsigned)iz * px_blocks) * kDirPx;
    const int pe = LINES ? (int)min((long long)kDirPx, (long long)np * e.nz - v0) : np;
    const int p0 = pb + lane;
    ff pz[LINES ? 4 : 1];
    int pixel[LINES ? 4 : 1];
    if (LINES) {
#pragma unroll
        for (int k = 0; k < (LINES ? 4 : 1); ++k) {
            const long long v = v0 + min(p0 + 32 * k, pe - 1);
            pixel[k] = (int)(v % np);
            pz[k] = ff_of(e.z0 + (double)(v / np) * e.dz);
        }
    } else {
        pz[0] = ff_of(e.z0 + iz * e.dz);
    }
    const int rows = e.n_f > kDirPoly ? 1 : min(32, kDirTerms / e.n_f);  // positions staged at a time
    // frequency of staged term `lane`, and its step over 32 terms (modulo n_f)
    const int lane_m = lane % e.n_f, step_m = 32 % e.n_f;
    float2 sum[2][2] = {{{0.f, 0.f}, {0.f, 0.f}}, {{0.f, 0.f}, {0.f, 0.f}}};   // [pair][re, im]
    for (int c = warp; c < e.n_chan; c += kDirWarps) {
        const float4 t = chff[2 * c], r = chff[2 * c + 1];
        ff rho_t[4], rho_r[MODE == 1 ? 4 : 1];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            // (past the image: the last pixel)
            const int p = LINES ? pixel[LINES ? k : 0] : min(p0 + 32 * k, np - 1);
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
                    const ff d = ff_sqr(ff_add(pz[0], ff_neg({zn.x, zn.y})));
                    sm_dz2[warp][lane] = LINES ? zn : make_float2(d.hi, d.lo);
                }
                __syncwarp();
                for (int n = 0; n < nr; ++n) {
                    ff dz2 = {sm_dz2[warp][n].x, sm_dz2[warp][n].y};
                    const ff zn = ff_neg(dz2);
                    float cs[4], sn[4], c0[4], s0[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        if (LINES) dz2 = ff_sqr(ff_add(pz[LINES ? k : 0], zn));
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
        if (pb + i >= pe) break;
        float2 g = part[i];
        for (int w = 1; w < kDirWarps; ++w) {
            g.x += part[w * kDirPx + i].x;
            g.y += part[w * kDirPx + i].y;
        }
        img[v0 + pb + i] = g;
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

}  // namespace

cudaError_t launch_exact_sum(const ExactDesc &e, const float2 *S, const float2 *kap,
                             const float *wum, const float4 *chff, float2 *G, cudaStream_t st) {
    // two buffers of 32 bytes a term
    const size_t smem = 2 * 32 * (size_t)(e.n_f < kExChunk ? e.n_f : kExChunk);
    const size_t blocks = (size_t)((e.nx * e.ny + kExThreads - 1) / kExThreads) * ((e.n_pad + 1) / 2);
    if (blocks > 0x7fffffffu) return cudaErrorInvalidValue;
    auto kern = e.mode == 1 ? k_exact_sum<1> : k_exact_sum<0>;
    kern<<<(unsigned)blocks, kExThreads, smem, st>>>(e, S, kap, wum, chff, G);
    return cudaGetLastError();
}

cudaError_t launch_bp_direct(const DirectDesc &e, const float2 *s, const float4 *chff,
                             const float2 *zs, const float2 *kff, float2 *img, cudaStream_t st) {
    if (e.uniform) {
        // planes of up to 64 pixels, half a block, as lines, once there are more
        // planes than SMs. Planes and lines, ms (120 channels, 48 positions, 51
        // frequencies): 1 x 1 x 16384 voxels 109 and 1.39, 5 x 5 x 8192 54.8 and
        // 11.9, 6 x 7 x 8192 54.8 and 19.3, 2 x 2 x 256 2.22 and 1.39, 5 x 5 x 128
        // 1.35 and 1.40.
        const int np = e.nx * e.ny;
        const bool lines = np <= kDirPx / 2 && e.nz > 152;
        auto kern = lines ? (e.mode == 1 ? k_bp_direct_uniform<1, true> : k_bp_direct_uniform<0, true>)
                          : (e.mode == 1 ? k_bp_direct_uniform<1, false> : k_bp_direct_uniform<0, false>);
        const long long blocks_ll = lines ? ((long long)np * e.nz + kDirPx - 1) / kDirPx
                                          : (long long)((np + kDirPx - 1) / kDirPx) * e.nz;
        if (blocks_ll > 0x7fffffffLL) return cudaErrorInvalidValue;
        const unsigned blocks = (unsigned)blocks_ll;
        kern<<<blocks, 32 * kDirWarps, 0, st>>>(e, s, chff, zs, kff, img);
        return cudaGetLastError();
    }
    const long long nv = (long long)e.nx * e.ny * e.nz;
    const unsigned blocks = (unsigned)((nv + 127) / 128);
    k_bp_direct<<<blocks, 128, 0, st>>>(e, s, chff, zs, kff, img);
    return cudaGetLastError();
}
