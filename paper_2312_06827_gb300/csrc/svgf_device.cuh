// Device code shared by the single-frame kernels (svgf_kernels.cu) and the batched persistent
// kernels (svgf_batch.cu): helpers, the storage policies of the workspace images, and one function
// per stage that processes one tile of one image:
//
//   temporal_tile          Sec. 3.4 forward map, Sec. 2 / Sec. 3 step 4 backward reprojection,
//                          Sec. 3.1 variance colour clamp, accumulation of colour and moments,
//                          temporal variance; flags tiles that hold short histories.
//   spatial_variance_tile  Sec. 2: 7x7 depth/normal-weighted moment variance for n < 4.
//   atrous_tile<MODE>      Sec. 2 Fig. 1 / Sec. 3 step 5 edge-avoiding a-trous iteration, 5x5
//                          (MODE 0) or the Sec. 3.3 separable horizontal (1) / vertical (2) pass,
//                          with the Sec. 3.2 adaptive start and, on the last pass, the Sec. 3.4
//                          inverse map fused into the store.
//
// One thread per pixel; a warp covers 32 consecutive pixels of a row so every tap load of a warp
// is one contiguous span.
//
// Accuracy notes (FP32 against the FP64 definition):
//  - the bilinear fraction of the reprojected position is taken from -mv alone (the pixel index
//    is an integer), so it does not lose the bits a large x would cost;
//  - the clamp's standard deviation is computed two-pass from the window in shared memory;
//  - moments are kept in central form (mu1, S = mu2 - mu1^2) with the exact exponential update
//    of S, so the variance never comes from a cancelling difference of FP32 second moments;
//  - the normal weight is (1 - t)^sigma_n with t = |n_p - n_q|^2 / 2: t is formed from differences
//    of nearby normals, which are exact or nearly so, instead of 1 - n_p.n_q whose rounding
//    sigma_n = 128 would amplify, and log2(1 - t) comes from a series near t = 0.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <math.h>

#include "svgf_internal.h"

namespace svgf {
namespace dev {


__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float lg2_approx(float x) {
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rcp_approx(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float sqrt_approx(float x) {
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Rec. 709 luma, Reinhard forward and inverse maps (Sec. 3.4).  Written as explicit fused
// multiply-adds: every kernel that evaluates them then rounds identically (the compiler may not
// contract a plain a * b + c the same way in two kernels).
__device__ __forceinline__ float luma(float r, float g, float b) {
    return fmaf(0.0722f, b, fmaf(0.7152f, g, 0.2126f * r));
}

__device__ __forceinline__ float3 tonemap(const Params& P, float3 c) {
    if (!P.tonemap) return c;
    const float r = 1.0f / fmaf(luma(c.x, c.y, c.z), P.luma_k, 1.0f);
    return make_float3(c.x * r, c.y * r, c.z * r);
}

__device__ __forceinline__ float3 inverse_tonemap(const Params& P, float3 c) {
    if (!P.tonemap) return c;
    float l = luma(c.x, c.y, c.z);
    float f;
    if (P.inverse_mode == 1) {
        f = (1.0f + l) * P.inv_weight;
    } else {
        float d = fmaf(-P.luma_k, l, 1.0f);
        d = d < 1e-6f ? 1e-6f : d;
        f = 1.0f / d;
    }
    return make_float3(c.x * f, c.y * f, c.z * f);
}

__device__ __forceinline__ float3 load_rgb(const float* __restrict__ p, long i) {
    return make_float3(__ldg(p + 3 * i), __ldg(p + 3 * i + 1), __ldg(p + 3 * i + 2));
}

// Central-difference depth gradient, one-sided at the borders, 0 along an axis of extent 1.
__device__ __forceinline__ float2 depth_grad(const float4* __restrict__ g, int x, int y, int W,
                                             int H) {
    float gx, gy;
    long row = (long)y * W;
    if (W == 1) gx = 0.f;
    else if (x == 0) gx = __ldg(&g[row + 1].w) - __ldg(&g[row].w);
    else if (x == W - 1) gx = __ldg(&g[row + W - 1].w) - __ldg(&g[row + W - 2].w);
    else gx = 0.5f * (__ldg(&g[row + x + 1].w) - __ldg(&g[row + x - 1].w));
    if (H == 1) gy = 0.f;
    else if (y == 0) gy = __ldg(&g[(long)W + x].w) - __ldg(&g[x].w);
    else if (y == H - 1) gy = __ldg(&g[(long)(H - 1) * W + x].w) - __ldg(&g[(long)(H - 2) * W + x].w);
    else gy = 0.5f * (__ldg(&g[(long)(y + 1) * W + x].w) - __ldg(&g[(long)(y - 1) * W + x].w));
    return make_float2(gx, gy);
}

// depth_grad for a pixel with all four neighbours in the image (same arithmetic, no branches).
__device__ __forceinline__ float2 depth_grad_interior(const float4* __restrict__ gp, int W) {
    return make_float2(0.5f * (__ldg(&gp[1].w) - __ldg(&gp[-1].w)),
                       0.5f * (__ldg(&gp[W].w) - __ldg(&gp[-W].w)));
}

__device__ __forceinline__ int start_level(const Params& P, const float* __restrict__ rough, long p) {
    if (!P.adaptive_start || rough == nullptr) return 0;
    return __ldg(rough + p) > P.rough_thr ? 1 : 0;
}

// [1 2 1] x [1 2 1] / 16 blur of the variance channel at (x, y), in-image taps renormalised.
template <class S>
__device__ __forceinline__ float var_prefilter(const typename S::Rec* __restrict__ cv, int x, int y,
                                               int W, int H) {
    float s = 0.f, ws = 0.f;
#pragma unroll
    for (int b = -1; b <= 1; ++b) {
        int yy = y + b;
        if (yy < 0 || yy >= H) continue;
#pragma unroll
        for (int a = -1; a <= 1; ++a) {
            int xx = x + a;
            if (xx < 0 || xx >= W) continue;
            float k = (a == 0 ? 0.5f : 0.25f) * (b == 0 ? 0.5f : 0.25f);
            s = fmaf(k, S::ld_var(cv, yy * W + xx), s);
            ws += k;
        }
    }
    return s / ws;
}

// var_prefilter for a pixel with its 3x3 neighbourhood in the image: the nine weights sum to 1
// exactly, so the same sum in the same order gives the same value.
template <class S>
__device__ __forceinline__ float var_prefilter_interior(const typename S::Rec* __restrict__ cp, int W) {
    float s = 0.f;
#pragma unroll
    for (int b = -1; b <= 1; ++b) {
#pragma unroll
        for (int a = -1; a <= 1; ++a) {
            const float k = (a == 0 ? 0.5f : 0.25f) * (b == 0 ? 0.5f : 0.25f);
            s = fmaf(k, S::ld_var(cp + b * W, a), s);
        }
    }
    return s;
}

// ------------------------------------------------------------------------- storage policies
//
// Workspace images: colour + variance (cv: r, g, b, var), colour history (hist: r, g, b, -) and
// moments (mom: mu1, S = mu2 - mu1^2, n, -).  StoreF32 keeps each pixel as a float4.  Store16<BF>
// packs each into 8 bytes: colour and mu1 as FP16 (BF = false) or BF16 (BF = true); the
// variance-type fields (var, S) always as BF16, whose 8-bit exponent keeps the small variances of
// the late a-trous passes that FP16 would flush to subnormals or zero; n as an exact 16-bit
// integer.  All arithmetic stays FP32: values are widened on load and rounded on store.
struct StoreF32 {
    using Rec = float4;
    __device__ static float4 ld_cv(const Rec* b, int i) { return __ldg(b + i); }
    __device__ static float ld_var(const Rec* b, int i) { return __ldg(&b[i].w); }
    __device__ static void st_cv(Rec* b, int i, float4 v) { b[i] = v; }
    __device__ static void st_var(Rec* b, int i, float v) { b[i].w = v; }
    __device__ static float4 ld_hist(const Rec* b, int i) { return __ldg(b + i); }
    __device__ static void st_hist(Rec* b, int i, float3 c) { b[i] = make_float4(c.x, c.y, c.z, 0.f); }
    __device__ static float4 ld_mom(const Rec* b, int i) { return __ldg(b + i); }
    __device__ static float ld_n(const Rec* b, int i) { return __ldg(&b[i].z); }
    __device__ static void st_mom(Rec* b, int i, float mu1, float S, float n) {
        b[i] = make_float4(mu1, S, n, 0.f);
    }
    __device__ static float4 round_cv(float4 v) { return v; }
};

template <bool BF>
struct Store16 {
    using Rec = uint2;
    __device__ static unsigned enc_c(float x) {
        return BF ? (unsigned)__bfloat16_as_ushort(__float2bfloat16_rn(x))
                  : (unsigned)__half_as_ushort(__float2half_rn(x));
    }
    __device__ static float dec_c(unsigned u) {
        return BF ? __uint_as_float(u << 16) : __half2float(__ushort_as_half((unsigned short)u));
    }
    __device__ static unsigned enc_v(float x) {
        return (unsigned)__bfloat16_as_ushort(__float2bfloat16_rn(x));
    }
    __device__ static float dec_v(unsigned u) { return __uint_as_float(u << 16); }
    __device__ static float4 ld_cv(const Rec* b, int i) {
        const uint2 u = __ldg(b + i);
        return make_float4(dec_c(u.x & 0xffffu), dec_c(u.x >> 16), dec_c(u.y & 0xffffu), dec_v(u.y >> 16));
    }
    __device__ static float ld_var(const Rec* b, int i) {
        return dec_v(__ldg(reinterpret_cast<const unsigned short*>(b) + 4 * i + 3));
    }
    __device__ static void st_cv(Rec* b, int i, float4 v) {
        b[i] = make_uint2(enc_c(v.x) | (enc_c(v.y) << 16), enc_c(v.z) | (enc_v(v.w) << 16));
    }
    __device__ static void st_var(Rec* b, int i, float v) {
        reinterpret_cast<unsigned short*>(b)[4 * i + 3] = (unsigned short)enc_v(v);
    }
    __device__ static float4 ld_hist(const Rec* b, int i) {
        const uint2 u = __ldg(b + i);
        return make_float4(dec_c(u.x & 0xffffu), dec_c(u.x >> 16), dec_c(u.y & 0xffffu), 0.f);
    }
    __device__ static void st_hist(Rec* b, int i, float3 c) {
        b[i] = make_uint2(enc_c(c.x) | (enc_c(c.y) << 16), enc_c(c.z));
    }
    __device__ static float4 ld_mom(const Rec* b, int i) {
        const uint2 u = __ldg(b + i);
        return make_float4(dec_c(u.x & 0xffffu), dec_v(u.x >> 16), (float)(u.y & 0xffffu), 0.f);
    }
    __device__ static float ld_n(const Rec* b, int i) {
        return (float)__ldg(reinterpret_cast<const unsigned short*>(b) + 4 * i + 2);
    }
    __device__ static void st_mom(Rec* b, int i, float mu1, float S, float n) {
        b[i] = make_uint2(enc_c(mu1) | (enc_v(S) << 16), (unsigned)n);
    }
    // The value a cv record would hold after a store and a load.
    __device__ static float4 round_cv(float4 v) {
        return make_float4(dec_c(enc_c(v.x)), dec_c(enc_c(v.y)), dec_c(enc_c(v.z)), dec_v(enc_v(v.w)));
    }
};

// ------------------------------------------------------------------------- temporal stage

// History rectification of h against the 3x3 box of centre m and half-extents e = gamma sigma
// (Sec. 3.1, Fig. 3).  mode 0 (clamping): each channel limited to [m - e, m + e].  mode 1
// (clipping): h moved toward m along the line from m until it lies in the box:
// h' = m + (h - m) / t, t = max_c |h_c - m_c| / e_c, when t > 1; a channel with h_c = m_c
// does not constrain, one with e_c = 0 and h_c != m_c gives t = inf, i.e. h' = m.
__device__ __forceinline__ float3 rectify(int mode, float3 h, const float* m, const float* e) {
    if (mode == 0)
        return make_float3(fminf(fmaxf(h.x, m[0] - e[0]), m[0] + e[0]),
                           fminf(fmaxf(h.y, m[1] - e[1]), m[1] + e[1]),
                           fminf(fmaxf(h.z, m[2] - e[2]), m[2] + e[2]));
    const float d[3] = {h.x - m[0], h.y - m[1], h.z - m[2]};
    float t = 0.f;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        if (d[c] == 0.f) continue;
        const float r = e[c] > 0.f ? fabsf(d[c]) / e[c] : INFINITY;
        t = fmaxf(t, r);
    }
    if (!(t > 1.0f)) return h;
    if (isinf(t)) return make_float3(m[0], m[1], m[2]);
    return make_float3(m[0] + d[0] / t, m[1] + d[1] / t, m[2] + d[2] / t);
}

// Two FP32 values in one 64-bit register pair and the packed operations on them: each rounds as
// the scalar operation does, in one issue slot instead of two.
using F2 = unsigned long long;
__device__ __forceinline__ F2 f2(float lo, float hi) {
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unf2(F2 v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ F2 add2(F2 a, F2 b) {
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ F2 sub2(F2 a, F2 b) {
    F2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ F2 mul2(F2 a, F2 b) {
    F2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// Shared-memory tile of the temporal stage: the tone-mapped colour of a TILE_X x TILE_Y tile with
// a one-pixel halo, red and green side by side for the packed window sums.
struct TemporalSmem {
    F2 rg[TILE_Y + 2][TILE_X + 2];
    float b[TILE_Y + 2][TILE_X + 2];
};

// Resident blocks per SM the temporal kernels' register budget is set for: 4 (64 registers).  With
// nothing of the gathers held across the barrier the single-frame kernel spills 48 bytes a thread in
// FP32 storage and 20 in 16 bits (the batched one: svgf_batch.cuh); 3 blocks (85 registers, none)
// measured 242 us a 4K frame against 216.
constexpr int kTemporalBlocksPerSM = 4;

// The temporal stage for the TILE_X x TILE_Y tile at (x0, y0) of a W x H image, by a block of
// TILE_X x TILE_Y threads.  *flag receives whether any pixel of the tile has a short history.
// Contains block-wide barriers: every thread of the block must call it.
//
// Bound by latency (the motion vector, then the gathers that depend on it) and issue.  Loads go
// out in dependency order, each group before the previous one is consumed: the pixel's G-buffer
// record, motion vector and noisy colour, the tile's halo, then the reprojection gathers, whose
// latency overlaps the tone map and fill of the tile; the gathers are blended down to six values
// before the block's barrier, so that nothing of them is held across it.  One reciprocal serves the
// blends, the window sums take two channels an instruction, and the halo is filled by three warps
// instead of a second pass of all eight.  4K frame 248 -> 216 us (4.4 TB/s of its 116 bytes a pixel),
// 16-bit storage 239 -> 195 us; 1080p 69 -> 62 us.
template <class S>
__device__ __forceinline__ void temporal_tile(
    const Params& P, int W, int H, int x0, int y0, int* flag, const float* __restrict__ noisy,
    const float4* __restrict__ gbuf, const float4* __restrict__ prev_gbuf,
    const float2* __restrict__ mv, const typename S::Rec* __restrict__ hist_prev,
    const typename S::Rec* __restrict__ mom_prev, int has_history,
    typename S::Rec* __restrict__ cv_out, typename S::Rec* __restrict__ mom_out,
    typename S::Rec* __restrict__ hist_accum_out, TemporalSmem& sm) {
    const int x = x0 + threadIdx.x;
    const int y = y0 + threadIdx.y;
    const bool inside = x < W && y < H;
    const long p = inside ? (long)y * W + x : 0;
    const float4 g = __ldg(&gbuf[p]);
    const float2 m = __ldg(&mv[p]);
    const float3 own = load_rgb(noisy, p);
    // the halo of the tile: its 2 x 34 + 2 x 8 pixels by the block's first threads
    constexpr int SX = TILE_X + 2, SY = TILE_Y + 2, kHalo = 2 * SX + 2 * TILE_Y;
    const int tid = threadIdx.y * TILE_X + threadIdx.x;
    int hx = 0, hy = 0;
    float3 hv = make_float3(0.f, 0.f, 0.f);
    if (tid < kHalo) {
        hy = tid < SX ? 0 : tid < 2 * SX ? SY - 1 : 1 + ((tid - 2 * SX) & (TILE_Y - 1));
        hx = tid < SX ? tid : tid < 2 * SX ? tid - SX : tid < 2 * SX + TILE_Y ? 0 : SX - 1;
        const int gx = x0 + hx - 1, gy = y0 + hy - 1;
        if (gx >= 0 && gy >= 0 && gx < W && gy < H) hv = load_rgb(noisy, (long)gy * W + gx);
    }

    // reprojection footprint: previous position p + 0.5 - mv, base floor(x - mv), fraction
    // frac(-mv); up to four taps, all their loads issued at once.  A tap outside the image or of
    // weight 0 reads record 0 and is skipped by its weight.
    const bool history = has_history && prev_gbuf != nullptr;   // uniform
    const bool reproject = inside && history && fabsf(m.x) < 1e7f && fabsf(m.y) < 1e7f;
    float4 tg[4], th[4], tmm[4];
    float twb[4];
    if (history) {
        const float ux = -m.x, uy = -m.y;
        const float flx = floorf(ux), fly = floorf(uy);
        const float fx = ux - flx, fy = uy - fly;
        const int bx = x + (int)flx, by = y + (int)fly;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int i = k & 1, j = k >> 1;
            const int tx = bx + i, ty = by + j;
            const float w = (i ? fx : 1.0f - fx) * (j ? fy : 1.0f - fy);
            const bool in = reproject && (unsigned)tx < (unsigned)W && (unsigned)ty < (unsigned)H && w > 0.f;
            twb[k] = in ? w : 0.f;
            const int t = in ? ty * W + tx : 0;
            tg[k] = __ldg(&prev_gbuf[t]);
            th[k] = S::ld_hist(hist_prev, t);
            tmm[k] = S::ld_mom(mom_prev, t);
        }
    }

    const float3 c = tonemap(P, own);
    {
        // pixels past the image's edge hold zeros, as the halo outside it does
        const float3 v = inside ? c : make_float3(0.f, 0.f, 0.f);
        sm.rg[threadIdx.y + 1][threadIdx.x + 1] = f2(v.x, v.y);
        sm.b[threadIdx.y + 1][threadIdx.x + 1] = v.z;
    }
    if (tid < kHalo) {
        const float3 v = tonemap(P, hv);
        sm.rg[hy][hx] = f2(v.x, v.y);
        sm.b[hy][hx] = v.z;
    }

    bool valid = false;
    float3 hist = make_float3(0.f, 0.f, 0.f);
    float mu1p = 0.f, Sp = 0.f, nprev = 0.f;
    if (reproject) {
        const float ztol = P.depth_rel_tol * g.w;
        float sw = 0.f;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float4 gp = tg[k];
            const float dz = fabsf(gp.w - g.w);
            const float ax = g.x - gp.x, ay = g.y - gp.y, az = g.z - gp.z;
            const float dn2 = fmaf(ax, ax, fmaf(ay, ay, az * az));
            // contributes: in the image, and consistent in depth and normal
            if (twb[k] > 0.f && dz <= ztol && dn2 <= P.normal_tol2) {
                const float w = twb[k];
                sw += w;
                hist.x = fmaf(w, th[k].x, hist.x);
                hist.y = fmaf(w, th[k].y, hist.y);
                hist.z = fmaf(w, th[k].z, hist.z);
                mu1p = fmaf(w, tmm[k].x, mu1p);
                nprev = fmaxf(nprev, tmm[k].z);
            } else {
                twb[k] = 0.f;
                tmm[k].x = 0.f;
                tmm[k].y = 0.f;
            }
        }
        if (sw >= P.disocc_w) {
            valid = true;
            const float rs = 1.0f / sw;
            hist = make_float3(hist.x * rs, hist.y * rs, hist.z * rs);
            // blended moments in central form: mean of mu1, and E[S] + Var[mu1] over taps
            mu1p *= rs;
            float sS = 0.f, sd = 0.f;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float d = tmm[k].x - mu1p;
                sS = fmaf(twb[k], tmm[k].y, sS);
                sd = fmaf(twb[k] * d, d, sd);
            }
            Sp = (sS + sd) * rs;
        }
    }
    __syncthreads();
    int short_history = 0;
    if (inside) {
        const int tx = threadIdx.x + 1, ty = threadIdx.y + 1;
        if (valid && P.clamp_enable) {
            // 3x3 box of the current tone-mapped colour, in-image pixels: mean and population
            // std-dev, two-pass, red and green packed
            float mb[3], sd[3];
            if (x > 0 && y > 0 && x + 1 < W && y + 1 < H) {
                F2 s2 = f2(0.f, 0.f);
                float s1 = 0.f;
#pragma unroll
                for (int b = -1; b <= 1; ++b)
#pragma unroll
                    for (int a = -1; a <= 1; ++a) {
                        s2 = add2(s2, sm.rg[ty + b][tx + a]);
                        s1 += sm.b[ty + b][tx + a];
                    }
                const F2 m2 = mul2(s2, f2(1.0f / 9.0f, 1.0f / 9.0f));
                const float m1 = s1 * (1.0f / 9.0f);
                F2 q2 = f2(0.f, 0.f);
                float q1 = 0.f;
#pragma unroll
                for (int b = -1; b <= 1; ++b)
#pragma unroll
                    for (int a = -1; a <= 1; ++a) {
                        const F2 d2 = sub2(sm.rg[ty + b][tx + a], m2);
                        const float d1 = sm.b[ty + b][tx + a] - m1;
                        q2 = fma2(d2, d2, q2);
                        q1 = fmaf(d1, d1, q1);
                    }
                unf2(m2, mb[0], mb[1]);
                mb[2] = m1;
                unf2(q2, sd[0], sd[1]);
                sd[2] = q1;
#pragma unroll
                for (int ch = 0; ch < 3; ++ch) sd[ch] = P.gamma * sqrtf(sd[ch] * (1.0f / 9.0f));
            } else {
                const bool xl = x > 0, xr = x + 1 < W, yu = y > 0, yd = y + 1 < H;
                const float inv_c = 1.0f / (float)((1 + xl + xr) * (1 + yu + yd));
                float s[3] = {0.f, 0.f, 0.f}, q[3] = {0.f, 0.f, 0.f};
                for (int pass = 0; pass < 2; ++pass) {
                    for (int b = yu ? -1 : 0; b <= (yd ? 1 : 0); ++b)
                        for (int a = xl ? -1 : 0; a <= (xr ? 1 : 0); ++a) {
                            float v[3];
                            unf2(sm.rg[ty + b][tx + a], v[0], v[1]);
                            v[2] = sm.b[ty + b][tx + a];
#pragma unroll
                            for (int ch = 0; ch < 3; ++ch) {
                                if (pass == 0) s[ch] += v[ch];
                                else q[ch] = fmaf(v[ch] - mb[ch], v[ch] - mb[ch], q[ch]);
                            }
                        }
#pragma unroll
                    for (int ch = 0; ch < 3; ++ch) {
                        if (pass == 0) mb[ch] = s[ch] * inv_c;
                        else sd[ch] = P.gamma * sqrtf(q[ch] * inv_c);
                    }
                }
            }
            hist = rectify(P.rectify_mode, hist, mb, sd);
        }

        const float nn = valid ? fminf(nprev + 1.0f, P.max_history) : 1.0f;
        const float inv_n = 1.0f / nn;
        const float a = fmaxf(P.alpha, inv_n);
        const float am = fmaxf(P.alpha_m, inv_n);
        float3 ci;
        if (valid) {
            ci = make_float3(fmaf(a, c.x - hist.x, hist.x), fmaf(a, c.y - hist.y, hist.y),
                             fmaf(a, c.z - hist.z, hist.z));
        } else {
            ci = c;
        }
        // Moments in central form (mu1, S = mu2 - mu1^2).  The exponential update of
        // (mu1, mu2) by l is, exactly, mu1' = mu1 + a d and S' = (1 - a)(S + a d^2), d = l - mu1;
        // it keeps S free of the cancellation that mu2 - mu1^2 suffers in FP32.
        const float l = luma(c.x, c.y, c.z);
        float mu1, Sv;
        if (valid) {
            const float d = l - mu1p;
            mu1 = fmaf(am, d, mu1p);
            Sv = (1.0f - am) * fmaf(am * d, d, Sp);
        } else {
            mu1 = l;
            Sv = 0.f;
        }
        float var = 0.f;
        if (nn >= P.min_temporal) {
            var = fmaxf(0.f, Sv);
        } else {
            short_history = 1;
        }
        S::st_cv(cv_out, (int)p, make_float4(ci.x, ci.y, ci.z, var));
        S::st_mom(mom_out, (int)p, mu1, Sv, nn);
        if (hist_accum_out) S::st_hist(hist_accum_out, (int)p, ci);
    }
    const int any_short = __syncthreads_or(short_history);
    if (threadIdx.x == 0 && threadIdx.y == 0) *flag = any_short;
}

// Largest spatial-variance radius (the configuration's range) and the window one tile reads:
// the tile with a margin of the radius on every side.
constexpr int kVarRadiusMax = 7;
constexpr int kVarWindowPx = (TILE_X + 2 * kVarRadiusMax) * (TILE_Y + 2 * kVarRadiusMax);
struct SpatialSmem {
    float4 g[kVarWindowPx];   // G-buffer (normal, depth)
    float2 m[kVarWindowPx];   // first two components of the moment record
};

// The weight of a spatial-variance tap is the a-trous weight without the luminance term, in natural
// units and to FP32 accuracy: a weighted variance magnifies a weight's relative error by up
// to max (x - m)^2 / var, and log2-unit weights took it past 1e-5 of the exact value.

// t = |n_p - n_q|^2 / 2 of the normal weight (1 - t)^sigma_n.
__device__ __forceinline__ float normal_t(const float4& g, const float4& gq) {
    const float ax = g.x - gq.x, ay = g.y - gq.y, az = g.z - gq.z;
    return 0.5f * fmaf(ax, ax, fmaf(ay, ay, az * az));
}

// log(1 - t) where nearly every tap lies, t <= kNearT (normals less than 14 degrees apart): the
// power series to t^5 (truncation below 5e-9 relative at 1/32; measured at most 1.10 u, log1pf 1.05).
// Elsewhere log1pf, -inf for t >= 1 and for a t that is not a number.
constexpr float kNearT = 0.03125f;
__device__ __forceinline__ float log1m_near(float t) {
    float p = fmaf(t, 1.0f / 5.0f, 1.0f / 4.0f);
    p = fmaf(t, p, 1.0f / 3.0f);
    p = fmaf(t, p, 0.5f);
    return -fmaf(t, __fmul_rn(t, p), t);
}
__device__ __forceinline__ float log1m_far(float t) { return t < 1.0f ? log1pf(-t) : -INFINITY; }

// exp(e) for e <= 0 as 2^(e log2 e), the exponent carried in two parts: h, the rounded product with
// log2 e to FP32, and r, the product's rounding error (exact by one fused multiply-add) plus the
// product with the remainder of log2 e (Dekker's splitting of a product); then
// 2^(h + r) = 2^h (1 + r ln 2) to first order, |r| < 2^-17, so what is left out is below 2^-35.  The
// exponential unit's own error remains: within 2.4 u (u = 2^-24), but on the low side, by 0.3 u on
// average near e = 0 and 0.85 u below -4, of which half a unit is put back.  Measured over [-87, 0] in
// 2^24 steps: at most 2.9 u, 0.75 u rms (expf 2.6 and 0.67; without the half unit 3.4 and 1.09).
// Below 2^-126, e < -87.3, it is 0.
__device__ __forceinline__ float exp_neg(float e) {
    const float h = __fmul_rn(e, 1.4426950216293335f);
    const float r = fmaf(e, 1.925963e-8f, fmaf(e, 1.4426950216293335f, -h));
    const float w = ex2_approx(h);
    return fmaf(w, fmaf(0.6931471805599453f, r, 0x1p-25f), w);
}

// The weight from l = log(1 - t): 0 where the normal weight is 0 or the weight is not a number (with
// sigma_z = infinity, a tap along which the depth has no gradient).  eps keeps the denominator within
// the reciprocal's range.
__device__ __forceinline__ float spatial_weight(const Params& P, float l, float zp, float zq, float2 gr,
                                                float dx, float dy) {
    const float den = fmaf(P.sigma_z, fabsf(fmaf(gr.x, dx, __fmul_rn(gr.y, dy))), fmaxf(P.eps, 1.17549435e-38f));
    const float depth = __fmul_rn(fabsf(zq - zp), rcp_approx(den));
    const float w = exp_neg(fmaf(P.sigma_n, l, -depth));
    return w > 0.f ? w : 0.f;
}

// The spatial variance of the pixels with a short history in the tile at (x0, y0) (a tile the
// temporal stage flagged).  The block first copies the tile's window of G-buffer and moments to
// shared memory (every load of the window in flight at once), then each short-history pixel
// sums its (2R + 1)^2 taps from there.  Called by every thread of the block (two barriers).
//
// E_w[mu2] - E_w[mu1]^2 = E_w[S] + Var_w[mu1], and Var_w[mu1] is formed without a difference of
// large sums, so it keeps its FP32 accuracy for wide windows: RC > 0 (the radius as a constant)
// takes the rows in a rolled loop, a row's mean and then its squared deviations from the weights
// in registers, and merges the rows by Chan's pairwise update.  The means are taken relative to the
// centre's, so that their roundings are of the size of the deviations: rounded at the size of the
// luminance, a row's mean cost accuracy wherever the noise is small against it (scattered normals,
// 1 % noise: 2-norm error of the variance 118 u with the per-tap update, 199 u with absolute row means,
// 2.3 u so, u = 2^-24).  Bound by instruction issue (78 % with every pixel short): about 52 instructions
// a tap, where the per-tap update with its division, log1pf and expf took about 95, and a body of one
// row, where 49 unrolled taps did not fit the instruction cache.  2560x1440 with every pixel short
// 556 -> 307 us, a steady 1080p frame (some 50 flagged tiles) 21.4 -> 15.9 us.  RC = 0 (the radius from P) keeps West's per-tap update.
template <class S, int RC>
__device__ __forceinline__ void spatial_variance_tile_r(const Params& P, int W, int H, int x0,
                                                        int y0, const float4* __restrict__ gbuf,
                                                        const typename S::Rec* __restrict__ mom,
                                                        typename S::Rec* __restrict__ cv,
                                                        SpatialSmem& sm) {
    const int R = RC > 0 ? RC : P.var_radius;
    const int HW = TILE_X + 2 * R, HH = TILE_Y + 2 * R;
    const int x = x0 + threadIdx.x, y = y0 + threadIdx.y, p = y * W + x;
    const bool work = x < W && y < H && S::ld_n(mom, p) < P.min_temporal;
    for (int i = threadIdx.y * TILE_X + threadIdx.x; i < HW * HH; i += TILE_X * TILE_Y) {
        const int yy = i / HW, xx = i - yy * HW;
        const int gx = x0 - R + xx, gy = y0 - R + yy;
        // outside the image: a normal that is no number, whose weight is 0
        float4 gq = make_float4(NAN, 0.f, 0.f, 0.f);
        if (gx >= 0 && gx < W && gy >= 0 && gy < H) {
            const int q = gy * W + gx;
            gq = __ldg(&gbuf[q]);
            const float4 mq = S::ld_mom(mom, q);
            sm.m[i] = make_float2(mq.x, mq.y);
        }
        sm.g[i] = gq;
    }
    __syncthreads();
    if (work) {
        const int c = (threadIdx.y + R) * HW + threadIdx.x + R;
        const float4 g = sm.g[c];
        const float2 gr = depth_grad(gbuf, x, y, W, H);
        float sw = 0.f, sS = 0.f, mean = 0.f, m2 = 0.f;
        if constexpr (RC > 0) {
            const float mc = sm.m[c].x;   // the centre's mean, which the taps' are taken relative to
#pragma unroll 1
            for (int b = -RC; b <= RC; ++b) {
                if (y + b < 0 || y + b >= H) continue;
                constexpr int N = 2 * RC + 1;
                const int q0 = c + b * HW - RC;
                float w[N], m[N], z[N];
                bool far = false;
#pragma unroll
                for (int a = 0; a < N; ++a) {
                    const float4 gq = sm.g[q0 + a];
                    z[a] = gq.w;
                    const float t = normal_t(g, gq);
                    far = far || !(t <= kNearT);
                    m[a] = t;
                    w[a] = log1m_near(t);
                }
                if (far) {
#pragma unroll
                    for (int a = 0; a < N; ++a)
                        if (!(m[a] <= kNearT)) w[a] = log1m_far(m[a]);
                }
                float rw = 0.f, rm = 0.f;
#pragma unroll
                for (int a = 0; a < N; ++a) {
                    w[a] = spatial_weight(P, w[a], g.w, z[a], gr, (float)(a - RC), (float)b);
                    // a tap of weight 0 adds nothing, whatever its moments hold
                    const float2 mq = w[a] > 0.f ? sm.m[q0 + a] : make_float2(mc, 0.f);
                    m[a] = mq.x - mc;
                    rw += w[a];
                    rm = fmaf(w[a], m[a], rm);
                    sS = fmaf(w[a], mq.y, sS);
                }
                if (!(rw > 0.f)) continue;
                const float row_mean = rm / rw;
                float r2 = 0.f;
#pragma unroll
                for (int a = 0; a < N; ++a) {
                    const float d = m[a] - row_mean;
                    r2 = fmaf(w[a] * d, d, r2);
                }
                const float t = sw + rw, d = row_mean - mean, f = __fdividef(rw, t);
                // (sw f d) d: 0 on the first row, where the square of d may overflow
                m2 += fmaf(__fmul_rn(__fmul_rn(sw, f), d), d, r2);
                mean = fmaf(d, f, mean);
                sw = t;
            }
        } else {
#pragma unroll 1
            for (int b = -R; b <= R; ++b) {
                if (y + b < 0 || y + b >= H) continue;
#pragma unroll 1
                for (int a = -R; a <= R; ++a) {
                    if (x + a < 0 || x + a >= W) continue;
                    const int q = c + b * HW + a;
                    const float4 gq = sm.g[q];
                    const float tn = normal_t(g, gq);
                    const float w = spatial_weight(P, tn <= kNearT ? log1m_near(tn) : log1m_far(tn), g.w, gq.w, gr,
                                                   (float)a, (float)b);
                    if (!(w > 0.f)) continue;   // a zero weight changes nothing (and would give 0/0 first)
                    const float2 mq = sm.m[q];
                    const float t = sw + w;
                    const float d = mq.x - mean;
                    const float r = __fdividef(d * w, t);
                    m2 = fmaf(sw * d, r, m2);
                    mean += r;
                    sw = t;
                    sS = fmaf(w, mq.y, sS);
                }
            }
        }
        S::st_var(cv, p, fmaxf(0.f, sS / sw + m2 / sw));
    }
    __syncthreads();   // the window is rewritten by the block's next tile
}

template <class S>
__device__ __forceinline__ void spatial_variance_tile(const Params& P, int W, int H, int x0,
                                                      int y0, const float4* __restrict__ gbuf,
                                                      const typename S::Rec* __restrict__ mom,
                                                      typename S::Rec* __restrict__ cv,
                                                      SpatialSmem& sm) {
    if (P.var_radius == 3) spatial_variance_tile_r<S, 3>(P, W, H, x0, y0, gbuf, mom, cv, sm);
    else spatial_variance_tile_r<S, 0>(P, W, H, x0, y0, gbuf, mom, cv, sm);
}

// ------------------------------------------------------------------------- a-trous
//
// The weight of tap q is w = h_jk * 2^E with E, in log2 units,
//   E = sigma_n log2(1 - t)  -  log2e |z_q - z_p| / (sigma_z |grad z_p . (p - q)| + eps)
//                            -  log2e |l_q - l_p| / (sigma_l sqrt(g(var)_p) + eps),
// t = |n_p - n_q|^2 / 2, so one ex2 per tap gives the product of the three edge functions.
//  - sigma_n log2(1 - t): the series -log2e (t + t^2/2 + t^3/3 + t^4/4) for t < 1/16, lg2 of
//    1 - t above, -inf for t >= 1.  The series' truncation error in the exponent is about
//    sigma_n t^5 / 5, so the weight's absolute error (relative to the centre tap) is at most
//    max_t sigma_n t^5/5 exp(-sigma_n t) = 625/sigma_n^4 e^-5 (1.6e-8 at sigma_n = 128; 2e-7 at
//    sigma_n = 1, reached at t = 1/16).  Above 1/16 the weight is below 2^(-0.093 sigma_n) and
//    lg2's absolute error (2^-22) is harmless;
//  - the depth denominator depends on the tap only through |j A + k B|, the same for the taps
//    (j, k) and (-j, -k): one reciprocal serves both;
//  - log2e is folded into the per-pixel constants.
// Blocks whose tile lies at least two maximal steps inside the image take a path without
// bounds checks (block-uniform branch).

constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;

// Per-launch constants of the tap weight, in log2 units.  With t2 = |n_p - n_q|^2 the normal
// weight is (1 - t2/2)^sigma_n, and sigma_n log2(1 - t2/2) = sum_m c_m t2^m with
// c_m = -sigma_n log2e / (m 2^m); the host computes c_1..c_4 into Params (as the launch
// parameters they cost the 5x5 pass no registers).
struct TapConsts {
    float c1, c2, c3, c4;
    float sigma_n;
};
__device__ __forceinline__ TapConsts tap_consts(const Params& P) {
    return {P.tc1, P.tc2, P.tc3, P.tc4, P.sigma_n};
}

// Normal edge-stopping weights this sharp or sharper take the series alone (NM = 2 below).
constexpr float kSeriesOnlySigma = 64.0f;

// log2 h + sigma_n log2(1 - t2/2) (-inf when the normal weight is 0).  Below t2 = 1/8 the
// degree-4 series keeps the relative accuracy that lg2.approx loses near 1.  NM = 0 branches to
// the lg2 form above; NM = 1 evaluates both forms and selects one (fewer control instructions,
// more arithmetic: faster for the two-tap separable passes, slower for the 24-tap 5x5 pass,
// where the lg2 form is rarely taken).  NM = 2, for sigma_n >= kSeriesOnlySigma, takes the
// series everywhere: its terms are all negative, so beyond t2 = 1/8 the weight it gives stays
// below exp(-sigma_n t2 / 2) and, like the exact weight, vanishes; the largest absolute error
// of the weight over t2 in [0, 4] is 2.2e-7 at sigma_n = 64 and 1.5e-8 at 128 (at t2 = 0.15
// and 0.08).
template <int NM>
__device__ __forceinline__ float normal_log2w(float t2, const TapConsts& T, float log2h) {
    if (NM == 2) return fmaf(t2, fmaf(t2, fmaf(t2, fmaf(t2, T.c4, T.c3), T.c2), T.c1), log2h);
    if (NM == 1) {
        const float series = fmaf(t2, fmaf(t2, fmaf(t2, fmaf(t2, T.c4, T.c3), T.c2), T.c1), log2h);
        const float direct = fmaf(T.sigma_n, lg2_approx(fmaf(t2, -0.5f, 1.0f)), log2h);
        return t2 < 0.125f ? series : (t2 < 2.0f ? direct : -INFINITY);
    }
    if (t2 < 0.125f) return fmaf(t2, fmaf(t2, fmaf(t2, fmaf(t2, T.c4, T.c3), T.c2), T.c1), log2h);
    return t2 < 2.0f ? fmaf(T.sigma_n, lg2_approx(fmaf(t2, -0.5f, 1.0f)), log2h) : -INFINITY;
}

// Tap pairs (j, k) with (-j, -k) as the partner: k > 0, or k == 0 and j > 0.
template <int MODE>
struct TapPairs;
template <>
struct TapPairs<0> {
    static constexpr int N = 12;
    __device__ static constexpr int j(int i) { return i < 2 ? i + 1 : ((i - 2) % 5) - 2; }
    __device__ static constexpr int k(int i) { return i < 2 ? 0 : (i < 7 ? 1 : 2); }
};
template <>
struct TapPairs<1> {
    static constexpr int N = 2;
    __device__ static constexpr int j(int i) { return i + 1; }
    __device__ static constexpr int k(int) { return 0; }
};
template <>
struct TapPairs<2> {
    static constexpr int N = 2;
    __device__ static constexpr int j(int) { return 0; }
    __device__ static constexpr int k(int i) { return i + 1; }
};

// log2 of the B3 taps 3/8, 1/4, 1/16
__device__ __forceinline__ constexpr float log2_b3(int j) {
    return j == 0 ? -1.4150374992788438f : ((j == 1 || j == -1) ? -2.0f : -4.0f);
}

struct AtrousAcc {
    float sw, sr, sg, sb, sv;
};

// One tap q of pixel p: cq, gq point at q's records.  The B3 weight h enters the exponent as
// log2 h, so w = 2^(log2 h + log2 w_n + log2 w_z + log2 w_l) is one ex2.
template <class S, int NM>
__device__ __forceinline__ void atrous_tap(const typename S::Rec* __restrict__ cq_ptr,
                                           const float4* __restrict__ gq_ptr, float log2h,
                                           float rden, const float4& g, float lp, float inv_dl2,
                                           const TapConsts& T, AtrousAcc& a) {
    const float4 cq = S::ld_cv(cq_ptr, 0);
    const float4 gq = __ldg(gq_ptr);
    const float ax = g.x - gq.x, ay = g.y - gq.y, az = g.z - gq.z;
    const float t2 = fmaf(ax, ax, fmaf(ay, ay, az * az));
    float e = normal_log2w<NM>(t2, T, log2h);
    e = fmaf(-fabsf(gq.w - g.w), rden, e);
    // the series-only form also folds -lp into the luminance's multiply-add chain
    const float dl = NM == 2 ? fmaf(0.0722f, cq.z, fmaf(0.7152f, cq.y, fmaf(0.2126f, cq.x, -lp)))
                             : luma(cq.x, cq.y, cq.z) - lp;
    e = fmaf(-fabsf(dl), inv_dl2, e);
    const float w = ex2_approx(e);
    a.sw += w;
    a.sr = fmaf(w, cq.x, a.sr);
    a.sg = fmaf(w, cq.y, a.sg);
    a.sb = fmaf(w, cq.z, a.sb);
    a.sv = fmaf(w * w, cq.w, a.sv);
}

// Output of one a-trous pass at pixel p: colour (and the history copy of it), or, for the last
// pass, the inverse tone-mapped FP32 colour with the variance.
template <class S>
__device__ __forceinline__ void atrous_store(const Params& P, int p, float4 v,
                                             typename S::Rec* __restrict__ cv_out,
                                             typename S::Rec* __restrict__ hist_out,
                                             float4* __restrict__ rgb_out) {
    if (hist_out) S::st_hist(hist_out, p, make_float3(v.x, v.y, v.z));
    if (rgb_out) {
        // the fused inverse map sees the colour at the storage precision, as the stage path does
        const float4 r = S::round_cv(v);
        const float3 o = inverse_tonemap(P, make_float3(r.x, r.y, r.z));
        rgb_out[p] = make_float4(o.x, o.y, o.z, r.w);
    } else {
        S::st_cv(cv_out, p, v);
    }
}

// Number of a-trous passes pixel p takes part in (Sec. 3.5): roughness <= t0 -> n0,
// <= t1 -> n1, otherwise all.
__device__ __forceinline__ int pass_budget(const Params& P, const float* __restrict__ rough, int p) {
    if (!P.iter_budget || rough == nullptr) return P.iter_all;
    const float r = __ldg(rough + p);
    return r <= P.iter_t0 ? P.iter_n0 : (r <= P.iter_t1 ? P.iter_n1 : P.iter_all);
}

// One pixel of one a-trous iteration at dilation `step`.  CHECK = false requires the whole 5x5
// footprint, the 3x3 prefilter and the gradient neighbours inside the image.  NS: the normal
// term by the series alone (sigma_n >= kSeriesOnlySigma).
template <int MODE, class S, bool CHECK, bool NS>
__device__ __forceinline__ void atrous_pixel(const Params& P, int W, int H, int step, int x, int y,
                                             const typename S::Rec* __restrict__ cv_in,
                                             const float4* __restrict__ gbuf,
                                             typename S::Rec* __restrict__ cv_out,
                                             typename S::Rec* __restrict__ hist_out,
                                             float4* __restrict__ rgb_out) {
    using Rec = typename S::Rec;
    const int p = y * W + x;
    const Rec* __restrict__ cvp = cv_in + p;
    const float4* __restrict__ gp = gbuf + p;
    const float4 g = __ldg(gp);
    const float2 gr = CHECK ? depth_grad(gbuf, x, y, W, H) : depth_grad_interior(gp, W);
    const float4 cp = S::ld_cv(cvp, 0);
    const float lp = luma(cp.x, cp.y, cp.z);
    const float vf = CHECK ? var_prefilter<S>(cv_in, x, y, W, H) : var_prefilter_interior<S>(cvp, W);
    // log2e / (sigma_l sqrt(g(var)) + eps): only scales an exponent, so the approximate square
    // root and reciprocal (a few ulp) are enough
    const float inv_dl2 = kLog2e * rcp_approx(fmaf(P.sigma_l, sqrt_approx(vf), P.eps));
    // |grad . offset| * sigma_z * ln2 = |j A + k B|; eps * ln2 keeps E in log2 units
    const float A = kLn2 * P.sigma_z * gr.x * (float)step;
    const float B = kLn2 * P.sigma_z * gr.y * (float)step;
    const float eps2 = kLn2 * P.eps;
    const TapConsts T = tap_consts(P);

    const float h0 = MODE == 0 ? 0.375f * 0.375f : 0.375f;
    AtrousAcc a = {h0, h0 * cp.x, h0 * cp.y, h0 * cp.z, h0 * h0 * cp.w};
#pragma unroll
    for (int i = 0; i < TapPairs<MODE>::N; ++i) {
        const int j = TapPairs<MODE>::j(i), k = TapPairs<MODE>::k(i);
        const float rden = rcp_approx(fabsf(fmaf((float)j, A, (float)k * B)) + eps2);
        const float log2h = MODE == 0 ? log2_b3(j) + log2_b3(k) : (MODE == 1 ? log2_b3(j) : log2_b3(k));
#pragma unroll
        for (int sgn = 1; sgn >= -1; sgn -= 2) {
            const int dx = sgn * j * step, dy = sgn * k * step;
            if (CHECK) {
                const int qx = x + dx, qy = y + dy;
                if (qx < 0 || qy < 0 || qx >= W || qy >= H) continue;
            }
            atrous_tap<S, NS ? 2 : (MODE != 0 ? 1 : 0)>((cvp + dy * W) + dx, (gp + dy * W) + dx, log2h,
                                                        rden, g, lp, inv_dl2, T, a);
        }
    }
    const float inv = 1.0f / a.sw;
    atrous_store<S>(P, p, make_float4(a.sr * inv, a.sg * inv, a.sb * inv,
                                      MODE == 1 ? cp.w : a.sv * (inv * inv)),
                    cv_out, hist_out, rgb_out);
}


// One a-trous iteration for a tile of TX columns from x0 and TY rows y0, y0 + ys, ...,
// y0 + (TY - 1) ys of a W x H image, by a block of TX x TY threads.  With ys = the pass's step
// the vertical taps of one row are the rows of the others (adaptive-start pixels, at twice the
// step, stay on the same lattice), so a block touches TY + 4 tap rows instead of 5 TY.  Tiles
// lying two maximal steps (plus the gradient/prefilter pixel) inside the image take the path
// without bounds checks; the branch is uniform over the block.  NS as for atrous_pixel.  MASK:
// only the pixels whose 32x32 tile is set in `need` (need_tx tiles a row) are computed; the rest
// of cv_out keeps what it held.
template <int MODE, class S, int TX, int TY, bool NS, bool MASK = false>
__device__ __forceinline__ void atrous_tile(const Params& P, int W, int H, int iter, int x0, int y0,
                                            int ys, const typename S::Rec* __restrict__ cv_in,
                                            const float4* __restrict__ gbuf,
                                            const float* __restrict__ rough,
                                            typename S::Rec* __restrict__ cv_out,
                                            typename S::Rec* __restrict__ hist_out,
                                            float4* __restrict__ rgb_out,
                                            const unsigned char* __restrict__ need = nullptr,
                                            int need_tx = 0) {
    pdl_wait();
    const int x = x0 + threadIdx.x, y = y0 + threadIdx.y * ys;
    if (MASK && (x >= W || y >= H || !need[(y >> 5) * need_tx + (x >> 5)])) return;
    const int reach = 2 << (iter + (P.adaptive_start && rough != nullptr ? 1 : 0));
    const int rx = MODE == 2 ? 1 : reach, ry = MODE == 1 ? 1 : reach;
    const bool interior = x0 - rx >= 1 && x0 + TX - 1 + rx < W - 1 && y0 - ry >= 1 &&
                          y0 + (TY - 1) * ys + ry < H - 1;
    if (P.iter_budget && x < W && y < H && iter >= pass_budget(P, rough, y * W + x)) {
        // past its pass budget: the pixel keeps its input (its neighbours still read it)
        const int p = y * W + x;
        atrous_store<S>(P, p, S::ld_cv(cv_in, p), cv_out, hist_out, rgb_out);
        return;
    }
    if (interior) {
        const int lvl = iter + start_level(P, rough, y * W + x);
        if (MODE == 0) {
            // the 24-tap pass with the step as a constant: each case inlines its own copy, so
            // every tap address is a row pointer plus an immediate (measured faster; the
            // two-tap separable passes gain nothing from it)
            switch (lvl) {
#define SVGF_ATROUS_AT(L)                                                                         \
    case L:                                                                                       \
        atrous_pixel<MODE, S, false, NS>(P, W, H, 1 << L, x, y, cv_in, gbuf, cv_out, hist_out, rgb_out); \
        return;
                SVGF_ATROUS_AT(0)
                SVGF_ATROUS_AT(1)
                SVGF_ATROUS_AT(2)
                SVGF_ATROUS_AT(3)
                SVGF_ATROUS_AT(4)
                SVGF_ATROUS_AT(5)
#undef SVGF_ATROUS_AT
                default: break;
            }
        }
        atrous_pixel<MODE, S, false, NS>(P, W, H, 1 << lvl, x, y, cv_in, gbuf, cv_out, hist_out, rgb_out);
    } else if (x < W && y < H) {
        atrous_pixel<MODE, S, true, NS>(P, W, H, 1 << (iter + start_level(P, rough, y * W + x)), x, y,
                                    cv_in, gbuf, cv_out, hist_out, rgb_out);
    }
}

}  // namespace dev
}  // namespace svgf
