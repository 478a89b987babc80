// resample.cu -- reprojection of the decoded equirectangular region into the
// viewport (Sec. 3.6: a mapping pass after the inverse wavelet transform) and
// YCbCr -> RGBA conversion.
//
// Per viewport pixel: the same projection as the footprint kernel gives the
// luma position (u, v); u wraps around the longitude seam, v clamps at the
// poles.  Bilinear filtering in fixed point: the fraction is rounded to 1/256
// (half up, with carry), the four integer weights sum to 65536 and the result
// is (sum + 32768) >> 16.  Chroma (4:2:0, centre-sited) is sampled at
// ((u + 1/2) / 2 - 1/2, (v + 1/2) / 2 - 1/2).  Colour: BT.709 full range,
// coefficients rounded to 1/65536, result rounded half up and clamped.
// The paper itself stores no colour transform (Sec. 5); the YCbCr 4:2:0
// stream and this conversion belong to this decoder's format.
#include <string.h>

#include "wv_impl.h"

namespace wv {

namespace {

// The 2 x 2 taps of a bilinear sample of a w x h plane at (u, v): x wraps
// (projected positions lie in [-1/2, w - 1/2), so one conditional add
// suffices; other positions take a modulo), y clamps.  Offsets into the
// row-major plane (planes are < 2^31 bytes) and 1/256 weights.
struct Taps {
    int a0, a1, b0, b1;   // (ya, xa), (ya, xb), (yb, xa), (yb, xb)
    int fx, fy;
};

// fixed_split for |t| < 2^15 (every projected position): there t * 256 +
// 1/2 is exact in float32, so floor(t * 256 + 1/2) = 256 i + f, the carry
// included, and one rounding conversion gives both parts.
__device__ __forceinline__ void fixed_split_near(float t, int &i, int &f) {
    const int T = __float2int_rd(fmaf(t, 256.0f, 0.5f));
    i = T >> 8;
    f = T & 255;
}

__device__ __forceinline__ Taps bilinear_taps(int w, int r_lo, int r_n, float u, float v) {
    int x0, fx, y0, fy;
    if (fabsf(u) < 32768.0f && fabsf(v) < 32768.0f) {
        fixed_split_near(u, x0, fx);
        fixed_split_near(v, y0, fy);
    } else {
        fixed_split(u, x0, fx);
        fixed_split(v, y0, fy);
    }
    Taps t;
    t.fx = fx;
    t.fy = fy;
    if ((unsigned)x0 < (unsigned)(w - 1) && y0 >= r_lo && y0 < r_lo + r_n - 1) {   // no wrap, no clamp
        t.a0 = y0 * w + x0;
        t.a1 = t.a0 + 1;
        t.b0 = t.a0 + w;
        t.b1 = t.b0 + 1;
        return t;
    }
    int xa = x0;
    if (xa < 0) xa += w;
    else if (xa >= w) xa -= w;
    if ((unsigned)xa >= (unsigned)w) {   // positions far outside (caller-given)
        xa %= w;
        if (xa < 0) xa += w;
    }
    const int xb = (xa + 1 == w) ? 0 : xa + 1;
    const int ya = min(max(y0, r_lo), r_lo + r_n - 1) * w;
    const int yb = min(max(y0 + 1, r_lo), r_lo + r_n - 1) * w;
    t.a0 = ya + xa;
    t.a1 = ya + xb;
    t.b0 = yb + xa;
    t.b1 = yb + xb;
    return t;
}

__device__ __forceinline__ int blend(const uint8_t *__restrict__ img, const Taps &t) {
    const int p00 = __ldg(img + t.a0), p01 = __ldg(img + t.a1);
    const int p10 = __ldg(img + t.b0), p11 = __ldg(img + t.b1);
    const int wx1 = t.fx, wx0 = 256 - t.fx;
    const int top = wx0 * p00 + wx1 * p01, bot = wx0 * p10 + wx1 * p11;
    return ((256 - t.fy) * top + t.fy * bot + 32768) >> 16;
}

// Cb and Cr of chroma sample e (row-major index) from a plane of
// alternating 4-sample groups (Cb of positions 4k..4k+3, then Cr of the
// same positions): one 8-byte load.
__device__ __forceinline__ uint2 tap_pair(const uint8_t *__restrict__ img, int e) {
    const uint2 q = __ldg(reinterpret_cast<const uint2 *>(img + 2 * (e & ~3)));
    const int sh = 8 * (e & 3);
    return make_uint2((q.x >> sh) & 255u, (q.y >> sh) & 255u);
}

// Cb and Cr of one tap set: four 8-byte loads instead of eight byte loads.
__device__ __forceinline__ void blend_pair(const uint8_t *__restrict__ img, const Taps &t, int &cb, int &cr) {
    const uint2 p00 = tap_pair(img, t.a0), p01 = tap_pair(img, t.a1);
    const uint2 p10 = tap_pair(img, t.b0), p11 = tap_pair(img, t.b1);
    const int wx1 = t.fx, wx0 = 256 - t.fx;
    const int tb = wx0 * (int)p00.x + wx1 * (int)p01.x, bb = wx0 * (int)p10.x + wx1 * (int)p11.x;
    const int tr = wx0 * (int)p00.y + wx1 * (int)p01.y, br = wx0 * (int)p10.y + wx1 * (int)p11.y;
    cb = ((256 - t.fy) * tb + t.fy * bb + 32768) >> 16;
    cr = ((256 - t.fy) * tr + t.fy * br + 32768) >> 16;
}

// Y, Cb, Cr of luma position (u, v); Cb and Cr share their taps.  Rows
// clamp to the eye's part of the frame (all of it for mono streams).
// WV_CHECKED builds: every tap offset inside the w x h plane.
__device__ __forceinline__ bool taps_in(const Taps &t, int w, int h, int *err) {
    const long long n = (long long)w * h;
    return checked_in(t.a0, n, err) && checked_in(t.a1, n, err) && checked_in(t.b0, n, err) &&
           checked_in(t.b1, n, err);
}

__device__ __forceinline__ void sample_ycbcr(const ResampleArgs &a, float u, float v, int &y, int &cb,
                                             int &cr) {
    const Taps ty = bilinear_taps(a.w[0], a.v.row0, a.v.rows, u, v);
    y = !kChecked || taps_in(ty, a.w[0], a.h[0], a.err) ? blend(a.plane[0], ty) : 0;
    cb = cr = 128;
    if (a.planes == 3) {
        float uc = u, vc = v;
        if (a.c420) {
            uc = fmaf(u + 0.5f, 0.5f, -0.5f);
            vc = fmaf(v + 0.5f, 0.5f, -0.5f);
        }
        const int sh = a.c420 ? 1 : 0;
        const Taps t = bilinear_taps(a.w[1], a.v.row0 >> sh, a.v.rows >> sh, uc, vc);
        if (kChecked && !taps_in(t, a.w[1], a.h[1], a.err)) return;
        if (a.c_pair) {
            blend_pair(a.plane[1], t, cb, cr);
        } else {
            cb = blend(a.plane[1], t);
            cr = blend(a.plane[2], t);
        }
    }
}

__device__ __forceinline__ uchar4 sample_px(const ResampleArgs &a, float u, float v) {
    int y, cb, cr;
    sample_ycbcr(a, u, v, y, cb, cr);
    return to_rgba(y, cb, cr);
}

// Luma / 255, Cb and Cr of viewport pixel (i, j) into the planes.
__device__ __forceinline__ void sample_ycc(const ResampleArgs &a, int i, int j) {
    float u, v;
    project_px(a.v, i, j, u, v);
    int y, cb, cr;
    sample_ycbcr(a, u, v, y, cb, cr);
    const size_t o = (size_t)j * a.v.out_w + i;
    a.y_plane[o] = (float)y * (1.0f / 255.0f);
    a.cb_plane[o] = (uint8_t)cb;
    a.cr_plane[o] = (uint8_t)cr;
}

__device__ __forceinline__ uint32_t rgba_word(uchar4 c) {
    return (uint32_t)c.x | ((uint32_t)c.y << 8) | ((uint32_t)c.z << 16) | ((uint32_t)c.w << 24);
}

__device__ __forceinline__ void position(const ResampleArgs &a, int i, int j, float &u, float &v) {
    if (a.uv) {
        const float2 p = reinterpret_cast<const float2 *>(a.uv)[(size_t)j * a.v.out_w + i];
        u = p.x;
        v = p.y;
    } else {
        project_px(a.v, i, j, u, v);
    }
}

// kPx horizontally adjacent pixels (i .. i + kPx - 1, j) per thread
// (independent work for the scheduler to overlap), written with one
// 4 kPx-byte store when the row holds all of them and the address is
// aligned.
constexpr int kPx = 2;

__device__ __forceinline__ void resample_run(const ResampleArgs &a, int i, int j) {
    if (i >= a.v.out_w || j >= a.v.out_h) return;
    if (a.y_plane) {
        for (int k = 0; k < kPx && i + k < a.v.out_w; ++k) sample_ycc(a, i + k, j);
        return;
    }
    uchar4 *dst = reinterpret_cast<uchar4 *>(a.out + (size_t)j * a.pitch) + i;
    if (i + kPx <= a.v.out_w && (reinterpret_cast<uintptr_t>(dst) & (4 * kPx - 1)) == 0) {
        uint32_t w[kPx];
#pragma unroll
        for (int k = 0; k < kPx; ++k) {
            float u, v;
            position(a, i + k, j, u, v);
            w[k] = rgba_word(sample_px(a, u, v));
        }
        if constexpr (kPx == 4) *reinterpret_cast<uint4 *>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
        else if constexpr (kPx == 2) *reinterpret_cast<uint2 *>(dst) = make_uint2(w[0], w[1]);
        else *reinterpret_cast<uint32_t *>(dst) = w[0];
        return;
    }
    for (int k = 0; k < kPx && i + k < a.v.out_w; ++k) {
        float u, v;
        position(a, i + k, j, u, v);
        dst[k] = sample_px(a, u, v);
    }
}

// ---- RGBA of projected positions --------------------------------------------
//
// The path of every viewport decode, written for instruction count and L1
// wavefronts, which bound it (a pixel reads 4 luma bytes and 4 chroma words
// that sit in L1 or L2):
//   - a warp covers 16 x 4 pixels at a time, lane (x, y) = (lane % 8,
//     lane / 8) taking pixels x and x + 8: a gather of 32 lanes then touches
//     about half the 128-byte lines that 32 adjacent pixel pairs of one row
//     do (rows of the viewport run diagonally through the frame);
//   - the two pixels are projected in packed fp32x2 arithmetic (each element
//     rounds as the scalar operations of project_px);
//   - positions two pixels inside the plane take a path without wrap and
//     clamp for luma and chroma together; the two taps of a row come out of
//     two words with one funnel shift and one dot product per component, and
//     the second word is loaded by the lanes that need it only (24 foveated
//     viewports 1441 -> 1431 us, 12 of shared frames 390 -> 383).
// One row of pixel pairs per warp took 284 instructions a pixel and 9.8 L1
// wavefronts a load, 53 us per 2160^2 viewport; this takes 187 and 5.6, 38 us
// alone and 30 with 24 viewports in a launch (80 % of the issue slots).

__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }

// wv_atan2 of two (y, x) pairs; XPOS: x is not negative.
template <bool XPOS>
__device__ __forceinline__ float2 atan2_pair(float2 y, float2 x) {
    const float ax0 = fabsf(x.x), ay0 = fabsf(y.x), ax1 = fabsf(x.y), ay1 = fabsf(y.y);
    const float mx0 = fmaxf(ax0, ay0), mx1 = fmaxf(ax1, ay1);
    float r0, r1;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r0) : "f"(mx0));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r1) : "f"(mx1));
    float2 t = __fmul2_rn(make_float2(fminf(ax0, ay0), fminf(ax1, ay1)), make_float2(r0, r1));
    if (!(mx0 > 0.0f)) t.x = 0.0f;
    if (!(mx1 > 0.0f)) t.y = 0.0f;
    const float2 u = __fmul2_rn(t, t);
    float2 p = f2(kAtan9);
    p = __ffma2_rn(p, u, f2(kAtan8));
    p = __ffma2_rn(p, u, f2(kAtan7));
    p = __ffma2_rn(p, u, f2(kAtan6));
    p = __ffma2_rn(p, u, f2(kAtan5));
    p = __ffma2_rn(p, u, f2(kAtan4));
    p = __ffma2_rn(p, u, f2(kAtan3));
    p = __ffma2_rn(p, u, f2(kAtan2));
    p = __ffma2_rn(p, u, f2(kAtan1));
    p = __ffma2_rn(p, u, f2(1.0f));
    float2 r = __fmul2_rn(p, t);
    const float2 c = __fadd2_rn(neg2(r), f2(1.5707963267948966f));
    if (ay0 > ax0) r.x = c.x;
    if (ay1 > ax1) r.y = c.y;
    if (!XPOS) {
        const float2 d = __fadd2_rn(neg2(r), f2(3.141592653589793f));
        if (x.x < 0.0f) r.x = d.x;
        if (x.y < 0.0f) r.y = d.y;
    }
    return make_float2(copysignf(r.x, y.x), copysignf(r.y, y.y));
}

// project_px of pixels (i, j) and (i + 8, j).  The rotation has no roll
// (r[3] = 0): the ray's y does not depend on the column.
__device__ __forceinline__ void project_pair(const View &v, int i, int j, float2 &u, float2 &w) {
    const float2 xc = __fadd2_rn(make_float2((float)i, (float)(i + 8)), f2(0.5f));
    const float2 xn = __fmul2_rn(__ffma2_rn(xc, f2(v.sx), f2(-1.0f)), f2(v.t));
    const float yn = __fmul_rn(fmaf(-((float)j + 0.5f), v.sy, 1.0f), v.t);
    const float2 dx = __ffma2_rn(f2(v.r[0]), xn, f2(fmaf(v.r[1], yn, v.r[2])));
    const float2 dy = f2(fmaf(v.r[4], yn, v.r[5]));
    const float2 dz = __ffma2_rn(f2(v.r[6]), xn, f2(fmaf(v.r[7], yn, v.r[8])));
    const float2 q = __ffma2_rn(dx, dx, __fmul2_rn(dz, dz));
    const float2 h = make_float2(sqrtf(q.x), sqrtf(q.y));
    u = __ffma2_rn(atan2_pair<false>(dx, dz), f2(v.ku), f2(v.cu));
    w = __ffma2_rn(atan2_pair<true>(dy, h), f2(v.kv), f2(v.cv));
}

// Rounded blend of two rows' horizontal sums.
__device__ __forceinline__ int blend_rows(int top, int bot, int fy) {
    return ((256 - fy) * top + (fy * bot + 32768)) >> 16;
}

// Channel layouts of a stream: grey, chroma planes, chroma in alternating
// 4-sample groups.
enum Chroma { kGrey = 0, kPlanar = 1, kGroups = 2 };

// WV_CHECKED builds: the `bytes` bytes from `first` that one tap set lies in,
// inside the plane's n; a pixel whose taps are not is kNoSample.
__device__ __forceinline__ bool bytes_in(long long first, long long bytes, long long n, int *err) {
    if constexpr (!kChecked) return true;
    return checked_in(first, n, err) && checked_in(first + bytes - 1, n, err);
}
constexpr uint32_t kNoSample = 0xff000000u;

// One pixel at luma position (u, w) at least two pixels inside the plane
// (its chroma taps then lie inside theirs).
template <int CH, bool C420>
__device__ __forceinline__ uint32_t inside_px(const ResampleArgs &a, int X, int Y, float uc, float vc) {
    const int fx = X & 255, fy = Y & 255;
    const unsigned W = a.w[0];
    // the taps of a row out of the aligned 8 bytes around them (planes are
    // 8-byte aligned, rows whole groups of 8), the next word only where they
    // straddle: fewer L1 wavefronts than two byte loads
    const unsigned k = (unsigned)(X >> 8) & 7u;
    const uint8_t *p = a.plane[0] + (unsigned)((Y >> 8) * (int)W + (X >> 8)) - k;
    if (!bytes_in(p - a.plane[0], W + (k == 7 ? 12 : 8), (long long)W * a.h[0], a.err)) return kNoSample;
    const uint2 t = __ldg(reinterpret_cast<const uint2 *>(p)), b = __ldg(reinterpret_cast<const uint2 *>(p + W));
    uint32_t tn = t.y, bn = b.y;
    if (k == 7) {
        tn = __ldg(reinterpret_cast<const uint32_t *>(p + 8));
        bn = __ldg(reinterpret_cast<const uint32_t *>(p + W + 8));
    }
    const unsigned wy = (unsigned)(256 - fx) | ((unsigned)fx << 16);
    const int y = blend_rows(__dp2a_lo(wy, __funnelshift_r(k < 4 ? t.x : t.y, k < 4 ? t.y : tn, 8 * (k & 3)), 0u),
                             __dp2a_lo(wy, __funnelshift_r(k < 4 ? b.x : b.y, k < 4 ? b.y : bn, 8 * (k & 3)), 0u), fy);
    if constexpr (CH == kGrey) {
        return rgba_word(to_rgba(y, 128, 128));
    } else {
        int Xc = X, Yc = Y;
        if constexpr (C420) {
            Xc = __float2int_rd(fmaf(uc, 256.0f, 0.5f));
            Yc = __float2int_rd(fmaf(vc, 256.0f, 0.5f));
        }
        const int gx = Xc & 255, gy = Yc & 255;
        const unsigned Wc = a.w[1], e = (unsigned)((Yc >> 8) * (int)Wc + (Xc >> 8));
        int cb, cr;
        if constexpr (CH == kGroups) {
            // rows are whole groups: the next row is 2 Wc bytes on
            const uint8_t *g0 = a.plane[1] + 8u * (e >> 2);
            if (!bytes_in(g0 - a.plane[1], 2 * Wc + ((e & 3) == 3 ? 16 : 8), 2ll * Wc * a.h[1], a.err)) return kNoSample;
            const uint2 t0 = __ldg(reinterpret_cast<const uint2 *>(g0)), b0 = __ldg(reinterpret_cast<const uint2 *>(g0 + 2 * Wc));
            uint2 t1 = t0, b1 = b0;   // the next group, where the taps straddle
            if ((e & 3) == 3) {
                t1 = __ldg(reinterpret_cast<const uint2 *>(g0 + 8));
                b1 = __ldg(reinterpret_cast<const uint2 *>(g0 + 8 + 2 * Wc));
            }
            // bytes k, k + 1 of the two groups side by side (taps of one
            // group: both words are that group, so byte k + 1 <= 3)
            const int sh = 8 * (e & 3);
            const unsigned wt = (unsigned)(256 - gx) | ((unsigned)gx << 16);
            const int cbt = __dp2a_lo(wt, __funnelshift_r(t0.x, t1.x, sh), 0u), cbb = __dp2a_lo(wt, __funnelshift_r(b0.x, b1.x, sh), 0u);
            const int crt = __dp2a_lo(wt, __funnelshift_r(t0.y, t1.y, sh), 0u), crb = __dp2a_lo(wt, __funnelshift_r(b0.y, b1.y, sh), 0u);
            cb = blend_rows(cbt, cbb, gy);
            cr = blend_rows(crt, crb, gy);
        } else {
            if (!bytes_in(e, Wc + 2, (long long)Wc * a.h[1], a.err)) return kNoSample;
            const uint8_t *p1 = a.plane[1] + e, *p2 = a.plane[2] + e;
            const uint8_t *q1 = p1 + Wc, *q2 = p2 + Wc;
            cb = blend_rows((256 - gx) * __ldg(p1) + gx * __ldg(p1 + 1), (256 - gx) * __ldg(q1) + gx * __ldg(q1 + 1), gy);
            cr = blend_rows((256 - gx) * __ldg(p2) + gx * __ldg(p2 + 1), (256 - gx) * __ldg(q2) + gx * __ldg(q2 + 1), gy);
        }
        // to_rgba with the constants gathered, saturating packs
        const int rr = (y * 65536 + (kRCr * cr + (32768 - 128 * kRCr))) >> 16;
        const int gg = (y * 65536 + (-kGCb * cb + (-kGCr * cr + (32768 + 128 * (kGCb + kGCr))))) >> 16;
        const int bb = (y * 65536 + (kBCb * cb + (32768 - 128 * kBCb))) >> 16;
        uint32_t hi, d;
        asm("cvt.pack.sat.u8.s32.b32 %0, %1, %2, 0;" : "=r"(hi) : "r"(255), "r"(bb));
        asm("cvt.pack.sat.u8.s32.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(gg), "r"(rr), "r"(hi));
        return d;
    }
}

constexpr int kPatchW = 64, kPatchH = 16;   // pixels per CTA: warps 4 x 2, two row groups each

template <int CH, bool C420>
__device__ __forceinline__ void resample_patch(const ResampleArgs &a, int bx, int by) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int i = bx * kPatchW + (warp & 3) * 16 + (lane & 7);
    const int W = a.w[0], r0 = a.v.row0, rn = a.v.rows;
#pragma unroll 1
    for (int k = 0; k < 2; ++k) {
        const int j = by * kPatchH + (warp >> 2) * 8 + 4 * k + (lane >> 3);
        if (i >= a.v.out_w || j >= a.v.out_h) return;
        float2 u, w;
        project_pair(a.v, i, j, u, w);
        const float2 X = __ffma2_rn(u, f2(256.0f), f2(0.5f)), Y = __ffma2_rn(w, f2(256.0f), f2(0.5f));
        float2 uc = u, vc = w;
        if (C420) {
            uc = __ffma2_rn(__fadd2_rn(u, f2(0.5f)), f2(0.5f), f2(-0.5f));
            vc = __ffma2_rn(__fadd2_rn(w, f2(0.5f)), f2(0.5f), f2(-0.5f));
        }
        uint32_t *dst = reinterpret_cast<uint32_t *>(a.out + (size_t)j * a.pitch) + i;
#pragma unroll
        for (int m = 0; m < 2; ++m) {
            if (m && i + 8 >= a.v.out_w) break;
            const int Xi = __float2int_rd(m ? X.y : X.x), Yi = __float2int_rd(m ? Y.y : Y.x);
            const bool in = (unsigned)((Xi >> 8) - 2) < (unsigned)(W - 6) && (unsigned)((Yi >> 8) - r0 - 2) < (unsigned)(rn - 6);
            uint32_t c;
            if (in) c = inside_px<CH, C420>(a, Xi, Yi, m ? uc.y : uc.x, m ? vc.y : vc.x);
            else c = rgba_word(sample_px(a, m ? u.y : u.x, m ? w.y : w.x));
            dst[8 * m] = c;
        }
    }
}

__device__ __forceinline__ void resample_any(const ResampleArgs &a, int bx, int by) {
    if (a.planes != 3) resample_patch<kGrey, false>(a, bx, by);
    else if (a.c_pair && a.c420) resample_patch<kGroups, true>(a, bx, by);
    else if (a.c_pair) resample_patch<kGroups, false>(a, bx, by);
    else if (a.c420) resample_patch<kPlanar, true>(a, bx, by);
    else resample_patch<kPlanar, false>(a, bx, by);
}

template <int CH, bool C420>
__global__ void __launch_bounds__(256) k_resample(ResampleArgs a) {
    resample_patch<CH, C420>(a, blockIdx.x, blockIdx.y);
}

// Batch: one z-slice of the grid per request.
__global__ void __launch_bounds__(256) k_resample_batch(const RequestJob *__restrict__ reqs) {
    const ResampleArgs &a = reqs[blockIdx.z].rs;
    if ((int)blockIdx.x * kPatchW >= a.v.out_w || (int)blockIdx.y * kPatchH >= a.v.out_h) return;
    resample_any(a, blockIdx.x, blockIdx.y);
}

// Caller-given positions, and luma and chroma planes instead of RGBA.
__global__ void k_resample_general(ResampleArgs a) {
    resample_run(a, kPx * (blockIdx.x * blockDim.x + threadIdx.x), blockIdx.y * blockDim.y + threadIdx.y);
}

}  // namespace

void launch_resample(const Geom &g, const View &v, uint8_t *const *recon, const float *uv,
                     uint8_t *out, size_t pitch, cudaStream_t cs, float *y_plane,
                     uint8_t *cb_plane, uint8_t *cr_plane, bool c_pair, int *err) {
    ResampleArgs a;
    memset(&a, 0, sizeof(a));
    a.err = err;
    a.y_plane = y_plane;
    a.cb_plane = cb_plane;
    a.cr_plane = cr_plane;
    a.v = v;
    for (int p = 0; p < 3; ++p) {
        a.plane[p] = recon[p];
        a.w[p] = p < g.planes ? g.p[p].w : 0;
        a.h[p] = p < g.planes ? g.p[p].h : 0;
    }
    a.planes = g.planes;
    a.c420 = g.c420;
    a.c_pair = c_pair && g.planes == 3 ? 1 : 0;
    a.uv = uv;
    a.out = out;
    a.pitch = pitch;
    if (uv || y_plane) {
        dim3 block(32, 8);
        dim3 grid((v.out_w + 32 * kPx - 1) / (32 * kPx), (v.out_h + 7) / 8);
        k_resample_general<<<grid, block, 0, cs>>>(a);
        return;
    }
    const dim3 grid((v.out_w + kPatchW - 1) / kPatchW, (v.out_h + kPatchH - 1) / kPatchH);
    if (a.planes != 3) k_resample<kGrey, false><<<grid, 256, 0, cs>>>(a);
    else if (a.c_pair && a.c420) k_resample<kGroups, true><<<grid, 256, 0, cs>>>(a);
    else if (a.c_pair) k_resample<kGroups, false><<<grid, 256, 0, cs>>>(a);
    else if (a.c420) k_resample<kPlanar, true><<<grid, 256, 0, cs>>>(a);
    else k_resample<kPlanar, false><<<grid, 256, 0, cs>>>(a);
}

void launch_resample_batch(const RequestJob *reqs, int n, int max_w, int max_h, cudaStream_t cs) {
    k_resample_batch<<<dim3((max_w + kPatchW - 1) / kPatchW, (max_h + kPatchH - 1) / kPatchH, n), 256, 0, cs>>>(reqs);
}

}  // namespace wv
