// pr_display.cu -- the display step after shading (Sec. 3.1.1, "Display"):
// the foveated framebuffer image I_f becomes the display image
// I_u(x) = I_f(q^-1(x)).  Two methods, as in the paper:
//
//  - MIP + cubic: a MIP pyramid of I_f (2x2 box averages, sizes halved
//    with ceil, blocks cut by the border averaged over their texels) is
//    sampled tri-linearly at the level of detail of the largest stretch of
//    q^-1 at x times the size ratio, each level with a 3-tap cubic filter
//    (the nearest texel and its two neighbours per axis, cubic B-spline
//    weights normalised by their sum, clamped to the edge);
//  - projected 5x5: the framebuffer pixel that holds q^-1(x) and its 5x5
//    neighbourhood, weighted by a Gaussian reconstruction filter of the
//    display-space distance between x and q of each pixel centre,
//    normalised (the paper's projection of the display's reconstruction
//    filter into the foveated domain); weights are taken relative to a
//    near sample, whose factor cancels, so they cannot all underflow.
//
// One thread per display pixel; planar rgb in and out.  What a tap reads
// lies together: the pyramid's texels above level 0 are (r, g, b, 0), and the
// projected filter first makes a table of (scale of q, r, g, b) per
// framebuffer pixel (direct_taps: not for small displays without foveation).
#include <algorithm>
#include <cstring>

#include "pr_launch.h"

namespace pr {

constexpr int kMaxMipLevels = 16;  // 16384 x 16384 needs 15

struct MipPyramid {
    // level 0 = the framebuffer image (planar); the others in the call's
    // scratch, a texel's (r, g, b, 0) side by side
    const float *rgb;
    float4 *lev[kMaxMipLevels];
    int w0, h0;                       // size of level 0; level k has ceil(w0 / 2^k) x ceil(h0 / 2^k) texels
    int L;
};

// Size of level k along one axis: halving with ceil k times.
__host__ __device__ __forceinline__ int mip_size(int n, int k) { return (n + (1 << k) - 1) >> k; }

// Display-step constants of a view (by value into the kernel).
struct DisplayView {
    int W, H, Wd, Hd;
    int fov;             // foveated or joint mode: q is the power map, else the identity
    float fx, fy;        // fovea
    float alpha, inv_alpha;
    const float *p_lut;  // or: the sampled p (then alpha is unused)
    int p_n;
    float rW, rH;        // 1 / W, 1 / H, correctly rounded (pixel_centre)
    float rWd, rHd;      // 1 / Wd, 1 / Hd, the same
    float scale;         // max(W / Wd, H / Hd)
    float sigma;         // projected filter width, display pixels
};

// The 2x2 block's mean of texels a, b (b beside a), c, d (below), over the
// texels of the block that exist (xr: the right ones do, yr: the lower ones
// do).  Scaling by 1, 1/2 or 1/4 is exact.
__device__ __forceinline__ float mip_mean(float a, float b, float c, float d, bool xr, bool yr)
{
    if (xr)
        a += b;
    if (yr) {
        a += c;
        if (xr)
            a += d;
    }
    return a * ((xr ? 0.5f : 1.f) * (yr ? 0.5f : 1.f));
}

// Levels 1 .. kTileLevels of a pyramid, a 64 x 64 tile of level 0 per CTA:
// each level is formed from the one below in shared memory, so a frame's
// pyramid takes two launches instead of one per level (stereo HMD frame: 54
// us in eleven launches, most of them a few texels and a launch's latency).
// Level 0 is read once; the bound is that read (DRAM).
constexpr int kTileLevels = 6, kTileSide = 1 << kTileLevels, kTileThreads = 256;

__device__ __forceinline__ void mip_tile(const MipPyramid &pyr, int tx, int ty)
{
    __shared__ float s_a[3][kTileSide / 2 * (kTileSide / 2)], s_b[3][kTileSide / 4 * (kTileSide / 4)];
    const int W = pyr.w0, H = pyr.h0;
    const int top = min(kTileLevels, pyr.L - 1);
    if (top >= 1) {  // level 1 from the image
        constexpr int side = kTileSide / 2, per = side * side / kTileThreads;
        const int w = mip_size(W, 1), h = mip_size(H, 1);
        const unsigned plane = (unsigned)W * (unsigned)H;  // <= 2^28
#pragma unroll
        for (int i = 0; i < per; ++i) {
            const int t = threadIdx.x + i * kTileThreads;
            const int x = tx * side + t % side, y = ty * side + t / side;
            if (x >= w || y >= h)
                continue;
            const bool xr = 2 * x + 1 < W, yr = 2 * y + 1 < H;
            const float *p = pyr.rgb + (unsigned)(2 * y * W + 2 * x);
            float v[3];
#pragma unroll
            for (int c = 0; c < 3; ++c, p += plane) {
                const float *p1 = p + W;
                v[c] = mip_mean(__ldg(p), xr ? __ldg(p + 1) : 0.f, yr ? __ldg(p1) : 0.f, xr && yr ? __ldg(p1 + 1) : 0.f,
                                xr, yr);
                s_a[c][t] = v[c];
            }
            pyr.lev[1][(unsigned)(y * w + x)] = make_float4(v[0], v[1], v[2], 0.f);
        }
        __syncthreads();
    }
    for (int k = 2; k <= top; ++k) {
        const int side = kTileSide >> k, lg = kTileLevels - k;  // the tile's texels of this level
        const int w = mip_size(W, k), h = mip_size(H, k), wb = mip_size(W, k - 1), hb = mip_size(H, k - 1);
        for (int t = threadIdx.x; t < side * side; t += kTileThreads) {
            const int ly = t >> lg, lx = t & (side - 1);
            const int x = (tx << lg) + lx, y = (ty << lg) + ly;
            if (x >= w || y >= h)
                continue;
            const bool xr = 2 * x + 1 < wb, yr = 2 * y + 1 < hb;
            float v[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const float *p = (k & 1 ? s_b[c] : s_a[c]) + 4 * side * ly + 2 * lx;  // odd levels sit in s_a, even in s_b
                v[c] = mip_mean(p[0], p[1], p[2 * side], p[2 * side + 1], xr, yr);
                if (k & 1)
                    s_a[c][t] = v[c];
                else
                    s_b[c][t] = v[c];
            }
            pyr.lev[k][(unsigned)(y * w + x)] = make_float4(v[0], v[1], v[2], 0.f);
        }
        __syncthreads();
    }
}

// The levels above, one CTA per pyramid: a few texels each (level 6 of a
// 2160^2 image is 34^2).
__device__ __forceinline__ void mip_top(const MipPyramid &pyr)
{
    for (int k = kTileLevels + 1; k < pyr.L; ++k) {
        const int w = mip_size(pyr.w0, k), h = mip_size(pyr.h0, k);
        const int wb = mip_size(pyr.w0, k - 1), hb = mip_size(pyr.h0, k - 1);
        const float4 *src = pyr.lev[k - 1], none = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int t = threadIdx.x; t < w * h; t += blockDim.x) {
            const int y = t / w, x = t - y * w;
            const bool xr = 2 * x + 1 < wb, yr = 2 * y + 1 < hb;
            const float4 *p = src + (size_t)(2 * y) * wb + 2 * x;
            const float4 a = p[0], b = xr ? p[1] : none, c = yr ? p[wb] : none, d = xr && yr ? p[wb + 1] : none;
            pyr.lev[k][t] = make_float4(mip_mean(a.x, b.x, c.x, d.x, xr, yr), mip_mean(a.y, b.y, c.y, d.y, xr, yr),
                                        mip_mean(a.z, b.z, c.z, d.z, xr, yr), 0.f);
        }
        __syncthreads();  // this level is the next one's source
    }
}

__global__ void __launch_bounds__(kTileThreads) k_mip_tile(const MipPyramid pyr)
{
    mip_tile(pyr, blockIdx.x, blockIdx.y);
}

__global__ void __launch_bounds__(512) k_mip_top(const MipPyramid pyr) { mip_top(pyr); }

// x^e of q; the linear factor of alpha = 2 without the general power (some
// eighty instructions; the same bits).
__device__ __forceinline__ float radial_pow(float x, float e) { return e == 1.f ? x : powf(x, e); }

// 2^x by the special-function unit alone: exp2f scales its argument around
// results below 2^-126, which a weight beside a sum of at least 2^-24 may lose.
// Against 64 bits (128 M display pixels of 192 sizes, widths, zooms and warps)
// the mean error is 1.0728e-5 with it, with exp2f and with expf (1.0729e-5 with
// expf and every weight from the nearest sample): the rounding of the samples'
// locations decides.  Projected filter 126 against 132 (exp2f) and 138 us
// (expf), 1440 x 1600 to 1800 x 2000.
__device__ __forceinline__ float exp2_ftz(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// What a tap of the projected filter reads of a framebuffer pixel c: the
// factor (|e|/D)^(alpha - 1) that q scales its offset e from the fovea by
// (1 without foveation, where offsets are taken from 0), and its colour.
__global__ void k_tap_table(const DisplayView dv, const float *__restrict__ rgb,
                            float4 *__restrict__ table)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y;
    if (i >= dv.W)
        return;
    const unsigned o = (unsigned)(j * dv.W + i), plane = (unsigned)dv.W * (unsigned)dv.H;  // <= 2^28
    const float r0 = rgb[o], g0 = rgb[plane + o], b0 = rgb[2 * plane + o];
    float s = 1.f;
    if (dv.fov) {
        const float e0 = pixel_centre(i, dv.W, dv.rW) - dv.fx, e1 = pixel_centre(j, dv.H, dv.rH) - dv.fy,
                    r = sqrtf(fmaf(e0, e0, e1 * e1));
        const SampledP sp{dv.p_lut, dv.p_n};
        s = r > 0.f ? (dv.p_lut ? sp.p(r) / r : radial_pow(r * (1.f / kSqrt2), dv.alpha - 1.f)) : 0.f;
    }
    table[o] = make_float4(s, r0, g0, b0);
}

// Cubic B-spline weights of the taps at -1, 0, 1 for a sample at d in
// [-1/2, 1/2] from the middle one: 2/3 - x^2 + x^3 / 2 within one texel,
// (2 - x)^3 / 6 beyond.  With m = 1 - |d| the nearer side tap has x = m, the
// farther one 2 - x = m.
__device__ __forceinline__ void bspline_taps(float d, float (&w)[3])
{
    const float a = fabsf(d), m = 1.f - a;
    const float m2 = m * m, m3 = m2 * m;
    const float near = fmaf(0.5f, m3, 2.f / 3.f - m2), far = m3 * (1.f / 6.f);
    w[0] = d < 0.f ? near : far;
    w[1] = fmaf(fmaf(0.5f, a, -1.f), a * a, 2.f / 3.f);
    w[2] = d < 0.f ? far : near;
}

// 3-tap cubic sample of one level at texel coordinates (s, t): the three
// taps of each row first, then the rows.  kPlanar: level 0, the image;
// otherwise a level of interleaved texels, where one 16-byte load serves a
// tap's three channels.
struct Texels {
    const float *img;
    const float4 *lev;
    unsigned plane;  // <= 2^28
};

template <bool kPlanar>
__device__ __forceinline__ float3 texel(const Texels &tx, unsigned o)
{
    if (kPlanar)
        return make_float3(__ldg(tx.img + o), __ldg(tx.img + tx.plane + o), __ldg(tx.img + 2 * tx.plane + o));
    const float4 v = __ldg(tx.lev + o);
    return make_float3(v.x, v.y, v.z);
}

__device__ __forceinline__ float3 taps3(const float (&w)[3], float3 a, float3 b, float3 c)
{
    return make_float3(fmaf(w[0], a.x, fmaf(w[1], b.x, w[2] * c.x)), fmaf(w[0], a.y, fmaf(w[1], b.y, w[2] * c.y)),
                       fmaf(w[0], a.z, fmaf(w[1], b.z, w[2] * c.z)));
}

template <bool kPlanar>
__device__ __forceinline__ void sample3(const Texels &tx, int w, int h, float s, float t, float out[3])
{
    const float fs = floorf(s + 0.5f), ft = floorf(t + 0.5f);
    float wx[3], wy[3];
    bspline_taps(s - fs, wx);
    bspline_taps(t - ft, wy);
    const float inv = 1.f / ((wx[0] + wx[1] + wx[2]) * (wy[0] + wy[1] + wy[2]));  // sums of about 1
    const int is = (int)fs, it = (int)ft;
    float3 row[3];
    if (is >= 1 && is < w - 1 && it >= 1 && it < h - 1) {
        // inside: the taps are neighbours
        const unsigned o = (unsigned)((it - 1) * w + is - 1);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const unsigned ok = o + (unsigned)(k * w);
            row[k] = taps3(wx, texel<kPlanar>(tx, ok), texel<kPlanar>(tx, ok + 1), texel<kPlanar>(tx, ok + 2));
        }
    } else {
        const int x0 = min(max(is - 1, 0), w - 1), x1 = min(max(is, 0), w - 1), x2 = min(max(is + 1, 0), w - 1);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const unsigned r = (unsigned)(min(max(it - 1 + k, 0), h - 1) * w);
            row[k] = taps3(wx, texel<kPlanar>(tx, r + x0), texel<kPlanar>(tx, r + x1), texel<kPlanar>(tx, r + x2));
        }
    }
    out[0] = fmaf(wy[2], row[2].x, fmaf(wy[1], row[1].x, wy[0] * row[0].x)) * inv;
    out[1] = fmaf(wy[2], row[2].y, fmaf(wy[1], row[1].y, wy[0] * row[0].y)) * inv;
    out[2] = fmaf(wy[2], row[2].z, fmaf(wy[1], row[1].z, wy[0] * row[0].z)) * inv;
}

// Where the projected filter's taps come from: the table, or (kDirect) the
// image itself, where q scales by 1.
template <bool kDirect>
struct TapSource {
    using Texel = float4;
    static __device__ __forceinline__ const float4 *base(const float4 *tab, const float *) { return tab; }
    static __device__ __forceinline__ float4 tap(const float4 *t, unsigned) { return __ldg(t); }
};
template <>
struct TapSource<true> {
    using Texel = float;
    static __device__ __forceinline__ const float *base(const float4 *, const float *rgb) { return rgb; }
    static __device__ __forceinline__ float4 tap(const float *t, unsigned plane)
    {
        return make_float4(1.f, __ldg(t), __ldg(t + plane), __ldg(t + 2 * plane));
    }
};

// Display pixel (a, b) of a view.  kDirect (the projected filter without
// foveation): the taps come from the image, there is no table.  kNarrow: a
// filter so narrow (narrow_filter) that the rounding of two equally near samples'
// locations could make an exponent large and positive; it is cut at 1.
template <int kMethod, bool kDirect = false, bool kNarrow = false>
__device__ __forceinline__ void unfoveate_pixel(const DisplayView &dv, const MipPyramid &pyr,
                                                const float4 *__restrict__ tab, float *__restrict__ out, int a, int b)
{
    const float x0 = pixel_centre(a, dv.Wd, dv.rWd), x1 = pixel_centre(b, dv.Hd, dv.rHd);
    // u = q^-1(x): the offset from the fovea scaled by (|e|/D)^(1/alpha - 1)
    float u0 = x0, u1 = x1, tang = 1.f, stretch = 1.f;
    if (dv.fov) {
        const float e0 = x0 - dv.fx, e1 = x1 - dv.fy, r = sqrtf(fmaf(e0, e0, e1 * e1));
        if (dv.p_lut) {  // the sampled p: tangential stretch p^-1(r)/r, radial the slope of p^-1
            const SampledP sp{dv.p_lut, dv.p_n};
            const float radial = sp.dpinv(r);
            tang = r > 0.f ? sp.pinv(r) / r : radial;
            stretch = fmaxf(tang, radial);
        } else {
            tang = r > 0.f ? powf(r * (1.f / kSqrt2), dv.inv_alpha - 1.f) : INFINITY;
            stretch = fmaxf(tang, tang * dv.inv_alpha);
        }
        const float s = r > 0.f ? tang : 0.f;
        u0 = fmaf(e0, s, dv.fx);
        u1 = fmaf(e1, s, dv.fy);
    }
    float res[3];
    if (kMethod == PR_UNFOVEATE_MIP_CUBIC) {
        // level of detail: the largest stretch of q^-1 (tangential for alpha >= 1)
        float lambda = log2f(stretch * dv.scale);
        lambda = fminf(fmaxf(lambda, 0.f), (float)(pyr.L - 1));  // NaN-free: tang >= 0
        const int k0 = (int)floorf(lambda), k1 = min(k0 + 1, pyr.L - 1);
        const float f = lambda - (float)k0;
        float s0[3], s1[3];
        const int w0 = mip_size(dv.W, k0), h0 = mip_size(dv.H, k0);
        const Texels tx0{pyr.rgb, pyr.lev[k0], (unsigned)dv.W * (unsigned)dv.H};
        const float c0 = fmaf(u0, (float)w0, -0.5f), c1 = fmaf(u1, (float)h0, -0.5f);
        if (k0 == 0)
            sample3<true>(tx0, w0, h0, c0, c1, s0);
        else
            sample3<false>(tx0, w0, h0, c0, c1, s0);
        if (f > 0.f) {
            const int w1 = mip_size(dv.W, k1), h1 = mip_size(dv.H, k1);
            const Texels tx1{nullptr, pyr.lev[k1], 0u};  // f > 0: k1 = k0 + 1
            sample3<false>(tx1, w1, h1, fmaf(u0, (float)w1, -0.5f), fmaf(u1, (float)h1, -0.5f), s1);
            for (int c = 0; c < 3; ++c)
                res[c] = fmaf(f, s1[c] - s0[c], s0[c]);
        } else {
            for (int c = 0; c < 3; ++c)
                res[c] = s0[c];
        }
    } else {
        const int i = min(max((int)floorf(u0 * (float)dv.W), 0), dv.W - 1);
        const int j = min(max((int)floorf(u1 * (float)dv.H), 0), dv.H - 1);
        // The window's part inside the framebuffer.  Weights are taken
        // relative to a reference sample m, whose factor cancels in the
        // normalisation: exp(k2 (d^2 - d_m^2)) with d^2 - d_m^2 =
        // (d - d_m)(d + d_m) per axis, where d - d_m comes from the difference
        // of the two samples' display locations.  The window's centre serves
        // where k2 d^2 of it is above -16, with the weights scaled by 2^shift,
        // about its own weight: none then exceeds 2, so that colours up to the
        // largest float over 50 stay in range, and the sum is at least
        // 2^-24.  Display pixels farther from their centre sample (beyond the
        // framebuffer's disc, or a display of far more pixels) look for the
        // nearest sample first, whose weight is 1.  (Up to -60 and unscaled: the
        // same time, 128 us, but weights of e^60 overflowed colours above 1e11.)
        // k2 is bounded so that its products with Wd^2, Hd^2 <= 2^28 and
        // locations stay finite (the reference's own offset 0 times an
        // infinite factor is not a number): a filter of sigma 2e-15 display
        // pixels is as narrow as any below it.
        const int dx0 = max(-2, -i), dx1 = min(2, dv.W - 1 - i), dy0 = max(-2, -j), dy1 = min(2, dv.H - 1 - j);
        const float k2 = fmaxf(-0.5f / (dv.sigma * dv.sigma), -1e29f);
        const float fWd = (float)dv.Wd, fHd = (float)dv.Hd;
        const unsigned plane = (unsigned)dv.W * (unsigned)dv.H;  // <= 2^28
        // offsets from the fovea (from 0 without foveation, so that q = c)
        const float fx = dv.fov ? dv.fx : 0.f, fy = dv.fov ? dv.fy : 0.f;
        using Src = TapSource<kDirect>;
        const float sm = kDirect ? 1.f : __ldg(&tab[(unsigned)(j * dv.W + i)].x);
        float qm0 = fmaf(pixel_centre(i, dv.W, dv.rW) - fx, sm, fx), qm1 = fmaf(pixel_centre(j, dv.H, dv.rH) - fy, sm, fy);
        float shift;
        {
            const float d0 = (x0 - qm0) * fWd, d1 = (x1 - qm1) * fHd, e = k2 * fmaf(d0, d0, d1 * d1);
            shift = ceilf(e * 1.44269504f);
            if (e < -16.f) {
                shift = 0.f;
                float d2min = INFINITY;
                for (int dy = dy0; dy <= dy1; ++dy) {
                    const float4 *tr = tab + (unsigned)((j + dy) * dv.W + i);
                    const float e1 = pixel_centre(j + dy, dv.H, dv.rH) - fy;
                    for (int dx = dx0; dx <= dx1; ++dx) {
                        const float s = kDirect ? 1.f : __ldg(&tr[dx].x);
                        const float q0 = fmaf(pixel_centre(i + dx, dv.W, dv.rW) - fx, s, fx), q1 = fmaf(e1, s, fy);
                        const float f0 = (x0 - q0) * fWd, f1 = (x1 - q1) * fHd;
                        const float q2 = fmaf(f0, f0, f1 * f1);
                        if (q2 < d2min) {
                            d2min = q2;
                            qm0 = q0;
                            qm1 = q1;
                        }
                    }
                }
            }
        }
        // weight of a sample at q: 2^((qm - q)(2 x - qm - q) . (kw, kh) + shift)
        const float2 qm2 = make_float2(qm0, qm1), far = make_float2(2.f * x0 - qm0, 2.f * x1 - qm1);
        const float kw = k2 * 1.44269504f * fWd * fWd, kh = k2 * 1.44269504f * fHd * fHd;  // exp as a power of two
        float acc[3] = {0.f, 0.f, 0.f}, wsum = 0.f;
        const float2 fov = make_float2(fx, fy);
        auto tap = [&](float e0, float e1, float4 c) {
            const float2 minus = make_float2(-1.f, -1.f), q = __ffma2_rn(make_float2(e0, e1), make_float2(c.x, c.x), fov);
            const float2 t = __fmul2_rn(__ffma2_rn(q, minus, qm2), __ffma2_rn(q, minus, far));
            const float x = fmaf(t.x, kw, fmaf(t.y, kh, shift));
            const float w = exp2_ftz(kNarrow ? fminf(x, 1.f) : x);
            wsum += w;
            acc[0] = fmaf(w, c.y, acc[0]);
            acc[1] = fmaf(w, c.z, acc[1]);
            acc[2] = fmaf(w, c.w, acc[2]);
        };
        const typename Src::Texel *tr = Src::base(tab, pyr.rgb) + (unsigned)((j + dy0) * dv.W + i + dx0);
        if (dx1 - dx0 == 4) {  // five taps a row (all but two columns at either side), their loads in flight together
            float e0[5];
#pragma unroll
            for (int dx = 0; dx < 5; ++dx)
                e0[dx] = pixel_centre(i - 2 + dx, dv.W, dv.rW) - fx;
#pragma unroll 1
            for (int dy = dy0; dy <= dy1; ++dy, tr += dv.W) {
                const float e1 = pixel_centre(j + dy, dv.H, dv.rH) - fy;
#pragma unroll
                for (int dx = 0; dx < 5; ++dx)
                    tap(e0[dx], e1, Src::tap(tr + dx, plane));
            }
        } else {
            for (int dy = dy0; dy <= dy1; ++dy, tr += dv.W) {
                const float e1 = pixel_centre(j + dy, dv.H, dv.rH) - fy;
                for (int dx = dx0; dx <= dx1; ++dx)
                    tap(pixel_centre(i + dx, dv.W, dv.rW) - fx, e1, Src::tap(tr + (dx - dx0), plane));
            }
        }
        const float inv = 1.f / wsum;
        for (int c = 0; c < 3; ++c)
            res[c] = acc[c] * inv;
    }
    const size_t dplane = (size_t)dv.Wd * dv.Hd, o = (size_t)b * dv.Wd + a;
    out[o] = res[0];
    out[dplane + o] = res[1];
    out[2 * dplane + o] = res[2];
}

// CTAs of the display kernels: 32 x 8 display pixels, six per SM, a warp's
// pixels 16 x 2.  Bound: the L1 data pipe for the MIP form (79 % busy, issue 66
// %), issue for the projected filter (84 %, L1 64 %).  q^-1
// is curved, so a row of 32 display pixels reads up to fifteen rows of
// texels, and every texel row of a tap is a cache line of its own: squarer
// warps meet fewer (32 x 1 / 16 x 2 / 8 x 4 with planar texels: projected
// filter, 1440 x 1600 to 1800 x 2000, 171 / 152 / 156 us a pass; MIP, 16
// views, 414 / 408 / 426), and so does one 16-byte load per tap instead of
// one per channel (and for q): 152 -> 132 and 408 -> 391 us.  Six CTAs per
// SM (40 registers) against four and five: 126 / 132 / 130 and 383 / 394 /
// 391 us.
constexpr int kDispW = 32, kDispH = 8;
constexpr int kWarpW = 16, kWarpH = 32 / kWarpW;
constexpr int kDispCtas = 6;

__device__ __forceinline__ int2 disp_pixel(int bx, int by)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, per = kDispW / kWarpW;
    return make_int2(bx * kDispW + (w % per) * kWarpW + lane % kWarpW, by * kDispH + (w / per) * kWarpH + lane / kWarpW);
}

template <int kMethod, bool kDirect = false, bool kNarrow = false>
__global__ void __launch_bounds__(kDispW *kDispH, kDispCtas) k_unfoveate(const DisplayView dv, const MipPyramid pyr,
                                                             const float4 *__restrict__ tab, float *__restrict__ out)
{
    const int2 at = disp_pixel(blockIdx.x, blockIdx.y);
    const int a = at.x, b = at.y;
    if (a >= dv.Wd || b >= dv.Hd)
        return;
    unfoveate_pixel<kMethod, kDirect, kNarrow>(dv, pyr, tab, out, a, b);
}

// ---- the batched display step (MIP): many views, two launches for their
// pyramids and one for the display pixels of all views.  A launch's blocks
// are numbered view after view (blk[q] = first block of view q, blk[n] =
// all); a block finds its view by a warp's ballot and runs the same
// per-texel and per-pixel code as the single-view kernels, so the results
// are the same.
struct DisplayBatchView {
    DisplayView dv;
    MipPyramid pyr;
    float *out;
    // block / blocks per row as (block * mul) >> 40: the round-up reciprocals
    // of Granlund and Montgomery (1994), exact for blocks < 2^23 and rows of
    // at most 2^11
    unsigned long long mul_disp, mul_tile;
};

// The view of block b (the same for every lane): the warp compares 32
// offsets at a time (find_view_warp).  Called by whole warps.
__device__ __forceinline__ int block_view(const long long *__restrict__ blk, int n, long long b)
{
    return find_view_warp(blk, n, b);
}

// Levels 1 .. kTileLevels of every view.
__global__ void __launch_bounds__(kTileThreads) k_mip_tile_batch(const DisplayBatchView *__restrict__ tab,
                                                                 const long long *__restrict__ blk, int n)
{
    const int q = block_view(blk, n, blockIdx.x);
    const DisplayBatchView &e = tab[q];
    const unsigned b = (unsigned)(blockIdx.x - blk[q]);
    const int ty = (int)((b * e.mul_tile) >> 40), tx = (int)b - ty * ((e.dv.W + kTileSide - 1) / kTileSide);
    mip_tile(e.pyr, tx, ty);
}

// The levels above (blockIdx.x: view).
__global__ void __launch_bounds__(512) k_mip_top_batch(const DisplayBatchView *__restrict__ tab)
{
    mip_top(tab[blockIdx.x].pyr);
}

// The display pixels of every view.
__global__ void __launch_bounds__(kDispW *kDispH, kDispCtas) k_unfoveate_mip_batch(const DisplayBatchView *__restrict__ tab,
                                                                          const long long *__restrict__ blk, int n)
{
    const int q = block_view(blk, n, blockIdx.x);
    const DisplayBatchView &e = tab[q];
    const DisplayView dv = e.dv;
    const unsigned t = (unsigned)(blockIdx.x - blk[q]);
    const int by = (int)((t * e.mul_disp) >> 40), bx = (int)t - by * ((dv.Wd + kDispW - 1) / kDispW);
    const int2 at = disp_pixel(bx, by);
    const int a = at.x, b = at.y;
    if (a >= dv.Wd || b >= dv.Hd)
        return;
    unfoveate_pixel<PR_UNFOVEATE_MIP_CUBIC>(dv, e.pyr, nullptr, e.out, a, b);
}

int mip_level_count(int W, int H)
{
    int L = 1;
    while (W > 1 || H > 1) {
        W = (W + 1) / 2;
        H = (H + 1) / 2;
        ++L;
    }
    return L;
}

// Scratch floats of a view's display step, four per texel: the levels above
// the image (MIP), or the tap table of the projected filter.
size_t display_scratch_floats(int method, int W, int H)
{
    if (method == PR_UNFOVEATE_PROJECTED)
        return (size_t)4 * W * H;
    size_t n = 0;
    while (W > 1 || H > 1) {
        W = (W + 1) / 2;
        H = (H + 1) / 2;
        n += (size_t)4 * W * H;
    }
    return n;
}

// Level pointers of a pyramid with its levels 1 .. L - 1 at `p` one after the
// other; false if it has more than kMaxMipLevels.
static bool fill_pyramid(MipPyramid &pyr, int W, int H, const float *rgb, float *p)
{
    pyr.L = mip_level_count(W, H);
    if (pyr.L > kMaxMipLevels)
        return false;
    pyr.w0 = W;
    pyr.h0 = H;
    pyr.rgb = rgb;
    pyr.lev[0] = nullptr;
    for (int k = 1; k < pyr.L; ++k) {
        pyr.lev[k] = reinterpret_cast<float4 *>(p);
        p += (size_t)4 * mip_size(W, k) * mip_size(H, k);
    }
    return true;
}

// Whether the projected filter takes its taps from the image: without
// foveation q is the identity, and the table (28 bytes moved per framebuffer
// pixel, to save two of a tap's three loads) pays only for about as many display
// pixels as the framebuffer has.  2160 x 2160 and 4096 x 4096, table / image, at
// 1/16 of its side 40 / 12 and 99 / 16 us, 1/4 51 / 20 and 145 / 54, 1/2 65 / 38
// and 196 / 111, 0.6 77 / 49 and 240 / 152; at the full side the image loses (125
// / 142 and 411 / 477 in a slower form of it, 108 / 96 at 0.8 of the side).
static bool direct_taps(const DisplayView &dv)
{
    return !dv.fov && 3ll * dv.Wd * dv.Hd <= 2ll * dv.W * dv.H;
}

// Whether a weight's exponent (qm - q)(2x - qm - q) k, k = Wd^2 / (2 sigma^2
// ln 2), of two samples equally near to x may come out as large as 10: |qm - q|
// is at most ten framebuffer pixels, and the second factor, 0 but for rounding,
// 2^-22.  The weights of wider filters need no cut, an instruction per tap.
static bool narrow_filter(const DisplayView &dv)
{
    const double k = 0.7214 * std::max((double)dv.Wd * dv.Wd, (double)dv.Hd * dv.Hd) / ((double)dv.sigma * dv.sigma);
    return 10.0 / std::min(dv.W, dv.H) * 2.4e-7 * k > 10.0;
}

cudaError_t launch_unfoveate(int method, int W, int H, int mode, float fx, float fy, float alpha, const float *p_lut,
                             int p_n, int Wd, int Hd, float sigma, const float *rgb, float *scratch, float *out,
                             cudaStream_t st)
{
    DisplayView dv;
    dv.W = W;
    dv.H = H;
    dv.Wd = Wd;
    dv.Hd = Hd;
    dv.rW = 1.f / (float)W;
    dv.rH = 1.f / (float)H;
    dv.rWd = 1.f / (float)Wd;
    dv.rHd = 1.f / (float)Hd;
    dv.fov = mode == PR_FOVEATED || mode == PR_BOTH;
    dv.fx = fx;
    dv.fy = fy;
    dv.alpha = alpha;
    dv.inv_alpha = 1.f / alpha;
    dv.p_lut = p_lut;
    dv.p_n = p_n;
    dv.scale = fmaxf((float)W / (float)Wd, (float)H / (float)Hd);
    dv.sigma = sigma;
    MipPyramid pyr;
    std::memset(&pyr, 0, sizeof pyr);
    const dim3 blk(kDispW * kDispH), grd((unsigned)((Wd + kDispW - 1) / kDispW), (unsigned)((Hd + kDispH - 1) / kDispH));
    if (method == PR_UNFOVEATE_MIP_CUBIC) {
        if (!fill_pyramid(pyr, W, H, rgb, scratch))
            return cudaErrorInvalidValue;
        if (pyr.L > 1)
            k_mip_tile<<<dim3((unsigned)((W + kTileSide - 1) / kTileSide), (unsigned)((H + kTileSide - 1) / kTileSide)),
                         kTileThreads, 0, st>>>(pyr);
        if (pyr.L > kTileLevels + 1)
            k_mip_top<<<1, 512, 0, st>>>(pyr);
        k_unfoveate<PR_UNFOVEATE_MIP_CUBIC><<<grd, blk, 0, st>>>(dv, pyr, nullptr, out);
    } else {
        pyr.rgb = rgb;
        const bool narrow = narrow_filter(dv);
        if (direct_taps(dv)) {
            if (narrow)
                k_unfoveate<PR_UNFOVEATE_PROJECTED, true, true><<<grd, blk, 0, st>>>(dv, pyr, nullptr, out);
            else
                k_unfoveate<PR_UNFOVEATE_PROJECTED, true><<<grd, blk, 0, st>>>(dv, pyr, nullptr, out);
            return cudaGetLastError();
        }
        float4 *tab = reinterpret_cast<float4 *>(scratch);
        const dim3 gq((unsigned)((W + 255) / 256), (unsigned)H);
        k_tap_table<<<gq, 256, 0, st>>>(dv, rgb, tab);
        if (narrow)
            k_unfoveate<PR_UNFOVEATE_PROJECTED, false, true><<<grd, blk, 0, st>>>(dv, pyr, tab, out);
        else
            k_unfoveate<PR_UNFOVEATE_PROJECTED><<<grd, blk, 0, st>>>(dv, pyr, tab, out);
    }
    return cudaGetLastError();
}

size_t display_batch_scratch_floats(int method, const DisplayEntry *e, int n)
{
    size_t f = 0;
    for (int q = 0; q < n; ++q) {
        const size_t v = display_scratch_floats(method, e[q].W, e[q].H);
        // every view's pyramid, side by side; one view's tap table at a time
        f = method == PR_UNFOVEATE_MIP_CUBIC ? f + v : std::max(f, v);
    }
    return f;
}

// Table layout (MIP): n DisplayBatchView, then two arrays of n + 1 block
// offsets: the display pixels', then the pyramid tiles'.
size_t display_batch_table_bytes(int n)
{
    const size_t views = ((sizeof(DisplayBatchView) * (size_t)n) + 15) & ~(size_t)15;
    return views + sizeof(long long) * 2 * (size_t)(n + 1);
}

cudaError_t launch_unfoveate_batch(int method, float sigma, const DisplayEntry *e, int n, float *scratch,
                                   void *h_table, void *d_table, cudaStream_t st)
{
    if (n <= 0)
        return cudaSuccess;
    if (method == PR_UNFOVEATE_PROJECTED) {
        // view after view with the single-view kernels (tap table, then the
        // filter), each view's table in the same scratch (with a table of 8
        // bytes per pixel, that of all views at once, or of L2-sized groups,
        // was measured slower)
        for (int q = 0; q < n; ++q) {
            const cudaError_t err = launch_unfoveate(method, e[q].W, e[q].H, e[q].mode, e[q].fx, e[q].fy, e[q].alpha,
                                                     e[q].p_lut, e[q].p_n, e[q].Wd, e[q].Hd, sigma, e[q].rgb, scratch,
                                                     e[q].out, st);
            if (err != cudaSuccess)
                return err;
        }
        return cudaSuccess;
    }
    const size_t views_bytes = ((sizeof(DisplayBatchView) * (size_t)n) + 15) & ~(size_t)15;
    DisplayBatchView *tab = static_cast<DisplayBatchView *>(h_table);
    long long *blk = reinterpret_cast<long long *>(static_cast<char *>(h_table) + views_bytes);
    bool any_tiles = false, any_top = false;
    float *p = scratch;
    for (int q = 0; q < n; ++q) {
        DisplayBatchView &t = tab[q];
        std::memset(&t, 0, sizeof t);
        DisplayView &dv = t.dv;
        dv.W = e[q].W;
        dv.H = e[q].H;
        dv.Wd = e[q].Wd;
        dv.Hd = e[q].Hd;
        dv.rW = 1.f / (float)dv.W;
        dv.rH = 1.f / (float)dv.H;
        dv.rWd = 1.f / (float)dv.Wd;
        dv.rHd = 1.f / (float)dv.Hd;
        dv.fov = e[q].mode == PR_FOVEATED || e[q].mode == PR_BOTH;
        dv.fx = e[q].fx;
        dv.fy = e[q].fy;
        dv.alpha = e[q].alpha;
        dv.inv_alpha = 1.f / e[q].alpha;
        dv.p_lut = e[q].p_lut;
        dv.p_n = e[q].p_n;
        dv.scale = fmaxf((float)dv.W / (float)dv.Wd, (float)dv.H / (float)dv.Hd);
        dv.sigma = sigma;
        t.out = e[q].out;
        // the view's scratch: its pyramid levels 1..
        float *lp = p;
        p += display_scratch_floats(method, dv.W, dv.H);
        if (!fill_pyramid(t.pyr, dv.W, dv.H, e[q].rgb, lp))
            return cudaErrorInvalidValue;
        any_tiles |= t.pyr.L > 1;
        any_top |= t.pyr.L > kTileLevels + 1;
        auto row_mul = [](long long per_row) { return ((1ull << 40) + per_row - 1) / (unsigned long long)per_row; };
        const long long dw = (dv.Wd + kDispW - 1) / kDispW, dh = (dv.Hd + kDispH - 1) / kDispH;
        const long long tw = (dv.W + kTileSide - 1) / kTileSide, th = (dv.H + kTileSide - 1) / kTileSide;
        t.mul_disp = row_mul(dw);
        t.mul_tile = row_mul(tw);
        if (q == 0)
            blk[0] = blk[n + 1] = 0;
        blk[q + 1] = blk[q] + dw * dh;
        blk[n + 1 + q + 1] = blk[n + 1 + q] + tw * th;
    }
    cudaError_t err = cudaMemcpyAsync(d_table, h_table, display_batch_table_bytes(n), cudaMemcpyHostToDevice, st);
    if (err != cudaSuccess)
        return err;
    const DisplayBatchView *dtab = static_cast<const DisplayBatchView *>(d_table);
    const long long *dblk = reinterpret_cast<const long long *>(static_cast<const char *>(d_table) + views_bytes);
    if (any_tiles)
        k_mip_tile_batch<<<(unsigned)blk[2 * n + 1], kTileThreads, 0, st>>>(dtab, dblk + n + 1, n);
    if (any_top)
        k_mip_top_batch<<<(unsigned)n, 512, 0, st>>>(dtab);
    if (blk[n] > 0)
        k_unfoveate_mip_batch<<<(unsigned)blk[n], kDispW * kDispH, 0, st>>>(dtab, dblk, n);
    return cudaGetLastError();
}

}  // namespace pr
