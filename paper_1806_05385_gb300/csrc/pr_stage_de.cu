// pr_stage_de.cu -- stage (d): deferred shading at the pixel time (Sec. 3.2,
// "Shading"), and stage (e): its adjoint with respect to the vertex colours,
// positions and velocities, with the visible triangle of every pixel held
// fixed.  Both recompute the pixel's time, ray, moved triangle and
// barycentrics from the id buffer instead of storing them.
#include "pr_launch.h"

#include <cstring>

namespace pr {

__device__ __forceinline__ float3 sub3(float3 a, float3 b) { return make_float3(a.x - b.x, a.y - b.y, a.z - b.z); }
__device__ __forceinline__ float dot3(float3 a, float3 b) { return fmaf(a.x, b.x, fmaf(a.y, b.y, a.z * b.z)); }
__device__ __forceinline__ float3 cross3(float3 a, float3 b)
{
    return make_float3(a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x);
}
// The same cross product with every rounding fixed (no contraction left to
// the compiler), so that every kernel that shades a pixel gets the same bits.
__device__ __forceinline__ float3 cross3_rn(float3 a, float3 b)
{
    return make_float3(fmaf(a.y, b.z, -__fmul_rn(a.z, b.y)), fmaf(a.z, b.x, -__fmul_rn(a.x, b.z)),
                       fmaf(a.x, b.y, -__fmul_rn(a.y, b.x)));
}
__device__ __forceinline__ float3 scale3(float3 a, float s) { return make_float3(a.x * s, a.y * s, a.z * s); }
__device__ __forceinline__ float3 add3(float3 a, float3 b) { return make_float3(a.x + b.x, a.y + b.y, a.z + b.z); }

// An 8-bit value b as b / 255 without the conversion pipe: 2^23 + b is exact
// in FP32 (its bits are 0x4B000000 | b), so subtracting 2^23 leaves b
// exactly; the product is the correctly rounded b * (1/255 in FP32), the
// same as (float)b * (1.f / 255.f).
__device__ __forceinline__ float u8_unit(unsigned char b)
{
    return (__uint_as_float(0x4B000000u | (unsigned)b) - 8388608.f) * (1.f / 255.f);
}

// Everything shading needs about the visible triangle at one pixel.
struct PixelHit {
    int ia, ib, ic;     // vertex indices
    float t;            // pixel time
    float3 dir;         // ray direction
    float3 A, B, C;     // triangle moved to t (camera space)
    float b0, b1, b2;   // barycentrics of the ray point
    float det;          // U + V + W of the watertight test
    float inv_det;      // 1 / det (0 if det = 0)
    float3 n;           // unit normal facing the viewer
    float inl;          // flip / |(B-A) x (C-A)| with flip = +-1 the sign applied (0 if degenerate)
    float3 l;           // unit light direction at t
    float ndl, sigma;   // n.l and k_a + k_d max(0, n.l)
    float3 hv;          // Blinn-Phong half vector normalize(l + v), v = the reversed ray
    float ndh, spec;    // n.h and k_s max(0, n.h)^shininess (0 without specular)
};

// Paths the shading kernels are built with: a view of the launch may have a
// specular term (k_s > 0), a view may use a sampled foveation function, a
// view may ask for the precision form.  The kernels built without a path
// are faster (fewer registers); the results of the views they shade are the
// same bits.
constexpr int kFeatSpec = 1, kFeatLut = 2, kFeatF64 = 4;

// Precision form of the shading: the FP32 barycentrics of a triangle that
// is small against its distance carry an error of about (coordinate error)
// x (sheared extent) / |det|, that is one coordinate ulp over the
// triangle's size; a pixel whose estimate exceeds kBaryRel takes its moved
// triangle, barycentrics and normal from FP64 instead (the FP32 coordinate
// error is taken as kRelCoordShade of the magnitudes it came from, about
// one ulp: measured colour errors of such triangles match it).
constexpr float kBaryRel = 2e-5f;
constexpr float kRelCoordShade = 6e-8f;

// The pixel's moved triangle, barycentrics and unit normal in FP64 from the
// scene's FP32 inputs (widened exactly), rounded to FP32 into h: the
// interpolation of M_s v_s and M_e v_e at the pixel time, the ray-plane
// barycentrics b_k = w_k / sum w with w_0 = dir.(B x C) (cyclically) and the
// face normal turned to face the viewer.
// Out of line, with a result struct of its own, so that the PixelHit of the
// callers stays in registers.
struct Hit64Out {
    float b0, b1, b2, det, inv_det;
    float3 n, A, B, C;
    float inl;
    int has_b, has_n;  // barycentrics / normal are defined
};
__device__ __noinline__ void pixel_hit64(const ViewDev &v, int i, int j, int ia, int ib, int ic, Hit64Out &o);

// Returns false, with h unfinished, for a pixel that needs FP64 when
// `defer64` (the caller leaves it to k_shade64).
template <int kFeat>
__device__ __forceinline__ bool pixel_hit(const ViewDev &v, int i, int j, unsigned id, PixelHit &h,
                                          bool defer64 = false)
{
    float x0, x1, dx, dy;
    pixel_ray<(kFeat & kFeatLut) != 0>(v, i, j, x0, x1, h.t, dx, dy);
    h.dir = make_float3(dx, dy, 1.f);
    const int4 tv = v.tri4[id];
    h.ia = tv.x;
    h.ib = tv.y;
    h.ic = tv.z;
    const float t = h.t;
    if (v.rec) {
        // the frame's own stage (a) record: S and D = E - S, the same bits
        // vertex_start_end gives, in 64 contiguous bytes
        const float4 *r = v.rec + ((size_t)v.tri_off + id) * kRecF4;
        const float4 r0 = r[0], r1 = r[1], r2 = r[2], r3 = r[3], r5 = r[5];
        h.A = make_float3(fmaf(t, r2.y, r0.x), fmaf(t, r2.z, r0.y), fmaf(t, r2.w, r0.z));
        h.B = make_float3(fmaf(t, r3.x, r0.w), fmaf(t, r3.y, r1.x), fmaf(t, r3.z, r1.y));
        h.C = make_float3(fmaf(t, r3.w, r1.z), fmaf(t, r5.z, r1.w), fmaf(t, r5.w, r2.x));
    } else {
        float3 S, E;
        vertex_start_end(v, h.ia, S, E);
        h.A = make_float3(fmaf(t, E.x - S.x, S.x), fmaf(t, E.y - S.y, S.y), fmaf(t, E.z - S.z, S.z));
        vertex_start_end(v, h.ib, S, E);
        h.B = make_float3(fmaf(t, E.x - S.x, S.x), fmaf(t, E.y - S.y, S.y), fmaf(t, E.z - S.z, S.z));
        vertex_start_end(v, h.ic, S, E);
        h.C = make_float3(fmaf(t, E.x - S.x, S.x), fmaf(t, E.y - S.y, S.y), fmaf(t, E.z - S.z, S.z));
    }
    // barycentrics from the sheared edge functions of the watertight test
    const float ax = fmaf(-dx, h.A.z, h.A.x), ay = fmaf(-dy, h.A.z, h.A.y);
    const float bx = fmaf(-dx, h.B.z, h.B.x), by = fmaf(-dy, h.B.z, h.B.y);
    const float cx = fmaf(-dx, h.C.z, h.C.x), cy = fmaf(-dy, h.C.z, h.C.y);
    const float U = __fsub_rn(__fmul_rn(cx, by), __fmul_rn(cy, bx));
    const float V = __fsub_rn(__fmul_rn(ax, cy), __fmul_rn(ay, cx));
    const float W = __fsub_rn(__fmul_rn(bx, ay), __fmul_rn(by, ax));
    h.det = U + V + W;
    const float inv = h.det != 0.f ? 1.f / h.det : 0.f;
    h.inv_det = inv;
    h.b0 = U * inv;
    h.b1 = V * inv;
    h.b2 = W * inv;
    float3 n = cross3_rn(sub3(h.B, h.A), sub3(h.C, h.A));
    const float flip = dot3(n, h.dir) > 0.f ? -1.f : 1.f;
    const float nn = dot3(n, n);
    const float rs = nn > 0.f ? rsqrtf(nn) : 0.f;
    h.inl = flip * rs;
    h.n = scale3(n, h.inl);
    if ((kFeat & kFeatF64) && v.fp64) {
        const float sm = fmaxf(fabsf(ax) + fabsf(ay), fmaxf(fabsf(bx) + fabsf(by), fabsf(cx) + fabsf(cy)));
        const float zm = fmaxf(fabsf(h.A.z), fmaxf(fabsf(h.B.z), fabsf(h.C.z)));
        const float mag = zm * (1.f + fabsf(dx) + fabsf(dy)) + sm;
        if (2.f * kRelCoordShade * mag * sm > kBaryRel * fabsf(h.det)) {
            if (defer64)
                return false;
            Hit64Out o;
            pixel_hit64(v, i, j, h.ia, h.ib, h.ic, o);
            if (o.has_b) {
                h.b0 = o.b0;
                h.b1 = o.b1;
                h.b2 = o.b2;
                h.det = o.det;
                h.inv_det = o.inv_det;
            }
            if (o.has_n) {
                h.n = o.n;
                h.inl = o.inl;
            }
            h.A = o.A;
            h.B = o.B;
            h.C = o.C;
        }
    }
    float3 l = make_float3(fmaf(t, v.l1[0] - v.l0[0], v.l0[0]), fmaf(t, v.l1[1] - v.l0[1], v.l0[1]),
                           fmaf(t, v.l1[2] - v.l0[2], v.l0[2]));
    h.l = scale3(l, rsqrtf(dot3(l, l)));
    h.ndl = dot3(h.n, h.l);
    h.sigma = fmaf(v.k_d, fmaxf(h.ndl, 0.f), v.k_a);
    h.spec = 0.f;
    h.ndh = 0.f;
    if ((kFeat & kFeatSpec) && v.k_s > 0.f) {
        // the eye at the pixel time is the camera origin: v = -dir / |dir|
        const float3 e = scale3(h.dir, -rsqrtf(dot3(h.dir, h.dir)));
        const float3 hh = add3(h.l, e);
        h.hv = scale3(hh, rsqrtf(fmaxf(dot3(hh, hh), 1e-30f)));
        h.ndh = dot3(h.n, h.hv);
        h.spec = h.ndh > 0.f ? v.k_s * powf(h.ndh, v.shininess) : 0.f;
    }
    return true;
}

__device__ __noinline__ void pixel_hit64(const ViewDev &v, int i, int j, int ia, int ib, int ic, Hit64Out &h)
{
    const Ray64 ry = pixel_ray64(v, i, j);
    const double d[3] = {ry.dx, ry.dy, 1.0};
    const int vid[3] = {ia, ib, ic};
    double P[3][3];
    for (int k = 0; k < 3; ++k) {
        const float4 va = v.vtx[2 * vid[k]], vb = v.vtx[2 * vid[k] + 1];
        const double p[3] = {va.x, va.y, va.z},
                     e[3] = {p[0] + (double)va.w, p[1] + (double)vb.x, p[2] + (double)vb.y};
        for (int r = 0; r < 3; ++r) {
            const double S = (double)v.R0[3 * r] * p[0] + (double)v.R0[3 * r + 1] * p[1] + (double)v.R0[3 * r + 2] * p[2] +
                             (double)v.T0[r];
            const double E = (double)v.R1[3 * r] * e[0] + (double)v.R1[3 * r + 1] * e[1] + (double)v.R1[3 * r + 2] * e[2] +
                             (double)v.T1[r];
            P[k][r] = (1.0 - ry.t) * S + ry.t * E;
        }
    }
    // w_0 = dir.(B x C) of the vertices sheared along the ray (x - dx z, y - dy z)
    double e[3][2], w[3];
    for (int k = 0; k < 3; ++k) {
        e[k][0] = P[k][0] - d[0] * P[k][2];
        e[k][1] = P[k][1] - d[1] * P[k][2];
    }
    for (int k = 0; k < 3; ++k) {
        const double *b = e[(k + 1) % 3], *c = e[(k + 2) % 3];
        w[k] = b[0] * c[1] - b[1] * c[0];
    }
    const double sw = w[0] + w[1] + w[2];
    h.has_b = sw != 0.0;
    if (sw != 0.0) {
        const double isw = 1.0 / sw;
        h.b0 = (float)(w[0] * isw);
        h.b1 = (float)(w[1] * isw);
        h.b2 = (float)(w[2] * isw);
        h.det = (float)(-sw);  // the watertight edge functions are -w
        h.inv_det = h.det != 0.f ? 1.f / h.det : 0.f;
    }
    const double e1[3] = {P[1][0] - P[0][0], P[1][1] - P[0][1], P[1][2] - P[0][2]};
    const double e2[3] = {P[2][0] - P[0][0], P[2][1] - P[0][1], P[2][2] - P[0][2]};
    const double n[3] = {e1[1] * e2[2] - e1[2] * e2[1], e1[2] * e2[0] - e1[0] * e2[2], e1[0] * e2[1] - e1[1] * e2[0]};
    const double nn = n[0] * n[0] + n[1] * n[1] + n[2] * n[2];
    h.has_n = nn > 0.0;
    if (nn > 0.0) {
        const double il = rsqrt(nn);
        const double s = n[0] * d[0] + n[1] * d[1] + n[2] * d[2] > 0.0 ? -il : il;
        h.n = make_float3((float)(n[0] * s), (float)(n[1] * s), (float)(n[2] * s));
        h.inl = (float)s;
    }
    h.A = make_float3((float)P[0][0], (float)P[0][1], (float)P[0][2]);
    h.B = make_float3((float)P[1][0], (float)P[1][1], (float)P[1][2]);
    h.C = make_float3((float)P[2][0], (float)P[2][1], (float)P[2][2]);
}

// Stages (d) and (e) run each warp over one strip of nsub pixel blocks of
// kBlkW x kBlkH (8 x 4) side by side: 32 x 4 pixels for nsub = 4, one block
// for nsub = 1 (strip_blocks: frames too small to fill the chip with
// strips).  First the whole strip is resolved row by row (every load of the
// strip in flight at once, rows coalesced): ids, depths, the background's
// colour and loss, the keys' reset.  Then its blocks that show a triangle
// are shaded one after the other, one pixel per lane (lane -> column
// lane % kBlkW, row lane / kBlkW), so that the lanes mostly share a
// triangle.  blk_offs[q] = first strip of view q in the batch.
// CTAs of the shading kernels: 64 threads (two warps), 20 resident per SM
// (48 registers; the precision form and the stand-alone adjoint 18, 56
// registers).  A CTA's slot frees only when its slowest warp finishes, and
// the warps of a CTA see different strips (background, one triangle,
// several), so small CTAs keep the SM fuller.  Training frame's shading, 64
// views / HMD frame: 1.29 / 0.126 ms with 20, 1.34 / 0.128 with 18, 1.37 /
// 0.127 with 16.  Precision form (with the FP64 launch), 1M-triangle stereo /
// HMD / 8 views: 424 / 204 / 206 us with 20, 415 / 200 / 209 with 18, 409 / 196
// / 212 with 16: 18 is within 2 % of the better on either kind.  The
// stand-alone adjoint of four views 0.0466 ms with 20, 0.0459 with 18.
constexpr int kShadeThreads = 64;
constexpr int kShadeWarps = kShadeThreads / 32;
constexpr int shade_ctas(int feat) { return feat & kFeatF64 ? 18 : 20; }
constexpr int kBackwardCtas = 18;

// The strip's visible ids in shared memory, rows apart by an odd multiple of
// eight words (a block's four rows of eight columns meet all banks).
constexpr int kIdPitch = 40;

// Position of a warp's strip.
struct Strip {
    int q;       // view
    int i0, j0;  // first pixel
    int sh;      // log2 of the strip's width
};

__device__ __forceinline__ Strip strip_of(const ViewDev *views, int nviews, const long long *blk_offs, long long b,
                                          int nsub)
{
    Strip s;
    s.q = find_view_warp(blk_offs, nviews, b);  // b is the warp's
    const ViewDev &v = views[s.q];
    s.sh = nsub == 1 ? 3 : 5;
    const int lb = (int)(b - v.blk_off);  // < 2^23 strips per view
    const int bw = (v.W + (1 << s.sh) - 1) >> s.sh;
    const int by = (int)(((unsigned long long)(unsigned)lb * v.bw_mul) >> 40);  // lb / bw
    s.i0 = (lb - by * bw) << s.sh;
    s.j0 = by * kBlkH;
    return s;
}

// Which of the strip's blocks the set lanes of a row's ballot belong to, as
// bits 0..3.
__device__ __forceinline__ unsigned blocks_of(unsigned lanes, int nsub)
{
    if (nsub == 1)
        return lanes ? 1u : 0u;
    return (lanes & 0xFFu ? 1u : 0u) | (lanes & 0xFF00u ? 2u : 0u) | (lanes & 0xFF0000u ? 4u : 0u) |
           (lanes & 0xFF000000u ? 8u : 0u);
}

// Vertex colours of the visible triangle and the interpolated albedo
// a = sum_k b_k col_k of the pixel (shared by the shading and the adjoint).
struct PixelAlbedo {
    float col[3][3];  // [vertex][channel]
    float a[3];
};

__device__ __forceinline__ void pixel_albedo(const ViewDev &v, const PixelHit &h, PixelAlbedo &pa)
{
    const int vid[3] = {h.ia, h.ib, h.ic};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float4 c = v.col4[vid[k]];
        pa.col[k][0] = c.x;
        pa.col[k][1] = c.y;
        pa.col[k][2] = c.z;
    }
#pragma unroll
    for (int c = 0; c < 3; ++c)
        pa.a[c] = fmaf(h.b0, pa.col[0][c], fmaf(h.b1, pa.col[1][c], h.b2 * pa.col[2][c]));
}

// The adjoint's sums over pixels.  A triangle has 27 gradient values: value
// 9k + c is d/dcol_k[c], 9k + 3 + c the sum of (1 - t) dL/dc_k[c] and
// 9k + 6 + c the sum of t dL/dc_k[c], with c_k the moved camera-space vertex
// k; the position and velocity gradients follow once per triangle from the
// last two: dc/dp = (1-t) R0 + t R1 and dc/dv = t R1, so dL/dp = R0^T sum
// (1-t) dL/dc + R1^T sum t dL/dc and dL/dv = R1^T sum t dL/dc.  Every value
// is a sum over pixels of a product x y of two of 17 per-pixel numbers:
// x = (g sigma)_c with y = b_k, or x = dL/dc_k[c] with y = 1 - t or t.
//
// So a block's pixels write those 17 numbers to the warp's rows in shared
// memory (as soon as each is known, which frees its register), and lane l
// then sums value l over the pixels with 16-byte loads of its two rows: 17
// stores, 16 loads and 32 multiply-adds per block, against 31 shuffles, 62
// selects and 31 adds for a shuffle reduce-scatter of the 27 products,
// which also had to live in registers at once (and spilled).  A value's sum
// is one register of one lane, kept while the warp's pixels stay on one
// triangle and written out when the triangle changes.
//
// Row numbers: the rows that eight neighbouring lanes read differ modulo 8
// (but for one pair), so the 16-byte loads meet different banks.
constexpr int kRowPitch = 36, kRows = 17;
__device__ __forceinline__ constexpr int row_gs(int c) { return c; }
__device__ __forceinline__ constexpr int row_b(int k) { return 8 + k; }
__device__ __forceinline__ constexpr int row_g(int k, int c)
{
    return k == 0 ? 3 + c : (k == 1 ? (c == 0 ? 11 : 5 + c) : (c == 0 ? 16 : 11 + c));
}
constexpr int kRowOmt = 14, kRowT = 15;

// What a lane sums: its two rows, and where the value goes.
struct ValueLane {
    int x, y;
};

__device__ __forceinline__ ValueLane value_lane()
{
    const int lane = threadIdx.x & 31;
    const int k = min(lane / 9, 2), r = min(lane - 9 * k, 8);
    ValueLane vl;
    const int c = r < 3 ? r : (r < 6 ? r - 3 : r - 6);
    vl.x = (r < 3 ? row_gs(c) : row_g(k, c)) * kRowPitch;
    vl.y = (r < 3 ? row_b(k) : (r < 6 ? kRowOmt : kRowT)) * kRowPitch;
    return vl;
}

// Adds a triangle's 27 sums (lane l: value l) to the gradients.
__device__ __forceinline__ void add_triangle(const ViewDev &v, unsigned id, float sum)
{
    const int lane = threadIdx.x & 31;
    const int k = min(lane / 9, 2), r = lane - 9 * k;
    const int base = 9 * k;
    const float o0 = __shfl_sync(0xffffffffu, sum, base + 3), o1 = __shfl_sync(0xffffffffu, sum, base + 4),
                o2 = __shfl_sync(0xffffffffu, sum, base + 5);
    const float t0 = __shfl_sync(0xffffffffu, sum, base + 6), t1 = __shfl_sync(0xffffffffu, sum, base + 7),
                t2 = __shfl_sync(0xffffffffu, sum, base + 8);
    if (lane < 27) {
        const int4 tv = v.tri4[id];
        const int c = r < 3 ? r : (r < 6 ? r - 3 : r - 6);
        const int vk = k == 0 ? tv.x : (k == 1 ? tv.y : tv.z);
        float val = sum;
        if (r >= 3) {
            val = fmaf(v.R1[c], t0, fmaf(v.R1[3 + c], t1, v.R1[6 + c] * t2));
            if (r < 6)
                val = fmaf(v.R0[c], o0, fmaf(v.R0[3 + c], o1, fmaf(v.R0[6 + c], o2, val)));
        }
        float *dst = r < 3 ? v.dcol : (r < 6 ? v.dpos : v.dvel);
        if (dst)
            atomicAdd(&dst[3 * vk + c], val);
    }
}

// Adjoint of rgb = a sigma + s, a = sum_k b_k col_k, sigma = k_a + k_d max(0, n.l),
// s = k_s max(0, n.h)^m (h depends only on the pixel's time and ray):
//  - d/dcol_k = g b_k sigma
//  - d/dn = (g . a) k_d l [n.l > 0] + (sum_c g_c) k_s m (n.h)^(m-1) h [n.h > 0]
//  - barycentrics b_k = w_k / sum w with w_0 = dir.(B x C), w_1 = dir.(C x A),
//    w_2 = dir.(A x B) (the watertight U, V, W are -w), so
//    d sum/dw_j = (gb_j - sum_k gb_k b_k) / sum w and dw_j/dA etc. are
//    cross products with dir;
//  - the unit normal n = flip (B-A)x(C-A) / |.|: dn gets (I - n n^T)/|.|;
//  - moved vertex c(t) = (1-t) S + t E with S = R0 p + T0, E = R1 (p + v) + T1
//    (applied per triangle after the sum, add_triangle).
// Writes the pixel's 17 numbers to column `lane` of the warp's rows.
template <int kFeat>
__device__ __forceinline__ void adjoint_rows(const ViewDev &v, const PixelHit &h, const PixelAlbedo &pa, float g0,
                                             float g1, float g2, float *col)
{
    const float b[3] = {h.b0, h.b1, h.b2};
    const float gs[3] = {g0 * h.sigma, g1 * h.sigma, g2 * h.sigma};
    float gb[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        col[row_gs(k) * kRowPitch] = gs[k];
        col[row_b(k) * kRowPitch] = b[k];
        gb[k] = fmaf(gs[0], pa.col[k][0], fmaf(gs[1], pa.col[k][1], gs[2] * pa.col[k][2]));
    }
    const float gsig = fmaf(g0, pa.a[0], fmaf(g1, pa.a[1], g2 * pa.a[2]));
    // barycentrics -> moved vertices: with w_0 = D.(B x C) etc.,
    // dL/dA = gw1 (D x C) + gw2 (B x D) = D x (gw1 C - gw2 B), cyclically
    const float gdotb = fmaf(gb[0], b[0], fmaf(gb[1], b[1], gb[2] * b[2]));
    const float isw = -h.inv_det;  // 1 / sum w, sum w = -det (exactly the negated reciprocal)
    const float gw0 = (gb[0] - gdotb) * isw, gw1 = (gb[1] - gdotb) * isw, gw2 = (gb[2] - gdotb) * isw;
    const float3 D = h.dir;
    float3 gA = cross3(D, sub3(scale3(h.C, gw1), scale3(h.B, gw2)));
    float3 gB = cross3(D, sub3(scale3(h.A, gw2), scale3(h.C, gw0)));
    float3 gC = cross3(D, sub3(scale3(h.B, gw0), scale3(h.A, gw1)));
    // normal -> moved vertices: the diffuse term through n.l, the
    // specular term k_s (n.h)^m (white) through n.h; the three
    // contributions (B-C) x gn, (C-A) x gn, (A-B) x gn sum to zero
    const bool dif = h.ndl > 0.f, spc = (kFeat & kFeatSpec) && h.spec > 0.f;
    if ((dif || spc) && h.inl != 0.f) {
        float3 gnh = scale3(h.l, dif ? gsig * v.k_d : 0.f);
        if (spc)
            gnh = add3(gnh, scale3(h.hv, (g0 + g1 + g2) * v.shininess * h.spec / h.ndh));
        const float pr = dot3(h.n, gnh);
        const float3 gnn = scale3(sub3(gnh, scale3(h.n, pr)), h.inl);
        const float3 na = cross3(sub3(h.B, h.C), gnn), nb = cross3(sub3(h.C, h.A), gnn);
        gA = add3(gA, na);
        gB = add3(gB, nb);
        gC = sub3(gC, add3(na, nb));
    }
    const float3 gk[3] = {gA, gB, gC};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        col[row_g(k, 0) * kRowPitch] = gk[k].x;
        col[row_g(k, 1) * kRowPitch] = gk[k].y;
        col[row_g(k, 2) * kRowPitch] = gk[k].z;
    }
    col[kRowOmt * kRowPitch] = 1.f - h.t;
    col[kRowT * kRowPitch] = h.t;
}

// A warp's running sums of one triangle of its view.
struct TriangleSum {
    float s;      // lane l: value l
    unsigned id;  // the triangle (0xFFFFFFFF: none)
};

// Adds the block's pixels (valid lanes, triangle id; their numbers in the
// warp's rows) to the running sum, triangle by triangle.  others: lanes that
// are not valid but whose columns are not zero.  Called by the whole warp.
//
// kUnroll: columns of several triangles, in groups of four, unrolled so that
// the next ones' loads go out during the sums (1 / 2 / 4 / 8 groups: HMD
// training frame 132 / 131 / 130 / 128 us, 64 views 1.307 / 1.290 / 1.281 /
// 1.280 ms, the adjoint of four views 49.4 / 49.3 / 46.6 / 47.2 us; the
// precision form's shading, with more registers in use, 415 us with 2 and 423
// with 8 on the 1M-triangle stereo frame, 200 / 201 on the HMD frame).
constexpr int sum_unroll(int feat) { return feat & kFeatF64 ? 2 : 8; }
template <int kUnroll>
__device__ __forceinline__ void sum_block(const ViewDev &v, const float *rows, const ValueLane &vl, bool valid,
                                          unsigned id, TriangleSum &ts, unsigned others = 0u)
{
    unsigned rem = __ballot_sync(0xffffffffu, valid);
    const unsigned all = rem | others;
    const float4 *x4 = reinterpret_cast<const float4 *>(rows + vl.x);
    const float4 *y4 = reinterpret_cast<const float4 *>(rows + vl.y);
    unsigned m = __ballot_sync(0xffffffffu, valid && id == ts.id);  // the running triangle first
    while (rem) {
        if (!m) {
            const unsigned tid = __shfl_sync(0xffffffffu, id, __ffs(rem) - 1);
            if (ts.id != 0xFFFFFFFFu)
                add_triangle(v, ts.id, ts.s);
            ts.id = tid;
            ts.s = 0.f;
            m = __ballot_sync(0xffffffffu, valid && id == tid);
        }
        float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
        if (m == all) {  // one triangle (the common case): the other lanes' columns are zero
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const float4 x = x4[q], y = y4[q];
                s0 = fmaf(x.x, y.x, s0);
                s1 = fmaf(x.y, y.y, s1);
                s2 = fmaf(x.z, y.z, s2);
                s3 = fmaf(x.w, y.w, s3);
            }
        } else {
#pragma unroll kUnroll
            for (int q = 0; q < 8; ++q) {
                const unsigned nib = (m >> (4 * q)) & 15u;
                if (!nib)
                    continue;  // warp-uniform
                const float4 x = x4[q], y = y4[q];
                if (nib & 1u)
                    s0 = fmaf(x.x, y.x, s0);
                if (nib & 2u)
                    s1 = fmaf(x.y, y.y, s1);
                if (nib & 4u)
                    s2 = fmaf(x.z, y.z, s2);
                if (nib & 8u)
                    s3 = fmaf(x.w, y.w, s3);
            }
        }
        ts.s += (s0 + s1) + (s2 + s3);
        rem &= ~m;
        m = 0u;
    }
}

__device__ __forceinline__ bool frame_overflowed(const Counters *frame_cnt)
{
    return frame_cnt && (frame_cnt->status & (ST_OVERFLOW_PAIRS | ST_OVERFLOW_ITEMS | ST_OVERFLOW_FLAGS | ST_TIMEOUT));
}

// Stage (d).  keys != null: the frame's packed depth|id keys are resolved
// here too (id and depth written, then shaded), saving a separate resolve
// pass.  kAdjoint (a training frame): for views with a gradient input, the
// stage (e) adjoint of the pixel follows from the same PixelHit -- with an
// L2 target, from the colour just computed -- so the frame needs no
// separate adjoint pass.  Whole warps run (the adjoint's sums).
// views: the device table, or the kernel's parameter table (k_shade_pv).
//
// Bound: the L1 data pipe (82 % busy on the HMD frame: the adjoint's rows and
// the spills), instruction issue (73 % of peak, DRAM 27 % on 64 views; 740 to
// 810 warp instructions per block that shows a triangle) and, on the
// background, DRAM writes.
//
// def.list (the precision form): pixels whose barycentrics need FP64 are not
// shaded here but listed for k_shade64.  An FP64 instruction holds the SM's
// unit as long for one lane as for 32, and the pixels that need it are few
// and scattered (1M-triangle stereo frame: 290,000 of 9.3 M pixels, most
// warps with one to three): run in place they took 0.18 of 0.47 ms, listed
// 0.155.
template <bool kAdjoint, int kFeat>
__device__ __forceinline__ void shade_body(const ViewDev *__restrict__ views, int nviews,
                                           const long long *__restrict__ blk_offs, long long nblocks, int nsub,
                                           unsigned long long *__restrict__ keys, int reset_keys,
                                           const Counters *__restrict__ frame_cnt, const Deferred64 def)
{
    __shared__ unsigned s_id[kShadeWarps][kBlkH * kIdPitch];
    __shared__ __align__(16) float s_rows[kAdjoint ? kShadeWarps : 1][kAdjoint ? kRows * kRowPitch : 4];
    const long long b0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (b0 >= nblocks)
        return;  // whole warps
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // a training frame whose forward overflowed is rerun by the host: its
    // adjoint must not accumulate
    const bool adjoint = kAdjoint && !frame_overflowed(frame_cnt);
    const Strip sp = strip_of(views, nviews, blk_offs, b0, nsub);
    const ViewDev &v = views[sp.q];
    const int W = v.W, H = v.H;
    const int plane = W * H;  // <= 2^28
    const bool grad = adjoint && (v.grad_in || v.target || v.target_u8);
    // a view with neither an image nor a gradient only needs the resolve
    const bool shaded = v.rgb_out || grad;
    float lsum = 0.f;  // the lane's share of the L2 loss (background: rgb = 0)
    unsigned live = 0u;  // blocks of the strip that show a triangle

    // the strip row by row: keys first, all in flight at once
    {
        const int col = sp.i0 + (lane & ((1 << sp.sh) - 1)), row0 = sp.j0 + (lane >> sp.sh), rstep = 32 >> sp.sh;
        unsigned long long key[kBlkH];
#pragma unroll
        for (int k = 0; k < kBlkH; ++k) {
            key[k] = ~0ull;
            const int j = row0 + k * rstep;
            if (k < nsub && col < W && j < H) {
                if (keys)
                    key[k] = keys[v.pix_off + j * W + col];
                else
                    key[k] = v.id_in[j * W + col] | 0xFFFFFFFF00000000ull;
            }
        }
#pragma unroll
        for (int k = 0; k < kBlkH; ++k) {
            if (k >= nsub)
                break;
            const int j = row0 + k * rstep, lin = j * W + col;
            const bool inside = col < W && j < H;
            const unsigned id = (unsigned)key[k];
            const bool hit = inside && id < (unsigned)v.T && shaded;
            if (inside) {
                if (keys) {
                    const bool bg = key[k] == ~0ull;
                    if (!bg && reset_keys)
                        keys[v.pix_off + lin] = ~0ull;  // left as the next frame wants it
                    if (v.id_out)
                        v.id_out[lin] = id;
                    if (v.depth_out)
                        v.depth_out[lin] = bg ? INFINITY : __uint_as_float((unsigned)(key[k] >> 32));
                }
                if (!hit) {
                    if (kAdjoint && grad && v.loss) {  // before the colour: rgb_out may be the target's own buffer
                        float e0, e1, e2;
                        if (v.target_u8) {
                            e0 = u8_unit(v.target_u8[lin]);
                            e1 = u8_unit(v.target_u8[plane + lin]);
                            e2 = u8_unit(v.target_u8[2 * plane + lin]);
                        } else {
                            e0 = v.target[lin];
                            e1 = v.target[plane + lin];
                            e2 = v.target[2 * plane + lin];
                        }
                        lsum += fmaf(e0, e0, fmaf(e1, e1, e2 * e2));
                    }
                    if (v.rgb_out) {
                        v.rgb_out[lin] = 0.f;
                        v.rgb_out[plane + lin] = 0.f;
                        v.rgb_out[2 * plane + lin] = 0.f;
                    }
                }
            }
            s_id[warp][(k * rstep + (lane >> sp.sh)) * kIdPitch + (lane & ((1 << sp.sh) - 1))] =
                hit ? id : 0xFFFFFFFFu;
            live |= blocks_of(__ballot_sync(0xffffffffu, hit), nsub);
        }
    }
    __syncwarp();

    // the blocks that show a triangle, one pixel per lane
    TriangleSum ts;
    ts.s = 0.f;
    ts.id = 0xFFFFFFFFu;
    const ValueLane vl = value_lane();
    float *rows = s_rows[kAdjoint ? warp : 0];
    for (; live; live &= live - 1u) {
        const int x = (__ffs(live) - 1) * kBlkW + lane % kBlkW, y = lane / kBlkW;
        const unsigned id = s_id[warp][y * kIdPitch + x];
        const int pi = sp.i0 + x, pj = sp.j0 + y, lin = pj * W + pi;
        bool done = false, later = false;
        if (id != 0xFFFFFFFFu) {
            // the upstream gradient (or L2 target) does not depend on the
            // hit: its loads go out first
            float gin[3] = {0.f, 0.f, 0.f};
            if (kAdjoint && grad) {
                if (v.target_u8) {
                    gin[0] = u8_unit(v.target_u8[lin]);
                    gin[1] = u8_unit(v.target_u8[plane + lin]);
                    gin[2] = u8_unit(v.target_u8[2 * plane + lin]);
                } else {
                    const float *gsrc = v.grad_in ? v.grad_in : v.target;
                    gin[0] = gsrc[lin];
                    gin[1] = gsrc[plane + lin];
                    gin[2] = gsrc[2 * plane + lin];
                }
            }
            PixelHit h;
            if (pixel_hit<kFeat>(v, pi, pj, id, h, (kFeat & kFeatF64) && def.list)) {
                PixelAlbedo pa;
                pixel_albedo(v, h, pa);
                const float rgb[3] = {fmaf(pa.a[0], h.sigma, h.spec), fmaf(pa.a[1], h.sigma, h.spec),
                                      fmaf(pa.a[2], h.sigma, h.spec)};
                if (v.rgb_out) {
                    v.rgb_out[lin] = rgb[0];
                    v.rgb_out[plane + lin] = rgb[1];
                    v.rgb_out[2 * plane + lin] = rgb[2];
                }
                if (kAdjoint && grad) {
                    if (!v.grad_in) {
                        // L2 loss sum (rgb - target)^2: its gradient from this frame's image
                        const float e0 = rgb[0] - gin[0], e1 = rgb[1] - gin[1], e2 = rgb[2] - gin[2];
                        lsum += fmaf(e0, e0, fmaf(e1, e1, e2 * e2));
                        gin[0] = 2.f * e0;
                        gin[1] = 2.f * e1;
                        gin[2] = 2.f * e2;
                    }
                    adjoint_rows<kFeat>(v, h, pa, gin[0], gin[1], gin[2], rows + lane);
                }
                done = true;
            } else {
                later = true;
            }
        }
        if (kFeat & kFeatF64) {
            const unsigned m = __ballot_sync(0xffffffffu, later);
            if (m) {
                unsigned long long base = 0;
                if (lane == __ffs(m) - 1)
                    base = atomicAdd(def.count, (unsigned long long)__popc(m));
                base = __shfl_sync(0xffffffffu, base, __ffs(m) - 1);
                if (later)
                    def.list[base + __popc(m & ((1u << lane) - 1u))] =
                        ((unsigned long long)(v.pix_off + lin) << 32) | id;
            }
        }
        if (kAdjoint && grad) {
            if (!done) {
#pragma unroll
                for (int r = 0; r < kRows; ++r)
                    rows[r * kRowPitch + lane] = 0.f;
            }
            __syncwarp();
            sum_block<sum_unroll(kFeat)>(v, rows, vl, done, id, ts);
            __syncwarp();  // the rows are written again by the next block
        }
    }
    if (kAdjoint && ts.id != 0xFFFFFFFFu)
        add_triangle(v, ts.id, ts.s);
    if (kAdjoint && adjoint && v.loss) {
        // one view per warp: a warp sum, then one atomic into one of the
        // view's partial sums (one address for every warp of a view would
        // serialise them)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
        if (lane == 0)
            atomicAdd(&v.loss_part[(unsigned)b0 & (kLossSlots - 1)], lsum);
    }
}

template <bool kAdjoint, int kFeat>
__global__ void __launch_bounds__(kShadeThreads, shade_ctas(kFeat))
    k_shade(const ViewDev *__restrict__ views, int nviews, const long long *__restrict__ blk_offs, long long nblocks, int nsub,
            unsigned long long *__restrict__ keys, int reset_keys, const Counters *__restrict__ frame_cnt,
            const Deferred64 def)
{
    shade_body<kAdjoint, kFeat>(views, nviews, blk_offs, nblocks, nsub, keys, reset_keys, frame_cnt, def);
}

template <int kN, bool kAdjoint, int kFeat>
__global__ void __launch_bounds__(kShadeThreads, shade_ctas(kFeat))
    k_shade_pv(const __grid_constant__ ParamViews<kN> pv, int nviews, const long long *__restrict__ blk_offs,
               long long nblocks, int nsub, unsigned long long *__restrict__ keys, int reset_keys,
               const Counters *__restrict__ frame_cnt, const Deferred64 def)
{
    shade_body<kAdjoint, kFeat>(pv.v, nviews, blk_offs, nblocks, nsub, keys, reset_keys, frame_cnt, def);
}

// The pixels that the shading kernels left to FP64, one lane each, so that
// every FP64 instruction serves 32 of them: the same pixel hit with its FP64
// path, colour, loss and adjoint.  Bound: the FP64 unit (225 FP64
// instructions per pixel at about 18 cycles of the SM per warp instruction:
// 0.120 of 0.155 ms for 290,000 pixels).  A warp's pixels are neighbours in the
// list, so most share a few triangles, summed as in the shading kernels
// (27 atomics per pixel instead: 0.287 against 0.155 ms for 290,000 pixels).
constexpr int kShade64Threads = 128, kShade64Ctas = 4;
template <bool kAdjoint, int kFeat>
__global__ void __launch_bounds__(kShade64Threads, kShade64Ctas)
    k_shade64(const ViewDev *__restrict__ views, int nviews, const long long *__restrict__ pix_offs,
              const Counters *__restrict__ frame_cnt, const Deferred64 def)
{
    __shared__ __align__(16) float s_rows[kAdjoint ? kShade64Threads / 32 : 1][kAdjoint ? kRows * kRowPitch : 4];
    const long long n = (long long)*def.count;
    const bool adjoint = kAdjoint && !frame_overflowed(frame_cnt);
    const int lane = threadIdx.x & 31;
    float *rows = s_rows[kAdjoint ? threadIdx.x >> 5 : 0];
    const ValueLane vl = value_lane();
    for (long long k0 = (long long)blockIdx.x * kShade64Threads + (threadIdx.x & ~31); k0 < n;
         k0 += (long long)gridDim.x * kShade64Threads) {
        int q = -1;  // the view of the lane's pixel, if it takes part in the adjoint
        unsigned id = 0xFFFFFFFFu;
        if (k0 + lane < n) {
            const unsigned long long e = def.list[k0 + lane];
            const long long g = (long long)(e >> 32);
            id = (unsigned)e;
            const int vq = find_view(pix_offs, nviews, g);
            const ViewDev &v = views[vq];
            const int lin = (int)(g - v.pix_off), plane = v.W * v.H, pj = lin / v.W, pi = lin - pj * v.W;
            const bool grad = kAdjoint && adjoint && (v.grad_in || v.target || v.target_u8);
            float gin[3] = {0.f, 0.f, 0.f};  // the gradient or target, before the colour: rgb_out may be its buffer
            if (grad) {
#pragma unroll
                for (int c = 0; c < 3; ++c)
                    gin[c] = v.target_u8 ? u8_unit(v.target_u8[c * plane + lin])
                                         : (v.grad_in ? v.grad_in : v.target)[c * plane + lin];
            }
            PixelHit h;
            PixelAlbedo pa;
            pixel_hit<kFeat>(v, pi, pj, id, h);
            pixel_albedo(v, h, pa);
            const float rgb[3] = {fmaf(pa.a[0], h.sigma, h.spec), fmaf(pa.a[1], h.sigma, h.spec),
                                  fmaf(pa.a[2], h.sigma, h.spec)};
            if (v.rgb_out) {
                v.rgb_out[lin] = rgb[0];
                v.rgb_out[plane + lin] = rgb[1];
                v.rgb_out[2 * plane + lin] = rgb[2];
            }
            if (grad) {
                q = vq;
                if (!v.grad_in) {
#pragma unroll
                    for (int c = 0; c < 3; ++c)
                        gin[c] = 2.f * (rgb[c] - gin[c]);
                }
                if (v.loss)  // sum (rgb - target)^2
                    atomicAdd(&v.loss_part[(unsigned)(k0 + lane) & (kLossSlots - 1)],
                              0.25f * fmaf(gin[0], gin[0], fmaf(gin[1], gin[1], gin[2] * gin[2])));
                adjoint_rows<kFeat>(v, h, pa, gin[0], gin[1], gin[2], rows + lane);
            }
        }
        if (kAdjoint && adjoint) {
            if (q < 0) {
#pragma unroll
                for (int r = 0; r < kRows; ++r)
                    rows[r * kRowPitch + lane] = 0.f;
            }
            __syncwarp();
            unsigned rem = __ballot_sync(0xffffffffu, q >= 0);
            const unsigned all = rem;
            while (rem) {  // view by view
                const int vq = __shfl_sync(0xffffffffu, q, __ffs(rem) - 1);
                const unsigned m = __ballot_sync(0xffffffffu, q == vq);
                TriangleSum ts;
                ts.s = 0.f;
                ts.id = 0xFFFFFFFFu;
                sum_block<sum_unroll(kFeat)>(views[vq], rows, vl, q == vq, id, ts, all & ~m);
                add_triangle(views[vq], ts.id, ts.s);
                rem &= ~m;
            }
            __syncwarp();  // the rows are written again by the next round
        }
    }
}

// A training frame's losses: one block per view sums the view's partial
// sums and adds them to the caller's loss (views without a loss: nothing).
__global__ void __launch_bounds__(kLossSlots) k_loss_finalize(const ViewDev *__restrict__ views,
                                                              const Counters *__restrict__ frame_cnt)
{
    const ViewDev &v = views[blockIdx.x];
    if (!v.loss || frame_overflowed(frame_cnt))
        return;  // an overflowed forward is rerun by the host: its loss must not count
    float s = v.loss_part[threadIdx.x];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        s += __shfl_xor_sync(0xffffffffu, s, o);
    __shared__ float ws[kLossSlots / 32];
    if ((threadIdx.x & 31) == 0)
        ws[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        float t = 0.f;
        for (int w = 0; w < kLossSlots / 32; ++w)
            t += ws[w];
        atomicAdd(v.loss, t);  // several views may share one loss
    }
}

cudaError_t launch_loss_finalize(const ViewDev *views, int nviews, const Counters *frame_cnt, cudaStream_t st)
{
    if (nviews > 0)
        k_loss_finalize<<<nviews, kLossSlots, 0, st>>>(views, frame_cnt);
    return cudaGetLastError();
}

// One warp per strip, kShadeThreads threads per CTA.
static unsigned shade_grid(long long nblocks)
{
    return (unsigned)((nblocks * 32 + kShadeThreads - 1) / kShadeThreads);
}

// The parameter table of a launch's views, from their host copy.
template <int kN>
static const ParamViews<kN> &param_views(const ViewDev *host_views, int nviews)
{
    static thread_local ParamViews<kN> pv;
    std::memcpy(pv.v, host_views, sizeof(ViewDev) * (size_t)nviews);
    return pv;
}

bool shade_reads_params(int nviews) { return nviews >= 1 && nviews <= kParamViews; }

template <bool kAdjoint, int kFeat>
static void launch_shade_one(unsigned g, const ViewDev *views, const ViewDev *host_views, int nviews,
                             const long long *blk_offs, long long nblocks, int nsub, unsigned long long *keys,
                             int reset_keys, const Counters *frame_cnt, const Deferred64 &def, cudaStream_t st)
{
    if (!host_views || !shade_reads_params(nviews))
        k_shade<kAdjoint, kFeat><<<g, kShadeThreads, 0, st>>>(views, nviews, blk_offs, nblocks, nsub, keys, reset_keys,
                                                              frame_cnt, def);
    else if (nviews <= kFewViews)
        k_shade_pv<kFewViews, kAdjoint, kFeat><<<g, kShadeThreads, 0, st>>>(
            param_views<kFewViews>(host_views, nviews), nviews, blk_offs, nblocks, nsub, keys, reset_keys, frame_cnt,
            def);
    else
        k_shade_pv<kParamViews, kAdjoint, kFeat><<<g, kShadeThreads, 0, st>>>(
            param_views<kParamViews>(host_views, nviews), nviews, blk_offs, nblocks, nsub, keys, reset_keys, frame_cnt,
            def);
}

template <bool kAdjoint>
static void launch_shade_t(int feat, unsigned g, const ViewDev *views, const ViewDev *pv, int nviews,
                           const long long *blk_offs, long long nblocks, int nsub, unsigned long long *keys, int reset_keys,
                           const Counters *frame_cnt, const Deferred64 &def, cudaStream_t st)
{
    if (feat == kFeatF64) {  // the precision form without the specular and sampled-foveation paths
        launch_shade_one<kAdjoint, kFeatF64>(g, views, pv, nviews, blk_offs, nblocks, nsub, keys, reset_keys, frame_cnt,
                                             def, st);
        return;
    }
    if (feat & kFeatF64) {  // the precision form with either: one variant with every path (same bits)
        launch_shade_one<kAdjoint, kFeatSpec | kFeatLut | kFeatF64>(g, views, pv, nviews, blk_offs, nblocks, nsub, keys,
                                                                    reset_keys, frame_cnt, def, st);
        return;
    }
    switch (feat) {
    case 0:
        launch_shade_one<kAdjoint, 0>(g, views, pv, nviews, blk_offs, nblocks, nsub, keys, reset_keys, frame_cnt,
                                             def, st);
        break;
    case kFeatSpec:
        launch_shade_one<kAdjoint, kFeatSpec>(g, views, pv, nviews, blk_offs, nblocks, nsub, keys, reset_keys, frame_cnt,
                                             def, st);
        break;
    case kFeatLut:
        launch_shade_one<kAdjoint, kFeatLut>(g, views, pv, nviews, blk_offs, nblocks, nsub, keys, reset_keys, frame_cnt,
                                             def, st);
        break;
    default:
        launch_shade_one<kAdjoint, kFeatSpec | kFeatLut>(g, views, pv, nviews, blk_offs, nblocks, nsub, keys, reset_keys,
                                                         frame_cnt, def, st);
    }
}

int shade_features(const ViewDev *vd, int n)
{
    int f = 0;
    for (int k = 0; k < n; ++k) {
        if (vd[k].k_s > 0.f)
            f |= kFeatSpec;
        if (vd[k].p_lut && (vd[k].mode == PR_FOVEATED || vd[k].mode == PR_BOTH))
            f |= kFeatLut;
        if (vd[k].fp64)
            f |= kFeatF64;
    }
    return f;
}

template <bool kAdjoint>
static void launch_shade64(int feat, const ViewDev *views, int nviews, const long long *pix_offs,
                           const Counters *frame_cnt, const Deferred64 &def, cudaStream_t st)
{
    static int grid = 0;
    if (grid == 0) {
        int dev = 0, sms = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        grid = sms * kShade64Ctas;
    }
    if (feat == kFeatF64)
        k_shade64<kAdjoint, kFeatF64><<<grid, kShade64Threads, 0, st>>>(views, nviews, pix_offs, frame_cnt, def);
    else
        k_shade64<kAdjoint, kFeatSpec | kFeatLut | kFeatF64>
            <<<grid, kShade64Threads, 0, st>>>(views, nviews, pix_offs, frame_cnt, def);
}

cudaError_t launch_shade(const ViewDev *views, int nviews, const long long *blk_offs, long long nblocks, int nsub,
                         unsigned long long *keys, bool reset_keys, bool adjoint, const Counters *frame_cnt, int feat,
                         cudaStream_t st, const ViewDev *host_views, const long long *pix_offs,
                         const Deferred64 &def)
{
    if (nblocks > 0) {
        const unsigned g = shade_grid(nblocks);
        const ViewDev *pv = host_views;
        if (adjoint)
            launch_shade_t<true>(feat, g, views, pv, nviews, blk_offs, nblocks, nsub, keys, reset_keys, frame_cnt, def,
                                 st);
        else
            launch_shade_t<false>(feat, g, views, pv, nviews, blk_offs, nblocks, nsub, keys, reset_keys, frame_cnt, def,
                                  st);
        if ((feat & kFeatF64) && def.list) {
            if (adjoint)
                launch_shade64<true>(feat, views, nviews, pix_offs, frame_cnt, def, st);
            else
                launch_shade64<false>(feat, views, nviews, pix_offs, frame_cnt, def, st);
        }
    }
    return cudaGetLastError();
}

// Stage (e) on its own: the adjoint of a shaded frame from its id buffer
// and an upstream gradient (grad_in of every view).
template <int kFeat>
__device__ __forceinline__ void backward_body(const ViewDev *__restrict__ views, int nviews,
                                              const long long *__restrict__ blk_offs, long long nblocks, int nsub)
{
    __shared__ unsigned s_id[kShadeWarps][kBlkH * kIdPitch];
    __shared__ __align__(16) float s_rows[kShadeWarps][kRows * kRowPitch];
    const long long b0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (b0 >= nblocks)
        return;  // whole warps
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const Strip sp = strip_of(views, nviews, blk_offs, b0, nsub);
    const ViewDev &v = views[sp.q];
    const int W = v.W, H = v.H;
    const int plane = W * H;  // <= 2^28
    unsigned live = 0u;
    {
        const int col = sp.i0 + (lane & ((1 << sp.sh) - 1)), row0 = sp.j0 + (lane >> sp.sh), rstep = 32 >> sp.sh;
        unsigned id[kBlkH];
#pragma unroll
        for (int k = 0; k < kBlkH; ++k) {
            id[k] = 0xFFFFFFFFu;
            const int j = row0 + k * rstep;
            if (k < nsub && col < W && j < H)
                id[k] = v.id_in[j * W + col];
        }
#pragma unroll
        for (int k = 0; k < kBlkH; ++k) {
            if (k >= nsub)
                break;
            const bool hit = id[k] < (unsigned)v.T;
            s_id[warp][(k * rstep + (lane >> sp.sh)) * kIdPitch + (lane & ((1 << sp.sh) - 1))] =
                hit ? id[k] : 0xFFFFFFFFu;
            live |= blocks_of(__ballot_sync(0xffffffffu, hit), nsub);
        }
    }
    __syncwarp();
    TriangleSum ts;
    ts.s = 0.f;
    ts.id = 0xFFFFFFFFu;
    const ValueLane vl = value_lane();
    float *rows = s_rows[warp];
    for (; live; live &= live - 1u) {
        const int x = (__ffs(live) - 1) * kBlkW + lane % kBlkW, y = lane / kBlkW;
        const unsigned id = s_id[warp][y * kIdPitch + x];
        const int pi = sp.i0 + x, pj = sp.j0 + y, lin = pj * W + pi;
        const bool hit = id != 0xFFFFFFFFu;
        if (hit) {
            const float g0 = v.grad_in[lin], g1 = v.grad_in[plane + lin], g2 = v.grad_in[2 * plane + lin];
            PixelHit h;
            PixelAlbedo pa;
            pixel_hit<kFeat>(v, pi, pj, id, h);
            pixel_albedo(v, h, pa);
            adjoint_rows<kFeat>(v, h, pa, g0, g1, g2, rows + lane);
        } else {
#pragma unroll
            for (int r = 0; r < kRows; ++r)
                rows[r * kRowPitch + lane] = 0.f;
        }
        __syncwarp();
        sum_block<sum_unroll(kFeat)>(v, rows, vl, hit, id, ts);
        __syncwarp();  // the rows are written again by the next block
    }
    if (ts.id != 0xFFFFFFFFu)
        add_triangle(v, ts.id, ts.s);
}

template <int kFeat>
__global__ void __launch_bounds__(kShadeThreads, kBackwardCtas)
    k_backward(const ViewDev *__restrict__ views, int nviews, const long long *__restrict__ blk_offs, long long nblocks,
               int nsub)
{
    backward_body<kFeat>(views, nviews, blk_offs, nblocks, nsub);
}

template <int kN, int kFeat>
__global__ void __launch_bounds__(kShadeThreads, kBackwardCtas)
    k_backward_pv(const __grid_constant__ ParamViews<kN> pv, int nviews, const long long *__restrict__ blk_offs,
                  long long nblocks, int nsub)
{
    backward_body<kFeat>(pv.v, nviews, blk_offs, nblocks, nsub);
}

template <int kFeat>
static void launch_backward_one(unsigned g, const ViewDev *views, const ViewDev *host_views, int nviews,
                                const long long *blk_offs, long long nblocks, int nsub, cudaStream_t st)
{
    if (!host_views || !shade_reads_params(nviews))
        k_backward<kFeat><<<g, kShadeThreads, 0, st>>>(views, nviews, blk_offs, nblocks, nsub);
    else if (nviews <= kFewViews)
        k_backward_pv<kFewViews, kFeat><<<g, kShadeThreads, 0, st>>>(param_views<kFewViews>(host_views, nviews), nviews,
                                                                     blk_offs, nblocks, nsub);
    else
        k_backward_pv<kParamViews, kFeat><<<g, kShadeThreads, 0, st>>>(param_views<kParamViews>(host_views, nviews),
                                                                       nviews, blk_offs, nblocks, nsub);
}

cudaError_t launch_backward(const ViewDev *views, int nviews, const long long *blk_offs, long long nblocks, int nsub,
                            int feat, cudaStream_t st, const ViewDev *host_views)
{
    if (nblocks > 0) {
        const unsigned g = shade_grid(nblocks);
        const ViewDev *pv = host_views;
        if (feat & kFeatF64) {
            launch_backward_one<kFeatSpec | kFeatLut | kFeatF64>(g, views, pv, nviews, blk_offs, nblocks, nsub, st);
            return cudaGetLastError();
        }
        switch (feat) {
        case 0:
            launch_backward_one<0>(g, views, pv, nviews, blk_offs, nblocks, nsub, st);
            break;
        case kFeatSpec:
            launch_backward_one<kFeatSpec>(g, views, pv, nviews, blk_offs, nblocks, nsub, st);
            break;
        case kFeatLut:
            launch_backward_one<kFeatLut>(g, views, pv, nviews, blk_offs, nblocks, nsub, st);
            break;
        default:
            launch_backward_one<kFeatSpec | kFeatLut>(g, views, pv, nviews, blk_offs, nblocks, nsub, st);
        }
    }
    return cudaGetLastError();
}

}  // namespace pr
